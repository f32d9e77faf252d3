"""Steps captured into a CUDA graph and replayed: each replay goes on from where the last step left the particles."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu

PHYSICS = {"default": {}, "paper": dict(gather="ngp", integrator="semi_implicit", drag="schiller_naumann"),
           "cic": dict(deposit="cic")}


def _sim(prec, physics, micro, K, stream, n=5000, N=16):
    from paper_2603_26691_gb300.sim import Sim

    pos, vel, d, _ = inputs.particles(1, 0, n, vmax=1.0)
    sim = Sim(N, precision=prec, stream=stream)
    sim.set_params(reorder_every=K)
    sim.set_physics(**PHYSICS[physics])
    sim.set_fluid(inputs.taylor_green(N))
    sim.add_particles(pos, d, vel)
    if micro:
        sim.set_microphysics(True)
        sim.set_thermo(np.full((N,) * 3, 285.0), np.full((N,) * 3, 0.0105))
    return sim


def _out(sim, stream):
    stream.synchronize()
    return [*sim.particles(), sim.sources(host=True)]


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("physics,micro", [("default", False), ("paper", False), ("cic", False), ("default", True)])
def test_captured_steps_up_to_a_sort(prec, physics, micro):
    """The captured steps are the last ones before a sort is due."""
    import torch

    out = []
    for captured in (False, True):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            sim = _sim(prec, physics, micro, 10, stream)
            sim.step(3, 1e-3)
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    sim.step(7, 1e-3)
                for _ in range(3):
                    graph.replay()
            else:
                sim.set_params(reorder_every=0)
                for _ in range(3):
                    sim.step(7, 1e-3)
            out.append(_out(sim, stream))
            sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("physics", ["paper", "cic"])
def test_captured_steps_after_a_sort(prec, physics):
    """The captured steps are the first ones after a sort that was asked for."""
    import torch

    out = []
    for captured in (False, True):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            sim = _sim(prec, physics, False, 4, stream)
            sim.step(4, 1e-3)
            sim.reorder()
            sim.set_params(reorder_every=0)
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    sim.step(2, 1e-3)
            for _ in range(3):
                if captured:
                    graph.replay()
                else:
                    sim.step(2, 1e-3)
            out.append(_out(sim, stream))
            sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
