"""Allocations that fail: the call reports it, or goes on without the buffers it can do without (the integer copy of an
FP64 field), with the same results to rounding."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu


class _Failing:
    """torch's allocator with the k-th call from now (or all from it on) returning nothing."""

    def __init__(self, monkeypatch):
        import torch

        self.alloc, self.left, self.rest, self.calls = torch.cuda.caching_allocator_alloc, -1, False, 0
        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", self)

    def arm(self, k, rest):
        self.left, self.rest = k, rest

    def __call__(self, *a):
        self.calls += 1
        if self.left >= 0:
            self.left -= 1
            if self.left < 0:
                self.left = 0 if self.rest else -1
                raise MemoryError
        return self.alloc(*a)


def _adjoint_sim(n):
    from paper_2603_26691_gb300.sim import Sim

    pos, vel, d, _ = inputs.particles(5, 0, n, vmax=1.0)
    sim = Sim(8, precision="fp64")
    sim.set_params(reorder_every=0)
    sim.set_fluid(inputs.taylor_green(8))
    sim.add_particles(pos, d, vel)
    return sim


@pytest.mark.parametrize("rest", [False, True])
@pytest.mark.parametrize("k", range(8))
def test_adjoint_backward_with_a_failing_allocation(monkeypatch, k, rest):
    """The k-th allocation of a backward pass with host outputs fails, once or with all after it."""
    fail = _Failing(monkeypatch)
    lam = np.random.default_rng(0).standard_normal((3, 512))
    sim = _adjoint_sim(1000)
    sim.adjoint_forward(12, 1e-3, 5)
    want = sim.adjoint_backward(lam)
    for attempt in range(2):
        fail.arm(k if attempt == 0 else -1, rest)  # the second attempt finds memory again
        try:
            got = sim.adjoint_backward(lam)
        except _lib.StError as e:
            assert attempt == 0 and rest and e.status == _lib.ST_ERR_OOM
            continue
        # the bounds of the adjoint's other tests
        for a, b in zip(want, got):
            assert np.abs(np.asarray(a) - np.asarray(b)).max() <= 1e-9 * np.abs(np.asarray(a)).max()
    fail.arm(-1, False)
    sim.close()


@pytest.mark.parametrize("rest", [False, True])
@pytest.mark.parametrize("k", range(12))
def test_couple_run_with_a_failing_allocation(monkeypatch, k, rest):
    """The k-th allocation of a first coupled run fails, its sort's among them."""
    fail = _Failing(monkeypatch)
    out = []
    for failing in (False, True):
        sim = _adjoint_sim(1000)
        sim.set_params(reorder_every=4)
        sim.couple_params(steps_per_interval=3)
        if failing:
            fail.arm(k, rest)
        try:
            sim.couple_run(1, 1e-3)
        except _lib.StError as e:
            assert failing and rest and e.status == _lib.ST_ERR_OOM
            fail.arm(-1, False)
            sim.close()
            return
        fail.arm(-1, False)
        pos, vel, _, ids = sim.particles()
        o = np.argsort(ids)
        out.append((pos[:, o], vel[:, o], sim.fluid(), sim.pending_sources()))
        sim.close()
    # FP64 throughout, a few steps: the parity bound of the FP64 tests
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-10 * np.abs(a).max()


def test_the_integer_field_stays_while_a_graph_may_read_it(monkeypatch):
    """A failing allocation after steps were captured is reported; the graph's field is not given up for it."""
    import torch

    from paper_2603_26691_gb300.sim import Sim

    fail = _Failing(monkeypatch)
    pos, vel, d, _ = inputs.particles(5, 0, 1000, vmax=1.0)
    out = []
    for captured in (False, True):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            sim = Sim(8, precision="fp64", stream=stream)
            sim.set_params(reorder_every=0)
            sim.set_fluid(inputs.taylor_green(8))
            sim.add_particles(pos, d, vel)
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    sim.step(3, 1e-3)
                fail.arm(0, False)
                with pytest.raises(_lib.StError) as e:
                    sim.sources(host=True)
                assert e.value.status == _lib.ST_ERR_OOM
                graph.replay()
                stream.synchronize()
            else:
                sim.step(3, 1e-3)
            out.append([*sim.particles(), sim.sources(host=True)])
            sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
def test_sorts_without_a_place_for_the_cells(monkeypatch, prec):
    """The last buffer of a first sort, which it can do without, is missing: the same results, and later sorts do not
    allocate (nor ask for it again)."""
    from paper_2603_26691_gb300.sim import Sim

    fail = _Failing(monkeypatch)
    pos, vel, d, _ = inputs.particles(7, 0, 5000, vmax=1.0)
    out, asked = [], []
    for k in (-1, 9):
        sim = Sim(16, precision=prec)
        sim.set_params(reorder_every=4)
        sim.set_fluid(inputs.taylor_green(16).astype(np.float32))
        sim.add_particles(pos, d, vel)
        fail.arm(k, False)
        calls = []
        for steps in (3, 4, 4, 4):  # each begins with a sort or has one inside
            before = fail.calls
            sim.step(steps, 1e-3)
            assert fail.left == -1
            calls.append(fail.calls - before)
        asked.append(calls)
        out.append([*sim.particles(), sim.sources(host=True)])
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert asked[0] == asked[1] and asked[0][2:] == [0, 0]


def test_small_reservations_do_not_reallocate_every_time(monkeypatch):
    from paper_2603_26691_gb300.sim import Sim

    fail = _Failing(monkeypatch)
    sim = Sim(8, precision="mixed_f32")
    fail.calls = 0
    sim.reserve(10_000)
    first = fail.calls
    for n in range(10_100, 40_000, 100):
        sim.reserve(n)
    # 1.5-fold growth from 1e4 to 4e4 takes four steps
    assert fail.calls <= 5 * first
    sim.close()
