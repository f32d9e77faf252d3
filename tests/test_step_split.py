"""A launch takes several steps: the state and the sources do not depend on how steps are split over calls."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu

PHYSICS = {
    "default": {},
    "cic": dict(deposit="cic"),
    "paper": dict(gather="ngp", integrator="semi_implicit", drag="schiller_naumann"),
    "ngp_cic": dict(gather="ngp", deposit="cic"),
}


def _run(prec, grid, n, K, physics, micro, split, dt, vmax, chunk):
    from paper_2603_26691_gb300.sim import Sim

    rng = np.random.default_rng(n)
    pos, vel, d, _ = inputs.particles(n, 0, n, vmax=vmax)
    sim = Sim(grid, chunk_edge=chunk, precision=prec)
    sim.set_params(reorder_every=K)
    sim.set_physics(**PHYSICS[physics])
    sim.set_fluid(rng.uniform(-1, 1, (grid[2], grid[1], grid[0], 3)).astype(np.float32))
    sim.add_particles(pos, d, vel)
    if micro:
        sim.set_microphysics(True)
        sim.set_thermo(rng.uniform(282, 288, grid[::-1]), rng.uniform(0.009, 0.012, grid[::-1]))
    for m in split:
        sim.step(m, dt)
    out = [*sim.particles(), sim.sources(host=True)]
    if micro:
        out += [sim.temperatures(), sim.micro_sources()]
    sim.close()
    return out


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("grid,chunk", [((16, 16, 16), 8), ((24, 16, 32), 8), ((64, 32, 32), 32), ((13, 9, 5), 4)])
@pytest.mark.parametrize("physics,micro", [("default", False), ("cic", False), ("paper", False), ("ngp_cic", False),
                                           ("default", True)])
@pytest.mark.parametrize("n,K", [(1, 4), (127, 0), (2049, 5), (40_001, 10)])
def test_results_do_not_depend_on_the_split(prec, grid, chunk, physics, micro, n, K):
    """Chunked grids of both kinds (powers of two or not) and a ragged one; n at the edges of a lane's, a warp's and
    a stage's share."""
    steps = 23
    args = (prec, grid, n, K, physics, micro)
    ref = _run(*args, [steps], 1e-3, 2.0, chunk)
    for split in ([1] * steps, [7, 16]):
        for a, b in zip(ref, _run(*args, split, 1e-3, 2.0, chunk)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("physics", ["default", "paper"])
@pytest.mark.parametrize("grid,vmax", [((64, 32, 32), 2.0), ((64, 32, 32), 200.0), ((16, 16, 16), 2.0)])
@pytest.mark.parametrize("n", [(1 << 23) - 1, (1 << 23) + 5])
def test_many_particles_in_single_steps(prec, physics, grid, vmax, n):
    """From 2^23 particles on a launch of one step is a kernel of its own: particles that stay near their units, that
    leave them, and units of more particles than its tile takes; steps before and after a sort."""
    args = (prec, grid, n, 4, physics, False)
    ref = _run(*args, [6], 1e-3, vmax, 8)
    for a, b in zip(ref, _run(*args, [1] * 6, 1e-3, vmax, 8)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("physics", ["default", "cic"])
def test_fast_particles_leave_their_tiles(prec, physics):
    """Moves of many cells and of whole boxes in a step: every particle commits outside its unit's tile."""
    args = (prec, (32, 16, 16), 5000, 10, physics, False)
    ref = _run(*args, [9], 0.05, 60.0, 8)
    for a, b in zip(ref, _run(*args, [1] * 9, 0.05, 60.0, 8)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [140_000])
def test_one_dense_cell(n):
    """All particles in one cell, more than a tile's digits take between flushes, against FP64 sums of the impulses
    the momentum budget gives."""
    from paper_2603_26691_gb300.sim import Sim

    N, dt, steps = 16, 1e-4, 4
    rng = np.random.default_rng(1)
    pos = (np.array([[5.0], [6.0], [7.0]]) + rng.uniform(0.3, 0.7, (3, n))) / N
    d = np.full(n, 20e-6)
    vel = np.zeros((3, n))
    sim = Sim(N, precision="mixed_f32")
    sim.set_fluid(inputs.uniform_field(N, (0.3, -0.2, 0.1)).astype(np.float32))
    sim.add_particles(pos, d, vel)
    sim.step(steps, dt)
    _, v, dd, _ = sim.particles()
    src = sim.sources(host=True)
    sim.close()
    m = 1000.0 * np.pi / 6.0 * dd ** 3
    g = np.array([0.0, 0.0, -9.81])
    expect = -(m * v).sum(1) + m.sum() * g * dt * steps
    cell = 5 + N * (6 + N * 7)
    # FP32 velocities (2^-24 each) and FP32 run sums, over steps of the same sign
    assert np.abs(src[:, cell] - expect).max() <= 2.0 ** -20 * np.abs(expect).max()
    assert np.abs(np.delete(src, cell, axis=1)).max() == 0.0
