"""The FP64 step's integer interpolation and its several steps per launch."""
import numpy as np
import pytest

import oracle
from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu


def _corner_max(U, pos, grid):
    """The largest corner magnitude of each particle's trilinear stencil, per component."""
    n = pos.shape[1]
    lo = [np.floor(pos[q] * grid[q] - 0.5).astype(int) for q in range(3)]
    m = np.zeros((3, n))
    for k in range(8):
        i, j, l = (np.mod(lo[q] + ((k >> q) & 1), grid[q]) for q in range(3))
        m = np.maximum(m, np.abs(U[l, j, i]).T)
    return m


@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 3, 5), (8, 8, 8), (7, 16, 9)])
@pytest.mark.parametrize("span", [0, 3, 40, 300])
def test_one_step_over_the_exponent_range(grid, span):
    """Cells whose values differ by up to `span` decades in either direction, zeros among them: the velocity the
    oracle gives, to the rounding of the largest corner."""
    from paper_2603_26691_gb300.sim import Sim

    rng = np.random.default_rng(span + grid[0])
    shape = (grid[2], grid[1], grid[0], 3)
    U = rng.uniform(-1, 1, shape) * 10.0 ** rng.uniform(-span, min(span, 2), shape)
    U[rng.random(shape) < 0.1] = 0.0
    n, dt = 3000, 1e-3
    pos, _, d, _ = inputs.particles(span, 0, n)
    pos[:, :8] = 0.0  # faces and the corner of the box
    pos[0, :grid[0]] = np.arange(grid[0]) / grid[0]
    vel = np.zeros((3, n))
    sim = Sim(grid, precision="fp64")
    sim.set_params(reorder_every=0, g=(0.0, 0.0, 0.0))
    sim.set_fluid(U)
    sim.add_particles(pos, d, vel)
    sim.step(1, dt)
    p, v, _, _ = sim.particles()
    sim.close()
    op, ov, _, _ = oracle.run(oracle.make_grid(grid, g=(0.0, 0.0, 0.0)), U, pos, vel, d, 1, dt)
    # the stencil's fractions differ by the rounding of a position in cells (up to 16 of them, 2^-48), which weighs
    # corner differences of twice the largest corner on three axes; every other rounding is smaller
    tol = 2.0 ** -45 * _corner_max(U, pos, grid)
    assert (np.abs(v - ov) <= tol).all(), (np.abs(v - ov) / np.maximum(tol, 1e-320)).max()
    dx = np.abs((p - op + 0.5) % 1.0 - 0.5)
    assert (dx <= 2.0 ** -50 + tol * dt).all()


@pytest.mark.parametrize("n", [1, 31, 4097])
@pytest.mark.parametrize("K", [0, 4])
def test_results_do_not_depend_on_the_split_over_calls(n, K):
    from paper_2603_26691_gb300.sim import Sim

    N, steps, dt = 8, 37, 2e-3
    pos, vel, d, _ = inputs.particles(n, 0, n, vmax=2.0)
    out = []
    for split in ([steps], [1] * steps, [5, 32]):
        sim = Sim(N, precision="fp64")
        sim.set_params(reorder_every=K)
        sim.set_fluid(inputs.taylor_green(N))
        sim.add_particles(pos, d, vel)
        for m in split:
            sim.step(m, dt)
        out.append((*sim.particles(), sim.sources(host=True)))
        sim.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)
