"""The adjoints' segments: sums of dL/dU over steps and lanes at the sizes and magnitudes where they end."""
import numpy as np
import pytest

import oracle
from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu


def _run(prec, grid, n, steps, every, lam, U, dt=1e-3, sort=False):
    from paper_2603_26691_gb300.sim import Sim

    pos, vel, d, _ = inputs.particles(5, 0, n, vmax=1.0)
    sim = Sim(grid, precision=prec)
    sim.set_params(reorder_every=0)
    sim.set_fluid(U)
    sim.add_particles(pos, d, vel)
    if sort:
        sim.reorder()
    sim.adjoint_forward(steps, dt, every)
    out = sim.adjoint_backward(lam)
    sim.close()
    return out


def _lam(rng, nc, decades):
    lam = rng.standard_normal((3, nc)) * 10.0 ** rng.uniform(-decades, decades, (3, nc))
    lam[:, rng.random(nc) < 0.2] = 0.0
    return lam


@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 5, 3), (16, 8, 8)])
@pytest.mark.parametrize("n", [1, 31, 33, 129])
@pytest.mark.parametrize("decades", [0, 9])
def test_fp64_segments_against_the_oracle(grid, n, decades):
    """Segments of one step, ragged ones and ones longer than a sum takes, dL/dJ zero in places and over 18 decades."""
    rng = np.random.default_rng(n + grid[0])
    U = rng.uniform(-1, 1, (grid[2], grid[1], grid[0], 3))
    lam = _lam(rng, grid[0] * grid[1] * grid[2], decades)
    pos, vel, d, _ = inputs.particles(5, 0, n, vmax=1.0)
    steps = 70
    ogd, oga, ogU = oracle.adjoint(oracle.make_grid(grid), U, pos, vel, d, steps, 1e-3, lam)
    for every in (1, 33, 70):
        gd, ga, gU = _run("fp64", grid, n, steps, every, lam, U)
        # the bounds of the adjoint's other tests
        assert np.abs(gd - ogd).max() <= 1e-9 * np.abs(ogd).max()
        assert abs(ga - oga) <= 1e-9 * max(abs(oga), np.abs(ogd).max() * d.max())
        assert np.abs(gU - ogU.reshape(gU.shape)).max() <= 1e-9 * np.abs(ogU).max()


@pytest.mark.parametrize("n", [1, 31, 33, 4097])
@pytest.mark.parametrize("decades", [0, 6])
def test_fp32_gradients_do_not_depend_on_the_segments(n, decades):
    grid = (8, 8, 8)
    rng = np.random.default_rng(n)
    U = rng.uniform(-1, 1, (8, 8, 8, 3)).astype(np.float32)
    lam = _lam(rng, 512, decades)
    for sort in (False, True):
        ref = _run("mixed_f32", grid, n, 70, 70, lam, U, sort=sort)
        for every in (1, 33):
            for a, b in zip(ref, _run("mixed_f32", grid, n, 70, every, lam, U, sort=sort)):
                assert np.array_equal(np.asarray(a), np.asarray(b))
