"""The general mixed-precision step at the sizes where its lanes and warps end."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu

GRID = (20, 12, 7)  # no chunk edge: the general kernel


def _run(prec, deposit, pos, vel, d, U):
    from paper_2603_26691_gb300.sim import Sim

    sim = Sim(GRID, precision=prec)
    sim.set_params(reorder_every=0)
    sim.set_physics(deposit=deposit)
    sim.set_fluid(U)
    sim.add_particles(pos, d, vel)
    sim.step(2, 1e-3)
    out = [*sim.particles(), sim.sources(host=True)]
    sim.close()
    return out


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("deposit", ["cell", "cic"])
@pytest.mark.parametrize("n", [1, 2, 3, 63, 65, 129, 257, 513, 40_001])
def test_parts_give_the_whole(prec, deposit, n):
    """Particles in one handle and in two (cut at whole warps): the same states, and sources that add up to rounding
    of the exact sums."""
    cut = 256 * (n // 512)
    pos, vel, d, _ = inputs.particles(3, 0, n, vmax=1.0)
    U = np.random.default_rng(n).uniform(-1, 1, (GRID[2], GRID[1], GRID[0], 3)).astype(np.float32)
    whole = _run(prec, deposit, pos, vel, d, U)
    parts = [_run(prec, deposit, pos[:, s], vel[:, s], d[s], U) for s in (slice(0, cut), slice(cut, n)) if len(d[s])]
    for i, a in enumerate(whole[:-1]):
        if a.dtype.kind == "f":  # the ids count from zero in each handle
            assert np.array_equal(a, np.concatenate([p[i] for p in parts], axis=-1))
    total = sum(p[-1] for p in parts)
    assert np.abs(whole[-1] - total).max() <= 1e-12 * np.abs(whole[-1]).max()
