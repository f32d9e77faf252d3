"""Cloud-in-cell deposit of dense and sparse units: the lanes' order of adds differs, the exact sums do not."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu


def _fixed(prec, pos, U):
    from paper_2603_26691_gb300.sim import Sim

    sim = Sim(16, precision=prec)
    sim.set_physics(deposit="cic")
    sim.set_fluid(U)
    sim.add_particles(pos, np.full(pos.shape[1], 20e-6))
    sim.step(3, 1e-3)
    w, E = sim.sources_fixed()
    w = w.cpu().numpy().astype(object)
    sim.close()
    return sum(w[..., k] * (1 << (32 * k)) for k in range(4)), E


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("n", [20_000, 140_000])
def test_dense_units_add_up_to_sparse_ones(prec, n):
    """2500 and 17500 particles to a unit of 512 cells in one handle, and a sixteenth of them each in others."""
    pos = inputs.particles(4, 0, n)[0]
    U = inputs.taylor_green(16).astype(np.float32)
    whole, E = _fixed(prec, pos, U)
    parts = [_fixed(prec, pos[:, i::16], U) for i in range(16)]
    assert all(e == E for _, e in parts)
    assert (whole == sum(p for p, _ in parts)).all()
