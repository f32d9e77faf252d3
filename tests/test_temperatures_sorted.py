"""Particle temperatures stay with their particles in sorts while the microphysics is off."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("physics", [{}, dict(deposit="cic"), dict(gather="ngp")])
def test_temperatures_follow_the_particles(physics):
    from paper_2603_26691_gb300.sim import Sim

    N, n = 16, 5000
    pos, vel, d, _ = inputs.particles(3, 0, n, vmax=2.0)
    sim = Sim(N, precision="mixed_f32")
    sim.set_params(reorder_every=4)
    sim.set_fluid(inputs.taylor_green(N))
    sim.add_particles(pos, d, vel)
    sim.set_microphysics(True)
    T = 280.0 + np.arange(n) * 2.0 ** -10  # exact in FP32 pairs
    sim.set_temperatures(T)
    sim.set_microphysics(False)
    sim.set_physics(**physics)
    for steps in (4, 3, 5):
        sim.step(steps, 1e-3)
        if steps == 4:
            sim.reorder()
        assert np.array_equal(sim.temperatures(), T[sim.particles()[3]])
    sim.close()
