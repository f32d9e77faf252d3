"""Particles read from a mixed handle: exact FP64 values of the stored FP32 state, from the arrays and from the
records a step before a sort leaves."""
import numpy as np
import pytest

from paper_2603_26691_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [8, 12, 16])
def test_exported_values_are_the_stored_ones(N):
    from paper_2603_26691_gb300.sim import Sim

    rng = np.random.default_rng(N)
    n = 1537
    # offsets at and around the sizes where the sum of cell and offset stops being exact, and faces
    off = np.concatenate([[0.0], 2.0 ** -np.arange(1, 60), rng.random(n - 60)])
    cell = rng.integers(0, N, (3, n))
    pos = (cell + rng.permuted(np.tile(off, (3, 1)), axis=1)) / N
    vel = rng.standard_normal((3, n))
    vel[0, :6] = [0.0, -0.0, 1e-40, -3e-45, 1.5e38, 2.0 ** -126]
    d = rng.uniform(1e-7, 1e-3, n)
    sim = Sim(N, precision="mixed_f32")
    sim.add_particles(pos, d, vel)
    p, v, dd, ids = sim.particles()
    s = pos * float(N)
    i = np.clip(np.floor(s), 0, N - 1)
    xi = (s - i).astype(np.float32)
    up = xi >= 1.0
    i, xi = np.where(up, (i + 1) % N, i), np.where(up, np.float32(0), xi)
    assert np.array_equal(p, (i + xi.astype(np.float64)) * (1.0 / N))
    assert np.array_equal(v, vel.astype(np.float32).astype(np.float64)) and np.array_equal(dd, d.astype(np.float32))
    assert np.array_equal(ids, np.arange(n))
    sim.close()


@pytest.mark.parametrize("prec", ["mixed_f32", "mixed_bf16"])
@pytest.mark.parametrize("micro", [False, True])
@pytest.mark.parametrize("n", [1, 5, 4097])
def test_records_and_arrays_read_the_same(prec, micro, n):
    from paper_2603_26691_gb300.sim import Sim

    N = 16
    pos, vel, d, _ = inputs.particles(21, 0, n, vmax=2.0)
    sim = Sim(N, precision=prec)
    sim.set_params(reorder_every=4)
    sim.set_fluid(inputs.taylor_green(N).astype(np.float32))
    sim.add_particles(pos, d, vel)
    if micro:
        sim.set_microphysics(True)
        sim.set_thermo(np.full((N,) * 3, 285.0), np.full((N,) * 3, 0.0105))
    sim.step(4, 1e-3)  # a sort is due: the state is records
    from_records = sim.particles()
    part = sim.particles(first=n // 3, count=n - n // 3)
    cells = sim.cells()
    sim.invariants()  # turns the records back into arrays
    for a, b, c in zip(from_records, sim.particles(), part):
        assert np.array_equal(a, b) and np.array_equal(a[..., n // 3:], c)
    assert np.array_equal(cells, sim.cells())
    sim.step(3, 1e-3)
    after = sim.particles()
    sim.close()
    # reading the records does not disturb the run that goes on from them
    sim = Sim(N, precision=prec)
    sim.set_params(reorder_every=4)
    sim.set_fluid(inputs.taylor_green(N).astype(np.float32))
    sim.add_particles(pos, d, vel)
    if micro:
        sim.set_microphysics(True)
        sim.set_thermo(np.full((N,) * 3, 285.0), np.full((N,) * 3, 0.0105))
    sim.step(4, 1e-3)
    sim.particles()
    sim.step(3, 1e-3)
    for a, b in zip(after, sim.particles()):
        assert np.array_equal(a, b)
    sim.close()
