"""dL/dU in cells that only small weights reach: each cell as accurate, relative to itself, as the products are."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N = 8


def _gradients(prec, pos, d, steps, every, lam, sort):
    from paper_2603_26691_gb300.sim import Sim

    sim = Sim(N, precision=prec)
    sim.set_params(reorder_every=0, g=(0.0, 0.0, 0.0))
    sim.set_fluid(np.zeros((N, N, N, 3)))
    sim.add_particles(pos, d)
    if sort:
        sim.reorder()
    p0, v0, d0, _ = sim.particles()  # the state as stored
    sim.adjoint_forward(steps, 1e-3, every)
    gU = sim.adjoint_backward(lam)[2]
    sim.close()
    G = oracle.make_grid((N, N, N), g=(0.0, 0.0, 0.0))
    return gU, oracle.adjoint(G, np.zeros((N, N, N, 3)), p0, v0, d0, steps, 1e-3, lam)[2].reshape(gU.shape)


@pytest.mark.parametrize("prec,rel", [("mixed_f32", 2.0 ** -19), ("fp64", 2.0 ** -46)])
@pytest.mark.parametrize("n", [1, 40])
@pytest.mark.parametrize("sort", [False, True])
@pytest.mark.parametrize("power", [2, 5, 9, 13, 20])
def test_each_cell_is_accurate(prec, rel, n, sort, power):
    """Particles at rest just beside the cell centres, so that the seven other corners have weights of 2^-power to
    2^(-3 power): below what a running sum holds too.  Everything is of one sign, so a cell's bound is that of its
    products: about ten roundings (of 2^-24, of 2^-53) in a weight and an adjoint velocity, over three steps; in FP64
    the oracle's own come on top."""
    rng = np.random.default_rng(power)
    f = 2.0 ** -power * (1.0 + rng.integers(0, 8, (3, n)) / 8.0)
    cell = np.array([[2], [3], [4]]) if n == 1 else rng.integers(0, 2, (3, n)) * 4
    pos = (cell + 0.5 + f) / N
    d = rng.uniform(20e-6, 40e-6, n)
    lam = rng.uniform(1.0, 2.0, (3, N ** 3))
    for every in (1, 3):
        got, want = _gradients(prec, pos, d, 3, every, lam, sort)
        assert (want != 0).sum() >= 24
        assert (np.abs(got - want) <= rel * np.abs(want)).all()


@pytest.mark.parametrize("n", [1, 31, 33, 4097])
@pytest.mark.parametrize("decades", [0, 9])
def test_fp64_gradients_do_not_depend_on_the_segments(n, decades):
    from paper_2603_26691_gb300 import inputs
    from paper_2603_26691_gb300.sim import Sim

    rng = np.random.default_rng(n)
    U = rng.uniform(-1, 1, (N, N, N, 3))
    lam = rng.standard_normal((3, N ** 3)) * 10.0 ** rng.uniform(-decades, decades, (3, N ** 3))
    lam[:, rng.random(N ** 3) < 0.2] = 0.0
    pos, vel, d, _ = inputs.particles(5, 0, n, vmax=1.0)
    for sort in (False, True):
        out = []
        for every in (70, 1, 33):
            sim = Sim(N, precision="fp64")
            sim.set_params(reorder_every=0)
            sim.set_fluid(U)
            sim.add_particles(pos, d, vel)
            if sort:
                sim.reorder()
            sim.adjoint_forward(70, 1e-3, every)
            out.append(sim.adjoint_backward(lam))
            sim.close()
        for o in out[1:]:
            for a, b in zip(out[0], o):
                assert np.array_equal(np.asarray(a), np.asarray(b))
