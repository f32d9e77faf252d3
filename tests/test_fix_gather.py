"""The FP64 step's interpolation on integers: exact for uniform fields, unbiased and rounded once for others.

Particles so light that they take the fluid's velocity in one step show the interpolated values themselves."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _interpolated(grid, U, pos):
    from paper_2603_26691_gb300.sim import Sim

    n = pos.shape[1]
    sim = Sim(grid, precision="fp64")
    sim.set_params(reorder_every=0, g=(0.0, 0.0, 0.0))
    sim.set_fluid(U)
    # e^{-a dt} = 0 in FP64: a dt = 18 mu dt / (rho_p d^2) = 3e4
    sim.add_particles(pos, np.full(n, 1e-7), np.zeros((3, n)))
    sim.step(1, 1e-3)
    v = sim.particles()[1]
    sim.close()
    return v


def _exact(N, U, pos):
    """The trilinear interpolation in extended precision at positions whose fractions of a cell are exact, and the
    largest corner of each."""
    n = pos.shape[1]
    s = pos * float(N)
    lo = np.floor(s - 0.5).astype(int)
    f = [np.longdouble(s[q]) - np.longdouble(lo[q]) - np.longdouble(0.5) for q in range(3)]
    want = np.zeros((3, n), np.longdouble)
    largest = np.zeros((3, n))
    for k in range(8):
        bit = [(k >> q) & 1 for q in range(3)]
        w = np.ones(n, np.longdouble)
        for q in range(3):
            w = w * (f[q] if bit[q] else 1 - f[q])
        i, j, l = (np.mod(lo[q] + bit[q], N) for q in range(3))
        want += w * U[l, j, i].T.astype(np.longdouble)
        largest = np.maximum(largest, np.abs(U[l, j, i].T))
    return want, largest


@pytest.mark.parametrize("grid", [(8, 8, 8), (7, 16, 9)])
def test_a_uniform_field_comes_out_exactly(grid):
    rng = np.random.default_rng(grid[0])
    pos = rng.random((3, 20_000))
    pos[:, 0] = 0.5 / np.array(grid)  # at a cell centre
    for size in (0.3, 1.0, 2.0, 4.0, 1e-5):
        u = size * (1.0 + rng.random(3)) * np.array([1, -1, 1])
        v = _interpolated(grid, np.broadcast_to(u, (grid[2], grid[1], grid[0], 3)).copy(), pos)
        assert np.array_equal(v, np.broadcast_to(u[:, None], v.shape))


def test_interpolation_is_rounded_once():
    """Corners of one size: FP64's rounding of the exact value (half a unit of the result); five roundings of weights, at
    most 0.75 of 2^-58 each, on differences of up to twice the largest corner (up to four times for the first), and two
    mantissa units of 2^-58 for the sum: below 2^-54 of it in all; no bias."""
    N, n = 16, 30_000
    rng = np.random.default_rng(2)
    U = rng.uniform(0.5, 1, (N, N, N, 3)) * rng.choice([-1.0, 1.0], (N, N, N, 3))
    pos = rng.integers(0, 2 ** 53, (3, n)) * 2.0 ** -53  # exact fractions of a cell
    v = _interpolated(N, U, pos)
    want, _ = _exact(N, U, pos)
    err = (np.longdouble(v) - want).astype(np.float64)
    assert (np.abs(err) <= np.spacing(np.abs(v)) / 2 + 2.0 ** -54).all()
    # in units of 2^-53: a sample's deviation is at most 0.3 (a rounding of values below 1), the mean's 0.3 / sqrt(3 n)
    assert abs(err.mean()) * 2.0 ** 53 <= 5 * 0.3 / np.sqrt(3 * n)


@pytest.mark.parametrize("span", [0, 1, 3, 9])
def test_no_less_accurate_than_fp64_lerps(span):
    """Cells over `span` decades, so that corners are aligned to the largest of their stencil: the errors' root mean
    square and largest value, in units of the largest corner, against those of three FP64 lerps."""
    N, n = 16, 30_000
    rng = np.random.default_rng(span)
    U = rng.uniform(0.5, 1, (N, N, N, 3)) * 10.0 ** rng.uniform(-span, 0, (N, N, N, 3)) * rng.choice([-1, 1], (N, N, N, 3))
    pos = rng.integers(0, 2 ** 53, (3, n)) * 2.0 ** -53
    v = _interpolated(N, U, pos)
    want, largest = _exact(N, U, pos)
    s = pos * float(N)
    lo = np.floor(s - 0.5).astype(int)
    c = [U[np.mod(lo[2] + (k >> 2), N), np.mod(lo[1] + ((k >> 1) & 1), N), np.mod(lo[0] + (k & 1), N)].T for k in range(8)]
    for q in range(3):
        f = s[q] - lo[q] - 0.5
        c = [c[2 * i] + f * (c[2 * i + 1] - c[2 * i]) for i in range(len(c) // 2)]
    err, lerps = (((np.longdouble(x) - want) / largest).astype(np.float64) for x in (v, c[0]))
    assert np.square(err).mean() <= np.square(lerps).mean()
    assert np.abs(err).max() <= np.abs(lerps).max()
