"""Velocities read back against plain division (GPU required).

lbm_get_moments divides the three momenta by the density through one
reciprocal and Markstein's residual correction.  The stored deviations and the
sums are formed here in the same order in IEEE binary64, so density must agree
to the bit and velocity with NumPy's correctly rounded quotient to the bit too
(tolerance zero where the density's reciprocal is a normal number and the
momentum is above 2^-968; Markstein's theorem), over densities near 1, a
thousand orders of two, a few units of 2^-52, huge ones, infinities and NaN.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (16, 20, 24)


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def weights():
    w1 = [1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0]
    return np.array([w1[i % 3] * w1[(i // 3) % 3] * w1[i // 9] for i in range(27)])


def expected(f):
    """Density and velocity of populations f[n][27], summed as the library sums them."""
    d = (f - weights()).T
    s = [(d[3 * j] + d[3 * j + 2]) + d[3 * j + 1] for j in range(9)]
    jx = np.zeros(f.shape[0])
    for j in range(9):
        jx = jx + (d[3 * j + 2] - d[3 * j])
    lo, mid, hi = (s[0] + s[3]) + s[6], (s[1] + s[4]) + s[7], (s[2] + s[5]) + s[8]
    jz = ((s[6] - s[0]) + (s[8] - s[2])) + (s[7] - s[1])
    rho = 1.0 + ((lo + hi) + mid)
    return rho, np.stack([jx, hi - lo, jz], 1), np.stack([jx / rho, (hi - lo) / rho, jz / rho], 1)


def near_one(rng, n):
    return weights() * (1.0 + 0.2 * (2.0 * rng.random((n, 27)) - 1.0))


def wide(rng, n):
    return rng.random((n, 27)) * np.exp2(rng.integers(-40, 1000, (n, 1)).astype(float))


def huge(rng, n):
    """One population alone, up to the largest exponents: velocities of magnitude 0 and 1."""
    f = np.zeros((n, 27))
    f[np.arange(n), rng.integers(0, 27, n)] = (1.0 + rng.random(n)) * np.exp2(rng.integers(1015, 1023, n).astype(float))
    return f


def small(rng, n):
    """Densities that cancel to a few units of 2^-52, and empty cells."""
    f = weights() * (1.0 + 1e-13 * rng.random((n, 27)))
    f[:, 13] -= 1.0 * (rng.random(n) < 0.9)
    f[::50] = 0.0
    return f


def broken(rng, n):
    f = near_one(rng, n)
    f[np.arange(n), rng.integers(0, 27, n)] = rng.choice([np.inf, -np.inf, np.nan, 0.0, 1.7e308, -1.7e308], n)
    return f


@pytest.mark.parametrize("make", [near_one, wide, huge, small, broken], ids=lambda m: m.__name__)
def test_velocity_is_the_correctly_rounded_quotient(lbm, make):
    n = int(np.prod(N))
    f = make(np.random.default_rng(7), n)
    with lbm.Lattice(np.ones(N, dtype=np.uint8), "fp64", periodic=7) as G:
        G.set_populations(f)
        rho, u = G.moments()
    with np.errstate(all="ignore"):
        want_rho, j, want = expected(f)
        assert np.array_equal(rho, want_rho, equal_nan=True)
        plain = (np.abs(j) > 2.0 ** -968) | (j == 0.0) | ~np.isfinite(j)
        assert np.array_equal(np.where(plain, u, 0.0), np.where(plain, want, 0.0), equal_nan=True)
