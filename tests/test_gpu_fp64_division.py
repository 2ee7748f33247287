"""The FP64 step's velocity u^eq = N / D (Eq. 3) is the correctly rounded
quotient, also where a division built from a reciprocal goes wrong: divisors
just below a power of two (mantissas near all ones), quotients close to the
middle between two doubles, and zeros.

Without couplings and with both relaxation times 1, N is the momentum and D
the density of the first species; populations are chosen so that D comes out
exactly as planned.  Velocities below 1/2, and up to 2^20, where the last bit
of u shows in every population.  Every operation of the step is one the oracle
performs too, in the same order, and the populations after a step are equal
bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def divisors(rng, n):
    u = 2.0 ** -52
    d = np.where(rng.random(n) < 0.7, 2.0 - u * rng.integers(1, 9, n), 1.0 + u * rng.integers(0, 9, n))
    return np.where(rng.random(n) < 0.2, 1.0 + u * rng.integers(0, 2 ** 52, n), d)


def numerators(rng, d, lo, hi):
    """Powers of two in (2^lo, 2^hi), products of d with the middle between two
    quotients there, and zeros."""
    n = d.size
    power = 2.0 ** rng.integers(lo + 1, hi, n)
    half = d * (rng.integers(2 ** 52, 2 ** 53, n) + 0.5) * 2.0 ** (rng.integers(lo, hi - 1, n) - 53.0)
    v = np.where(rng.random(n) < 0.5, power, half)
    return np.where(rng.random(n) < 0.1, 0.0, v)


def planned(nx, ny, seed, fast):
    rng = np.random.default_rng(seed)
    n = nx * ny
    d = divisors(rng, n)
    f = np.zeros((2, 9, n))
    if fast:      # an opposite pair cancels in the density, the diagonal pair holds it
        v = 0.5 * numerators(rng, d, 4, 20) * np.where(rng.random(n) < 0.5, 1.0, -1.0)
        along_x = rng.random(n) < 0.5
        for a, on in ((0, along_x), (1, ~along_x)):
            f[0, 1 + a] = np.where(on, v, 0.0)
            f[0, 3 + a] = np.where(on, -v, 0.0)
        f[0, 5] = f[0, 7] = 0.5 * d
    else:         # momenta on the grid of the density's last bit, so that both are exact
        for a in range(2):
            j = np.round(np.minimum(numerators(rng, d, -20, -1), 0.49) * 2.0 ** 52) * 2.0 ** -52
            f[0, 0] -= j
            plus = rng.random(n) < 0.5
            f[0, 1 + a] = np.where(plus, j, 0.0)
            f[0, 3 + a] = np.where(plus, 0.0, j)
        f[0, 0] += d
    s = f[0, 0].copy()
    for i in range(1, 9):
        s += f[0, i]
    assert np.array_equal(s, d)
    return f.reshape(2, 9, ny, nx)


@pytest.mark.parametrize("nx,ny", [(70, 37), (300, 90)])   # row by row (k_small64), and in tiles
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("fast", [False, True])
def test_velocity_is_the_rounded_quotient(oracle_mod, nx, ny, mode, fast):
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    kw = dict(tau=(1.0, 1.0), G_AB=0.0, G1=0.0, G2=0.0)
    for seed in range(4):
        f = planned(nx, ny, seed, fast)
        o = oracle_mod.OracleSim(nx, ny, **kw)
        o.set_f(f)
        o.step(1)
        L = lb.Lattice(nx, ny, **kw)
        L.set_config(mode, 8)
        L.set_populations(np.ascontiguousarray(f))
        L.step(1)
        a, b = L.get_populations(), o.get_f().reshape(2, 9, ny, nx)
        L.close()
        assert np.isfinite(b).all()
        assert np.array_equal(a, b), int((a != b).sum())
