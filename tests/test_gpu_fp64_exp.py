"""The FP64 step's exp(-rho) (table-driven, csrc/lb_f64.cuh) over and beyond the
densities its table covers: a uniform mixture at rest has forces of zero
beyond rounding, so a density ramp is used instead: one step of smooth random
densities in [lo, hi] against the oracle, 1e-13 of the largest population (one
step; the only differing roundings are exp()'s last bit)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C6 = dict(G_AB=3.0, G1=-7.4, G2=6.4)


@pytest.mark.parametrize("lo,hi", [(0.0, 1e-3), (0.01, 1.2), (0.9, 1.1), (1.5, 2.5), (2.0, 6.0), (-0.05, 0.05), (20.0, 30.0)])
@pytest.mark.parametrize("nx,ny,mode", [(70, 37, 0), (230, 75, 0), (230, 75, 2)])
def test_one_step(oracle_mod, lo, hi, nx, ny, mode):
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    rng = np.random.default_rng(1)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).reshape(1, 9, 1, 1)
    f = w * rng.uniform(lo, hi, (2, 1, ny, nx))
    f[1] = w * rng.uniform(0.5, 1.0, (1, ny, nx))
    kw = dict(tau=(1.0, 2.0), **C6)
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
    assert np.max(np.abs(a - b)) <= 1e-13 * np.max(np.abs(b))
