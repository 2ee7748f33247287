"""The FP64 step forms its products in integer arithmetic where every value
lies in the range that arithmetic covers, and on the FP64 pipe elsewhere
(csrc/lb_f64.cuh); both have the bits of the IEEE product.

A body force of 1e-70 lies outside the range of the lattice's constants, so
such a lattice takes the FP64 pipe at every node, and is too small to change
a force: its populations equal those of the lattice without it bit for bit.
Against the oracle the tolerance is 1e-13 of the largest population: three
steps, whose only differing roundings are the last bit of exp()."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C6 = dict(G_AB=3.0, G1=-7.4, G2=6.4)
# a lattice stepped row by row (k_small64), and one stepped in tiles
SIZES = [(70, 37), (230, 75)]


@pytest.fixture(scope="module")
def lbmod():
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    return lb


def populations(nx, ny, seed, kind="wide"):
    """Populations of a mixture near equilibrium, node densities over two
    decades; "ties": mantissas of few bits, whose products are ties and exact
    results."""
    rng = np.random.default_rng(seed)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).reshape(1, 9, 1, 1)
    f = w * rng.uniform(0.1, 1.0, (2, 1, ny, nx)) * rng.uniform(0.8, 1.2, (2, 9, ny, nx))
    f *= np.where(rng.random((2, 1, ny, nx)) < 0.2, 0.05, 1.0)
    return np.round(f * 4096.0) / 4096.0 if kind == "ties" else f


@pytest.mark.parametrize("mode,height", [(0, 2), (0, 4), (0, 8), (1, 8), (2, 2), (2, 4), (2, 8)])
@pytest.mark.parametrize("kind,walls,wall_mode", [("wide", 0, 0), ("wide", 1, 0), ("ties", 1, 1), ("ties", 0, 0)])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_integer_products_equal_the_fp64_pipe(lbmod, mode, height, kind, walls, wall_mode, nx, ny):
    got = []
    for g in ((0.0, 0.0), (1e-70, 1e-70)):
        L = lbmod.Lattice(nx, ny, tau=(0.83, 2.7), g=g, walls=walls, wall_mode=wall_mode, wall_rho=(0.03, 1.0), **C6)
        L.set_config(mode, height)
        L.set_populations(populations(nx, ny, 11, kind))
        L.step(3)
        got.append(L.get_populations())
        L.close()
    assert np.isfinite(got[0]).all()
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("scale", [1.0, 1e-40, 1e-62, 1e-306, 1e60, 1e140])
@pytest.mark.parametrize("what", ["uniform", "one species", "random"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_values_at_and_beyond_the_covered_range(oracle_mod, lbmod, mode, scale, what, nx, ny):
    f = populations(nx, ny, 5)
    if what == "uniform":                     # forces and velocities exactly zero
        w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).reshape(1, 9, 1, 1)
        f = np.broadcast_to(w, f.shape).copy()
    elif what == "one species":
        f[0] = 0.0
    f *= scale
    kw = dict(tau=(1.0, 2.0), **C6)
    o = oracle_mod.OracleSim(nx, ny, **kw)
    o.set_f(f)
    L = lbmod.Lattice(nx, ny, **kw)
    L.set_config(mode, 8)
    L.set_populations(f)
    o.step(3)
    L.step(3)
    a, b = L.get_populations(), o.get_f().reshape(2, 9, ny, nx)
    L.close()
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    ok = np.isfinite(b)
    if ok.any():
        assert np.max(np.abs(a[ok] - b[ok])) <= 1e-13 * np.max(np.abs(b[ok]))


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e300])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_a_bad_node_spreads_as_in_the_oracle(oracle_mod, lbmod, mode, bad, nx, ny):
    f = populations(nx, ny, 7)
    f[0, 3, 9, 33] = bad
    kw = dict(tau=(1.0, 2.0), **C6)
    o = oracle_mod.OracleSim(nx, ny, **kw)
    o.set_f(f)
    L = lbmod.Lattice(nx, ny, **kw)
    L.set_config(mode, 8)
    L.set_populations(f)
    o.step(2)
    L.step(2)
    a, b = L.get_populations(), o.get_f().reshape(2, 9, ny, nx)
    L.close()
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    ok = np.isfinite(b) & (np.abs(b) < 1e10)
    assert np.max(np.abs(a[ok] - b[ok])) <= 1e-13 * np.max(np.abs(b[ok]))
