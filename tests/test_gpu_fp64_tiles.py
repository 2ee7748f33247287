"""The tile kernels of both passes and of the one-pass step, beyond the sizes that
FP64 lattices step row by row and at every tile height.

- A batch of more rows than that (and one of velocity-shift lattices, which never
  step by rows, on both sides of the choice of the two-pass step's tile height):
  every mode and height gives the same populations, in two chains and alone, and
  the oracle's to 1e-12 (the tolerance of the batched parity test).
- lb_profile steps with the kernels of its mode and height, the two passes among
  them: the populations are those of lb_step, bit for bit.
- With a body force of 1e-70 (no integer products) the tile kernels give the
  populations of the lattice without it."""
import numpy as np
import pytest

from paper_1806_06943_gb300 import workloads as W

pytestmark = pytest.mark.gpu

C6 = dict(G_AB=3.0, G1=-7.4, G2=6.4)
BIG = [
    dict(nx=230, ny=75, tau=(1.0, 1.0)),
    dict(nx=96, ny=33, tau=(0.6, 1.2), walls=1, wall_mode=1, wall_rho=(0.03, 1.0), g=(1e-5, 0.0)),
    dict(nx=130, ny=46, tau=(1.3, 0.9), walls=1, wall_mode=0, g=(2e-5, 0.0)),
]
SHIFT = dict(G_AB=1.0, G1=-2.0, G2=1.5, forcing=1)
CONFIGS = [(m, ty) for m in (0, 1, 2) for ty in (2, 4, 8)]


@pytest.fixture(scope="module")
def lbmod():
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    return lb


def field(s, i):
    return W.droplet(s["nx"], s["ny"], min(s["nx"], s["ny"]) / 4, seed=300 + i, periodic=not s.get("walls", 0))


def oracle_fields(oracle_mod, s, rho, steps, common):
    kw = {k: v for k, v in s.items() if k not in ("nx", "ny")}
    o = oracle_mod.OracleSim(s["nx"], s["ny"], **kw, **common)
    o.set_fields(rho)
    o.step(steps)
    return o.fields()


@pytest.mark.parametrize("common,specs", [(C6, BIG), (SHIFT, [dict(nx=70, ny=45, tau=(1.0, 0.8))]),
                                          (SHIFT, [dict(nx=230, ny=81, tau=(1.0, 0.8))])])
def test_modes_and_heights_agree(lbmod, oracle_mod, common, specs):
    steps = 2 * 64 + 3
    rhos = [field(s, i) for i, s in enumerate(specs)]
    ref = []
    for s, r in zip(specs, rhos):
        kw = {k: v for k, v in s.items() if k not in ("nx", "ny")}
        L = lbmod.Lattice(s["nx"], s["ny"], **kw, **common)
        L.set_fields(r)
        L.step(steps)
        ref.append(L.fields())
        L.close()
        fo = oracle_fields(oracle_mod, s, r, steps, common)
        assert np.max(np.abs(ref[-1]["rho"] - fo["rho"])) <= 1e-12 * np.max(np.abs(fo["rho"]))
    for cfg in CONFIGS:
        b = lbmod.Batch(specs, **common)
        b.set_config(*cfg)
        for i, r in enumerate(rhos):
            b.set_fields(i, r)
        b.step(steps)
        for i in range(len(specs)):
            got = b.fields(i)
            for k in ("rho", "mom"):
                assert np.array_equal(got[k], ref[i][k]), (cfg, i, k)
        b.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("spec", [dict(nx=70, ny=37, tau=(2.0, 1.0))] + BIG)
def test_profiled_steps_are_steps(lbmod, precision, spec):
    nx, ny, rho = spec["nx"], spec["ny"], field(spec, 9)
    spec = {k: v for k, v in spec.items() if k not in ("nx", "ny")}
    ref = None
    for cfg in CONFIGS + ([(3, ty) for ty in (2, 4, 8)] if precision else []):
        L = lbmod.Lattice(nx, ny, precision=precision, **spec, **C6)
        L.set_fields(rho)
        if ref is None:
            L.step(9)
            ref = L.get_populations()
            L.set_fields(rho)
        L.set_config(*cfg)
        L.step(1)            # an odd step first: both parities are profiled
        L.profile(8)
        assert L.t == 9
        assert np.array_equal(L.get_populations(), ref), cfg
        L.close()


@pytest.mark.parametrize("height", [2, 4, 8])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("walls,wall_mode", [(0, 0), (1, 0), (1, 1)])
def test_integer_products_of_the_tile_kernels(lbmod, mode, height, walls, wall_mode):
    nx, ny = 230, 85
    rng = np.random.default_rng(17)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).reshape(1, 9, 1, 1)
    f = w * rng.uniform(0.1, 1.0, (2, 1, ny, nx)) * rng.uniform(0.8, 1.2, (2, 9, ny, nx))
    got = []
    for g in ((0.0, 0.0), (1e-70, 1e-70)):
        L = lbmod.Lattice(nx, ny, tau=(0.83, 2.7), g=g, walls=walls, wall_mode=wall_mode, wall_rho=(0.03, 1.0), **C6)
        L.set_config(mode, height)
        L.set_populations(f)
        L.profile(3)
        got.append(L.get_populations())
        L.close()
    assert np.isfinite(got[0]).all()
    assert np.array_equal(got[0], got[1])
