"""The transpose of one time step near walls whose ghost rows mirror the fluid
(their adjoint goes to the fluid node a ghost copies) and on lattices with
ragged tiles: <J v, w> = <v, J^T w> with J v by central differences of the
FP64 forward step (eps = 1e-6), to 1e-7 relative, the bound of the same check
elsewhere."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,walls,wall_mode", [(20, 16, 1, 0), (33, 5, 1, 0), (5, 5, 0, 0), (65, 13, 0, 0), (40, 6, 1, 1)])
def test_step_vjp(nx, ny, walls, wall_mode):
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    from paper_1806_06943_gb300 import workloads as W
    kw = dict(tau=(0.9, 1.3), G_AB=3.0, G1=-7.4, G2=6.4, walls=walls, wall_mode=wall_mode, wall_rho=(0.03, 1.0),
              g=(1e-5, 2e-6))
    L = lb.Lattice(nx, ny, **kw)
    L.set_fields(W.droplet(nx, ny, min(nx, ny) / 3.0, seed=7, periodic=not walls))
    L.step(10)
    f0 = L.get_populations()
    rng = np.random.default_rng(ny)
    v = rng.standard_normal(f0.shape) * np.max(np.abs(f0))
    w = rng.standard_normal(f0.shape)

    def step_from(f):
        K = lb.Lattice(nx, ny, **kw)
        K.set_populations(np.ascontiguousarray(f))
        K.step(1)
        return K.get_populations()

    eps = 1e-6
    Jv = (step_from(f0 + eps * v) - step_from(f0 - eps * v)) / (2 * eps)
    JTw, _ = L.step_vjp(w)
    lhs, rhs = float(np.sum(Jv * w)), float(np.sum(v * JTw))
    assert abs(lhs - rhs) <= 1e-7 * abs(rhs), (lhs, rhs)
