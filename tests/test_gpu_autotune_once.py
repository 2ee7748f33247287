"""The autotuner times a step that several (mode, tile height) pairs share once:
a small FP64 lattice steps row by row in LB_MODE_LAUNCH and LB_MODE_FUSED at every
height, so its choice is always the first of these, LB_MODE_LAUNCH at the height
that mode takes there, and not whichever of six equal timings came out lowest."""
import pytest

from paper_1806_06943_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(32, 32), (64, 64), (70, 45), (96, 60)])
def test_shared_steps_are_timed_once(nx, ny):
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    L = lb.Lattice(nx, ny, tau=(1.0, 1.0), G_AB=3.0, G1=-7.4, G2=6.4)
    L.set_fields(W.droplet(nx, ny, min(nx, ny) / 4, seed=5))
    for _ in range(3):
        L.autotune(64)
        assert L.config() == (lb.LB_MODE_LAUNCH, 4)
    L.close()
