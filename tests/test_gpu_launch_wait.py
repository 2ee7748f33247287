"""An FP32 step of LB_MODE_LAUNCH that is staged by TMA (12 or more tiles of
32 x 8 per SM): lb_batch_set_wait_limit belongs to LB_MODE_PERSISTENT and
LB_MODE_TMA, so neither a limit of one clock nor the drop hook reaches it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_launch_mode_takes_no_wait_limit():
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    nx, ny = 1024, 512
    y, x = np.mgrid[0:ny, 0:nx]
    wave = np.cos(2 * np.pi * x / nx) * np.cos(2 * np.pi * y / ny)
    rho = np.stack([0.7 + 0.5 * wave, 0.7 - 0.5 * wave])
    out = []
    for mode, limit in ((lb.LB_MODE_LAUNCH, 1e-9), (lb.LB_MODE_FUSED, None)):
        b = lb.Batch([dict(nx=nx, ny=ny, tau=(1.0, 1.0))], precision=lb.LB_FP32, G_AB=3.0, G1=-7.4, G2=6.4)
        b.set_config(mode, 8)
        b.set_fields(0, rho)
        if limit is not None:
            b.set_wait_limit(limit, drop_tile=18)
        b.step(4)
        b.synchronize()
        out.append(b.fields(0))
        b.close()
    assert np.array_equal(out[0]["rho"], out[1]["rho"]) and np.array_equal(out[0]["mom"], out[1]["mom"])
