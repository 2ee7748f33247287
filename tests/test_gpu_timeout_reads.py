"""A bounded wait that ran out (here: a tile whose copy is never started, or that
never reports) is reported by the next call that reads the state, the fields
among them, and once."""
import pytest

from paper_1806_06943_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SPECS = [dict(nx=96, ny=48, tau=(1.0, 1.0)), dict(nx=64, ny=40, tau=(1.5, 1.0))]


@pytest.mark.parametrize("mode", ["TMA", "PERSISTENT"])
@pytest.mark.parametrize("read", ["fields", "observables", "pressure_tensor"])
def test_a_read_reports_the_expired_wait(mode, read):
    from paper_1806_06943_gb300 import build
    build.build()
    from paper_1806_06943_gb300 import lb
    b = lb.Batch(SPECS, precision=lb.LB_FP32, G_AB=3.0, G1=-7.4, G2=6.4)
    b.set_config(getattr(lb, "LB_MODE_" + mode), 8)
    rhos = [W.droplet(s["nx"], s["ny"], 10.0, seed=i) for i, s in enumerate(SPECS)]
    call = {"fields": lambda: b.fields(0), "observables": b.observables, "pressure_tensor": lambda: b.pressure_tensor(0)}[read]
    for i, r in enumerate(rhos):
        b.set_fields(i, r)
    b.set_wait_limit(0.05, drop_tile=2)
    b.step(4)
    with pytest.raises(lb.LBError) as ei:
        call()
    assert ei.value.code == lb.LB_ETIMEOUT
    b.set_wait_limit(2.0, drop_tile=-1)
    for i, r in enumerate(rhos):
        b.set_fields(i, r)
    b.step(40)
    call()
    b.synchronize()
    b.close()
