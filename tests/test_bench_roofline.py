"""The FP64 roofline's fraction is that of the FP64 pipe: one where the kernel's
FP64 instructions alone take the launch's time at the measured rate, whatever
part of the step's products runs on other pipes."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


@pytest.mark.parametrize("kernel", ["k_fused<double, 8>", "k_collide<double, 4>"])
@pytest.mark.parametrize("busy", [1.0, 0.86])
def test_fp64_fraction_counts_the_pipes_instructions(busy, kernel):
    import bench
    peak_tflops, nodes = 1.256, 10 ** 6
    ops = bench.FP64_PIPE_OPS_PER_NODE[kernel.split("<")[0]]
    ms = ops * nodes / (peak_tflops * 1e12 / 2) * 1e3 / busy
    r = bench.alu_roofline(kernel, nodes, ms, peak_tflops, 6800.0)
    assert r["frac"] == pytest.approx(busy) and r["frac"] == pytest.approx(r["achieved"] / r["peak"])
    assert r["plain_evaluation_tflops"] == pytest.approx(bench.FP64_FLOPS_PER_NODE * nodes / (ms * 1e-3) / 1e12)
