"""The length the passes transform at, as a plan reports it and as the bench uses it."""

import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_bench_counts_bytes_and_names_kernels_at_the_transform_length():
    import sys
    sys.path.insert(0, ROOT)
    import bench
    with open(os.path.join(ROOT, "bench.py")) as f:
        src = f.read()
    assert "plan.L" not in src and "L = plan.transform_length" in src
    # n = 260 runs 576-point passes: T2 = n 576^2, not n 1024^2
    n, M = 260, 576
    assert bench.alg_bytes("yinv", n, M, 8) == 8.0 * (n * M * M + n * n * M)
    pers = {"yfwd": 0, "zconv": 0, "yinv": 0}
    assert bench.fp32_kernel_name("zconv", 576, pers) == "k_zconv_mix<576>"
    assert bench.fp32_kernel_name("yfwd", 576, pers) == "k_yfwd_pipe<float, 576, 8, 24>"
    assert bench.fp32_kernel_name("yinv", 400, dict(pers, yinv=1)) == "k_yinv_pipe<400, 16, 20>"
    assert bench.fp32_kernel_name("yfwd", 200, pers) == "k_yfwd_pipe<float, 200, 8, 20>"
    assert bench.fp32_kernel_name("xfwd", 800, pers) == "k_xfwd_pipe<800, 8>"
    with open(os.path.join(ROOT, "paper_1602_04691_gb300", "csrc", "common.cuh")) as f:
        mix = {int(L): int(L1) for L, L1 in re.findall(r"struct MixRad<(\d+)> .*L1 = (\d+);", f.read())}
    assert bench.MIXED_L1 == mix


@pytest.mark.gpu
@pytest.mark.parametrize("n,min_L,L,M", [(12, 0, 32, 32), (64, 0, 128, 128), (65, 0, 256, 144), (100, 0, 256, 200),
                                         (101, 0, 256, 256), (100, 256, 256, 256), (100, 512, 512, 512),
                                         (130, 0, 512, 288), (160, 0, 512, 400)])
def test_a_plan_reports_its_transform_length(n, min_L, L, M):
    import torch
    from paper_1602_04691_gb300 import Plan, inputs
    h, N = inputs.random_h_N(n, n)
    plan = Plan(n, 1.0, torch.from_numpy(h).cuda(), torch.from_numpy(N).cuda(), min_L=min_L)
    assert (plan.L, plan.transform_length) == (L, M)
    assert len(plan.save_spectrum()) == 576 + 16 * (M // 2 + 1) ** 3
    plan.close()
