"""Rounding errors of the FFT passes: the paired-FP32 renormalisations and the
twiddle constants of the transform lengths between the powers of two."""

import math

import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 64, 144, 200, 260, 280])
def test_paired_fp32_operator_keeps_its_renormalisations(n):
    """Error of the paired-FP32 operator against the FP64 one (1e-15 itself) with
    the convolution 1e6 times the identity term, root mean square over four
    media.  At lengths that are powers of two and fully used (n = 64, 128, 256,
    512), with every value renormalised after eight points, it was 0.85 to
    1.05e-14, and 0.84e-14 at n = 32; bound 1.1e-14 everywhere."""
    import torch
    from paper_1602_04691_gb300 import Plan
    errs = []
    for seed in range(4):
        g = torch.Generator(device="cuda").manual_seed(1000 * n + seed)
        u = lambda: torch.rand(n ** 3, generator=g, device="cuda", dtype=torch.float64) + 0.5   # noqa: E731
        h = torch.complex(u(), u())
        N = u()
        x = torch.randn(n ** 3, generator=g, device="cuda", dtype=torch.complex128)
        plan = Plan(n, 3.0, h, N, c_S=4 * math.pi * 1e8)
        ref = plan.matvec(x, form="A", precision="fp64")
        y = plan.matvec(x, form="A", precision="df")
        errs.append(float((y - ref).norm() / ref.norm()))
        plan.close()
    assert np.sqrt(np.mean(np.square(errs))) < 1.1e-14, errs
