"""The kernels of 256, 512 and 1024 points.  Most grids between the powers of
two run at other transform lengths; min_L asks for the power of two, so that
every launch variant, the TILES kernels, the FP64 and the paired-FP32 passes are
held to the oracle at these lengths too, on grids that fill them in part."""

import itertools

import numpy as np
import pytest

import oracle as O
from paper_1602_04691_gb300 import inputs


def rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.gpu
@pytest.mark.parametrize("n,L", [(100, 256), (117, 256), (200, 512), (231, 512), (260, 1024), (403, 1024)])
def test_every_kernel_of_a_power_of_two_matches_the_oracle(n, L):
    """FP64 against the oracle's direct sums on rows of every tile class (1e-12);
    paired FP32 (1e-12) and every FP32 schedule (1e-5) against it in every cell."""
    import torch
    from paper_1602_04691_gb300 import Plan
    k = 3.0
    h, N = inputs.random_h_N(n, 190 + n)
    x = inputs.random_complex(n ** 3, 191 + n)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()               # noqa: E731
    plan = Plan(n, k, dev(h), dev(N), min_L=L)
    assert plan.transform_length == L
    rng = np.random.default_rng(n)
    rows = np.unique(np.concatenate([[0, n - 1, n * n - 1, n ** 3 - 1, n ** 3 - n, (n // 2) * (n * n + n + 1)],
                                     rng.choice(n ** 3, 8, replace=False)]))
    S = O.sqrt_hN(h, N)
    ref = x[rows] + S[rows] * (O.C_S_SPHERE / n ** 3) * O.offdiag_sum_rows_octant(S * x, rows, n, k,
                                                                                octant=O.kernel_octant(n, k))
    xd = dev(x)
    y64 = plan.matvec(xd, form="B", precision="fp64")
    y = y64.cpu().numpy()[rows]
    assert np.linalg.norm(y - ref) / np.linalg.norm(ref) < 1e-12
    assert rel(plan.matvec(xd, form="B", precision="df"), y64) < 1e-12
    default = plan.schedule()
    x32 = xd.to(torch.complex64)
    schedules = [{}] + [{f: v} for f in ("yfwd_variant", "zconv_variant", "yinv_variant") for v in range(3)]
    schedules += [dict(yfwd_variant=v, zconv_variant=v, yinv_variant=v, ctas_per_sm=c) for v in range(3) for c in (0, 1)]
    schedules += [dict(yfwd=a, zconv=b, yinv=c) for a, b, c in itertools.product((0, 1), repeat=3)]
    for sch in schedules:
        plan.set_schedule(dict(default, **sch))
        assert rel(plan.matvec32(x32, form="B").to(torch.complex128), y64) < 1e-5, sch
    if n < 300:
        for sch in ({}, dict(zconv_variant=0, yfwd_variant=0, yinv_variant=0), dict(zconv_variant=1), dict(yfwd=1, zconv=1, yinv=1)):
            plan.set_schedule(dict(default, **sch))
            _, info = plan.solve(tol=1e-6)
            assert info["status"] == 0 and info["relres"] <= 1e-6, sch
    plan.close()
