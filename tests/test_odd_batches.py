"""Batches on grids with an odd number of cells: every second system's FP32
vectors start 8 bytes off a 16-byte boundary."""

import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_update_accesses_are_aligned_and_cover_every_cell():
    """The kernel's own expressions (read from the source) for its first element,
    the number of 16-byte pairs and the lone element, over systems and sizes."""
    with open(os.path.join(ROOT, "paper_1602_04691_gb300", "csrc", "vector_kernels.cuh")) as f:
        src = f.read()
    body = src[src.index("k_cocg_update<float>("):]
    base = re.search(r"float4\* x4 = reinterpret_cast<float4\*>\((.*?)\);", body).group(1)
    pairs = re.search(r"const long long nv = (.*?);", body).group(1).replace("/", "//")
    lone = re.search(r"const long long i = (n3 - 1|head \? 0 : n3 - 1);", body).group(1)
    for n3 in (1, 8, 27, 729, 1000, 65 ** 3):
        for rb in range(4):
            env = {"n3": n3, "head": (rb * n3) & 1, "x": 0}
            start = eval(base, {}, env)
            nv = eval(pairs, {}, env)
            assert (rb * n3 + start) % 2 == 0, (n3, rb)                  # 16-byte accesses
            last = (0 if env["head"] else n3 - 1) if "?" in lone else n3 - 1
            cells = [start + i for i in range(2 * nv)] + ([last] if n3 & 1 else [])
            assert sorted(cells) == list(range(n3)), (n3, rb)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3, 9, 17, 33, 65])
def test_odd_batches_match_single_solves(n):
    """Each system of a mixed-precision batch against its own FP64 solve; both meet
    their tolerances, and the condition number of these systems is of order 1."""
    import torch
    from paper_1602_04691_gb300 import Plan, inputs
    h, N = inputs.random_h_N(n, 70 + n)
    plan = Plan(n, [1.0, 3.0], torch.from_numpy(h).cuda(), torch.from_numpy(N).cuda())
    dirs = [(0.0, 0.0, 1.0), (0.6, 0.8, 0.0), (1.0, 0.0, 0.0)]
    u, infos = plan.solve_batch(dirs, tol=1e-6)
    ref, _ = plan.solve_batch(dirs, tol=1e-11, precision="fp64")
    assert all(i["status"] == 0 for i in infos)
    d = (u - ref).reshape(6, -1).norm(dim=1) / ref.reshape(6, -1).norm(dim=1)
    assert np.all(d.cpu().numpy() < 2e-5)
    plan.close()
