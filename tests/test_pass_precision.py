"""Rounding errors of the FFT passes: the paired-FP32 renormalisations and the
twiddle constants of the transform lengths between the powers of two."""

import math
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1602_04691_gb300", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_twiddles_of_the_mixed_lengths_are_rounded_once(tmp_path):
    """The table of every mixed length and the constants of the 3- to 40-point
    transforms, compiled from the sources: within half a unit in the last place of
    [1/2, 1) of the exact values (and a little for the reference's own rounding)."""
    with open(os.path.join(CSRC, "common.cuh")) as f:
        common = f.read()
    with open(os.path.join(CSRC, "ori_api.cu")) as f:
        api = f.read()
    series = common[common.index("constexpr double kPi"):common.index("// cos/sin of 2 pi j / 64")]
    consts = common[common.index("constexpr bool is_pow2"):common.index("// a + s t and m")]
    table = re.search(r"(static CosSin rounded_cos_sin.*?\n)?static void host_twiddles\(.*?\n\}\n", api, re.S).group(0)
    radices = (3, 5, 6, 10, 12, 20, 24, 40)
    lengths = (144, 200, 288, 400, 576, 800)
    main = "int main() {\n" + "".join(                      # the constants at compile time, as the kernels take them
        f"  {{ constexpr double c = TwR<{R}, double>::c({j}), s = TwR<{R}, double>::s({j});\n"
        f"    std::printf(\"{R} {j} %.17g %.17g\\n\", c, s); }}\n" for R in radices for j in range(R)) + "".join(
        f"  {{ static cpx<double> t[{L}]; host_twiddles({L}, t);\n"
        f"    for (int j = 0; j < {L}; ++j) std::printf(\"{L} %d %.17g %.17g\\n\", j, t[j].x, t[j].y); }}\n" for L in lengths) + "}\n"
    src = tmp_path / "tw.cpp"
    src.write_text("#include <cmath>\n#include <cstdio>\ntemplate <class T> struct cpx { T x, y; };\n" + series + consts +
                   "constexpr bool is_mixed_len(int L) { return !is_pow2(L); }\n" + table + main)
    exe = str(tmp_path / "tw")
    subprocess.run(["g++", "-std=c++17", "-O2", "-o", exe, str(src)], check=True)
    rows = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]
    assert len(rows) == sum(radices) + sum(lengths)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    for row in rows:
        n, j, c, s = row.split()
        a = 2 * pi * np.longdouble(int(j)) / np.longdouble(int(n))
        assert abs(np.longdouble(float(c)) - np.cos(a)) < 5.6e-17 and abs(np.longdouble(float(s)) - np.sin(a)) < 5.6e-17, row


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
