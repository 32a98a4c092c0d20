"""A complex64 vector of a caller may start 8 bytes off a 16-byte boundary (a
view into a larger tensor): the passes that copy in 16-byte pieces leave such
vectors to those that read element by element."""

import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sixteen_byte_staging_asks_for_the_alignment():
    with open(os.path.join(ROOT, "paper_1602_04691_gb300", "csrc", "passes_impl.cuh")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    ok = re.search(r"inline bool xfwd_pipe_ok\(.*?\n\}", src, re.S).group(0)
    for p in ("a.x", "a.scale", "a.p"):
        assert f"reinterpret_cast<uintptr_t>({p})" in ok
    assert "& 15u) == 0" in ok
    staged = re.search(r"const bool staged = (.*?);", src, re.S).group(1)
    assert all(f"reinterpret_cast<uintptr_t>({p})" in staged for p in ("a.xin", "a.scale")) and "& 15u) == 0" in staged


@pytest.mark.gpu
@pytest.mark.parametrize("n", [12, 40, 70, 100, 128, 130, 300])
def test_matvec32_of_a_view_at_an_odd_element(n):
    """The same operator whatever the alignment of x and y; the two X kernels round
    differently, bound 1e-5 as for every FP32 operator."""
    import torch
    from paper_1602_04691_gb300 import Plan, inputs
    h, N = inputs.random_h_N(n, 30 + n)
    plan = Plan(n, 2.0, torch.from_numpy(h).cuda(), torch.from_numpy(N).cuda())
    buf = torch.randn(n ** 3 + 1, device="cuda", dtype=torch.complex64)
    out = torch.zeros(n ** 3 + 2, device="cuda", dtype=torch.complex64)
    x, y = buf[1:], out[1:-1]
    assert x.data_ptr() % 16 == 8 and y.data_ptr() % 16 == 8
    for form in ("A", "B"):
        ref = plan.matvec32(x.clone(), form=form)
        plan.matvec32(x, form=form, out=y)
        assert float((y - ref).norm() / ref.norm()) < 1e-5
        assert out[0] == 0 and out[-1] == 0
    plan.close()
