"""Which saved spectra a plan takes: those of its padded length L and those of the
transform length of its n, as when both were one length."""

import ctypes
import struct

import numpy as np
import pytest


def header(n, L, c_S, side=1.0):
    H = L // 2 + 1
    h = struct.pack("<8siiiiddQ", b"ORISPEC\0", 1, n, L, 1, c_S, side, H ** 3) + struct.pack("<d", 1.0) + bytes(63 * 8)
    return h.ljust(576, b"\0")


@pytest.mark.parametrize("n,saved,min_L,accepted", [
    (100, 200, 0, True), (100, 256, 0, True), (100, 256, 256, True),
    (100, 200, 256, True), (100, 200, 64, True), (100, 256, 64, True),      # min_L does not raise the length
    (100, 200, 512, False), (100, 256, 512, False), (100, 512, 512, True), (100, 512, 0, False),
    (100, 400, 0, False), (100, 144, 0, False), (64, 128, 128, True), (64, 144, 0, False), (260, 576, 1024, True)])
def test_lengths_are_checked_on_the_host(n, saved, min_L, accepted):
    """A file that holds nothing but its header: refused for its length, or for being short."""
    from paper_1602_04691_gb300 import _lib
    lib = _lib.load()
    dom = _lib.Domain()
    dom.side = 1.0
    po = _lib.PlanOpts()
    lib.ori_default_plan_opts(ctypes.byref(po))
    po.min_L = min_L
    data = header(n, saved, po.c_S)
    plan = ctypes.c_void_p()
    st = lib.ori_plan_from_spectrum(n, ctypes.byref(dom), 1, 1, ctypes.byref(po), data, len(data), None, ctypes.byref(plan))
    assert st == _lib.ORI_ERR_INVALID_ARG
    assert (b"truncated" if accepted else b"padded length") in lib.ori_last_error()


@pytest.mark.gpu
def test_a_spectrum_saved_without_min_L_loads_with_one_that_changes_nothing():
    import torch
    from paper_1602_04691_gb300 import Plan, inputs
    n = 70
    h, N = inputs.random_h_N(n, 7)
    h, N = torch.from_numpy(h).cuda(), torch.from_numpy(N).cuda()
    plan = Plan(n, 2.0, h, N)
    x = torch.from_numpy(inputs.random_complex(n ** 3, 8)).cuda()
    q = Plan(n, 0.0, h, N, spectrum=plan.save_spectrum(), min_L=256)
    assert (q.L, q.transform_length) == (256, 144)
    for prec in ("fp32", "df", "fp64"):
        assert bool((q.matvec(x, "B", prec) == plan.matvec(x, "B", prec)).all())
    assert np.isfinite(float(q.solve(tol=1e-6)[1]["relres"]))
