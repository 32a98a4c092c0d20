"""Calls of one plan from several streams.  The calls share the plan's scratch
cubes, so each is ordered behind the plan's last work on whatever stream that
ran: operator calls launch on the caller's stream, the others on the plan's."""

import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_entered_call_marks_its_end_on_every_way_out():
    """The end of a call's work is marked by a scope guard, so an error return
    with launches in flight marks it too; no call enters without the guard."""
    with open(os.path.join(ROOT, "paper_1602_04691_gb300", "csrc", "ori_api.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    guard = re.search(r"\nstruct Handoff \{.*?\n\};\n", src, re.S)
    assert guard and re.search(r"~Handoff\(\) \{\s*if \(p != nullptr && close\(\)", guard.group(0))
    rest = src.replace(guard.group(0), "")
    assert "cudaEventRecord(p->ev" not in re.sub(r"cudaEventRecord\(p->ev[01],", "", rest)   # recorded by the guard alone
    calls = re.findall(r"(\w+[.>]*)\benter\(p, ", rest)
    assert len(calls) >= 9 and set(calls) == {"io."}
    assert len(re.findall(r"\bHandoff io;", rest)) == len(calls)


@pytest.fixture(scope="module")
def problem():
    import torch
    from paper_1602_04691_gb300 import Plan, inputs
    n = 128
    h, N = inputs.random_h_N(n, 61)
    plan = Plan(n, 2.0, torch.from_numpy(h).cuda(), torch.from_numpy(N).cuda())
    g = torch.Generator(device="cuda").manual_seed(62)
    xs = [torch.randn(n ** 3, generator=g, device="cuda", dtype=torch.complex64) for _ in range(4)]
    ref = [plan.matvec32(x, form="B") for x in xs]
    x64 = xs[0].to(torch.complex128)
    df = plan.matvec(x64, form="A", precision="df")
    u, _ = plan.solve(tol=1e-6)
    torch.cuda.synchronize()
    yield plan, xs, ref, x64, df, u
    plan.close()


@pytest.mark.gpu
def test_calls_from_two_streams_follow_one_another(problem):
    """Bitwise the serial results, whichever stream each call comes from, with no synchronisation between."""
    import torch
    plan, xs, ref, x64, df, u = problem
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    out = []
    for rep in range(8):
        for i, s in ((0, a), (1, b), (2, a), (3, b)):
            with torch.cuda.stream(s):
                out.append((ref[i], plan.matvec32(xs[i], form="B")))
        with torch.cuda.stream(a if rep % 2 else b):
            out.append((df, plan.matvec(x64, form="A", precision="df")))
    with torch.cuda.stream(a):
        ys = [plan.matvec32(xs[1], form="B") for _ in range(20)]
    with torch.cuda.stream(b):
        ub, _ = plan.solve(tol=1e-6)
        out.append((ref[2], plan.matvec32(xs[2], form="B")))
    torch.cuda.synchronize()
    assert bool((ub == u).all())
    for r, y in out + [(ref[1], y) for y in ys]:
        assert bool((y == r).all())


@pytest.mark.gpu
def test_captured_operator_calls_replay(problem):
    import torch
    plan, xs, ref, x64, df, _ = problem
    x, y = xs[0].clone(), torch.empty_like(xs[0])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.matvec32(x, form="B", out=y)
        y64 = plan.matvec(x64, form="A", precision="df")
    for i in (0, 2, 3):
        x.copy_(xs[i])
        y.zero_()
        g.replay()
        after = plan.matvec32(xs[1], form="B")      # a direct call behind the replay
        torch.cuda.synchronize()
        assert bool((y == ref[i]).all()) and bool((y64 == df).all()) and bool((after == ref[1]).all())
