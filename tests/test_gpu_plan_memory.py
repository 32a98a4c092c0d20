"""Device memory while a plan is made."""

import threading

import pytest

from paper_1602_04691_gb300 import inputs


@pytest.mark.gpu
@pytest.mark.parametrize("n,min_L", [(100, 1024), (128, 0), (140, 0)])
def test_the_spectrum_build_and_the_scratch_are_not_held_together(n, min_L):
    """Peak of the device memory in use, sampled while the plan is made: no more than
    the plan's arrays with the build's own cubes, or with the pass scratch, whichever
    is larger.  With a min_L that makes the spectrum larger than the scratch the two
    used to add up (n = 100, 1024 points: 1.9 GB on top)."""
    import torch
    from paper_1602_04691_gb300 import Plan
    h, N = inputs.random_h_N(n, 5)
    h, N = torch.from_numpy(h).cuda(), torch.from_numpy(N).cuda()
    Plan(n, 1.0, h, N, min_L=min_L).close()              # contexts, modules and pools are set up
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    low, stop = [free0], threading.Event()

    def watch():
        torch.cuda.set_device(0)
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])

    t = threading.Thread(target=watch)
    t.start()
    plan = Plan(n, 1.0, h, N, min_L=min_L)
    torch.cuda.synchronize()
    stop.set()
    t.join()
    M = plan.transform_length
    H = M // 2 + 1
    held = free0 - torch.cuda.mem_get_info()[0]
    scratch = 16 * (n * n * M + n * M * M) + n ** 3 * (6 * 16 + 4 * 8)
    build = 16 * (H ** 3 + 2 ** 26)
    fits = n * M * M >= H ** 3 + M * H
    bound = held if fits else max(held, held - scratch + build)
    assert free0 - low[0] <= bound + (64 << 20), (free0 - low[0], held, bound)
    plan.close()
