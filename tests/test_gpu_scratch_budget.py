"""Device memory of the scratch that one-pair calls of few large tiles take (needs
a GPU): beside the host workspace it stays inside the context's budget, it makes
room for what the context allocates later, and calls in flight on many streams
share one bounded pool.  Memory is what the device reports free before and
after, within SLACK: allocations are whole 2 MB pages, and other processes
leave the GPU alone."""
import numpy as np
import pytest

import parity
from paper_2501_10653_gb300 import synth

pytestmark = pytest.mark.gpu

PARAMS = {"C1": 1e-6, "C2": 1e-6, "C": 1e-6, "D": 0.0}
MB = 1 << 20
SLACK = 16 * MB


@pytest.fixture(scope="module")
def loaded():
    """Kernels loaded and their local memory in place before any measurement."""
    import torch
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    x, y = synth.paper_pair(N=1031)
    for budget in (0, 1 << 20):
        ctx = iqa.iqa_create(0, budget)
        for dt in (np.float32, np.float16):
            parity.gpu_maps(ctx, x.astype(dt), y.astype(dt), 1031, PARAMS)
        iqa.iqa_destroy(ctx)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _host(ctx, x, y, NT):
    from paper_2501_10653_gb300 import iqa
    T = x.shape[0] // NT
    out = [np.full(T * T, np.nan, np.float32) for _ in range(2)]
    iqa.iqa_both_host(ctx, x, y, iqa.IQA_F32, x.shape[0], NT, PARAMS, *out)
    return out


def test_workspace_and_scratch_fit_the_budget(loaded):
    """One tile of 5639 x 5639 elements: a workspace of 255 MB and scratch of 64
    MB, which together exceed a budget of 270 MB but not one of 600 MB."""
    from paper_2501_10653_gb300 import iqa
    N = 5639
    rng = np.random.default_rng(2)
    x, y = (rng.random((N, N), dtype=np.float32) * 1e-3 for _ in range(2))
    got = []
    for budget in (270 * MB, 600 * MB):
        before = _free()
        ctx = iqa.iqa_create(0, budget)
        got.append(_host(ctx, x, y, N))
        assert before - _free() <= budget + SLACK
        iqa.iqa_destroy(ctx)
    assert np.array_equal(got[0], got[1])


def test_scratch_gives_way_to_a_workspace(loaded):
    """The pool is in use on a stream that is still busy when a host call needs
    the budget; both give the values they give alone."""
    import torch
    from paper_2501_10653_gb300 import iqa
    N, NH = 2039, 7168
    budget = 420 * MB  # the workspace takes 411 MB
    x, y = synth.paper_pair(N=N)
    dx, dy = parity.to_device(x), parity.to_device(y)
    rng = np.random.default_rng(3)
    hx, hy = (rng.random((NH, NH), dtype=np.float32) * 1e-3 for _ in range(2))
    alone = iqa.iqa_create(0, 0)
    want = parity.gpu_maps(alone, x, y, N, PARAMS, dx=dx, dy=dy)
    want_h = _host(alone, hx, hy, 64)
    iqa.iqa_destroy(alone)
    maps = torch.full((2, 1), float("nan"), device="cuda")
    sums = torch.full((1, 4), float("nan"), dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    before = _free()
    ctx = iqa.iqa_create(0, budget)
    with torch.cuda.stream(side):
        torch.cuda._sleep(50_000_000)
        iqa.iqa_both(ctx, dx, dy, iqa.IQA_F32, N, N, PARAMS, maps[0], maps[1], sums, side)
    got_h = _host(ctx, hx, hy, 64)
    assert before - _free() <= budget + SLACK
    for g, w in zip((maps[0], maps[1], sums), want):
        assert np.array_equal(g.cpu().numpy().ravel(), w.ravel())
    assert all(np.array_equal(g, w) for g, w in zip(got_h, want_h))
    # and a call after it, which finds no room for scratch
    got = parity.gpu_maps(ctx, x, y, N, PARAMS, dx=dx, dy=dy)
    assert all(np.array_equal(g, w) for g, w in zip(got, want))
    assert before - _free() <= budget + SLACK
    iqa.iqa_destroy(ctx)


def test_streams_share_a_bounded_pool(loaded):
    """Six calls of 200 MB of scratch held back on six streams at once: 512 MB of
    device memory at most, and every call gives the bits of the others."""
    import torch
    from paper_2501_10653_gb300 import iqa
    N, calls = 10007, 6
    gen = torch.Generator(device="cuda").manual_seed(9)
    x, y = ((torch.rand((N, N), generator=gen, device="cuda") * 1e-3).half() for _ in range(2))
    out = torch.full((calls, 2), float("nan"), device="cuda")
    sums = torch.full((calls, 4), float("nan"), dtype=torch.float64, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(calls)]
    before = _free()
    ctx = iqa.iqa_create(0, 0)
    for st in streams:
        with torch.cuda.stream(st):
            torch.cuda._sleep(200_000_000)
    for k, st in enumerate(streams):
        iqa.iqa_both(ctx, x, y, iqa.IQA_F16, N, N, PARAMS, out[k, :1], out[k, 1:], sums[k], st)
    used = before - torch.cuda.mem_get_info()[0]
    torch.cuda.synchronize()
    iqa.iqa_destroy(ctx)
    assert used <= 512 * MB + SLACK
    assert torch.isfinite(sums).all()
    assert all(torch.equal(out[k], out[0]) and torch.equal(sums[k], sums[0])
               for k in range(1, calls))
