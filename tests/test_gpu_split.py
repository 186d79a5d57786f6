"""Few large tiles split over the GPU (needs a GPU): bit for bit what the
one-pair kernel gives without the split (a context whose budget leaves no room
for scratch, and a captured call), and the oracle's values."""
import numpy as np
import pytest

import parity
from paper_2501_10653_gb300 import synth

pytestmark = pytest.mark.gpu

PARAMS = {"C1": 1e-6, "C2": 1e-6, "C": 1e-6, "D": 0.0}


@pytest.fixture(scope="module")
def contexts():
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    free, bound = iqa.iqa_create(0, 0), iqa.iqa_create(0, 1 << 20)
    yield free, bound
    iqa.iqa_destroy(free)
    iqa.iqa_destroy(bound)


# one tile, 4 and 9 tiles; whole vectors, and elements (odd sides); a side with
# no divisor up to 8 (one CTA a tile), last batches of few threads
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("N,NT", [(1536, 1536), (2048, 1024), (1536, 512), (2500, 500), (1031, 1031),
                                  (2022, 1011), (1533, 511), (2056, 2056)])
def test_split_gives_the_bits_of_the_whole(contexts, orc, dt, N, NT):
    free, bound = contexts
    x, y = synth.paper_pair(N=N, dtype=dt)
    dx, dy = parity.to_device(x), parity.to_device(y)
    for which in ("both", "lisi", "aug", "both_nosums"):
        got = parity.gpu_maps(free, x, y, NT, PARAMS, which, dx=dx, dy=dy)
        want = parity.gpu_maps(bound, x, y, NT, PARAMS, which, dx=dx, dy=dy)
        for g, w in zip(got, want):
            assert (g is None) == (w is None)
            assert g is None or np.array_equal(g, w)
    parity.assert_parity(parity.gpu_maps(free, x, y, NT, PARAMS, dx=dx, dy=dy),
                         parity.oracle_maps(orc, x, y, NT, PARAMS), PARAMS)


def test_captured_call_runs_without_scratch(contexts):
    import torch
    from paper_2501_10653_gb300 import iqa
    ctx = contexts[0]
    N = 1536
    x, y = synth.paper_pair(N=N)
    dx, dy = parity.to_device(x), parity.to_device(y)
    want = parity.gpu_maps(ctx, x, y, N, PARAMS, dx=dx, dy=dy)
    lisi, aug = torch.full((2, 1), float("nan"), device="cuda")
    sums = torch.full((1, 4), float("nan"), dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        iqa.iqa_both(ctx, dx, dy, iqa.IQA_F32, N, N, PARAMS, lisi, aug, sums,
                     torch.cuda.current_stream())
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    for g, w in zip((lisi, aug, sums), want):
        assert np.array_equal(g.cpu().numpy().ravel(), w.ravel())


def test_another_stream_under_capture():
    """The first split call of a context (which makes its pool) while another
    stream is being captured: the call runs at once, the capture is whole."""
    import torch
    from paper_2501_10653_gb300 import iqa
    ctx = iqa.iqa_create(0, 0)
    N = 1536
    x, y = synth.paper_pair(N=N)
    dx, dy = parity.to_device(x), parity.to_device(y)
    maps = torch.full((2, 2), float("nan"), device="cuda")
    sums = torch.full((2, 4), float("nan"), dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        iqa.iqa_both(ctx, dx, dy, iqa.IQA_F32, N, N, PARAMS, maps[0, :1], maps[0, 1:],
                     sums[0], side)
        iqa.iqa_both(ctx, dx, dy, iqa.IQA_F32, N, N, PARAMS, maps[1, :1], maps[1, 1:],
                     sums[1], torch.cuda.current_stream())
    graph.replay()
    torch.cuda.synchronize()
    iqa.iqa_destroy(ctx)
    assert torch.isfinite(sums).all() and torch.equal(sums[0], sums[1])
    assert torch.isfinite(maps).all() and torch.equal(maps[0], maps[1])


def test_two_streams_share_no_scratch(contexts):
    """Calls in flight on two streams at once, ten each: every result as alone."""
    import torch
    from paper_2501_10653_gb300 import iqa
    ctx = contexts[0]
    N = 1536
    pairs = [synth.paper_pair(pair_index=i, N=N) for i in range(2)]
    dev = [(parity.to_device(x), parity.to_device(y)) for x, y in pairs]
    want = [parity.gpu_maps(ctx, x, y, N, PARAMS, dx=d[0], dy=d[1])
            for (x, y), d in zip(pairs, dev)]
    streams = [torch.cuda.Stream() for _ in dev]
    outs = [[torch.full((6,), float("nan"), dtype=torch.float64, device="cuda")
             for _ in range(10)] for _ in dev]
    maps = [[torch.full((2,), float("nan"), device="cuda") for _ in range(10)] for _ in dev]
    torch.cuda.synchronize()
    for k in range(10):
        for (dx, dy), st, o, m in zip(dev, streams, outs, maps):
            iqa.iqa_both(ctx, dx, dy, iqa.IQA_F32, N, N, PARAMS, m[k][:1], m[k][1:],
                         o[k][:4], st)
    torch.cuda.synchronize()
    for w, o, m in zip(want, outs, maps):
        for k in range(10):
            assert np.array_equal(o[k][:4].cpu().numpy(), w[2].ravel())
            assert np.array_equal(m[k].cpu().numpy(), np.concatenate([w[0].ravel(),
                                                                      w[1].ravel()]))
