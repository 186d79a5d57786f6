"""Which one-pair calls are split over the GPU (needs a GPU): shapes just inside and
just outside the rule, by the context's route counts, each with the bits of a
context whose budget leaves no room for scratch (asserted not to split)."""
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


# (dtype, N, N_T, elements that y lies off a 16-byte boundary, split).  Vectors:
# units of 100K pixels (16 bits); 32K where rows lie 2 KB apart, 50K where units
# are at most 16, else 100K (FP32); none of either in clusters of eight with a
# third to two thirds of a unit per SM, but of 16 bits from 400K pixels on, nor
# with one and more.
# Elements: 40K pixels, and 192 less the units, times a unit's pixels, above 4.2M
# (16 bits) or 3.4M (FP32).
CASES = [
    ("f32", 1536, 1536, 0, True), ("f32", 2048, 1024, 0, True), ("f32", 800, 800, 0, True),
    ("f32", 600, 600, 0, False), ("f32", 2480, 1240, 0, True), ("f32", 1600, 800, 0, False),
    ("f32", 1536, 512, 0, True), ("f32", 3072, 1024, 0, False), ("f32", 2048, 512, 0, True),
    ("f32", 2560, 512, 0, False), ("f32", 2500, 500, 0, False), ("f32", 1024, 256, 0, False),
    ("f32", 1536, 1536, 1, True), ("f32", 1031, 1031, 0, True), ("f32", 2022, 1011, 0, True),
    ("f32", 1626, 542, 0, True), ("f32", 1533, 511, 0, False), ("f32", 844, 211, 0, True),
    ("f32", 1477, 211, 0, True), ("f32", 2321, 211, 0, False), ("f32", 1788, 298, 0, True),
    ("f32", 2384, 298, 0, False), ("f32", 2052, 684, 0, False), ("f32", 3852, 1284, 0, True),
    ("f16", 1536, 1536, 0, True), ("f16", 1600, 800, 0, False), ("f16", 1536, 512, 0, False),
    ("f16", 3072, 1024, 0, False), ("f16", 1031, 1031, 0, True), ("f16", 1600, 800, 3, True),
    ("f16", 1533, 511, 0, False), ("f16", 1477, 211, 0, True), ("f16", 2384, 298, 0, False),
    ("f16", 1652, 826, 0, True),
    ("bf16", 2048, 1024, 0, True), ("bf16", 1626, 542, 0, True), ("bf16", 1536, 512, 0, False),
]


@pytest.mark.parametrize("dt,N,NT,shift,split", CASES)
def test_route_and_bits(contexts, dt, N, NT, shift, split):
    import torch
    from paper_2501_10653_gb300 import iqa
    free, bound = contexts
    x, y = synth.paper_pair(N=N, dtype=dt)
    dx, flat = parity.to_device(x), parity.to_device(y).reshape(-1)
    buf = torch.zeros(flat.numel() + shift, dtype=flat.dtype, device="cuda")
    buf[shift:] = flat
    dy = buf[shift:]
    whiches = ("both", "lisi", "aug", "both_nosums")
    before = [sum(iqa.iqa_debug_routes(c)) for c in contexts], \
        [iqa.iqa_debug_routes(c)[2] for c in contexts]
    for which in whiches:
        got = parity.gpu_maps(free, x, y, NT, PARAMS, which, dx=dx, dy=dy)
        want = parity.gpu_maps(bound, x, y, NT, PARAMS, which, dx=dx, dy=dy)
        for g, w in zip(got, want):
            assert (g is None) == (w is None)
            assert g is None or np.array_equal(g, w)
    calls = [sum(iqa.iqa_debug_routes(c)) - b for c, b in zip(contexts, before[0])]
    splits = [iqa.iqa_debug_routes(c)[2] - b for c, b in zip(contexts, before[1])]
    assert calls == [len(whiches)] * 2
    assert splits == [len(whiches) if split else 0, 0]


def test_pinned_shape_is_not_split(contexts):
    from paper_2501_10653_gb300 import iqa
    ctx, N = contexts[0], 1536
    x, y = synth.paper_pair(N=N)
    want = parity.gpu_maps(ctx, x, y, N, PARAMS)
    key = (ctx, iqa.IQA_F32, N, N, iqa.MAPS_BOTH)
    before = iqa.iqa_debug_routes(ctx)[2]
    iqa.iqa_set_config(*key, iqa.iqa_get_config(*key))
    got = parity.gpu_maps(ctx, x, y, N, PARAMS)
    iqa.iqa_set_config(*key, None)
    assert iqa.iqa_debug_routes(ctx)[2] == before
    assert all(np.array_equal(g, w) for g, w in zip(got, want))


def test_streams_split_side_by_side(contexts):
    """Ten calls on each of two streams: every one is split."""
    import torch
    from paper_2501_10653_gb300 import iqa
    ctx, N = contexts[0], 1536
    x, y = synth.paper_pair(N=N)
    dx, dy = parity.to_device(x), parity.to_device(y)
    maps = torch.full((2, 10, 2), float("nan"), device="cuda")
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    before = iqa.iqa_debug_routes(ctx)[2]
    for k in range(10):
        for s, st in enumerate(streams):
            iqa.iqa_both(ctx, dx, dy, iqa.IQA_F32, N, N, PARAMS, maps[s, k, :1], maps[s, k, 1:],
                         None, st)
    torch.cuda.synchronize()
    assert iqa.iqa_debug_routes(ctx)[2] - before == 20
    assert torch.isfinite(maps).all() and (maps == maps[0, 0]).all()
