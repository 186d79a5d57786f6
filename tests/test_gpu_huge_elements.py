"""Element-order units whose offsets need 64 bits (needs a GPU with 20 GB free): one
tile of 46349 x 46349 pixels (a prime side, so one CTA's unit and no vectors), in
which rows from 46334 on begin 2^31 elements and more past the first.  The scratch
of a split would exceed its limit, so the one-pair kernel runs (asserted).  The
last 64 rows hold more than half of Sx and B, so a wrapped offset cannot hide.
Tolerance: tests/parity.py."""
import pytest

import parity

pytestmark = pytest.mark.gpu

N = 46349
PARAMS = {"C1": 0.5, "C2": 0.5, "C": 0.5, "D": 0.25}


@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
def test_one_unit_past_32_bit_offsets(dt):
    import torch
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    tdt, code = {"f32": (torch.float32, iqa.IQA_F32), "f16": (torch.float16, iqa.IQA_F16),
                 "bf16": (torch.bfloat16, iqa.IQA_BF16)}[dt]
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 2 * N * N * tdt.itemsize + (2 << 30):
        pytest.skip("needs 20 GB of free device memory")
    x = torch.full((N, N), 1.0, dtype=tdt, device="cuda")
    y = torch.full((N, N), 0.5, dtype=tdt, device="cuda")
    last = 64  # rows at the end
    x[-last:] = 2048.0
    ctx = iqa.iqa_create(0, 0)
    try:
        st = torch.cuda.current_stream()
        out = {k: torch.full((1,), float("nan"), device="cuda") for k in ("l", "a", "l1", "a1")}
        sums = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
        iqa.iqa_both(ctx, x, y, code, N, N, PARAMS, out["l"], out["a"], sums, st)
        iqa.iqa_lisi(ctx, x, y, code, N, N, PARAMS, out["l1"], None, st)
        iqa.iqa_auglisi(ctx, x, y, code, N, N, PARAMS, out["a1"], None, st)
        torch.cuda.synchronize()
        assert iqa.iqa_debug_routes(ctx) == (3, 0, 0)
    finally:
        iqa.iqa_destroy(ctx)
        del x, y
        torch.cuda.empty_cache()
    rest, end = float(N) * (N - last), float(N) * last
    A = rest * 1.5 / 1.0 + end * 2048.5 / 2048.0
    B = rest * 1.5 * 0.5 + end * 2048.5 * 2047.5
    Sx, Sy = rest + 2048.0 * end, 0.5 * (rest + end)
    assert 2048.0 * end > rest
    for g, w in zip(sums.cpu().numpy(), (A, B, Sx, Sy)):
        assert abs(g - w) <= parity.REL * w
    lisi = 0.25 * A / (max(Sx, Sy) + 0.5)
    r = B / (Sx + Sy + 0.5)
    for k in ("l", "l1"):
        assert abs(float(out[k]) - lisi) <= parity.REL * lisi
    for k in ("a", "a1"):
        assert abs(float(out[k]) - (1.0 - r)) <= parity.REL * max(abs(1.0 - r), r)
