"""Units of 2^31 and more loads a CTA (needs a GPU with 70 GB free): one tile of
131072 x 131072 16-bit pixels in one CTA's unit, 2^31 vectors of eight.

The pixels are powers of two and small multiples of them, so every partial sum
of Sx, Sy and B is a multiple of its unit in the last place whatever the order:
these three come out exact.  A and the maps: 1e-5 relative (tests/parity.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 131072
PARAMS = {"C1": 0.5, "C2": 0.5, "C": 0.5, "D": 0.25}


@pytest.mark.parametrize("dt", ["f16", "bf16"])
def test_one_cta_unit_of_two_to_the_31_vectors(dt):
    import torch
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    need = 2 * 2 * N * N
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < need + (2 << 30):
        pytest.skip("needs 70 GB of free device memory")
    tdt, code = {"f16": (torch.float16, iqa.IQA_F16), "bf16": (torch.bfloat16, iqa.IQA_BF16)}[dt]
    x = torch.full((N, N), 1.0, dtype=tdt, device="cuda")
    y = torch.full((N, N), 0.5, dtype=tdt, device="cuda")
    x[-1] = 3.0  # the last row, which a count cut short would miss
    ctx = iqa.iqa_create(0, 0)
    try:
        iqa.iqa_set_config(ctx, code, N, N, iqa.MAPS_BOTH,
                           {"variant": 0, "threads": 512, "ilp": 8, "tiles_across": 1,
                            "split": 1, "vector": 1})
        lisi, aug = torch.full((2, 1), float("nan"), device="cuda")
        sums = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
        iqa.iqa_both(ctx, x, y, code, N, N, PARAMS, lisi, aug, sums, torch.cuda.current_stream())
        torch.cuda.synchronize()
    finally:
        iqa.iqa_destroy(ctx)
        del x, y
        torch.cuda.empty_cache()
    rest, row = float(N) * (N - 1), float(N)
    A = rest * 1.5 / 1.0 + row * 3.5 / 3.0
    B = rest * 1.5 * 0.5 + row * 3.5 * 2.5
    Sx, Sy = rest + 3.0 * row, 0.5 * (rest + row)
    got = sums.cpu().numpy()
    assert tuple(got[1:]) == (B, Sx, Sy)
    assert abs(got[0] - A) <= 1e-5 * A
    want = 0.25 * A / (max(Sx, Sy) + 0.5)
    assert abs(float(lisi[0]) - want) <= 1e-5 * want
    r = B / (Sx + Sy + 0.5)
    assert abs(float(aug[0]) - (1.0 - r)) <= 1e-5 * max(1.0 - r, r)
    assert np.isfinite(got).all()
