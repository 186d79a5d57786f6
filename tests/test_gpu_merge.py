"""Every merge kernel against the same sums in numpy (needs a GPU): block widths
at the edges of each kernel's range, last CTAs with fewer blocks, tables and
outputs off a 32-byte and a 16-byte boundary, zero tiles and values outside
float32's range.  Sums are FP64 in another order: m^2 additions of nonnegative
terms, within m^2 2^-53 relative; ratios round once to float32, half an ulp, and
a quotient formed in float32 with an FP64 residual adds less than 2^-40."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PARAMS = {"C1": 1e-6, "C2": 1e-6, "C": 1e-6, "D": 0.0}


@pytest.fixture(scope="module")
def ctx():
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    h = iqa.iqa_create(0, 0)
    yield h
    iqa.iqa_destroy(h)


def _run(ctx, tiles, T, m, shift):
    import torch
    from paper_2501_10653_gb300 import iqa
    M = T // m
    buf = torch.zeros(tiles.size + shift, dtype=torch.float64, device="cuda")
    buf[shift:] = torch.from_numpy(tiles.ravel()).cuda()
    out = torch.full((4 * M * M + shift,), float("nan"), dtype=torch.float64, device="cuda")
    lisi, aug = torch.full((2, M * M), float("nan"), device="cuda")
    iqa.iqa_merge(ctx, buf[shift:], T, m, PARAMS, lisi, aug, out[shift:],
                  torch.cuda.current_stream())
    torch.cuda.synchronize()
    return lisi.cpu().numpy(), aug.cpu().numpy(), out[shift:].cpu().numpy().reshape(-1, 4)


def _check(got, tiles, T, m):
    M = T // m
    want = tiles.reshape(M, m, M, m, 4).astype(np.longdouble).sum(axis=(1, 3)).reshape(-1, 4)
    lisi, aug, sums = got
    assert np.all(np.abs(sums - want) <= m * m * 2.0 ** -53 * want)
    A, B, Sx, Sy = want.T
    eps = 2.0 ** -24 * (1 + 2.0 ** -16) + m * m * 2.0 ** -50
    ratio = np.longdouble(0.5e-6) * A / (np.maximum(Sx, Sy) + np.longdouble(1e-6))
    assert np.all(np.abs(lisi - ratio) <= eps * np.abs(ratio))
    d = Sx + Sy + np.longdouble(1e-6)
    assert np.all(np.abs(aug - (1 - B / d)) <= eps * np.abs(1 - B / d) + m * m * 2.0 ** -50 * B / d)


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("T,m", [(1, 1), (37, 1), (64, 2), (33, 3), (20, 4), (5, 5), (65, 5),
                                 (63, 7), (120, 8), (136, 8), (45, 15), (48, 16), (93, 31),
                                 (96, 32), (33, 33), (99, 33), (91, 91), (256, 128)])
def test_every_width(ctx, T, m, shift):
    rng = np.random.default_rng(T * 100 + m)
    tiles = rng.uniform(0.5, 1.5, (T * T, 4)) * np.array([4e4, 1e-5, 0.02, 0.02])
    tiles[rng.random(T * T) < 0.2] = 0.0
    _check(_run(ctx, tiles, T, m, shift), tiles, T, m)


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e20, 1e36])
def test_values_outside_the_range_of_the_float32_quotient(ctx, scale):
    """Scaled tiles: the FP64 quotient takes over, zeros included."""
    T, m = 32, 8
    rng = np.random.default_rng(3)
    tiles = rng.uniform(0.5, 1.5, (T * T, 4)) * np.array([scale, 1e-2, 1.0, 1.0])
    tiles.reshape(4, 8, 4, 8, 4)[1] = 0.0
    _check(_run(ctx, tiles, T, m, 0), tiles, T, m)
