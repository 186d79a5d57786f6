"""The two quotients of a merged tile (needs a GPU) against the same FP64
operations in numpy: sums that are infinite or NaN, and quotients next to the
middle between two float32 numbers, where only an FP64 quotient rounds the right
way.  One tile a block (m = 1), so the sums are the inputs, exact: LISI has to be
float32(D * A / (max(Sx, Sy) + C2)) bit for bit, and augLISI float32(1 - B /
(Sx + Sy + C))."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    h = iqa.iqa_create(0, 0)
    yield h
    iqa.iqa_destroy(h)


def _merge(ctx, tiles, T, m, params):
    import torch
    from paper_2501_10653_gb300 import iqa
    n = (T // m) ** 2
    lisi, aug = torch.full((2, n), 7.0, device="cuda")
    iqa.iqa_merge(ctx, torch.from_numpy(np.ascontiguousarray(tiles)).cuda(), T, m, params, lisi,
                  aug, None, torch.cuda.current_stream())
    torch.cuda.synchronize()
    return lisi.cpu().numpy(), aug.cpu().numpy()


def _want(tiles, params):
    A, B, Sx, Sy = tiles.T
    with np.errstate(all="ignore"):
        return ((params["D"] * A / (np.fmax(Sx, Sy) + params["C2"])).astype(np.float32),
                (1.0 - B / (Sx + Sy + params["C"])).astype(np.float32))


def _special_tiles():
    """Every combination of ordinary, zero, huge, infinite and NaN sums."""
    v = np.array([0.0, 0.375, 3e38, 1e200, np.inf, np.nan])
    return np.stack([g.ravel() for g in np.meshgrid(v, v, v, v, indexing="ij")], axis=1)


@pytest.mark.parametrize("C", [1e-6, 0.0])
@pytest.mark.parametrize("m", [1, 4, 5, 16, 33])
def test_infinite_and_nan_sums(ctx, m, C):
    """The same tile in one place of each block, zeros elsewhere: sums of a block
    are that tile's in every kernel."""
    tiles = _special_tiles()
    M = 36  # 36 * 36 = 6^4 blocks
    params = {"C1": 1e-6, "C2": C, "C": C, "D": 0.5e-6}
    table = np.zeros((M, m, M, m, 4))
    table[:, m - 1, :, m // 2] = tiles.reshape(M, M, 4)
    got = _merge(ctx, table.reshape(-1, 4), M * m, m, params)
    for g, w in zip(got, _want(tiles, params)):
        np.testing.assert_array_equal(g, w)


def test_equal_bright_pixels_whose_sum_overflows(ctx):
    """Maps and merge agree on a tile whose pixel sums are infinite: B = 0 and
    Sx = Sy = inf give augLISI 1."""
    import torch
    from paper_2501_10653_gb300 import iqa
    N = NT = 64
    x = torch.full((N, N), 3e36, device="cuda")
    aug, merged = torch.full((2, 1), 7.0, device="cuda")
    sums = torch.zeros((1, 4), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    iqa.iqa_both(ctx, x, x, iqa.IQA_F32, N, NT, None, None, aug, sums, st)
    iqa.iqa_merge(ctx, sums, 1, 1, None, None, merged, None, st)
    torch.cuda.synchronize()
    assert torch.isinf(sums[0, 2:]).all() and float(sums[0, 1]) == 0.0
    assert float(aug[0]) == 1.0 and float(merged[0]) == 1.0


@pytest.mark.parametrize("k", [34, 40, 44, 46, 48, 50])
def test_quotients_beside_the_middle_of_two_floats(ctx, k):
    """Quotients 2^-k off the middle, either side.  numpy's FP64 operations round
    as the GPU's, and augLISI's quotient of 1/2 to 1 keeps 2^-52 of itself."""
    T = 256
    rng = np.random.default_rng(k)
    n = T * T
    mid = (rng.integers(1 << 23, 1 << 24, n) + 0.5) * 2.0 ** -24  # in [1/2, 1)
    q = mid * (1 + rng.choice([-1.0, 1.0], n) * 2.0 ** -k)
    d = rng.uniform(0.01, 2.0, n)
    tiles = np.zeros((n, 4))
    tiles[:, 0] = q * d
    tiles[:, 1] = d * (1.0 - q)
    tiles[:, 2] = d
    # C2 = C = 0 and D = 1: the quotients are A / Sx and 1 - B / Sx
    params = {"C1": 1e-6, "C2": 0.0, "C": 0.0, "D": 1.0}
    lisi, aug = _merge(ctx, tiles, T, 1, params)
    want_l, want_a = _want(tiles, params)
    assert np.array_equal(lisi, want_l)
    if k <= 48:
        assert np.array_equal(aug, want_a)
