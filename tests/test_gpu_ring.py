"""The one-pair kernel's shared-memory ring (needs a GPU): against the oracle
where a thread's vectors are fewer than, equal to and more than the ring's
entries and the last batch is partial, and bit for bit against the same units
summed from registers."""
import numpy as np
import pytest

import parity
from paper_2501_10653_gb300 import synth

pytestmark = pytest.mark.gpu

PARAMS = {"C1": 1e-6, "C2": 1e-6, "C": 1e-6, "D": 0.0}


@pytest.fixture(scope="module")
def ctx():
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    h = iqa.iqa_create(0, 0)
    yield h
    iqa.iqa_destroy(h)


# 16-bit units of eight-vector batches always take the ring: N_T = 16 leaves
# most threads without a vector, 48 / 80 / 96 give ragged counts, 256 with one
# CTA many batches, split 2 a cluster
@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("N,NT,across,split", [
    (64, 16, 1, 1), (480, 48, 1, 1), (400, 80, 1, 1), (384, 96, 1, 2), (512, 64, 4, 1),
    (512, 256, 1, 1), (512, 512, 1, 8)])
@pytest.mark.parametrize("threads", [128, 256, 512])
def test_ring_against_oracle(ctx, orc, dt, N, NT, across, split, threads):
    from paper_2501_10653_gb300 import iqa
    x, y = synth.paper_pair(N=N, dtype=dt)
    code = parity.dtype_code(x)
    cfg = dict(variant=0, threads=threads, ilp=8, tiles_across=across, split=split)
    want = parity.oracle_maps(orc, x, y, NT, PARAMS)
    for which, maps in (("both", iqa.MAPS_BOTH), ("lisi", iqa.MAPS_LISI),
                        ("aug", iqa.MAPS_AUGLISI)):
        iqa.iqa_set_config(ctx, code, N, NT, maps, cfg)
        try:
            got = parity.gpu_maps(ctx, x, y, NT, PARAMS, which)
        finally:
            iqa.iqa_set_config(ctx, code, N, NT, maps, None)
        parity.assert_parity(got, want, PARAMS)


@pytest.mark.parametrize("threads,across", [(128, 1), (128, 2), (256, 2), (512, 1)])
def test_fp32_ring_gives_the_bits_of_the_register_path(ctx, threads, across):
    """2048 units and more of FP32 take the ring, fewer registers: the tiles of
    an image's corner come out the same from the whole image and alone."""
    from paper_2501_10653_gb300 import iqa
    NT = 32
    big, small = 64 * NT, 16 * NT
    rng = np.random.default_rng(17)
    x = rng.normal(0.0, 1e-3, (big, big)).astype(np.float32)
    y = rng.normal(0.0, 1e-3, (big, big)).astype(np.float32)
    maps = {}
    for N in (big, small):
        cfg = dict(variant=0, threads=threads, ilp=8, tiles_across=across)
        if N == small:
            assert (N // NT) ** 2 // across < 2048
        iqa.iqa_set_config(ctx, iqa.IQA_F32, N, NT, iqa.MAPS_BOTH, cfg)
        try:
            maps[N] = parity.gpu_maps(ctx, np.ascontiguousarray(x[:N, :N]),
                                      np.ascontiguousarray(y[:N, :N]), NT, PARAMS)
        finally:
            iqa.iqa_set_config(ctx, iqa.IQA_F32, N, NT, iqa.MAPS_BOTH, None)
    T, t = big // NT, small // NT
    for k in range(2):
        assert np.array_equal(maps[big][k][:t, :t], maps[small][k])
    assert np.array_equal(maps[big][2].reshape(T, T, 4)[:t, :t], maps[small][2].reshape(t, t, 4))
