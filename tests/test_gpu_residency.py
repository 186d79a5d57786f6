"""16-bit units whose kernel is compiled for more than one number of CTAs on an SM
(needs a GPU): unit counts around each line of the choice, every map, stream
ordered and independent calls, against the oracle and each other.  Tolerance:
tests/parity.py."""
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


def _check(ctx, orc, N, NT, dt, ilp):
    from paper_2501_10653_gb300 import iqa
    x, y = synth.paper_pair(N=N, dtype=dt)
    code = parity.dtype_code(x)
    assert iqa.iqa_get_config(ctx, code, N, NT, iqa.MAPS_BOTH).ilp == ilp
    dx, dy = parity.to_device(x), parity.to_device(y)
    want = parity.gpu_maps(ctx, x, y, NT, PARAMS, dx=dx, dy=dy)
    parity.assert_parity(want, parity.oracle_maps(orc, x, y, NT, PARAMS), PARAMS)
    for independent in (0, 1):
        iqa.iqa_set_option(ctx, iqa.IQA_OPT_INDEPENDENT_CALLS, independent)
        for which in ("lisi", "aug", "both_nosums"):
            got = parity.gpu_maps(ctx, x, y, NT, PARAMS, which, dx=dx, dy=dy)
            for g, w in zip(got, want):
                assert g is None or np.array_equal(g, w)
    iqa.iqa_set_option(ctx, iqa.IQA_OPT_INDEPENDENT_CALLS, 0)


# batches of two; 1152, 1250, 1352 and 1849 units: up to eight, nine and more on
# each of 152 SMs
@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("N,NT", [(256, 16), (1536, 32), (1600, 32), (1664, 32), (1376, 32)])
def test_batches_of_two(ctx, orc, dt, N, NT):
    _check(ctx, orc, N, NT, dt, 2)


# the ring: 8 to 9 vectors a thread with 625, 722 and 882 units (five and six per
# SM), 16 with 900 and 1024 (six and seven); 512 threads with 128 and 200
@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("N,NT", [(2400, 96), (2432, 64), (2688, 64), (3840, 64), (4096, 128),
                                  (2912, 728), (3640, 728)])
def test_ring(ctx, orc, dt, N, NT):
    _check(ctx, orc, N, NT, dt, 8)
