"""Element-order launches of few units (needs a GPU), which ask for shared memory
so that no SM holds more than their even share: unit counts around a quarter of
152 SMs and around one, two and three units per SM, and clusters that fit one CTA
an SM or do not, alone and back to back on outputs that differ, against the
oracle.  Tolerance: tests/parity.py."""
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


# T^2 = 36, 49, 144, 169, 289, 324, 441, 484 units of one CTA; clusters of two, three
# and seven: 98 and 162, 147 and 300, 63 and 112 CTAs
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("T,NT", [(6, 33), (7, 33), (12, 33), (13, 33), (17, 33), (18, 33),
                                  (21, 33), (22, 33), (7, 202), (9, 202), (7, 177), (10, 177),
                                  (3, 301), (4, 301)])
def test_few_element_units(ctx, orc, dt, T, NT):
    import torch
    from paper_2501_10653_gb300 import iqa
    N = NT * T
    x, y = synth.paper_pair(N=N, dtype=dt)
    dx, dy = parity.to_device(x), parity.to_device(y)
    want = parity.gpu_maps(ctx, x, y, NT, PARAMS, dx=dx, dy=dy)
    parity.assert_parity(want, parity.oracle_maps(orc, x, y, NT, PARAMS), PARAMS)
    outs = torch.full((12, 2, T * T), float("nan"), device="cuda")
    for o in outs:
        iqa.iqa_both(ctx, dx, dy, parity.dtype_code(x), N, NT, PARAMS, o[0], o[1], None,
                     torch.cuda.current_stream())
    torch.cuda.synchronize()
    for o in outs.cpu().numpy():
        assert np.array_equal(o[0], want[0].ravel()) and np.array_equal(o[1], want[1].ravel())
