"""Element-order units (needs a GPU): tiles and images that are not whole aligned
16-byte vectors, at the counts where a thread's batches end (none, one element,
a full batch, a last partial one), with the two images offset differently, in
several tiles across a unit and in clusters.  Tolerance: tests/parity.py."""
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


def _shifted(a, elements):
    import torch
    flat = parity.to_device(a).reshape(-1)
    buf = torch.zeros(flat.numel() + elements, dtype=flat.dtype, device="cuda")
    buf[elements:] = flat
    return buf[elements:]


# 256 threads, batches of 8: 45^2 = 2025 elements end inside the first batch,
# 46^2 = 2116 begin a second, 91^2 = 8281 a fifth; 64 and 16 with images off
# the vector boundary put several tiles in a unit; 210 and 214 are split over a
# cluster; 3 and 15 leave most threads without an element
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("N,NT,sx,sy", [
    (9, 3, 0, 0), (45, 15, 1, 0), (90, 45, 0, 0), (92, 46, 0, 3), (182, 91, 1, 1),
    (256, 64, 1, 1), (128, 16, 3, 2), (420, 210, 0, 1), (642, 214, 1, 1), (255, 255, 0, 0)])
def test_elements_against_oracle(ctx, orc, dt, N, NT, sx, sy):
    x, y = synth.paper_pair(N=N, dtype=dt)
    want = parity.oracle_maps(orc, x, y, NT, PARAMS)
    dx, dy = _shifted(x, sx), _shifted(y, sy)
    for which in ("both", "lisi", "aug"):
        parity.assert_parity(parity.gpu_maps(ctx, x, y, NT, PARAMS, which, dx=dx, dy=dy), want,
                             PARAMS)
