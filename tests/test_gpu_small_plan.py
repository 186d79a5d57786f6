"""Plans of few units: units fewer than the launch's CTAs are made smaller, by
tile rows only (needs a GPU)."""
import numpy as np
import pytest

from test_gpu_batch import PARAMS, Batch, _plan_with_shape, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

# one tile; one unit row (nothing to halve); ragged tile sizes; unequal pairs; 16
# bits; a plan that already has more units than CTAs
CASES = [
    ([(256, 256)], "f32"),
    ([(512, 64)], "f32"),
    ([(640, 80), (768, 96), (256, 32)], "f32"),
    ([(1024, 32), (256, 128), (512, 16)], "f16"),
    ([(512, 32)] * 9, "bf16"),
    ([(1024, 16)] * 24, "f32"),
]


@pytest.mark.parametrize("specs,dt", CASES)
@pytest.mark.parametrize("launches,independent", [(1, False), (3, True)])
def test_smaller_units_change_no_bit(ctx, specs, dt, launches, independent):  # noqa: F811
    """The width of a unit decides the order of a tile's sums, and it is not
    touched: the default plan gives the bits of the same shape set by hand (which
    keeps its unit size), and never fewer units."""
    from paper_2501_10653_gb300 import iqa
    code = {"f32": 0, "f16": 1, "bf16": 2}[dt]
    flags = iqa.IQA_PLAN_GRAPH | (iqa.IQA_PLAN_INDEPENDENT if independent else 0)
    b = Batch(specs, dtype=dt, seed=61)
    small = _run(ctx, b, flags=flags, dtype_code=code, launches=launches)
    got = [b.results(i) for i in range(len(specs))]
    c = small.config
    plain = _plan_with_shape(ctx, b, {"threads": c.threads, "unit_kpx": c.unit_kpx},
                             flags=flags, dtype_code=code, launches=launches)
    assert small.total_units >= plain.total_units
    for i in range(len(specs)):
        for u, v in zip(got[i], b.results(i)):
            assert np.array_equal(u, v), i
