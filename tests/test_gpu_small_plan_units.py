"""How many units a plan of few units has (needs a GPU): halved in tile rows while
they are no more than the launch's 456 CTAs (three on each of 152 SMs; half of
them for an independent plan), as the host-only geometry query counts them, and
the bits of the plan whose shape is set by hand, which keeps its units."""
import numpy as np
import pytest

from test_gpu_batch import Batch, _plan_with_shape, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

# (pairs, dtype, units of the shape as it is, of the plan, of an independent plan):
# rows halved to one; halved until more would be too many; one tile row a unit
# already; more units than CTAs already
CASES = [
    ([(256, 16)], "f32", 2, 16, 16),
    ([(1024, 16), (512, 32)], "f32", 40, 144, 144),
    ([(512, 32)] * 9, "bf16", 18, 144, 144),
    ([(512, 32)] * 48, "f16", 96, 384, 192),
    ([(1024, 16)] * 5, "f32", 160, 320, 160),
    ([(512, 64)] * 3, "f32", 24, 24, 24),
    ([(1024, 16)] * 15, "f32", 480, 480, 480),
]


def test_units_of_a_tuned_context(ctx):  # noqa: F811
    """A shape tuned on a large plan serves a later plan of one small pair, whose
    units are halved all the same: 16 of one tile row, whatever the unit size of
    the tuned shape (4K to 128K pixel pairs), with the bits of that shape set by
    hand."""
    import torch
    from paper_2501_10653_gb300 import iqa
    own = iqa.iqa_create(0, 0)
    large = Batch([(1024, 64)] * 24, seed=63)
    plan = iqa.iqa_plan_create(own, large.pairs(), iqa.IQA_F32, None, 0)
    tuned = iqa.iqa_plan_autotune(plan, torch.cuda.current_stream(), 3)
    assert iqa.iqa_plan_info(plan).config.unit_kpx == tuned.unit_kpx
    iqa.iqa_plan_destroy(plan)
    small = Batch([(256, 16)], seed=64)
    info = _run(own, small)
    got = small.results(0)
    assert info.config.unit_kpx == tuned.unit_kpx and info.config.threads == tuned.threads
    assert info.total_units == 16
    _plan_with_shape(own, small, tuned)
    for u, v in zip(got, small.results(0)):
        assert np.array_equal(u, v)
    iqa.iqa_destroy(own)


@pytest.mark.parametrize("specs,dt,plain_units,units,units_independent", CASES)
@pytest.mark.parametrize("independent", [False, True])
def test_units(ctx, specs, dt, plain_units, units, units_independent, independent):  # noqa: F811
    from paper_2501_10653_gb300 import iqa
    code = {"f32": 0, "f16": 1, "bf16": 2}[dt]
    flags = iqa.IQA_PLAN_INDEPENDENT if independent else iqa.IQA_PLAN_GRAPH
    b = Batch(specs, dtype=dt, seed=62)
    small = _run(ctx, b, flags=flags, dtype_code=code)
    got = [b.results(i) for i in range(len(specs))]
    c = small.config
    shape = {"threads": c.threads, "unit_kpx": c.unit_kpx}
    assert sum(iqa.iqa_plan_unit_shape(code, N, NT, shape)[2] for N, NT in specs) == plain_units
    assert small.total_units == (units_independent if independent else units)
    plain = _plan_with_shape(ctx, b, shape, flags=flags, dtype_code=code)
    assert plain.total_units == plain_units
    for i in range(len(specs)):
        for u, v in zip(got[i], b.results(i)):
            assert np.array_equal(u, v), i
