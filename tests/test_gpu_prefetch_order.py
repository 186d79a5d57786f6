"""One-pair calls that bring their pixels to L2 before the kernel just before them,
which writes those pixels, has ended (needs a GPU): they must see what it wrote.
The maps of one call are the images of the next, of 8 MB and more, so that the
second call prefetches (asserted), back to back over inputs that change every
time; the same calls with the device idle in between give the expected bytes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PARAMS = {"C1": 1e-2, "C2": 1e-2, "C": 1e-2, "D": 0.0}

# side and tile side of the first call, dtype and tile side of the second.  FP32:
# units of several tiles from registers, at 8 MB and at 33 MB; the shared-memory
# ring (2048 units and more); a cluster; element order, one and several tiles a
# unit.  16 bits: the bytes of both maps, an image of twice their side, for x and
# y: the ring, and element order.
CASES = [
    (8192, 8, "f32", 64), (8192, 4, "f32", 64), (8192, 4, "f32", 16), (8192, 4, "f32", 256),
    (8192, 2, "f32", 16), (8160, 4, "f32", 85), (8160, 4, "f32", 51), (8184, 4, "f32", 31),
    (8192, 8, "f16", 64), (8192, 4, "f16", 128), (8192, 4, "f16", 16), (8184, 4, "f16", 93),
]


@pytest.mark.parametrize("N,NT,dt,NT2", CASES)
def test_prefetching_call_sees_what_the_kernel_before_wrote(N, NT, dt, NT2):
    import torch
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    ctx = iqa.iqa_create(0, 0)
    st = torch.cuda.current_stream()
    n = N // NT
    gen = torch.Generator(device="cuda").manual_seed(5)
    inputs = [torch.rand((2, N, N), generator=gen, device="cuda") * 0.1 for _ in range(3)]
    first = torch.zeros((2, n, n), device="cuda")
    if dt == "f32":
        x, y, side, code = first[0], first[1], n, iqa.IQA_F32
    else:
        x, y, side, code = first, first, 2 * n, iqa.IQA_F16
    t = (side // NT2) ** 2
    outs = torch.full((24, 2 * t + 8 * t), float("nan"), device="cuda")

    def call(k, out):
        i = inputs[k % 3]
        iqa.iqa_both(ctx, i[0], i[1], iqa.IQA_F32, N, NT, PARAMS, first[0], first[1], None, st)
        iqa.iqa_both(ctx, x, y, code, side, NT2, PARAMS, out[8 * t:9 * t], out[9 * t:],
                     out[:8 * t], st)

    want = []
    for k in range(3):
        call(k, outs[0])
        torch.cuda.synchronize()
        want.append(outs[0].clone())
    assert not torch.equal(want[0].view(torch.int32), want[1].view(torch.int32))
    before = iqa.iqa_debug_routes(ctx)
    for k in range(len(outs)):
        call(k, outs[k])
    after = iqa.iqa_debug_routes(ctx)
    torch.cuda.synchronize()
    # the first call of each two is above the sizes that prefetch
    assert [b - a for a, b in zip(before, after)] == [len(outs), len(outs), 0]
    for k in range(len(outs)):
        assert torch.equal(outs[k].view(torch.int32), want[k % 3].view(torch.int32))
    values = want[0][8 * t:].cpu().numpy()
    assert np.isfinite(values).mean() > 0.5
    iqa.iqa_destroy(ctx)
