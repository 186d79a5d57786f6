"""A one-pair call whose images the kernel just before it writes (needs a GPU):
its CTAs are scheduled, and ask for their pixels in L2, while that kernel still
runs, and must see what it wrote.  Maps of one call are the images of the next,
back to back with nothing in between, over inputs that change every time."""
import numpy as np
import pytest

from paper_2501_10653_gb300 import synth

pytestmark = pytest.mark.gpu


# the second call: vector units from registers, 16-byte rows in units of several
# tiles, element-order units, a cluster
@pytest.mark.parametrize("N,NT,NT2", [(8192, 16, 64), (8192, 16, 16), (8160, 16, 85),
                                      (4096, 8, 256), (8184, 22, 31)])
def test_reads_what_the_kernel_before_wrote(N, NT, NT2):
    import torch
    from paper_2501_10653_gb300 import build, iqa
    build.build()
    ctx = iqa.iqa_create(0, 0)
    st = torch.cuda.current_stream()
    n = N // NT
    gen = torch.Generator(device="cuda").manual_seed(5)
    inputs = [torch.rand((2, N, N), generator=gen, device="cuda") * 0.1 for _ in range(3)]
    first = torch.zeros((2, n, n), device="cuda")
    t = n // NT2
    outs = [torch.full((2, t, t), float("nan"), device="cuda") for _ in range(24)]
    params = {"C1": 1e-2, "C2": 1e-2, "C": 1e-2, "D": 0.0}

    def call(k, out):
        x = inputs[k % 3]
        iqa.iqa_both(ctx, x[0], x[1], iqa.IQA_F32, N, NT, params, first[0], first[1], None, st)
        iqa.iqa_both(ctx, first[0], first[1], iqa.IQA_F32, n, NT2, params, out[0], out[1], None,
                     st)

    want = []
    for k in range(3):
        call(k, outs[0])
        torch.cuda.synchronize()
        want.append(outs[0].cpu().numpy().copy())
    assert not np.array_equal(want[0], want[1])
    for k, out in enumerate(outs):
        call(k, out)
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        assert np.array_equal(out.cpu().numpy(), want[k % 3])
    iqa.iqa_destroy(ctx)
