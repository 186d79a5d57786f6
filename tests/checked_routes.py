"""Launches for the bounds-checked library (libiqa_checked.so) over the routes that
the battery of checked_battery.py has no shape for: split tiles, the shared-memory
ring with more vectors a thread than ring entries, prefetching calls, and merges
by columns whose width is no power of two.  Run in its own process with
IQA_LIBRARY set (see test_gpu_checked_routes.py); exits non-zero on the first
group with a failed check or a wrong map."""
import sys

import numpy as np

import parity
from checked_battery import PARAMS, _violations
from paper_2501_10653_gb300 import iqa, synth


def _expect(ctx, orc, N, NT, dt, route, shift=0):
    import torch
    x, y = synth.paper_pair(N=N, dtype=dt)
    flat = parity.to_device(y).reshape(-1)
    buf = torch.zeros(flat.numel() + shift, dtype=flat.dtype, device="cuda")
    buf[shift:] = flat
    before = iqa.iqa_debug_routes(ctx)
    for which in ("lisi", "aug", "both"):
        got = parity.gpu_maps(ctx, x, y, NT, PARAMS, which, dy=buf[shift:])
    counts = [a - b for a, b in zip(iqa.iqa_debug_routes(ctx), before)]
    if counts[route] != 3:
        print("N=%d NT=%d %s: calls by route %s" % (N, NT, dt, counts))
        sys.exit(1)
    parity.assert_parity(got, parity.oracle_maps(orc, x, y, NT, PARAMS), PARAMS)


def main():
    import torch
    import oracle
    orc = oracle.Oracle()
    ctx = iqa.iqa_create(0, 0)
    st = torch.cuda.current_stream()
    _violations("start")

    # vectors with long and short chains, elements, several tiles
    for N, NT, shift in ((1536, 1536, 0), (2048, 1024, 0), (1031, 1031, 0), (1626, 542, 0),
                         (1536, 1536, 1)):
        for dt in ("f32", "f16", "bf16"):
            _expect(ctx, orc, N, NT, dt, 2, shift)
    _violations("split tiles")

    # ring: FP32 from 2048 units on, 16 bits always; 33 MB and 8 MB images
    # prefetch, the others do not
    for N, NT, dt, route in ((2048, 16, "f32", 1), (2048, 64, "f32", 1), (2048, 64, "f16", 1),
                             (768, 48, "bf16", 0), (1024, 256, "f16", 0), (1800, 75, "f32", 1),
                             (2001, 69, "bf16", 1)):
        _expect(ctx, orc, N, NT, dt, route)
    # 3072 units of one tile, 18 vectors a thread
    x, y = synth.paper_pair(N=6144)
    dx, dy = parity.to_device(x), parity.to_device(y)
    NT = 96
    T = 6144 // NT
    want = parity.gpu_maps(ctx, x, y, NT, PARAMS, dx=dx, dy=dy)
    iqa.iqa_set_config(ctx, iqa.IQA_F32, 6144, NT, iqa.MAPS_BOTH,
                       dict(variant=0, threads=128, ilp=8, tiles_across=1))
    got = parity.gpu_maps(ctx, x, y, NT, PARAMS, dx=dx, dy=dy)
    assert T * T > 2048 and all(np.allclose(g, w, rtol=1e-5) for g, w in zip(got, want))
    _violations("ring and prefetching calls")

    # column merges, last CTAs with fewer blocks
    for T, m in ((65, 5), (63, 7), (45, 15), (93, 31), (33, 3), (99, 33)):
        rng = np.random.default_rng(T)
        tiles = rng.uniform(0.5, 1.5, (T, T, 4))
        M = T // m
        out = torch.empty((M * M, 4), dtype=torch.float64, device="cuda")
        iqa.iqa_merge(ctx, torch.from_numpy(tiles).cuda(), T, m, PARAMS,
                      torch.empty(M * M, device="cuda"), torch.empty(M * M, device="cuda"), out,
                      st)
        sums = tiles.reshape(M, m, M, m, 4).sum(axis=(1, 3)).reshape(-1, 4)
        assert np.allclose(out.cpu().numpy(), sums, rtol=1e-12)
    _violations("column merges")
    iqa.iqa_destroy(ctx)
    print("checked routes: no failed checks", flush=True)


if __name__ == "__main__":
    main()
