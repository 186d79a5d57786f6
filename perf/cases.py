"""The workloads that performance is measured on.

Each case is one call, or one short sequence of calls, that a program using
``paper_2501_10653_gb300`` makes through its public entry points: maps of one
image pair, of many pairs in one batched launch, from host memory, merged maps,
and served requests.  Sizes follow the tests, the benchmark and the paper's own
(N = 2048, N_T from 16 to 256), plus image sides and tile sides that are not
powers of two, as image cut-outs have them.
"""
import math

import numpy as np
import torch

from paper_2501_10653_gb300 import iqa

C = 1e-6  # C1 = C2 = C, the library's default; D = C1 / 2
DTYPES = {"f32": (iqa.IQA_F32, torch.float32), "f16": (iqa.IQA_F16, torch.float16),
          "bf16": (iqa.IQA_BF16, torch.bfloat16)}
SERVE_SIDES = (512, 1024, 2048, 4096)
MAX_BYTES = 2 * 8192 * 8192 * 4  # input of the largest listed case


def listed():
    return [
        # the smallest calls: LISI, then augLISI of a 256 x 256 cut-out (the
        # paper computes the two separately); launch and host cost
        {"name": "pair_small_f32", "kind": "pair", "N": 256, "NT": 64, "dtype": "f32",
         "maps": "each", "sums": False},
        # the paper's own pair, one call per pair as epochs arrive
        {"name": "pair_paper_f32", "kind": "pair", "N": 2048, "NT": 64, "dtype": "f32",
         "maps": "both", "sums": False},
        # a wide-field mosaic, one pair per call
        {"name": "pair_large_f32", "kind": "pair", "N": 8192, "NT": 64, "dtype": "f32",
         "maps": "both", "sums": False},
        # the same stored in 16 bits, coarse tiles, augLISI alone with its sums
        # (augLISI is the map to read in 16-bit storage)
        {"name": "pair_large_f16", "kind": "pair", "N": 8192, "NT": 128, "dtype": "f16",
         "maps": "aug", "sums": True},
        # an image side and tile side that are no multiple of a 16-byte vector
        {"name": "pair_ragged_f32", "kind": "pair", "N": 3000, "NT": 75, "dtype": "f32",
         "maps": "both", "sums": False},
        # an odd image side in 16-bit storage: every row starts at another
        # alignment
        {"name": "pair_odd_bf16", "kind": "pair", "N": 2001, "NT": 69, "dtype": "bf16",
         "maps": "both", "sums": False},
        # Eq. 1 / Eq. 2 of the whole image: one tile
        {"name": "pair_whole_f32", "kind": "pair", "N": 4096, "NT": 4096, "dtype": "f32",
         "maps": "both", "sums": True},
        # a night's epochs of several fields in one launch, graph-captured plan
        {"name": "batch_mixed_f32", "kind": "batch", "count": 12, "N": 1024, "N2": 4096,
         "NT": 32, "NT2": 128, "dtype": "f32", "independent": False},
        # many small cut-outs in 16-bit storage, launched back to back
        {"name": "batch_small_f16", "kind": "batch", "count": 48, "N": 512, "N2": 512,
         "NT": 32, "NT2": 32, "dtype": "f16", "independent": True},
        # Eq. 3 / Eq. 4: coarser maps of an N = 8192, N_T = 16 pair from its sums
        {"name": "merge_m8", "kind": "merge", "T": 512, "m": 8},
        # a pair in page-locked host memory, maps back to the host
        {"name": "host_pair_f32", "kind": "host", "N": 2048, "NT": 64, "dtype": "f32",
         "count": 1},
        # a burst of served requests: second epochs rendered on the device
        # against resident references, FP16
        {"name": "serve_burst_f16", "kind": "serve", "count": 12, "N": 4096, "NT": 64,
         "dtype": "f16"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair"] * 7 + ["batch"] * 3 + ["merge", "host", "serve"])
    dtype = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind == "pair":
        shape = rng.choice(["power", "power", "ragged", "ragged", "coarse"])
        if shape == "power":
            NT = rng.choice([16, 32, 64, 128, 256])
        elif shape == "ragged":
            NT = rng.randint(9, 250)
        else:
            NT = rng.choice([rng.randint(400, 2000), 512, 1024, 2048, 4096])
        T = max(1, _log_int(rng, 256, 8192) // NT)
        return {"kind": kind, "N": NT * T, "NT": NT, "dtype": dtype,
                "maps": rng.choice(["both", "both", "both", "lisi", "aug", "each"]),
                "sums": rng.random() < 0.3}
    if kind == "batch":
        NT, NT2 = (rng.choice([16, 32, 48, 64, 96, 128, 256]) for _ in range(2))
        N, N2 = (max(256, 256 * round(_log_int(rng, 256, 4096) / 256)) for _ in range(2))
        most = max(1, MAX_BYTES // (N * N + N2 * N2 + 1) // 4)
        return {"kind": kind, "count": min(_log_int(rng, 2, 64), most), "N": N, "N2": N2,
                "NT": NT, "NT2": NT2, "dtype": dtype, "independent": rng.random() < 0.5}
    if kind == "merge":
        m = rng.choice([2, 3, 4, 5, 8, 16, 32])
        return {"kind": kind, "T": m * max(1, _log_int(rng, 32, 1024) // m), "m": m}
    if kind == "host":
        NT = rng.choice([32, 64, 128, 75])
        return {"kind": kind, "N": NT * max(1, _log_int(rng, 256, 3000) // NT), "NT": NT,
                "dtype": dtype, "count": rng.randint(1, 4)}
    return {"kind": kind, "count": rng.randint(1, 16), "N": rng.choice(SERVE_SIDES[1:]),
            "NT": rng.choice([32, 64, 128]), "dtype": "f16"}


# --- inputs -------------------------------------------------------------------

_ctx = None


def _context():
    """The library context, one for the process."""
    global _ctx
    if _ctx is None:
        _ctx = iqa.iqa_create(0, 0)
    return _ctx


def _sky_pair(N, seed, index, dtype):
    """Two epochs of one synthetic sky on the GPU: Gaussian-beam sources of 4
    pixels FWHM over noise of 2e-4; the second epoch lacks the faintest tenth
    and has noise of its own."""
    rng = np.random.default_rng([seed, index])
    n = max(1, round(33 * (N / 2048) ** 2))
    flux = np.sort(np.exp(rng.uniform(math.log(0.005), math.log(2.0), n)))
    where = rng.integers(0, N, (n, 2))
    gone = math.ceil(0.1 * n)
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 62)))
    x = torch.randn((N, N), generator=gen, device="cuda") * 2e-4
    y = torch.randn((N, N), generator=gen, device="cuda") * 2e-4
    h = 11
    sigma = 4.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    g = np.exp(-np.arange(-h, h + 1) ** 2 / (2.0 * sigma * sigma))
    beam = torch.from_numpy(np.outer(g, g)).float().cuda()
    for i in range(n):
        r, c = (int(v) for v in where[i])
        r0, r1, c0, c1 = max(0, r - h), min(N, r + h + 1), max(0, c - h), min(N, c + h + 1)
        spot = beam[r0 - r + h:r1 - r + h, c0 - c + h:c1 - c + h] * float(flux[i])
        x[r0:r1, c0:c1] += spot
        if i >= gone:
            y[r0:r1, c0:c1] += spot
    t = DTYPES[dtype][1]
    return x.to(t), y.to(t)


def _batch_shapes(case):
    """(N, N_T) of each pair: the two sizes in turn; where a tile side does not
    divide its image side, the next smaller image side that it divides."""
    shapes = []
    for i in range(case["count"]):
        N, NT = (case["N"], case["NT"]) if i % 2 == 0 else (case["N2"], case["NT2"])
        shapes.append((N // NT * NT, NT))
    return shapes


class _Held:
    """A plan or server, destroyed with the state that holds it."""

    def __init__(self, handle, destroy):
        self.handle, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.handle)


def _serve_requests(case, seed):
    """References (side, catalogue, seed) and requests of a burst."""
    rng = np.random.default_rng([seed, 77])
    refs = []
    sigma = 4.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    h = math.ceil(6.0 * sigma)
    prof = np.exp(-np.arange(-h, h + 1, dtype=np.float64) ** 2
                  / (2.0 * sigma * sigma)).astype(np.float32)
    for N in SERVE_SIDES[:SERVE_SIDES.index(case["N"]) + 1]:
        n = max(2, round(33 * (N / 2048) ** 2))
        cat = {"N": N, "x": rng.integers(0, N, n).astype(np.int32),
               "y": rng.integers(0, N, n).astype(np.int32),
               "flux": np.exp(rng.uniform(math.log(0.005), math.log(2.0), n)).astype(np.float32),
               "half": np.full(n, h, np.int32),
               "profile_off": np.arange(n, dtype=np.int32) * (2 * h + 1),
               "profile": np.tile(prof, n), "noise_sigma": np.float32(2e-4)}
        refs.append((N, cat, int(rng.integers(1 << 40))))
    requests = []
    for i in range(case["count"]):
        k = i % len(refs)
        N, cat = refs[k][:2]
        drop = [int(v) for v in rng.choice(len(cat["x"]), min(2, len(cat["x"]) - 1),
                                           replace=False)]
        add = None
        if i % 2:
            add = (int(rng.integers(len(cat["x"]))), int(rng.integers(N)),
                   int(rng.integers(N)), float(np.float32(rng.uniform(0.01, 1.0))))
        requests.append((k, int(rng.integers(1 << 40)), drop, add))
    return refs, requests


def prepare(case, seed):
    ctx = _context()
    kind = case["kind"]
    s = {"case": case, "ctx": ctx, "stream": torch.cuda.current_stream(),
         "params": iqa.iqa_default_params()}
    if kind == "pair":
        N, T = case["N"], case["N"] // case["NT"]
        s["x"], s["y"] = _sky_pair(N, seed, 0, case["dtype"])
        s["lisi"] = torch.zeros((T, T), device="cuda") if case["maps"] != "aug" else None
        s["aug"] = torch.zeros((T, T), device="cuda") if case["maps"] != "lisi" else None
        s["sums"] = (torch.zeros((T * T, 4), device="cuda", dtype=torch.float64)
                     if case["sums"] else None)
    elif kind == "batch":
        # one buffer for all LISI maps and one for all augLISI maps
        shapes = _batch_shapes(case)
        tiles = [(N // NT) ** 2 for N, NT in shapes]
        s["images"], pairs, at = [], [], 0
        s["lisi"], s["aug"] = torch.zeros((2, sum(tiles)), device="cuda")
        for i, ((N, NT), n) in enumerate(zip(shapes, tiles)):
            x, y = _sky_pair(N, seed, i, case["dtype"])
            s["images"].append((x, y))
            pairs.append(iqa.make_pair(x, y, N, NT, s["lisi"][at:at + n], s["aug"][at:at + n]))
            at += n
        flags = iqa.IQA_PLAN_INDEPENDENT if case["independent"] else iqa.IQA_PLAN_GRAPH
        torch.cuda.synchronize()
        s["plan"] = _Held(iqa.iqa_plan_create(ctx, pairs, DTYPES[case["dtype"]][0],
                                              s["params"], flags), iqa.iqa_plan_destroy)
    elif kind == "merge":
        T, M = case["T"], case["T"] // case["m"]
        gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 11)
        r = torch.rand((T * T, 4), generator=gen, device="cuda", dtype=torch.float64)
        # per-tile sums of 16 x 16 pixels of noise with sources here and there
        scale = torch.tensor([4e4, 1e-5, 0.02, 0.02], device="cuda", dtype=torch.float64)
        s["tiles"] = (0.5 + r) * scale
        s["lisi"], s["aug"] = torch.zeros((2, M, M), device="cuda")
        s["sums"] = torch.zeros((M * M, 4), device="cuda", dtype=torch.float64)
    elif kind == "host":
        N, T = case["N"], case["N"] // case["NT"]
        s["images"], s["outputs"], s["pairs"] = [], [], []
        for i in range(case["count"]):
            x, y = (v.cpu().pin_memory() for v in _sky_pair(N, seed, i, case["dtype"]))
            lisi, aug = np.zeros((2, T, T), np.float32)
            s["images"].append((x, y))
            s["outputs"].append((lisi, aug))
            s["pairs"].append(iqa.make_host_pair(x, y, N, case["NT"], lisi, aug))
    else:
        refs, requests = _serve_requests(case, seed)
        srv = iqa.iqa_server_create(ctx, iqa.IQA_F16, max_pairs_per_step=16,
                                    max_inflight_steps=4, pool_bytes=1 << 28,
                                    max_step_bytes=1 << 30, params=s["params"])
        s["server"] = _Held(srv, iqa.iqa_server_destroy)
        for k, (N, cat, ref_seed) in enumerate(refs):
            iqa.iqa_server_add_reference(srv, k, cat, ref_seed)
        s["requests"] = [iqa.make_request(k, case["NT"], q, drop, add)
                         for k, q, drop, add in requests]
        s["outputs"] = []
        for k, *_ in requests:
            T = refs[k][0] // case["NT"]
            s["outputs"].append((np.zeros((T, T), np.float32), np.zeros((T, T), np.float32)))
    return s


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "pair":
        dt = DTYPES[case["dtype"]][0]
        if case["maps"] == "both":
            iqa.iqa_both(ctx, s["x"], s["y"], dt, case["N"], case["NT"], s["params"],
                         s["lisi"], s["aug"], s["sums"], s["stream"])
        if case["maps"] in ("lisi", "each"):
            iqa.iqa_lisi(ctx, s["x"], s["y"], dt, case["N"], case["NT"], s["params"],
                         s["lisi"], s["sums"], s["stream"])
        if case["maps"] in ("aug", "each"):
            iqa.iqa_auglisi(ctx, s["x"], s["y"], dt, case["N"], case["NT"], s["params"],
                            s["aug"], s["sums"], s["stream"])
        return [v for v in (s["lisi"], s["aug"], s["sums"]) if v is not None]
    if kind == "batch":
        iqa.iqa_plan_launch(s["plan"].handle, s["stream"])
        return [s["lisi"], s["aug"]]
    if kind == "merge":
        iqa.iqa_merge(ctx, s["tiles"], case["T"], case["m"], s["params"], s["lisi"], s["aug"],
                      s["sums"], s["stream"])
        return [s["lisi"], s["aug"], s["sums"]]
    if kind == "host":
        if case["count"] == 1:
            (x, y), (lisi, aug) = s["images"][0], s["outputs"][0]
            iqa.iqa_both_host(ctx, x, y, DTYPES[case["dtype"]][0], case["N"], case["NT"],
                              s["params"], lisi, aug)
        else:
            iqa.iqa_both_host_many(ctx, s["pairs"], DTYPES[case["dtype"]][0], s["params"])
        return s["outputs"]
    srv = s["server"].handle
    handles = [iqa.iqa_submit(srv, r) for r in s["requests"]]
    for h, (lisi, aug) in zip(handles, s["outputs"]):
        if iqa.iqa_poll(srv, h, 5_000_000) != iqa.IQA_OK:
            raise RuntimeError("a served request did not finish")
        iqa.iqa_result(srv, h, lisi, aug)
    return s["outputs"]


# --- the work of a pass -----------------------------------------------------------

def work(case):
    """Each pixel read once and each output written once; about ten operations
    a pixel pair (two clamps, sum, difference, divide, four accumulations)."""
    kind = case["kind"]
    es = 4 if case.get("dtype", "f32") == "f32" else 2
    if kind == "merge":
        tiles, merged = case["T"] ** 2, (case["T"] // case["m"]) ** 2
        return {"bytes": 32 * tiles + 40 * merged, "flops": 4 * tiles + 8 * merged}
    if kind == "serve":
        # the reference is read; the second epoch exists only on the device
        sides = SERVE_SIDES[:SERVE_SIDES.index(case["N"]) + 1]
        sides = [sides[i % len(sides)] for i in range(case["count"])]
        px = sum(N * N for N in sides)
        return {"bytes": es * px + sum(8 * (N // case["NT"]) ** 2 for N in sides),
                "flops": 24 * px}
    if kind == "batch":
        shapes = _batch_shapes(case)
    else:
        shapes = [(case["N"], case["NT"])] * case.get("count", 1)
    px = sum(N * N for N, _ in shapes)
    out = 8 if case.get("maps", "both") in ("both", "each") else 4
    out += 32 if case.get("sums") else 0
    return {"bytes": 2 * es * px + sum(out * (N // NT) ** 2 for N, NT in shapes),
            "flops": 10 * px}


# --- the same in 64 bits ----------------------------------------------------------

def _maps64(x, y, NT):
    """Eq. 1, Eq. 2 and the four sums of every tile, in float64 on the GPU, a
    tile row at a time."""
    N, T = x.shape[0], x.shape[0] // NT
    rows = []
    for r in range(T):
        a = x[r * NT:(r + 1) * NT].double()
        b = y[r * NT:(r + 1) * NT].double()
        a, b = (torch.where(v > 0, v, torch.zeros_like(v)) for v in (a, b))
        total, diff = a + b, (a - b).abs()
        terms = torch.stack([total / (diff + C), total * diff, a, b])
        rows.append(terms.view(4, NT, T, NT).sum(dim=(1, 3)).t())
    sums = torch.cat(rows)
    return _ratios(sums, T) + (sums,)


def _ratios(sums, T):
    A, B, Sx, Sy = sums.unbind(1)
    lisi = 0.5 * C * A / (torch.maximum(Sx, Sy) + C)
    return lisi.view(T, T), (1.0 - B / (Sx + Sy + C)).view(T, T)


def _philox(q, seed):
    """Philox4x32-10 (Salmon, Moraes, Dror and Shaw, SC'11): the four words of
    counter (q, 0, 0x5EED, 0) under the 64-bit key `seed`."""
    low = 0xFFFFFFFF  # products wrap modulo 2^64: their 64 bits are exact
    c = [q, torch.zeros_like(q), torch.full_like(q, 0x5EED), torch.zeros_like(q)]
    k0, k1 = seed & low, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & low) ^ c[1] ^ k0, p1 & low,
             ((p0 >> 32) & low) ^ c[3] ^ k1, p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c


def _epoch(cat, seed, drop=(), add=None):
    """The served sky as the library states it (include/iqa.h): float32 sources
    and noise, stored as float16."""
    N = cat["N"]
    sky = torch.zeros((N, N), device="cuda")
    spots = [(i, int(cat["x"][i]), int(cat["y"][i]), cat["flux"][i])
             for i in range(len(cat["x"])) if i not in drop]
    if add is not None:
        spots.append((add[0], add[1], add[2], np.float32(add[3])))
    for i, cx, cy, flux in spots:
        h, at = int(cat["half"][i]), int(cat["profile_off"][i])
        g = cat["profile"][at:at + 2 * h + 1]
        r0, r1, c0, c1 = max(0, cy - h), min(N, cy + h + 1), max(0, cx - h), min(N, cx + h + 1)
        spot = (np.float32(flux) * g[r0 - cy + h:r1 - cy + h])[:, None] \
            * g[c0 - cx + h:c1 - cx + h][None, :]
        sky[r0:r1, c0:c1] += torch.from_numpy(spot).cuda()
    noise = torch.empty((N * N // 4, 4), device="cuda")
    scale = float(np.float32(1.7320508075688772) / np.float32(256.0))
    for k, w in enumerate(_philox(torch.arange(N * N // 4, device="cuda"), seed)):
        noise[:, k] = (sum((w >> (8 * b)) & 0xFF for b in range(4)) - 510).float() * scale
    return (sky + noise.view(N, N) * float(cat["noise_sigma"])).half()


def exact(case, seed):
    kind = case["kind"]
    if kind == "pair":
        lisi, aug, sums = _maps64(*_sky_pair(case["N"], seed, 0, case["dtype"]), case["NT"])
        return [v for v, wanted in ((lisi, case["maps"] != "aug"), (aug, case["maps"] != "lisi"),
                                    (sums, case["sums"])) if wanted]
    if kind == "batch":
        maps = [_maps64(*_sky_pair(N, seed, i, case["dtype"]), NT)
                for i, (N, NT) in enumerate(_batch_shapes(case))]
        return [torch.cat([m[k].reshape(-1) for m in maps]) for k in (0, 1)]
    if kind == "merge":
        T, m = case["T"], case["m"]
        M = T // m
        sums = prepare(case, seed)["tiles"].view(M, m, M, m, 4).sum(dim=(1, 3)).view(-1, 4)
        return [*_ratios(sums, M), sums]
    if kind == "host":
        return [_maps64(*_sky_pair(case["N"], seed, i, case["dtype"]), case["NT"])[:2]
                for i in range(case["count"])]
    refs, requests = _serve_requests(case, seed)
    first = [_epoch(cat, ref_seed) for _, cat, ref_seed in refs]
    return [_maps64(first[k], _epoch(refs[k][1], q, drop, add), case["NT"])[:2]
            for k, q, drop, add in requests]
