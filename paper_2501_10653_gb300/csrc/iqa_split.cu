// iqa_split.cu -- split tiles: the chains over the batch sums, the end of a
// tile, and the host side (iqa_split.cuh says how the work is divided).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "iqa.h"
#include "iqa_ctx.h"
#include "iqa_split.cuh"

namespace iqa {

// blockIdx.y = unit, blockIdx.x = sum * (TH / kSplitThreads) + slice: a GPU
// thread per thread of the unit adds its batches of one sum in order, and the
// warp's totals go through the tree of reduce_unit.  Bound by the chain, four
// dependent additions a batch (N = N_T = 4096 FP32: 128 batches), as long as its
// loads arrive in time: AHEAD of them are on their way while the previous AHEAD
// are added.  Eight at a time, waited for each time, left the whole N = N_T =
// 4096 call at 51.5 us (32.7 with 32 ahead); units of few batches take 8, whose
// registers let more CTAs run at once (N = 4096, N_T = 1024: 30.6 against 40.4).
template <int AHEAD>
__global__ void __launch_bounds__(kSplitThreads) iqa_split_chain_kernel(const SplitArgs p)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int slices = p.TH / kSplitThreads;
    const int q = blockIdx.x / slices, slice = blockIdx.x - q * slices;
    if ((q == 0 && !(p.maps & MAPS_A)) || (q == 1 && !(p.maps & MAPS_B))) return;
    const int tid = slice * kSplitThreads + threadIdx.x;
    const int lc = blockIdx.y;
    const int items = p.t.RH * p.t.LPU;
    int nb = (items_from(tid, p.TH, items) + kSplitIlp - 1) / kSplitIlp;
    // the unit, its threads, batches and warps have a place in the scratch
    // (checked build only)
    const bool warp_ok = IQA_CHECK(lc < p.t.T * p.t.T * p.t.S && q < 4 && tid < p.TH);
    if (!IQA_CHECK(nb <= p.NB) || !warp_ok) nb = 0;
    const float *in = p.parts + ((long long)lc * p.NB * 4 + q) * p.TH + tid;
    const long long step = 4LL * p.TH;
    Kahan k;
    float v[2][AHEAD];
    const auto load = [&](int b, float (&to)[AHEAD]) {
#pragma unroll
        for (int i = 0; i < AHEAD; ++i)
            if (b + i < nb) to[i] = __ldcg(in + (b + i) * step);
    };
    const auto add = [&](int b, const float (&from)[AHEAD]) {
#pragma unroll
        for (int i = 0; i < AHEAD; ++i)
            if (b + i < nb) k.add(from[i]);
    };
    load(0, v[0]);
    for (int b = 0; b < nb; b += 2 * AHEAD) {
        load(b + AHEAD, v[1]);
        add(b, v[0]);
        load(b + 2 * AHEAD, v[0]);
        add(b + AHEAD, v[1]);
    }
    const float s = warp_sum(k.value());
    if ((tid & 31) == 0 && warp_ok) p.warps[((long long)lc * 4 + q) * (p.TH / 32) + tid / 32] = s;
}

// A warp per tile.
__global__ void __launch_bounds__(32) iqa_split_tile_kernel(const SplitArgs p)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int tile = blockIdx.x, lane = threadIdx.x;
    const int warps = p.TH / 32;
    // the tile has a place in the map, a unit's warps one in the warp (checked
    // build only)
    if (!IQA_CHECK(tile < p.t.T * p.t.T && warps <= 32 && p.t.S <= kMaxCluster)) return;
    // all loads first: one latency, not one per unit
    float v[kMaxCluster][4];
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool formed = (q != 0 || (p.maps & MAPS_A)) && (q != 1 || (p.maps & MAPS_B));
            const float *w = p.warps + (((long long)tile * p.t.S + r) * 4 + q) * warps;
            v[r][q] = formed && r < p.t.S && lane < warps ? __ldcg(w + lane) : 0.0f;
        }
    }
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r) {
        if (r < p.t.S) {
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] += warp_sum(v[r][q]);
        }
    }
    if (lane != 0) return;
    combine_tile(p.t.lisi, p.t.aug, tile, s[0], s[1], s[2], s[3], p.t.C2f, p.t.Cf, p.t.Df,
                 p.t.Cd);
    if (p.t.sums) {
        for (int q = 0; q < 4; ++q) p.t.sums[4LL * tile + q] = s[q];
    }
}

namespace {

template <typename Kernel>
cudaError_t launch_after(Kernel kern, const SplitArgs &p, dim3 grid, int threads, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

// Scratch of one call, from the context's stream-ordered pool, which holds at
// most kPoolMost bytes for all streams together, keeps at most kScratchMost of
// them between calls and is given back with the context.  Sizes are powers of
// two, so that one stream's calls of any sizes fit the pool (their blocks add up
// to less than twice the largest).  nullptr where there is none:
//   * above kScratchMost, or with calls of other streams in flight that hold
//     too much of the pool;
//   * under a budget that leaves less than kScratchMost beside what the context
//     holds otherwise (charge_memory);
//   * while the stream is being captured: an allocation in a graph would belong
//     to the graph, beyond the reach of the pool's limit and the budget;
//   * out of memory.
constexpr size_t kScratchMost = 256u << 20;
constexpr size_t kPoolMost = 2 * kScratchMost;
constexpr size_t kScratchLeast = 2u << 20;

// Another stream may be under capture in the mode that forbids every thread
// the calls that could wait for it, among them this stream's allocation and
// release of scratch, which do not.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// ctx->pool_mu is held.
float *scratch_alloc(iqa_ctx *ctx, size_t bytes, cudaStream_t st)
{
    if (bytes > kScratchMost || ctx->pool_failed) return nullptr;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return nullptr;
    }
    if (!ctx->pool) {
        size_t most = kPoolMost;
        if (ctx->budget) {
            const size_t room = ctx->budget > ctx->held ? ctx->budget - ctx->held : 0;
            most = std::min(most, room / kScratchLeast * kScratchLeast);
            if (most < kScratchMost) return nullptr;
        }
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = ctx->device;
        props.maxSize = most;
        unsigned long long keep = kScratchMost;
        int no = 0;  // never makes one stream wait for another
        if (cudaMemPoolCreate(&ctx->pool, &props) != cudaSuccess ||
            cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolAttrReleaseThreshold, &keep) !=
                cudaSuccess ||
            cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolReuseAllowInternalDependencies, &no) !=
                cudaSuccess) {
            cudaGetLastError();
            ctx->pool_failed = true;
            return nullptr;
        }
        ctx->pool_most = most;
    }
    size_t size = kScratchLeast;
    while (size < bytes) size *= 2;
    void *p = nullptr;
    if (cudaMallocFromPoolAsync(&p, size, ctx->pool, st) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return static_cast<float *>(p);
}

// Releases the scratch behind the calls enqueued on st; under a budget also
// records where they end, for charge_memory.  ctx->pool_mu is held.
cudaError_t scratch_free(iqa_ctx *ctx, float *p, cudaStream_t st)
{
    const cudaError_t e = cudaFreeAsync(p, st);
    if (e != cudaSuccess || !ctx->budget) return e;
    std::vector<cudaEvent_t> &busy = ctx->scratch_busy, &idle = ctx->scratch_idle;
    for (size_t i = 0; i < busy.size();) {
        if (cudaEventQuery(busy[i]) == cudaSuccess) {
            idle.push_back(busy[i]);
            busy[i] = busy.back();
            busy.pop_back();
        } else {
            ++i;
        }
    }
    cudaGetLastError();  // of an event not reached yet
    if (idle.empty()) {
        cudaEvent_t ev;
        const cudaError_t ec = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (ec != cudaSuccess) return ec;
        idle.push_back(ev);
    }
    busy.push_back(idle.back());
    idle.pop_back();
    return cudaEventRecord(busy.back(), st);
}

}  // namespace

// Counts `bytes` that the context is about to allocate against its budget.  The
// scratch pool has to give way: where both do not fit, it is given back, once
// the calls that use it have ended.
void charge_memory(iqa_ctx *ctx, size_t bytes)
{
    std::lock_guard<std::mutex> g(ctx->pool_mu);
    ctx->held += bytes;
    if (!ctx->pool || !ctx->budget || ctx->held + ctx->pool_most <= ctx->budget) return;
    const RelaxedCapture relaxed;
    for (cudaEvent_t ev : ctx->scratch_busy) {
        cudaEventSynchronize(ev);
        ctx->scratch_idle.push_back(ev);
    }
    ctx->scratch_busy.clear();
    cudaMemPoolDestroy(ctx->pool);
    ctx->pool = nullptr;
}

// Bytes charged before and given back since.
void credit_memory(iqa_ctx *ctx, size_t bytes)
{
    std::lock_guard<std::mutex> g(ctx->pool_mu);
    ctx->held -= bytes;
}

// Whether the units of shape c (one-pair kernel) leave so many SMs idle for so
// long that three launches are faster.  Measured one-pair kernel against split,
// in us, back to back / a call alone:
//   * element order (256 threads, 4 or 2 bytes a load), spread one to an SM
//     up to 152 units (spread_smem): the split takes its three launches and the
//     image's bytes, the units the time of one.  N = 401, one tile of 161K pixels:
//     31.3 / 45 against 8.6 / 23; tiles of N_T = 211 (45K): 9 units 13.1 / 24
//     against 9.9 / 25, 36 18.3 / 24 and 15.0 / 28, 64 15.1 / 29 and 17.9 / 30, 144
//     20.0 / 30 and 23.3 / 39.  So fewer units the smaller they are: 192 less one
//     for each unit, times a unit's pixels, above 4.2M for 16 bits, 3.4M for FP32,
//     which leaves to the split what it is faster at with inputs in L2 (N_T = 233,
//     100 of 54K FP32 23.1 / 33 and 20.2 / 34; N_T = 609, 112 of 53K FP16 24.6 / 34
//     and 22.4 / 37) or not (N_T = 422, 128 of 89K FP32 37.9 / 51 and 33.9 / 48; N_T =
//     801, 147 of 214K 100 / 106 and 74.7 / 89; N_T = 298, 128 of 44K 21.4 / 33 and
//     21.5 / 36).
//   * vectors: not from one unit per SM on (FP32 N = 3072, N_T = 512, 288 units:
//     18.5 / 26 against 20.5 / 31; N = 6200, N_T = 1240: 55.7 / 69 and 62.2 / 77; FP16
//     N = 8192, N_T = 1024, 512 units: 42.8 / 57 and 57.3 / 68).  With a third to two
//     thirds of a unit per SM full clusters find an SM for each CTA, and the
//     split pays for few shapes (72 units of 131K pixels: FP32 18.7 / 30 against
//     20.7 / 31, FP16 12.8 / 25 and 15.4 / 28; of 524K FP16 38.3 / 52 and 37.0 / 48);
//     with two thirds to one it pays again (128 units of 131K: FP32 35.0 / 42
//     against 30.6 / 42, FP16 24.5 / 36 and 21.1 / 33).
//     - 16 bits: from 100K pixels (one tile N = 1024: 11.6 / 24 against 8.9 / 22;
//       below, N = 800: 8.4 / 21 and 8.5 / 22, 4 tiles N = 1600: 9.2 / 22 and 11.5 /
//       24).
//     - FP32, whose units keep more bytes in flight: from 32K pixels where rows
//       lie multiples of 2 KB apart (N = 1536, N_T = 512: 14.9 / 22 against 11.7 /
//       23; N = 2048: 17.7 / 23 and 13.2 / 26), from 50K where units are at most 16
//       (N = 728, one tile: 11.1 / 22 and 8.4 / 22; below, N = 600: 7.7 / 20 and 8.4 /
//       21), else from 100K (4 tiles N = 1600, 80K: 11.0 / 24 and 11.1 / 24).
bool split_pays(iqa_ctx *ctx, int N, int NT, iqa_dtype dtype, const TileConfig &c)
{
    if (c.variant != 0 || c.TX != 1 || c.ilp != kSplitIlp || c.threads % kSplitThreads != 0)
        return false;
    const long long T = N / NT, units = T * T * c.S;
    const long long unit_px = (long long)NT * NT / c.S;
    const long long sms = ctx->num_sms > 0 ? ctx->num_sms : 152;
    if (c.vec == 1) {
        const long long least = dtype == IQA_F32 ? 3400000 : 4200000;
        return unit_px >= 40000 && (sms + sms / 4 + 2 - units) * unit_px > least;
    }
    if (units >= sms || unit_px < 32768) return false;
    const bool one_an_sm = c.S == kMaxCluster && 3 * units > sms && 3 * units <= 2 * sms;
    if (dtype != IQA_F32) return unit_px >= (one_an_sm ? 400000 : 100000);
    if (unit_px >= 100000) return !one_an_sm;
    return N % 512 == 0 || (units <= 16 && unit_px >= 50000);
}

// One pair in the order of the one-pair kernel's shape c; `a` as for
// launch_tiles.  *done is false, and nothing was launched, without scratch.
iqa_status run_split(iqa_ctx *ctx, const TileArgs &a, const TileConfig &c, iqa_dtype dtype,
                     int maps, cudaStream_t st, bool *done)
{
    *done = false;
    SplitArgs p;
    p.t = a;
    p.maps = maps;
    p.TH = c.threads;
    const long long units = (long long)a.T * a.T * a.S;
    const long long items = (long long)a.RH * a.LPU;
    const long long batch = (long long)p.TH * kSplitIlp;
    const long long NB = (items + batch - 1) / batch;
    if (items > 0x7fffffffLL - batch) return IQA_OK;
    p.NB = (int)NB;
    // about two waves of the six CTAs that an SM holds
    const long long sms = ctx->num_sms > 0 ? ctx->num_sms : 152;
    const long long slices = units * (p.TH / kSplitThreads);
    const long long pieces = std::min(NB, std::max(1LL, (12 * sms + slices - 1) / slices));
    p.PB = (int)((NB + pieces - 1) / pieces);
    p.pieces = (int)((NB + p.PB - 1) / p.PB);
    const size_t n_parts = (size_t)units * NB * 4 * p.TH, n_warps = (size_t)units * 4 * (p.TH / 32);
    const RelaxedCapture relaxed;
    std::unique_lock<std::mutex> lock(ctx->pool_mu);
    p.parts = scratch_alloc(ctx, (n_parts + n_warps) * sizeof(float), st);
    if (!p.parts) return IQA_OK;
    if (!ctx->budget) lock.unlock();  // nothing takes the pool away
    p.warps = p.parts + n_parts;
    cudaError_t e = dtype == IQA_F32   ? launch_split_sums_f32(p, c.vec, maps, st)
                    : dtype == IQA_F16 ? launch_split_sums_f16(p, c.vec, maps, st)
                                       : launch_split_sums_bf16(p, c.vec, maps, st);
    if (e == cudaSuccess)
        e = launch_after(p.NB > 32 ? iqa_split_chain_kernel<32> : iqa_split_chain_kernel<8>, p,
                         dim3((unsigned)(4 * (p.TH / kSplitThreads)), (unsigned)units),
                         kSplitThreads, st);
    if (e == cudaSuccess)
        e = launch_after(iqa_split_tile_kernel, p, dim3((unsigned)(a.T * a.T)), 32, st);
    const cudaError_t ef = scratch_free(ctx, p.parts, st);
    if (e == cudaSuccess) e = ef;
    if (e != cudaSuccess) return cuda_fail(ctx, e, "tile kernel launch");
    *done = true;
    return IQA_OK;
}

}  // namespace iqa

IQA_VIOLATION_READER(iqa_read_violations_split)
