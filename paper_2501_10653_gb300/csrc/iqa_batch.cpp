// iqa_batch.cpp -- batched form: many image pairs (any mix of N and N_T) in
// ONE persistent launch of iqa_stream_kernel over a (pair, unit) work list,
// optionally captured as a CUDA graph, with a per-plan autotuner.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>
#include <numeric>
#include <utility>
#include <vector>

#include "iqa.h"
#include "iqa_ctx.h"
#include "iqa_stream.cuh"

using namespace iqa;

struct iqa_plan {
    iqa_ctx *ctx = nullptr;
    iqa_dtype dtype = IQA_F32;
    iqa_params P{};
    TileConfig cfg;          // shared by all pairs (TX is chosen per pair)
    int maps = MAPS_AB;
    std::vector<iqa_pair> pairs;  // in work-list order (largest units first)
    PairDesc *h_table = nullptr;  // 128-byte aligned host copy
    PairDesc *d_table = nullptr;
    unsigned long long *d_sched = nullptr;
    long long total_units = 0;
    int head_units = 1;  // units of each CTA's static first grab
    bool shrink = false; // units may be smaller than cfg's (plan_build)
    int grid = 0;
    size_t table_bytes = 0;
    size_t charged = 0;  // device bytes counted against the context's budget
    unsigned long long input_bytes = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int flags = 0;
};

namespace iqa {

static iqa_status check_pair(iqa_ctx *ctx, const iqa_pair &p, iqa_dtype dtype, int i)
{
    if (!p.x || !p.y) {
        set_error(ctx, "pair %d: x and y must be device pointers", i);
        return IQA_ERR_INVALID_ARG;
    }
    if (!p.lisi_map && !p.aug_map && !p.sums) {
        set_error(ctx, "pair %d: no output requested", i);
        return IQA_ERR_INVALID_ARG;
    }
    iqa_status s = check_shape(ctx, p.N, p.NT);
    if (s != IQA_OK) return s;
    const int V = 16 / elem_size(dtype);
    if (((uintptr_t)p.x & 15u) || ((uintptr_t)p.y & 15u) || p.NT % V || p.NT > 256) {
        set_error(ctx, "pair %d: the batched kernel needs 16-byte aligned images and "
                       "NT a multiple of 16 bytes, at most 256 (N=%d NT=%d)",
                  i, p.N, p.NT);
        return IQA_ERR_UNSUPPORTED;
    }
    return IQA_OK;
}

// Bytes of each image in every CTA's static first grab: what an independent
// launch streams while the previous launch drains.  Measured on GB300 (32
// N=2048 pairs per launch, same box, alternated): 256 KB against 64 KB gives
// FP16 N_T = 16 / 64 +2.6% / +3.4% and FP32 about the same; 512 KB gives FP16
// N_T = 32 / 64 a further +1% but loses 4% on FP32 N_T = 32 and 64 (the
// static grabs then unbalance the CTAs), so 16-bit storage takes 512 KB.
// (Capping the static grabs at a quarter of the work instead cost FP16 up to
// 0.8% at N = 1024 ... 4096.)  With 16-bit units of 128K pixel pairs (256 KB
// of each image) 512 KB is still best: 256 KB lost 2.5% and 1 MB 6% at
// N_T = 32 and 64.  FP32 with units of 32K or 64K: 128 KB is within 0.2% of
// 256 KB, and 512 KB 0.4-0.6% slower.
static long long head_bytes(iqa_dtype dtype) { return elem_size(dtype) == 2 ? 524288 : 262144; }

// Halvings of the unit size, in tile rows only (the width stays that of cfg,
// so every tile is summed in the same order whatever else the plan holds), for
// a plan whose units are fewer than its CTAs: as many as still give every unit a
// CTA of its own.  A unit is a serial chain for its CTA (128K pixel pairs take
// about 30 us), so with few of them the launch lasts as long as one.  Launches of
// an independent plan overlap, each with the CTAs that the last one leaves, and
// smaller units cost them more than they save: as many halvings as leave half
// of the CTAs to the next launch.  Measured in us, back to back with inputs not
// in L2 / a launch alone, by units:
//   * graph replays of 48 pairs of N = 512, N_T = 32 FP16: 96 units of 128K 26.7 /
//     35, 192 22.6 / 31, 384 20.6 / 29, 768 22.8 / 32; of 8 pairs 16 units 23.1 / 32,
//     128 10.3 / 20;
//   * the same as independent launches: 96 units 7.8 / 37, 192 8.6 / 32, 384 10.6 /
//     32, 768 13.5 / 32; of 24 pairs 48 units 4.6 / 35, 96 4.4 / 27, 192 5.2 / 26,
//     384 7.3 / 25; of 8 pairs 16 units 3.3 / 33, 128 3.6 / 20.
static int shrink_units(const iqa_plan *pl, const TileConfig &cfg)
{
    long long slots =
        (long long)(pl->ctx->num_sms > 0 ? pl->ctx->num_sms : 152) * cfg.ctas_per_sm;
    if (pl->flags & IQA_PLAN_INDEPENDENT) slots /= 2;
    const auto units_at = [&](int halvings) {
        long long units = 0;
        for (const iqa_pair &p : pl->pairs) {
            TileConfig c = cfg;
            stream_unit_shape(c, p.N, p.NT, pl->dtype, halvings);
            units += pair_units(p.N, p.NT, c);
        }
        return units;
    };
    int best = 0;
    for (int h = 1; h <= 8 && units_at(h) <= slots; ++h) best = h;
    return best;
}

// (Re)build the descriptor table for cfg and upload it; `shrink`: cfg is the
// built-in one or was tuned on another plan, and its units may be made smaller
// (shrink_units).  A shape set by hand, or tuned on this plan, stays as it is.
static iqa_status plan_build(iqa_plan *pl, const TileConfig &cfg, bool shrink = false)
{
    iqa_ctx *ctx = pl->ctx;
    std::string why;
    const int n = (int)pl->pairs.size();
    const int halvings = shrink ? shrink_units(pl, cfg) : 0;
    long long units = 0;
    for (int i = 0; i < n; ++i) {
        const iqa_pair &p = pl->pairs[i];
        TileConfig c = cfg;
        stream_unit_shape(c, p.N, p.NT, pl->dtype, halvings);
        if (!stream_config_valid(p.N, p.NT, pl->dtype, c, &why)) {
            set_error(ctx, "pair %d (N=%d NT=%d): %s", i, p.N, p.NT, why.c_str());
            return IQA_ERR_INVALID_ARG;
        }
        iqa_status s = fill_pair_desc(ctx, &pl->h_table[i], p.x, p.y, p.N, p.NT, pl->dtype,
                                      c, pl->P, p.lisi_map, p.aug_map, p.sums, units);
        if (s != IQA_OK) return s;
        units += pair_units(p.N, p.NT, c);
    }
    cudaError_t e = cudaMemcpy(pl->d_table, pl->h_table, pl->table_bytes,
                               cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "descriptor upload");
    pl->cfg = cfg;
    pl->shrink = shrink;
    pl->total_units = units;
    pl->grid = stream_grid(ctx, cfg, units);
    // each CTA's first grab spans about head_bytes() of each image (at most
    // 8 units), counted on the first pair's units (the largest); one unit of
    // 16K-128K pixel pairs alone is 32-256 KB; no more than an even share of
    // the units, or the CTAs past the last static grab would have nothing
    if (n > 0) {
        const PairDesc &d0 = pl->h_table[0];
        const long long unit_bytes =
            (long long)d0.RH * d0.TX * d0.NT * d0.NT * elem_size(pl->dtype);
        pl->head_units = (int)std::max<long long>(
            1, std::min<long long>({8, units / pl->grid,
                                    head_bytes(pl->dtype) /
                                        std::max<long long>(1, unit_bytes)}));
    }
    return IQA_OK;
}

static StreamParams plan_params(const iqa_plan *pl)
{
    StreamParams sp;
    std::memset(&sp, 0, sizeof sp);
    sp.descs = pl->d_table;
    sp.npairs = (int)pl->pairs.size();
    sp.stage_bytes = pl->cfg.stage_kb * 1024;
    sp.stages = pl->cfg.stages;
    sp.head_units = pl->head_units;
    sp.total_units = pl->total_units;
    sp.status = pl->ctx->d_status;
    sp.timeout_ns = pl->ctx->wait_timeout_ns;
    sp.sched = pl->d_sched;
    sp.inject_stall = pl->ctx->inject_stall;
    sp.overlap_head = (pl->flags & IQA_PLAN_INDEPENDENT) ? 1 : 0;
    return sp;
}

static cudaError_t plan_launch_direct(iqa_plan *pl, cudaStream_t st)
{
    StreamParams sp = plan_params(pl);
    return launch_stream(sp, pl->dtype, pl->cfg, pl->maps, pl->grid, st);
}

static void plan_drop_graph(iqa_plan *pl)
{
    if (pl->exec) cudaGraphExecDestroy(pl->exec);
    if (pl->graph) cudaGraphDestroy(pl->graph);
    pl->exec = nullptr;
    pl->graph = nullptr;
}

static iqa_status plan_capture(iqa_plan *pl)
{
    plan_drop_graph(pl);
    cudaStream_t s = pl->ctx->s_comp;
    cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(pl->ctx, e, "graph capture begin");
    cudaError_t el = plan_launch_direct(pl, s);
    e = cudaStreamEndCapture(s, &pl->graph);
    if (el != cudaSuccess) {
        plan_drop_graph(pl);
        return cuda_fail(pl->ctx, el, "captured launch");
    }
    if (e != cudaSuccess) return cuda_fail(pl->ctx, e, "graph capture end");
    e = cudaGraphInstantiate(&pl->exec, pl->graph, 0);
    if (e != cudaSuccess) {
        plan_drop_graph(pl);
        return cuda_fail(pl->ctx, e, "graph instantiate");
    }
    return IQA_OK;
}

// Batched-kernel shape when nothing was tuned: the autotuner's usual choice on
// GB300 (three CTAs per SM, each a 128-thread consumer group with a two-stage
// ring of 16 KB per image), with units of 32K pixel pairs for FP32 (128 KB of
// each image) and 128K for 16-bit storage (256 KB).  Measured on 32 N=2048
// pairs, same box: FP32 units of 32K against 16K stream 1.4% faster at
// N_T = 64 and 0.9% at N_T = 16, and 64K or more no faster (128K: 0.6%
// slower); 16-bit units of 64K against 32K 1.9% faster at N_T = 64 and 1.3% at
// N_T = 32 (a unit row of 1024 pixels, 2 KB, instead of 512), and 128K another
// 1.2% and 1.5% (two tile rows of 1024 pixels).
TileConfig default_batch_config(iqa_dtype dtype)
{
    TileConfig c;
    c.variant = 1;
    c.threads = 128;
    c.stages = 2;
    c.stage_kb = 16;
    c.ctas_per_sm = 3;
    c.unit_kpx = elem_size(dtype) == 2 ? 128 : 32;
    return c;
}

}  // namespace iqa

extern "C" {

iqa_status iqa_plan_create(iqa_ctx *ctx, const iqa_pair *pairs, int npairs, iqa_dtype dtype,
                           const iqa_params *params, int flags, iqa_plan **out)
{
    if (!ctx) return IQA_ERR_INVALID_ARG;
    if (!out || !pairs || npairs < 1) {
        set_error(ctx, "need out, pairs and npairs >= 1");
        return IQA_ERR_INVALID_ARG;
    }
    *out = nullptr;
    if (!dtype_ok(dtype)) {
        set_error(ctx, "unknown dtype %d", (int)dtype);
        return IQA_ERR_INVALID_ARG;
    }
    if (flags & ~(IQA_PLAN_GRAPH | IQA_PLAN_INDEPENDENT)) {
        set_error(ctx, "unknown plan flags 0x%x", flags);
        return IQA_ERR_INVALID_ARG;
    }
    iqa_params P;
    iqa_status s = resolve_params(ctx, params, &P);
    if (s != IQA_OK) return s;
    for (int i = 0; i < npairs; ++i) {
        s = check_pair(ctx, pairs[i], dtype, i);
        if (s != IQA_OK) return s;
    }
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ctx->device);

    iqa_plan *pl = new iqa_plan();
    pl->ctx = ctx;
    pl->dtype = dtype;
    pl->P = P;
    pl->flags = flags;
    // largest units first, so the dynamic schedule ends evenly
    std::vector<int> order(npairs);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return pairs[a].NT > pairs[b].NT;
    });
    int maps = 0;
    for (int i : order) {
        pl->pairs.push_back(pairs[i]);
        const iqa_pair &p = pairs[i];
        if (p.sums) maps = MAPS_AB;
        if (p.lisi_map) maps |= MAPS_A;
        if (p.aug_map) maps |= MAPS_B;
        pl->input_bytes += 2ull * p.N * p.N * elem_size(dtype);
    }
    pl->maps = maps;
    pl->table_bytes = sizeof(PairDesc) * (size_t)npairs;
    pl->h_table = static_cast<PairDesc *>(
        ::operator new(pl->table_bytes, std::align_val_t(alignof(PairDesc))));
    const size_t need = pl->table_bytes + 256;
    if (ctx->budget && need > ctx->budget) {
        set_error(ctx, "plan tables need %zu bytes, over the HBM budget", need);
        iqa_plan_destroy(pl);
        cudaSetDevice(prev);
        return IQA_ERR_NOMEM;
    }
    charge_memory(ctx, need);
    pl->charged = need;
    cudaError_t e = cudaMalloc(&pl->d_table, pl->table_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&pl->d_sched, 256);
    if (e == cudaSuccess) e = cudaMemset(pl->d_sched, 0, 256);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error(ctx, "plan allocation failed: %s", cudaGetErrorString(e));
        iqa_plan_destroy(pl);
        cudaSetDevice(prev);
        return IQA_ERR_NOMEM;
    }
    TileConfig cfg = default_batch_config(dtype);
    {
        std::lock_guard<std::mutex> g(ctx->cfg_mu);
        if (ctx->has_batch_cfg[dtype]) cfg = ctx->batch_cfg[dtype];
    }
    s = plan_build(pl, cfg, true);
    if (s == IQA_OK && (flags & IQA_PLAN_GRAPH)) s = plan_capture(pl);
    cudaSetDevice(prev);
    if (s != IQA_OK) {
        iqa_plan_destroy(pl);
        return s;
    }
    *out = pl;
    return IQA_OK;
}

iqa_status iqa_plan_launch(iqa_plan *plan, iqa_stream stream)
{
    if (!plan) return IQA_ERR_INVALID_ARG;
    cudaError_t e = plan->exec ? cudaGraphLaunch(plan->exec, (cudaStream_t)stream)
                               : plan_launch_direct(plan, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(plan->ctx, e, "plan launch");
    return IQA_OK;
}

void iqa_plan_destroy(iqa_plan *plan)
{
    if (!plan) return;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(plan->ctx->device);
    plan_drop_graph(plan);
    if (plan->d_table) cudaFree(plan->d_table);
    if (plan->d_sched) cudaFree(plan->d_sched);
    credit_memory(plan->ctx, plan->charged);
    cudaSetDevice(prev);
    if (plan->h_table)
        ::operator delete(plan->h_table, std::align_val_t(alignof(PairDesc)));
    delete plan;
}

iqa_status iqa_plan_info(const iqa_plan *plan, iqa_plan_stats *out)
{
    if (!plan || !out) return IQA_ERR_INVALID_ARG;
    out->npairs = (int)plan->pairs.size();
    out->total_units = plan->total_units;
    out->grid = plan->grid;
    out->input_bytes = plan->input_bytes;
    out->graph = plan->exec ? 1 : 0;
    out->config.variant = 1;
    out->config.threads = plan->cfg.threads;
    out->config.ilp = 0;
    out->config.tiles_across = 0;
    out->config.split = 1;
    out->config.vector = 1;
    out->config.stages = plan->cfg.stages;
    out->config.stage_kb = plan->cfg.stage_kb;
    out->config.ctas_per_sm = plan->cfg.ctas_per_sm;
    out->config.unit_kpx = plan->cfg.unit_kpx;
    return IQA_OK;
}

iqa_status iqa_plan_set_config(iqa_plan *plan, const iqa_launch_config *cfg)
{
    if (!plan) return IQA_ERR_INVALID_ARG;
    iqa_ctx *ctx = plan->ctx;
    if (!cfg || cfg->variant != 1 || cfg->unit_kpx < 1 || cfg->unit_kpx > 1024) {
        set_error(ctx, "a plan takes a variant 1 shape with unit_kpx in 1..1024");
        return IQA_ERR_INVALID_ARG;
    }
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ctx->device);
    const TileConfig keep = plan->cfg;
    const bool keep_shrink = plan->shrink;
    TileConfig c = keep;
    c.threads = cfg->threads;
    c.stages = cfg->stages;
    c.stage_kb = cfg->stage_kb;
    c.ctas_per_sm = cfg->ctas_per_sm;
    c.unit_kpx = cfg->unit_kpx;
    iqa_status s = plan_build(plan, c);
    if (s != IQA_OK) {
        // back to the previous shape, keeping the error message of this one;
        // if even that fails (a CUDA error), its status is returned and the
        // plan can only be destroyed
        std::string msg;
        {
            std::lock_guard<std::mutex> g(ctx->err_mu);
            msg = ctx->last_error;
        }
        const iqa_status r = plan_build(plan, keep, keep_shrink);
        if (r == IQA_OK) set_error(ctx, "%s", msg.c_str());
        else s = r;
    }
    if (s == IQA_OK && plan->exec) s = plan_capture(plan);
    cudaSetDevice(prev);
    return s;
}

iqa_status iqa_plan_unit_shape(iqa_dtype dtype, int N, int NT, const iqa_launch_config *cfg,
                               int *tiles_across, int *tile_rows, long long *units)
{
    if (!cfg || !tiles_across || !tile_rows || !units) {
        set_error(nullptr, "need cfg and the three outputs");
        return IQA_ERR_INVALID_ARG;
    }
    if (!dtype_ok(dtype)) {
        set_error(nullptr, "unknown dtype %d", (int)dtype);
        return IQA_ERR_INVALID_ARG;
    }
    if (check_shape(nullptr, N, NT) != IQA_OK) return IQA_ERR_INVALID_ARG;
    const int V = 16 / elem_size(dtype);
    if (NT % V || NT > 256) {
        set_error(nullptr, "the batched kernel needs NT a multiple of 16 bytes, at most 256 "
                           "(NT=%d)", NT);
        return IQA_ERR_INVALID_ARG;
    }
    if (cfg->variant != 1 || cfg->unit_kpx < 1 || cfg->unit_kpx > 1024) {
        set_error(nullptr, "a plan takes a variant 1 shape with unit_kpx in 1..1024");
        return IQA_ERR_INVALID_ARG;
    }
    TileConfig c = default_batch_config(dtype);
    c.threads = cfg->threads;
    c.stages = cfg->stages;
    c.stage_kb = cfg->stage_kb;
    c.ctas_per_sm = cfg->ctas_per_sm;
    c.unit_kpx = cfg->unit_kpx;
    stream_unit_shape(c, N, NT, dtype);
    std::string why;
    if (!stream_config_valid(N, NT, dtype, c, &why)) {
        set_error(nullptr, "N=%d NT=%d: %s", N, NT, why.c_str());
        return IQA_ERR_INVALID_ARG;
    }
    *tiles_across = c.TX;
    *tile_rows = c.RH;
    *units = pair_units(N, NT, c);
    return IQA_OK;
}

iqa_status iqa_plan_autotune(iqa_plan *plan, iqa_stream stream, int iters,
                             iqa_launch_config *best_out)
{
    if (!plan || iters < 1) return IQA_ERR_INVALID_ARG;
    iqa_ctx *ctx = plan->ctx;
    const TileConfig keep = plan->cfg;
    const bool keep_shrink = plan->shrink;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    TileConfig best = keep;
    const int threads_c[] = {128, 256};
    // {stages, stage_kb, ctas_per_sm, unit_kpx}
    const int shape_c[][4] = {{3, 16, 2, 16}, {2, 16, 2, 16}, {2, 16, 2, 4},
                              {3, 16, 2, 4},  {6, 8, 2, 4},   {4, 8, 3, 4},
                              {2, 16, 3, 4},  {4, 16, 1, 16}, {8, 8, 1, 4},
                              {3, 8, 4, 4},   {2, 8, 4, 4},   {2, 16, 3, 16},
                              {2, 16, 3, 32}, {3, 16, 2, 32}, {2, 16, 3, 64},
                              {4, 8, 3, 64},  {2, 16, 3, 128}};
    iqa_status s = IQA_OK;
    // time of `n` back-to-back launches of the plan built for c, after one
    // untimed launch; < 0 when the plan cannot take c (s is set on a CUDA error)
    const auto time_shape = [&](const TileConfig &c, int n) -> float {
        if (plan_build(plan, c) != IQA_OK) return -1.0f;
        cudaError_t e = plan_launch_direct(plan, (cudaStream_t)stream);  // warm-up
        if (e == cudaSuccess) e = cudaEventRecord(e0, (cudaStream_t)stream);
        for (int i = 0; i < n && e == cudaSuccess; ++i)
            e = plan_launch_direct(plan, (cudaStream_t)stream);
        if (e == cudaSuccess) e = cudaEventRecord(e1, (cudaStream_t)stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        if (e != cudaSuccess) {
            s = cuda_fail(ctx, e, "autotune launch");
            return -1.0f;
        }
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    // first pass: every shape, `iters` launches each
    std::vector<std::pair<float, TileConfig>> timed;
    for (int th : threads_c) {
        for (const auto &sh : shape_c) {
            TileConfig c = keep;
            c.threads = th;
            c.stages = sh[0];
            c.stage_kb = sh[1];
            c.ctas_per_sm = sh[2];
            c.unit_kpx = sh[3];
            const float ms = time_shape(c, iters);
            if (s != IQA_OK) break;
            if (ms >= 0.0f) timed.emplace_back(ms, c);
        }
        if (s != IQA_OK) break;
    }
    // second pass: the three fastest again, 3 * iters launches each, slowest
    // first, the fastest of them kept (shapes within a percent of each other
    // are ordered by more than one short sample)
    std::stable_sort(timed.begin(), timed.end(),
                     [](const std::pair<float, TileConfig> &a,
                        const std::pair<float, TileConfig> &b) { return a.first < b.first; });
    const int finalists = (int)std::min<size_t>(3, timed.size());
    float best_ms = 1e30f;
    for (int k = finalists - 1; k >= 0 && s == IQA_OK; --k) {
        const float ms = time_shape(timed[k].second, 3 * iters);
        if (ms >= 0.0f && ms < best_ms) {
            best_ms = ms;
            best = timed[k].second;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    iqa_status s2 = s == IQA_OK ? plan_build(plan, best) : plan_build(plan, keep, keep_shrink);
    if (s == IQA_OK) s = s2;
    if (s == IQA_OK && plan->exec) s = plan_capture(plan);
    if (s == IQA_OK) {
        std::lock_guard<std::mutex> g(ctx->cfg_mu);
        ctx->batch_cfg[plan->dtype] = plan->cfg;
        ctx->has_batch_cfg[plan->dtype] = true;
    }
    if (s == IQA_OK && best_out) {
        iqa_plan_stats st;
        iqa_plan_info(plan, &st);
        *best_out = st.config;
    }
    return s;
}

}  // extern "C"
