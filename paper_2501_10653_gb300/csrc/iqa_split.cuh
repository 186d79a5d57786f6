// iqa_split.cuh -- tiles so few and large that the CTAs of the one-pair kernel
// (at most kMaxCluster a tile) would leave most SMs without work: the same sums
// in the same order, bit for bit, spread over the whole GPU.
//
// What fixes the bits in iqa_tiles_kernel is, per thread of a unit, the order
// of the pixels inside a batch (ILP items added one after the other) and the
// compensated additions of the batches, one after the other; then the trees
// over the threads.  Only the compensated additions are a serial chain, so:
//   1. iqa_split_sums_kernel forms the batch sums, any batch of any thread on
//      any SM (all of the reading and arithmetic per pixel), and leaves them in
//      a scratch buffer: 16 bytes per batch, 1/16 of the bytes read for FP32
//      vectors, 1/4 for FP32 elements;
//   2. iqa_split_chain_kernel adds each thread's batches in order, one GPU
//      thread per thread and sum, and each warp's totals with the shuffle tree
//      of reduce_unit;
//   3. iqa_split_tile_kernel finishes each tile: the tree over a unit's warps,
//      the units of a tile in rank order, Eq. 1 and Eq. 2.
// The three launches overlap by programmatic dependent launch.  Bound by the
// first one's reads and, for small images, by the launches (about 8 us in all).
// Against the one-pair kernel's CTAs: N = N_T = 4096 FP32 30.0 us against 193,
// FP16 20.5 against 137; N = N_T = 8192 FP32 104 against 734; N = 4095, N_T = 1365
// FP32 (elements) 45 against 100.
#pragma once

#include "iqa_internal.h"

namespace iqa {

constexpr int kSplitIlp = 8;  // items of a batch: only units of this shape

struct SplitUnit {
    long long row0, col0;  // top-left pixel
};

__device__ __forceinline__ SplitUnit split_unit(const SplitArgs &p, int lc)
{
    // unit lc = tile * S + rank
    const int tile = lc / p.t.S, rank = lc - tile * p.t.S;
    const int r = tile / p.t.T, c = tile - r * p.t.T;
    return {(long long)r * p.t.NT + (long long)rank * p.t.RH, (long long)c * p.t.NT};
}

// Batches [PB * piece, PB * (piece + 1)) of kSplitThreads consecutive threads of
// unit blockIdx.y.
template <typename T, int VEC, bool DO_A, bool DO_B>
__global__ void __launch_bounds__(kSplitThreads) iqa_split_sums_kernel(const SplitArgs p)
{
    extern __shared__ __align__(16) unsigned char ring[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int slices = p.TH / kSplitThreads;
    const int piece = blockIdx.x / slices, slice = blockIdx.x - piece * slices;
    const int tid = slice * kSplitThreads + threadIdx.x;  // thread of the unit
    const int lc = blockIdx.y;
    const SplitUnit un = split_unit(p, lc);
    const long long N = p.t.N;
    const T *const xu = static_cast<const T *>(p.t.x) + un.row0 * N + un.col0;
    const T *const yu = static_cast<const T *>(p.t.y) + un.row0 * N + un.col0;
    const int items = p.t.RH * p.t.LPU;
    const int b0 = piece * p.PB;
    const int first = tid + b0 * kSplitIlp * p.TH;
    int n = min(items_from(first, p.TH, items), p.PB * kSplitIlp);
    // the unit lies inside the image (checked build only)
    if (!IQA_CHECK(un.row0 + p.t.RH <= N && un.col0 + (long long)p.t.LPU * VEC <= N &&
                   (n == 0 || b0 + (n - 1) / kSplitIlp < p.NB)))
        n = 0;
    float *out = p.parts + ((long long)lc * p.NB + b0) * 4 * p.TH + tid;
    const auto sink = [&](float a, float b, float x, float y) {
        if (DO_A) out[0] = a;
        if (DO_B) out[p.TH] = b;
        out[2 * p.TH] = x;
        out[3 * p.TH] = y;
        out += 4 * p.TH;
    };
    if constexpr (VEC > 1) {
        // (the policy: N = N_T = 4096 FP32 31.4 us without and 30.0 with, FP16 20.3 and
        // 20.7)
        sum_vectors_ring<T, VEC, kSplitIlp, kSplitThreads, kSplitDepth, DO_A, DO_B, VEC == 4>(
            xu, yu, N, p.t.LPU, first, p.TH, n, p.t.C1f,
            (uint32_t)__cvta_generic_to_shared(ring) + threadIdx.x * 16, sink);
    } else {
        // elements of any alignment, from registers
        const int W = p.t.LPU;
        int row = first / W, col = first - row * W;
        const int drow = p.TH / W, dcol = p.TH - drow * W;
        for (int j = 0; j < n; j += kSplitIlp) {
            Raw<T, 1> rx[kSplitIlp], ry[kSplitIlp];
#pragma unroll
            for (int u = 0; u < kSplitIlp; ++u) {
                if (j + u < n) {
                    const long long off = (long long)row * N + col;
                    rx[u] = load_raw<T, 1>(xu + off);
                    ry[u] = load_raw<T, 1>(yu + off);
                } else {
                    rx[u] = zero_raw<T, 1>();
                    ry[u] = zero_raw<T, 1>();
                }
                col += dcol;
                row += drow;
                if (col >= W) {
                    col -= W;
                    ++row;
                }
            }
            Sums2 q;
            q.zero();
#pragma unroll
            for (int u = 0; u < kSplitIlp; ++u)
                vector_terms<T, 1, DO_A, DO_B>(rx[u], ry[u], p.t.C1f, q);
            sink(q.a.x + q.a.y, q.b.x + q.b.y, q.x.x + q.x.y, q.y.x + q.y.y);
        }
    }
}

template <typename T, int VEC>
static cudaError_t launch_split_sums_v(const SplitArgs &p, int maps, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.pieces * (p.TH / kSplitThreads)),
                       (unsigned)(p.t.T * p.t.T * p.t.S), 1);
    cfg.blockDim = dim3(kSplitThreads, 1, 1);
    cfg.dynamicSmemBytes = VEC > 1 ? kSplitDepth * kSplitThreads * 32 : 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    switch (maps) {
    case MAPS_A: return cudaLaunchKernelEx(&cfg, iqa_split_sums_kernel<T, VEC, true, false>, p);
    case MAPS_B: return cudaLaunchKernelEx(&cfg, iqa_split_sums_kernel<T, VEC, false, true>, p);
    default: return cudaLaunchKernelEx(&cfg, iqa_split_sums_kernel<T, VEC, true, true>, p);
    }
}

template <typename T>
static cudaError_t launch_split_sums_t(const SplitArgs &p, int vec, int maps, cudaStream_t st)
{
    return vec == 1 ? launch_split_sums_v<T, 1>(p, maps, st)
                    : launch_split_sums_v<T, Elem<T>::VEC>(p, maps, st);
}

}  // namespace iqa
