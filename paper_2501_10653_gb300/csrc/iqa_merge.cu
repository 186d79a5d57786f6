// iqa_merge.cu -- Eq. 3 / Eq. 4 (arxiv 2501.10653, Section 3): the LISI and
// augLISI of larger tiles formed by merging m x m blocks of tiles, up to the
// whole image, rebuilt from the per-tile sums without re-reading any pixel.
//
// Eq. 3 multiplies each lisi_t by (max(Sx_t, Sy_t) + C2), which by Eq. 1 is
// D * A_t; Eq. 4 multiplies each auglisi_t by (Sx_t + Sy_t + C), which by Eq. 2
// is Sx_t + Sy_t + C - B_t, and removes the (n - 1) extra C.  Both therefore
// equal Eq. 1 / Eq. 2 applied to the block's summed (A, B, Sx, Sy); the kernels
// sum the four per-tile sums of each block in FP64, in an order fixed by the
// launch shape (so results repeat bit for bit), and apply Eq. 1 / Eq. 2 once.
//
// What bounds the kernels is the FP64 pipe (T = 512, m = 8: busy half of the
// cycles in which an SM works), then the 32 bytes read per tile: an FP64
// instruction holds an SM's pipe for about 16 cycles, whatever the number of its
// active lanes.  So sums are formed with full warps, and the two quotients of a
// merged tile in float32 with one FP64 residual each, to the same rounding
// (ratio()).  By block width m, measured back to back with all outputs, in us,
// against one thread (m <= 4), warp (m <= 90) or cluster per merged tile with
// 64-bit index divisions and FP64 quotients:
//   * m <= 4: a thread per merged tile, its tiles in 32-byte loads (T = 512: m =
//     1 9.4 against 17.7, m = 2 11.7 / 23.2, m = 4 6.9 / 11.3; without a stated
//     residency the compiler kept 32 registers and loads waited: m = 2 15.6);
//   * m <= kColsMax: a thread per tile column and kColsRows rows (consecutive
//     threads read consecutive tiles); the column sums meet in shared memory
//     (T = 512: m = 8 7.4 / 20.5, m = 16 10.5 / 25.4, m = 32 8.2 / 17.4; T =
//     1024: m = 8 14.3 / 54.8);
//   * larger blocks, up to the whole image: a cluster of kClusterCtas CTAs per
//     merged tile whose partial sums meet in distributed shared memory (T =
//     512: m = 64 11.9 / 54.4, m = 256 14.5 / 18.8; T = m = 1024 163 / 302).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "iqa.h"
#include "iqa_ctx.h"

namespace cg = cooperative_groups;

namespace iqa {

constexpr int kMergeThreads = 256;   // cluster kernel
constexpr int kClusterCtas = 8;
constexpr int kThreadThreads = 128;  // thread kernel
constexpr int kColsMax = 32;          // widest block of the column kernel
constexpr int kColsThreads = 512;     // most threads of its CTAs
constexpr int kColsRows = 4;          // most rows of its threads

struct MergeArgs {
    const double *sums;
    int T, m, M;  // tiles per row, merge factor, merged tiles per row
    int nb;       // column kernel: blocks across a CTA
    int RG;       // column kernel: row groups of a CTA (nb * m threads each)
    double C2, C, D;
    float *lisi;
    float *aug;
    double *out_sums;
};

// A tile's four sums: one 32-byte load where the table is 32-byte aligned
// (WIDE), else four of 8.  Volatile, so that a batch of them is issued before
// the first addition that needs one.
template <bool WIDE>
__device__ __forceinline__ void load_tile(double (&v)[4], const MergeArgs &a, int row, int col)
{
    const double *p = a.sums + 4 * ((long long)row * a.T + col);
    // the tile lies in the table (checked build only)
    if (!IQA_CHECK(row < a.T && col < a.T)) p = a.sums;
    if constexpr (WIDE) {
        asm volatile("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
                     : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                     : "l"(p));
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v[k]) : "l"(p + k));
    }
}

// The FP64 quotient n / d rounded to float32 in *q, from the quotient of the
// rounded operands and its FP64 residual n - q d (one step of iterative
// refinement).  The correction c is at most 1.5 2^-23 of q (two rounded operands
// and the division), itself off by at most 1.5 2^-22 of itself (rounded residual,
// rounded divisor, __fdividef's 2 ulp), so q + c lies within 2^-43 of n / d, and
// within that of its FP64 rounding.  Where q + c rounds the same over twice that
// range, it is the float32 that the FP64 quotient rounds to.  Otherwise (once
// in about 2^17 quotients), and where an operand or the quotient is outside the
// range in which float32 keeps its precision (zeros, infinities and NaN among
// them), the result is false and the caller forms the FP64 quotient.  Without the
// test of the range, quotients 2^-44 and less beside the middle of two floats
// rounded to the wrong one.
__device__ __forceinline__ bool ratio(double n, double d, float *q)
{
    const float fn = __double2float_rn(n), fd = __double2float_rn(d);
    const float q0 = __fdiv_rn(fn, fd);
    const float an = fabsf(fn), aq = fabsf(q0);
    if (!(an > 1e-30f && an < 1e30f && fd > 1e-30f && fd < 1e30f && aq > 1e-30f && aq < 1e30f))
        return false;
    const float c = __fdividef(__double2float_rn(__fma_rn(-(double)q0, d, n)), fd);
    const float e = aq * 0x1p-42f;
    *q = __fadd_rn(q0, __fadd_rn(c, -e));
    return *q == __fadd_rn(q0, __fadd_rn(c, e));
}

__device__ __forceinline__ void write_merged(const MergeArgs &a, long long b, const double (&t)[4])
{
    if (!IQA_CHECK(b < (long long)a.M * a.M)) return;
    const double A = t[0], B = t[1], Sx = t[2], Sy = t[3];
    float q;
    if (a.lisi) {
        const double n = a.D * A, d = fmax(Sx, Sy) + a.C2;
        a.lisi[b] = ratio(n, d, &q) ? q : (float)(n / d);
    }
    if (a.aug) {
        // 1 - B / d; where d is infinite and B is not, (d - B) / d would be NaN
        const double d = Sx + Sy + a.C;
        a.aug[b] = ratio(d - B, d, &q) ? q : (float)(1.0 - B / d);
    }
    if (a.out_sums) {
        double *o = a.out_sums + 4 * b;
        if (((uintptr_t)a.out_sums & 15u) == 0) {
            reinterpret_cast<double2 *>(o)[0] = make_double2(A, B);
            reinterpret_cast<double2 *>(o)[1] = make_double2(Sx, Sy);
        } else {
            o[0] = A;
            o[1] = B;
            o[2] = Sx;
            o[3] = Sy;
        }
    }
}

// Programmatic dependent launch: the next kernel in the stream may be
// scheduled as this grid drains, and this one waits for the previous grid
// (which wrote the per-tile sums) before its first read.
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Blocks of M_ <= 4 tiles across: a thread per merged tile, its M_ x M_ tiles
// loaded a row (one or two: all of them) at a time.
template <int M_, bool WIDE>
__global__ void __launch_bounds__(kThreadThreads, 8) iqa_merge_thread_kernel(const MergeArgs a)
{
    pdl_enter();
    const int b = blockIdx.x * kThreadThreads + threadIdx.x;
    if (b >= a.M * a.M) return;
    const int R = b / a.M, Cc = b - R * a.M;
    constexpr int ROWS = M_ <= 2 ? M_ : 1;  // rows in flight
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int r = 0; r < M_; r += ROWS) {
        double v[ROWS * M_][4];
#pragma unroll
        for (int i = 0; i < ROWS * M_; ++i)
            load_tile<WIDE>(v[i], a, R * M_ + r + i / M_, Cc * M_ + i % M_);
#pragma unroll
        for (int i = 0; i < ROWS * M_; ++i) {
#pragma unroll
            for (int k = 0; k < 4; ++k) s[k] = r + i == 0 ? v[i][k] : s[k] + v[i][k];
        }
    }
    write_merged(a, b, s);
}

// Blocks of 4 < m <= kColsMax: CTA (x, y) takes merged tiles [nb x, nb x + nb) of
// merged row y.  Thread (rg, c) sums tile column c of rows rg, rg + RG, ...;
// then a thread (or, from 16 columns on, a warp) per (merged tile, sum) adds
// the block's RG x m column sums in order, and thread i writes merged tile i.
template <bool WIDE>
__global__ void __launch_bounds__(kColsThreads, 1) iqa_merge_cols_kernel(const MergeArgs a)
{
    __shared__ double part[4][kColsThreads];
    __shared__ double total[4][kColsThreads];
    pdl_enter();
    const int tid = threadIdx.x, threads = blockDim.x;
    const int m = a.m;
    const int first = blockIdx.x * a.nb;
    const int blocks = min(a.nb, a.M - first);
    const int width = a.nb * m;
    const int rg = tid / width, c = tid - rg * width;
    const bool mine = rg < a.RG && c < blocks * m;
    const int row0 = blockIdx.y * m, col = first * m + c;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (mine) {
        double v[kColsRows][4];
        const int n = (m - rg + a.RG - 1) / a.RG;  // rows of this thread, <= kColsRows
#pragma unroll
        for (int i = 0; i < kColsRows; ++i)
            if (i < n) load_tile<WIDE>(v[i], a, row0 + rg + i * a.RG, col);
#pragma unroll
        for (int i = 0; i < kColsRows; ++i) {
            if (i < n) {
#pragma unroll
                for (int k = 0; k < 4; ++k) s[k] += v[i][k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) part[k][tid] = s[k];
    __syncthreads();
    const int tasks = 4 * blocks;
    if (m < 16) {
        for (int i = tid; i < tasks; i += threads) {
            const int k = i & 3, b = i >> 2;
            double t = 0.0;
            for (int g = 0; g < a.RG; ++g)
                for (int j = 0; j < m; ++j) t += part[k][g * width + b * m + j];
            total[k][b] = t;
        }
    } else {
        const int lane = tid & 31;
        for (int i = tid >> 5; i < tasks; i += threads >> 5) {
            const int k = i & 3, b = i >> 2;
            double t = 0.0;
            if (lane < m)
                for (int g = 0; g < a.RG; ++g) t += part[k][g * width + b * m + lane];
            t = warp_sum_d(t);
            if (lane == 0) total[k][b] = t;
        }
    }
    __syncthreads();
    if (tid < blocks) {
        const double t[4] = {total[0][tid], total[1][tid], total[2][tid], total[3][tid]};
        write_merged(a, (long long)blockIdx.y * a.M + first + tid, t);
    }
}

// Larger blocks: cluster b (kClusterCtas CTAs) takes merged tile b; CTA rank q
// sums its tiles i = q * kMergeThreads + tid + j * kClusterCtas *
// kMergeThreads in row-major order, reduces them in shared memory (four warps,
// one per sum), and rank 0 adds the ranks' partials in rank order through
// distributed shared memory.
template <bool WIDE>
__global__ void __launch_bounds__(kMergeThreads) iqa_merge_cluster_kernel(const MergeArgs a)
{
    __shared__ double red[4][kMergeThreads];
    __shared__ double part[4];
    pdl_enter();
    cg::cluster_group cluster = cg::this_cluster();
    const int q = (int)cluster.block_rank();
    const int b = blockIdx.x / kClusterCtas;
    const int R = b / a.M, Cc = b - R * a.M;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    // tile (r, c) of the block, stepped without divisions
    const int step = kClusterCtas * kMergeThreads;
    const int dr = step / a.m, dc = step - dr * a.m;
    int r = (q * kMergeThreads + tid) / a.m, c = q * kMergeThreads + tid - r * a.m;
    while (r < a.m) {
        double v[4][4];
        int n = 0;  // tiles of this batch
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (r < a.m) {
                load_tile<WIDE>(v[i], a, R * a.m + r, Cc * a.m + c);
                n = i + 1;
            }
            r += dr;
            c += dc;
            if (c >= a.m) {
                c -= a.m;
                ++r;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < n) {
#pragma unroll
                for (int k = 0; k < 4; ++k) s[k] += v[i][k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) red[k][tid] = s[k];
    __syncthreads();
    if (warp < 4) {
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < kMergeThreads; i += 32) t += red[warp][i + lane];
        t = warp_sum_d(t);
        if (lane == 0) part[warp] = t;
    }
    cluster.sync();
    if (q == 0 && tid == 0) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k = 0; k < kClusterCtas; ++k) {
            const double *rp = cluster.map_shared_rank(part, k);
#pragma unroll
            for (int j = 0; j < 4; ++j) t[j] += rp[j];
        }
        write_merged(a, b, t);
    }
    cluster.sync();  // keep every rank's shared memory alive until read
}

}  // namespace iqa

IQA_VIOLATION_READER(iqa_read_violations_merge)

using namespace iqa;

extern "C" iqa_status iqa_merge(iqa_ctx *ctx, const double *sums, int T, int m,
                                const iqa_params *params, float *merged_lisi,
                                float *merged_aug, double *merged_sums, iqa_stream stream)
{
    if (!ctx) return IQA_ERR_INVALID_ARG;
    if (!sums || (!merged_lisi && !merged_aug && !merged_sums)) {
        set_error(ctx, "need per-tile sums and at least one output");
        return IQA_ERR_INVALID_ARG;
    }
    if (T < 1 || m < 1 || m > T || T % m) {
        set_error(ctx, "need 1 <= m <= T with m dividing T (T=%d, m=%d)", T, m);
        return IQA_ERR_INVALID_ARG;
    }
    const long long M = T / m;
    if (M * M * kClusterCtas > 0x7fffffffLL) {
        set_error(ctx, "too many merged tiles");
        return IQA_ERR_UNSUPPORTED;
    }
    iqa_params P;
    iqa_status s = resolve_params(ctx, params, &P);
    if (s != IQA_OK) return s;
    MergeArgs a{sums, T, m, (int)M, 0, 0, P.C2, P.C, P.D, merged_lisi, merged_aug, merged_sums};
    const bool wide = ((uintptr_t)sums & 31u) == 0;
    cudaStream_t st = (cudaStream_t)stream;
    // every shape launches with programmatic stream serialization (see
    // pdl_enter); the cluster shape adds its cluster dimension
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    if (m <= 4) {
        cfg.blockDim = dim3(kThreadThreads);
        cfg.gridDim = dim3((unsigned)((M * M + kThreadThreads - 1) / kThreadThreads));
        const auto launch = [&](auto wide_kernel, auto kernel) {
            return wide ? cudaLaunchKernelEx(&cfg, wide_kernel, a)
                        : cudaLaunchKernelEx(&cfg, kernel, a);
        };
        switch (m) {
        case 1:
            e = launch(iqa_merge_thread_kernel<1, true>, iqa_merge_thread_kernel<1, false>);
            break;
        case 2:
            e = launch(iqa_merge_thread_kernel<2, true>, iqa_merge_thread_kernel<2, false>);
            break;
        case 3:
            e = launch(iqa_merge_thread_kernel<3, true>, iqa_merge_thread_kernel<3, false>);
            break;
        default:
            e = launch(iqa_merge_thread_kernel<4, true>, iqa_merge_thread_kernel<4, false>);
        }
    } else if (m <= kColsMax) {
        // kColsRows rows a thread; as many blocks across as 128 columns
        // hold, fewer while that leaves SMs without a CTA
        a.RG = (m + kColsRows - 1) / kColsRows;
        a.nb = std::max(1, std::min(128 / m, kColsThreads / (a.RG * m)));
        const long long sms = ctx->num_sms > 0 ? ctx->num_sms : 152;
        while (a.nb > 1 && (M + a.nb - 1) / a.nb * M < 2 * sms && a.nb * m > 32) a.nb /= 2;
        cfg.blockDim = dim3((unsigned)((a.RG * a.nb * m + 31) / 32 * 32));
        cfg.gridDim = dim3((unsigned)((M + a.nb - 1) / a.nb), (unsigned)M);
        e = wide ? cudaLaunchKernelEx(&cfg, iqa_merge_cols_kernel<true>, a)
                 : cudaLaunchKernelEx(&cfg, iqa_merge_cols_kernel<false>, a);
    } else {
        cfg.blockDim = dim3(kMergeThreads);
        cfg.gridDim = dim3((unsigned)(M * M * kClusterCtas));
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = kClusterCtas;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
        e = wide ? cudaLaunchKernelEx(&cfg, iqa_merge_cluster_kernel<true>, a)
                 : cudaLaunchKernelEx(&cfg, iqa_merge_cluster_kernel<false>, a);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "merge kernel launch");
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(ctx, e, "merge kernel launch");
    return IQA_OK;
}
