// iqa_tiles.cuh -- the plain-path kernel: one launch computes the LISI (Eq. 1)
// and/or augLISI (Eq. 2) map of one image pair, reading every pixel once.
//
// Grid: x = unit column (TX whole tiles each), y = tile row * S + part, where a
// tile taller than one unit is split over S CTAs that form a thread-block
// cluster along y; the S partial sums meet in distributed shared memory and
// the cluster's rank-0 CTA writes the tile.  Launched with programmatic
// dependent launch: every CTA waits for the previous grid in the stream before
// its first access (the first ones of a launch may bring their pixels to L2
// before that, and independent calls wait only before they write: Order).
// Included once per storage type.
#pragma once

#include <cooperative_groups.h>

#include <atomic>

#include "iqa_internal.h"

namespace iqa {

namespace cg = cooperative_groups;

// Reduces the CTA's sums and writes its tiles; with S > 1 the CTAs of the
// tile form one cluster, whose rank 0 combines and writes.
template <int THREADS, bool OVERLAP>
__device__ __forceinline__ void finish_unit(const TileArgs &p, const float (&acc)[4],
                                            int tile_row, int tile_col0,
                                            float (*red)[THREADS], float *part)
{
    reduce_unit<THREADS>(acc, p.TX, p.LPU, p.LPT, red, part, CtaBarrier());
    if constexpr (OVERLAP) asm volatile("griddepcontrol.wait;" ::: "memory");

    const long long t0 = (long long)tile_row * p.T + tile_col0;
    const bool out_ok = IQA_CHECK(t0 + p.TX <= (long long)p.T * p.T && p.TX <= kMaxTX);
    if (p.S == 1) {
        for (int tl = threadIdx.x; tl < p.TX && out_ok; tl += THREADS)
            write_tile(p, t0 + tl, part[tl * 4 + 0], part[tl * 4 + 1],
                       part[tl * 4 + 2], part[tl * 4 + 3]);
        return;
    }
    // S > 1: the CTAs of this tile form one cluster; combine in rank order.
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (cluster.block_rank() == 0 && out_ok) {
        for (int tl = threadIdx.x; tl < p.TX; tl += THREADS) {
            float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            for (int r = 0; r < p.S; ++r) {
                const float *rp = cluster.map_shared_rank(part, r);
#pragma unroll
                for (int k = 0; k < 4; ++k) s[k] += rp[tl * 4 + k];
            }
            write_tile(p, t0 + tl, s[0], s[1], s[2], s[3]);
        }
    }
    // keep every CTA's shared memory alive until rank 0 has read it
    cluster.sync();
}

// Whether a launch of vector units streams its pixels through a ring in shared
// memory (accumulate_unit_ring) or in batches of loads to registers
// (accumulate_unit); both sum in the same order, bit for bit.  Measured back to
// back, registers against ring, in us:
//   * 16-bit storage, eight or more vectors a thread (ILP 8): ring.  N = 4096,
//     N_T = 16 / 64 / 128 / 256: 17.9 / 18.0 / 17.8 / 27.8 against 14.7 / 15.0
//     / 14.5 / 14.2; N = 8192: 48.9 / 60.9 / 61.1 / 57.7 against 44.8 / 44.2 /
//     44.3 / 47.7.  With fewer vectors the ring's set-up is not repaid (N =
//     512, N_T = 16: 3.4 against 4.4).
//   * FP32, whose eight-vector batches the compiler keeps in flight: ring from
//     kRingUnits units on, where every SM has several CTAs to run one after the
//     other (N = 8192, N_T = 16 / 64 / 256: 83.6 / 79.3 / 87.5 against 77.0 /
//     75.7 / 77.7; N = 4096, N_T = 16: 25.1 / 22.7); with fewer, registers (N =
//     4096, N_T = 64: 22.2 against 22.8; N = 2048: 8.1 against 9.1).
constexpr long long kRingUnits = 2048;

// A unit of 2^31 vectors and more, whose items the ring counts in 32 bits (one
// CTA for a 16-bit tile of 131072 pixels a side), takes registers, which walk
// rows and columns: counted in 64 bits the 16-bit ring compiled to 84 registers
// in place of 102, and N = 8192, N_T = 64 / 128 took 47.2 us in place of 44.0.
template <int VEC> inline bool use_ring(const TileArgs &p, int ilp, int rows)
{
    if (VEC == 1 || ilp != 8 || (long long)p.RH * p.LPU > 0x7fffffffLL - 512) return false;
    return VEC == 8 || (long long)(p.T / p.TX) * rows * p.S >= kRingUnits;
}

// Ring entries: 32 KB of shared memory for 128 threads (six CTAs, 192 KB in
// flight on an SM), 64 KB for wider CTAs, which come alone or in twos or
// threes.  Sixteen entries measured slower (N = 8192, N_T = 16 FP16: 53.7
// against 43.3), four 1-2% slower.
__host__ __device__ constexpr int ring_depth(int threads) { return threads == 512 ? 4 : 8; }

// Whether the ring's copies carry a policy for L2 (l2_policy): FP32, and 16 bits
// with six CTAs.  The 16-bit build for four then takes 118 registers in
// place of 102 and is 1-2% slower back to back (N = 8192, N_T = 128 FP16 43.8 and
// 44.3), though faster on images just made (71.6 and 68.6).
template <int VEC, int CTAS> constexpr bool kL2Hint = VEC == 4 || CTAS == 6;

// Resident CTAs to compile for.  Left to itself the compiler aims at a residency
// of its own and sinks loads between their arithmetic for it; stated, it keeps a
// batch in flight.  Measured back to back, in us:
//   * FP32 batches of eight in registers: five CTAs of 128 threads (96
//     registers), with which the one-wave rule of the launch shapes counts.
//     Four (114 registers) gain where a launch still fits one wave (N = 2048, N_T
//     = 64 8.8 and 8.1) and lose a wave where it does not (N = 4608, N_T = 64 27.5
//     and 34.2);
//   * shorter batches: as many CTAs as hold their registers without spills;
//     fewer leave small units waiting (N = 3936, N_T = 16 BF16 60.7 and 69.8).
//     16-bit batches of two keep more in flight with fewer, so launches whose
//     units all fit at once take eight or nine (by_maps: inputs not in L2, ten /
//     nine / eight: N = 1536, N_T = 32 FP16, 1152 units 5.9 / 5.6 / 5.1, N = 1440,
//     N_T = 48, 900 units 5.3 / 5.2 / 4.6, N = 1664, N_T = 32, 1352 units 6.0 / 5.7 /
//     6.2; N = 3232, N_T = 32, 10201 units 17.3 / 18.0 / 18.8);
//   * element order, four (56): N = 8001, N_T = 63 BF16 136 without and 92 with;
//     N = 3000, N_T = 75 FP32 19.4 and 15.3 (two or three: the same; five: 16.7);
//   * 16-bit ring, one (102, so four CTAs of 128 threads): N = 2048, N_T = 128 7.2
//     without and 5.6 with; N = 8192, N_T = 64 49.0 and 44.2.  That suits long units.
//     With few vectors a thread a CTA's start and end weigh more, and six (72
//     registers, as many as the shared memory lets in) cover them: from six units
//     per SM on, with fewer than 16 vectors always (four and six: N = 3456, N_T =
//     64 BF16 12.4 and 10.9, N = 5504 26.8 and 22.6; with five per SM N = 2400, N_T =
//     96 7.2 and 8.1), with fewer than 32 but for seven to nine per SM, which make
//     a second, nearly empty wave of six (N = 3840, N_T = 64 BF16, six 12.9 and
//     10.7; N = 4864, ten 20.2 and 17.3; but N = 4096, N_T = 128 FP16, seven 12.8 and
//     13.2).  A CTA of 512 threads has an SM to itself; two (64 registers) where
//     that leaves a second wave (N = 4368, N_T = 728 FP16 24.7 and 17.1; N = 4800,
//     N_T = 800 BF16 27.3 and 19.4);
//   * FP32 ring, as many as its shared memory lets in: N = 8192, N_T = 64 / 256 76.9
//     / 79.2 without and 75.8 / 77.2 with (one CTA: 78.2 / 85.6).
template <int VEC, int ILP, bool STREAMED> constexpr int min_ctas(int threads)
{
    if (VEC == 1) return 4;
    if (ILP == 2) return threads == 128 ? 10 : threads == 256 ? 5 : 2;
    if (ILP == 4) return threads == 128 ? 8 : threads == 256 ? 4 : 2;
    if (!STREAMED) return threads == 128 ? 5 : threads == 256 ? 2 : 1;
    if (VEC == 8) return 1;
    return threads == 128 ? 6 : threads == 256 ? 3 : 2;
}

// How a launch stands to the kernel before it in the stream.
enum Order {
    ORDER_WAIT,      // every access after it
    ORDER_PREFETCH,  // the same, with the first CTAs' units brought to L2 before
    ORDER_OVERLAP    // an independent call: only writes after it
};

template <typename T, int VEC, int ILP, int THREADS, bool DO_A, bool DO_B, int ORDER,
          bool STREAMED, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS)
    iqa_tiles_kernel(const TileArgs p)
{
    extern __shared__ __align__(16) unsigned char ring[];
    __shared__ float red[4][THREADS];
    __shared__ float part[kMaxTX * 4];

    // programmatic dependent launch: let the next kernel in the stream be
    // scheduled as this grid drains, and wait for the previous one (which may
    // have written these images or maps) before the first access -- or, for
    // an independent call, only before the first write, so the loads stream
    // while that kernel drains
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (ORDER == ORDER_WAIT) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int tile_col0 = blockIdx.x * p.TX;
    // (small element-order units notice the two divisions, vector units do not)
    const int tile_row_s = VEC == 1 && p.S == 1 ? blockIdx.y : blockIdx.y / p.S;
    const int srank = VEC == 1 && p.S == 1 ? 0 : blockIdx.y % p.S;
    const int tile_row = p.tile_row0 + tile_row_s;
    const long long row0 = (long long)tile_row * p.NT + (long long)srank * p.RH;
    const long long col0 = (long long)tile_col0 * p.NT;
    const T *xu = static_cast<const T *>(p.x) + row0 * p.N + col0;
    const T *yu = static_cast<const T *>(p.y) + row0 * p.N + col0;

    if constexpr (ORDER == ORDER_PREFETCH) {
        if ((int)(blockIdx.y * gridDim.x + blockIdx.x) < p.prefetch_ctas &&
            IQA_CHECK(tile_row < p.T && row0 + p.RH <= p.N &&
                      col0 + (long long)p.TX * p.NT <= p.N)) {
            for (long long r = threadIdx.x; r < p.RH; r += THREADS) {
                prefetch_l2(xu + r * p.N, (unsigned)(p.LPU * VEC * (int)sizeof(T)));
                prefetch_l2(yu + r * p.N, (unsigned)(p.LPU * VEC * (int)sizeof(T)));
            }
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }

    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    // the unit lies inside the image (checked build only)
    if (IQA_CHECK(tile_row < p.T && row0 + p.RH <= p.N &&
                  col0 + (long long)p.TX * p.NT <= p.N && p.LPU * VEC == p.TX * p.NT))
    {
        if constexpr (VEC > 1 && STREAMED)
            accumulate_unit_ring<T, VEC, ILP, THREADS, ring_depth(THREADS), DO_A, DO_B,
                                 kL2Hint<VEC, CTAS>>(
                xu, yu, p.N, p.RH, p.LPU, p.C1f,
                (uint32_t)__cvta_generic_to_shared(ring) + threadIdx.x * 16, acc);
        else if constexpr (STREAMED)
            accumulate_elements<T, ILP, THREADS, DO_A, DO_B>(xu, yu, (int)p.N, p.RH, p.LPU,
                                                             p.drow, p.dcol, p.inv_lpu, p.C1f,
                                                             acc);
        else
            accumulate_unit<T, VEC, ILP, THREADS, DO_A, DO_B>(
                xu, yu, p.N, p.RH, p.LPU, p.drow, p.dcol, p.inv_lpu, p.C1f, acc);
    }
    finish_unit<THREADS, ORDER == ORDER_OVERLAP>(p, acc, tile_row, tile_col0, red, part);
}

// Launches `kern` over the units of rows x T / TX tiles, the S CTAs of a tile
// as a cluster; `raised` holds the devices on which its dynamic shared memory
// limit was raised to kMaxRing.
constexpr int kMaxRing = 160 * 1024;

template <typename Kernel>
static cudaError_t launch_units(Kernel kern, std::atomic<unsigned long long> &raised,
                                const TileArgs &p, int rows, int threads, size_t smem,
                                cudaStream_t st)
{
    if (smem > 32768) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
        if (!(raised.load(std::memory_order_acquire) & bit)) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxRing);
            if (e != cudaSuccess) return e;
            raised.fetch_or(bit, std::memory_order_release);
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.T / p.TX), (unsigned)(rows * p.S), 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.S > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 1;
        attr[1].val.clusterDim.y = (unsigned)p.S;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kern, p);
}

// Element-order launches of up to three units per SM are spread: they ask for as
// much dynamic shared memory as lets an SM's 228 KB hold `ctas` CTAs, their even
// share, beside the static part and the 1 KB that each is charged.  A launch
// whose CTAs are placed while the kernel before it drains otherwise fills
// whichever SMs have room, with up to four CTAs on one and none on others, and
// lasts as long as the fullest.  Back to back, in us, placed freely and spread: 81
// units N = 1287, N_T = 143 FP32 11.8 and 6.1, N = 1089, N_T = 121 FP16 9.7 and 4.8;
// 324 units N = 2250, N_T = 125 FP32 12.8 and 10.1; 400 units N = 1800, N_T = 90 BF16
// 6.9 and 5.7; but 36 units N = 858, N_T = 143 FP16 7.7 and 8.2, which leave room
// for two launches side by side.  Isolated launches are spread anyway.  (An SM
// whose last kernel had another split of L1 and shared memory is reconfigured:
// after each of a caller's own elementwise kernels the 81 units take 0.7 us more.)
constexpr int kSpreadMost = 3;

constexpr int spread_smem(int threads, int ctas)
{
    return 228 * 1024 / (ctas + 1) - (4 * threads + 4 * kMaxTX) * (int)sizeof(float);
}

// An independent call (p.overlap) runs the ORDER_OVERLAP instantiation, which
// only the 16-byte vector paths have.
template <typename T, int VEC, int ILP, int THREADS, bool DO_A, bool DO_B, int ORDER,
          bool STREAMED, int CTAS>
static cudaError_t launch_one(const TileArgs &p, int rows, cudaStream_t st)
{
    static std::atomic<unsigned long long> raised{0};
    int smem = VEC > 1 && STREAMED ? ring_depth(THREADS) * THREADS * 32 : 0;
    if (VEC == 1 && p.per_sm >= 1 && p.per_sm <= kSpreadMost)
        smem = spread_smem(THREADS, p.per_sm);
    return launch_units(
        iqa_tiles_kernel<T, VEC, ILP, THREADS, DO_A, DO_B, ORDER, STREAMED, CTAS>, raised, p, rows,
        THREADS, smem, st);
}

template <typename T, int VEC, int ILP, int THREADS, int ORDER, bool STREAMED,
          int CTAS = min_ctas<VEC, ILP, STREAMED>(THREADS)>
static cudaError_t by_maps_o(const TileArgs &p, int maps, int rows, cudaStream_t st)
{
    switch (maps) {
    case MAPS_A:
        return launch_one<T, VEC, ILP, THREADS, true, false, ORDER, STREAMED, CTAS>(p, rows, st);
    case MAPS_B:
        return launch_one<T, VEC, ILP, THREADS, false, true, ORDER, STREAMED, CTAS>(p, rows, st);
    default:
        return launch_one<T, VEC, ILP, THREADS, true, true, ORDER, STREAMED, CTAS>(p, rows, st);
    }
}

template <typename T, int VEC, int ILP, int THREADS, bool STREAMED,
          int CTAS = min_ctas<VEC, ILP, STREAMED>(THREADS)>
static cudaError_t by_order(const TileArgs &p, int maps, int rows, cudaStream_t st)
{
    if (VEC > 1 && p.overlap)
        return by_maps_o<T, VEC, ILP, THREADS, (VEC > 1 ? ORDER_OVERLAP : ORDER_WAIT), STREAMED,
                         CTAS>(p, maps, rows, st);
    // (16-bit batches of two never prefetch)
    if constexpr (VEC != 8 || ILP != 2) {
        if (p.prefetch_ctas > 0)
            return by_maps_o<T, VEC, ILP, THREADS, ORDER_PREFETCH, STREAMED, CTAS>(p, maps, rows,
                                                                                  st);
    }
    return by_maps_o<T, VEC, ILP, THREADS, ORDER_WAIT, STREAMED, CTAS>(p, maps, rows, st);
}

template <typename T, int VEC, int ILP, int THREADS>
static cudaError_t by_maps(const TileArgs &p, int maps, int rows, cudaStream_t st)
{
    if constexpr (VEC > 1 && ILP == 8) {
        if (use_ring<VEC>(p, ILP, rows)) {
            if constexpr (VEC == 8 && THREADS == 128) {
                const int vectors = p.RH * p.LPU / THREADS;  // a thread's
                const bool waves = p.per_sm == 6 || p.per_sm > 9;
                if (p.S == 1 && p.per_sm > 5 && (vectors < 16 || (vectors < 32 && waves)))
                    return by_order<T, VEC, ILP, THREADS, true, 6>(p, maps, rows, st);
            }
            if constexpr (VEC == 8 && THREADS == 512) {
                if (p.per_sm > 1) return by_order<T, VEC, ILP, THREADS, true, 2>(p, maps, rows, st);
            }
            return by_order<T, VEC, ILP, THREADS, true>(p, maps, rows, st);
        }
    }
    if constexpr (VEC == 8 && ILP == 2 && THREADS == 128) {
        if (p.per_sm <= 8) return by_order<T, VEC, ILP, THREADS, false, 8>(p, maps, rows, st);
        if (p.per_sm == 9) return by_order<T, VEC, ILP, THREADS, false, 9>(p, maps, rows, st);
    }
    if constexpr (VEC == 1) {
        // 32-bit offsets wherever a unit's fit
        if ((long long)(p.RH + THREADS) * p.N < 0x7fffffffLL)
            return by_order<T, VEC, ILP, THREADS, true>(p, maps, rows, st);
    }
    // (16-bit: units of 2^31 vectors only, a long serial work of one CTA, for
    // which the instantiation that waits for the kernel before it is enough)
    if constexpr (VEC == 8 && ILP == 8)
        return by_maps_o<T, VEC, ILP, THREADS, ORDER_WAIT, false>(p, maps, rows, st);
    else return by_order<T, VEC, ILP, THREADS, false>(p, maps, rows, st);
}

template <typename T, int VEC, int ILP>
static cudaError_t by_threads(const TileArgs &p, const TileConfig &c, int maps,
                              int rows, cudaStream_t st)
{
    switch (c.threads) {
    case 128: return by_maps<T, VEC, ILP, 128>(p, maps, rows, st);
    case 256: return by_maps<T, VEC, ILP, 256>(p, maps, rows, st);
    case 512: return by_maps<T, VEC, ILP, 512>(p, maps, rows, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
static cudaError_t launch_tiles_t(const TileArgs &p, const TileConfig &c,
                                  int maps, int rows, cudaStream_t st)
{
    constexpr int V = Elem<T>::VEC;
    if (c.vec == 1) {
        // scalar path for unaligned images or tiles that are not a whole
        // number of 16-byte vectors wide: one launch shape only
        if (c.threads != 256 || c.ilp != 8) return cudaErrorInvalidValue;
        return by_maps<T, 1, 8, 256>(p, maps, rows, st);
    }
    if (c.vec != V) return cudaErrorInvalidValue;
    switch (c.ilp) {
    case 2: return by_threads<T, V, 2>(p, c, maps, rows, st);
    case 4: return by_threads<T, V, 4>(p, c, maps, rows, st);
    case 8: return by_threads<T, V, 8>(p, c, maps, rows, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace iqa
