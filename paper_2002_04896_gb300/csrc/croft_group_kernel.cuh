// croft_group_kernel.cuh - one pass over the pencils of many grids that share
// the axis length N (the grouped schedule of batched plans).
//
// A batch of uneven grids has few distinct axis lengths.  The grouped schedule
// launches, for each pass and each length N, one kernel over the tiles of every
// grid whose axis of that pass has length N; the launches of one pass are
// independent and run concurrently (sibling nodes of a CUDA graph).  Each kernel
// is the single-grid pass kernel specialised on N (compile-time radix schedule
// and tile width) with a per-CTA lookup of its grid: CTA b works on tile
// b - first_tile of the last segment with first_tile <= b.  The segments lie in the kernel's
// parameters (constant bank; up to kGroupSegs of them, a pass with more grids of a length takes another launch)
// and are searched there: a few hundred cycles less before a CTA's first load than a map and a table in memory,
// two dependent loads - 9 % of the life of a CTA of a short pass.
#pragma once
#include "croft_fft_core.cuh"
#include "croft_internal.h"
#include "croft_two_stage_kernel.cuh"

namespace croft {

struct GroupSeg {
    const float2* in;   // pass input of this grid (the exec's `in` for the grid's first pass)
    float2* out;
    long long M;        // element stride of the axis (1 for a ROW pass)
    long long ncols;    // pencils of this grid along the axis
    CroftColDiv cdiv;   // COL: col / M as a multiply-high (croft_coldiv.h; m = 0: divide)
};

constexpr int kGroupSegs = 32;  // a power of two

struct GroupArgs {
    const float2* tw;               // twiddle table of N (two-stage: N entries; else N-1)
    int W;                          // ROW, not two-stage: pencils per CTA
    float isign;                    // +1 forward, -1 backward
    int first_tile[kGroupSegs];     // first CTA of each grid in the launch (INT_MAX past the last)
    GroupSeg seg[kGroupSegs];
};

// The segment of this CTA (binary search; the same in all threads).
__device__ __forceinline__ int group_seg(const GroupArgs& A) {
    int k = 0;
#pragma unroll
    for (int step = kGroupSegs / 2; step >= 1; step /= 2)
        if (A.first_tile[k + step] <= (int)blockIdx.x) k += step;
    return k;
}

// Batch row and column of pencil `col` of a COL segment.
__device__ __forceinline__ long long group_col_base(const GroupSeg& S, long long col, int n) {
    long long b, m;
    if (S.cdiv.m) {
        const unsigned q = croft_coldiv_q(S.cdiv.m, S.cdiv.s1, S.cdiv.s2, (unsigned)col);
        b = q;
        m = (unsigned)col - q * (unsigned)S.M;
    } else {
        b = col / S.M;
        m = col - b * S.M;
    }
    return b * (long long)n * S.M + m;
}

// The two-stage passes (croft_two_stage_kernel.cuh) of the lengths that have them: the same tiles
// and arithmetic as a single grid's passes.
template <int LAYOUT, int N>
constexpr CroftTwo group_two() { return croft_two_batch(N, LAYOUT == LAYOUT_ROW); }

template <int LAYOUT, int N>
__global__ void __launch_bounds__(group_two<LAYOUT, N>().w* group_two<LAYOUT, N>().t, group_two<LAYOUT, N>().minb)
    croft_group_two_kernel(const __grid_constant__ GroupArgs A) {
    constexpr CroftTwo K = group_two<LAYOUT, N>();
    using C = typename TwoComplex<K.packed != 0>::type;
    extern __shared__ __align__(16) float2 two_raw[];
    C* two_smem = reinterpret_cast<C*>(two_raw);
    C* buf = two_smem + (K.stage ? croft_two_pad(N) : 0);
    pdl_allow_dependents();
    const C* tw = two_twiddles<N, K.stage != 0>(A.tw, two_smem, K.w * K.t);
    const int k = group_seg(A);
    const GroupSeg& S = A.seg[k];
    const long long tile = (int)blockIdx.x - A.first_tile[k];
    pdl_wait();
    if constexpr (LAYOUT == LAYOUT_ROW) {
        const int c = threadIdx.x / K.t, lane = threadIdx.x % K.t;
        const long long col = tile * K.w + c;
        const long long base = col * N;
        two_pencil<N, K.r1, K.t>(GlobalInUnitT<C>{reinterpret_cast<const C*>(S.in) + base, A.isign},
                             GlobalOutUnitT<C>{reinterpret_cast<C*>(S.out) + base, A.isign},
                                 TwoExRow<K.r1, C>{buf + c * K.ld}, tw, lane, col < S.ncols);
    } else {
        const int c = threadIdx.x % K.w, lane = threadIdx.x / K.w;
        const long long col = tile * K.w + c;
        const long long base = group_col_base(S, col, N);
        two_pencil<N, K.r1, K.t>(GlobalInT<C>{reinterpret_cast<const C*>(S.in) + base, S.M, A.isign},
                             GlobalOutT<C>{reinterpret_cast<C*>(S.out) + base, S.M, A.isign},
                                 TwoExCol<K.r1, K.w, C>{buf + c}, tw, lane, col < S.ncols);
    }
}

// The other lengths (one stage, or no two-stage kernel).  ROW launches: W = 256 / T pencils per
// CTA; COL launches: the compile-time width croft_col_width(N).
template <int LAYOUT, int N>
__global__ void __launch_bounds__(256) croft_group_kernel(const __grid_constant__ GroupArgs A) {
    constexpr int T = croft_threads_per_pencil(N);
    constexpr int TW_PAD = ((N + 1) / 2) * 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* stw = reinterpret_cast<float2*>(smem_raw);
    float2* sbuf = stw + TW_PAD;
    pdl_allow_dependents();
    if (croft_make_sched(N).count > 1)
        for (int i = threadIdx.x; i < N - 1; i += blockDim.x) stw[i] = A.tw[i];
    const int k = group_seg(A);
    const GroupSeg& S = A.seg[k];
    const long long tile = (int)blockIdx.x - A.first_tile[k];
    pdl_wait();
    if constexpr (LAYOUT == LAYOUT_ROW) {
        const int c = threadIdx.x / T;
        const int lane = threadIdx.x - c * T;
        const long long col = tile * A.W + c;
        const bool ok = col < S.ncols;
        const long long base = col * N;
        fft_pencil_row<N, T>(GlobalInUnit{S.in + base, A.isign}, sbuf + c * croft_row_ld_staged(N),
                             GlobalOutUnit{S.out + base, A.isign}, stw, lane, ok);
    } else {
        constexpr int WC = croft_col_width(N, 8);
        const int c = threadIdx.x % WC;
        const int lane = threadIdx.x / WC;
        const long long col = tile * WC + c;
        const bool ok = col < S.ncols;
        const long long base = group_col_base(S, col, N);
        fft_pencil<N, T>(GlobalIn{S.in + base, S.M, A.isign}, SmemColFixed<float2, WC>{sbuf + c},
                         GlobalOut{S.out + base, S.M, A.isign}, stw, lane, ok);
    }
}

}  // namespace croft
