// croft_two_stage_kernel.cuh - a pass whose 1D transforms take two stages, N = R1 * R2 with
// radices of up to 32 points, and one exchange through shared memory between them.
//
// Paper mapping: the batched 1D FFTs of Sec. 4.1 (steps 1, 5, 9) with the rearrangement fused
// into the gather, as croft_pass_kernel.cuh; one Cooley-Tukey step per pencil:
//   stage 1: butterfly b < R2 reads x[b + j*R2] (j < R1) from HBM, radix-R1 DFT, stores
//            element b*R1 + j of the exchange buffer;
//   stage 2: butterfly k < R1 reads elements k + j*R1 (j < R2), multiplies by w_N^{jk}, radix-R2
//            DFT, writes y[k + j*R1] to HBM.
//
// What bounds it: HBM for most lengths (6.7-7.1 TB/s of 6.8 measured by a plain copy on row and
// short-stride column passes), the latency of one load - compute - store round per CTA for the
// 300..1024-point column passes (5.6-6.9 TB/s).  Why two large radices: with radices of at most
// 16 these lengths take three stages, that is two exchanges and two barriers, and the passes
// stood at 3.9-6.2 TB/s on the shared-memory queue and the barriers while a strided copy with
// the same tiles moves 6.6 TB/s and more; 16 to 32 points per thread in registers replace one of
// the exchanges.  Lengths, radices, tiles and launch bounds: croft_two_stage.h, with the
// throughput of both kinds of pass beside each.
//
// Twiddles w_N^{jk}, j < R2, k < R1 at tw[j*R1 + k] (N entries): staged in shared memory at
// entry, or read through L1 where that measured faster (512-point column pass, 2 MB strides:
// 366 -> 338 us per 2.1 GB; the staging load precedes every load of the tile).
#pragma once
#include "croft_fft_core.cuh"
#include "croft_internal.h"
#include "croft_two_stage.h"

namespace croft {

// Radix-R DFTs of this thread's butterflies lane, lane + T, ... < NB after their twiddles (tw:
// row j, column the butterfly's index, PITCH entries per row; null for the first stage).
template <int R, int NB, int T, int PITCH, bool TWIDDLE, int Q, class C>
__device__ __forceinline__ void two_butterflies(C (&v)[Q][R], const C* tw, int lane) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int b = lane + q * T;
        if (NB % T == 0 || b < NB) {
            if constexpr (TWIDDLE) {
#pragma unroll
                for (int j = 1; j < R; ++j) v[q][j] = cmul(v[q][j], tw[j * PITCH + b]);
            }
            dft<R>(v[q]);
        }
    }
}

// One pencil: T threads (this one is `lane`), in and out with element strides as Src / Dst have
// them, the exchange buffer through Ex (Ex::at(b, j): the slot of element b*R1 + j).
template <int N, int R1, int T, class Src, class Dst, class Ex>
__device__ __forceinline__ void two_pencil(const Src& src, const Dst& dst, const Ex& ex,
                                           const typename Src::value_type* tw, int lane, bool ok) {
    using C = typename Src::value_type;
    constexpr int R2 = N / R1;
    static_assert(R1 * R2 == N, "two stages");
    constexpr int Q1 = (R2 + T - 1) / T, Q2 = (R1 + T - 1) / T;
    {
        C v[Q1][R1];
#pragma unroll
        for (int q = 0; q < Q1; ++q) {
            const int b = lane + q * T;
            if (ok && (R2 % T == 0 || b < R2)) {
#pragma unroll
                for (int j = 0; j < R1; ++j) v[q][j] = src.load(b + j * R2);
            }
        }
        two_butterflies<R1, R2, T, 1, false>(v, tw, lane);
#pragma unroll
        for (int q = 0; q < Q1; ++q) {
            const int b = lane + q * T;
            if (R2 % T == 0 || b < R2) {
#pragma unroll
                for (int j = 0; j < R1; ++j) *ex.at(b, j) = v[q][j];
            }
        }
    }
    __syncthreads();
    {
        C v[Q2][R2];
#pragma unroll
        for (int q = 0; q < Q2; ++q) {
            const int k = lane + q * T;
            if (R1 % T == 0 || k < R1) {
#pragma unroll
                for (int j = 0; j < R2; ++j) v[q][j] = *ex.at(j, k);
            }
        }
        two_butterflies<R2, R1, T, R1, true>(v, tw, lane);
#pragma unroll
        for (int q = 0; q < Q2; ++q) {
            const int k = lane + q * T;
            if (ok && (R1 % T == 0 || k < R1)) {
#pragma unroll
                for (int j = 0; j < R2; ++j) dst.store(k + j * R1, v[q][j]);
            }
        }
    }
}

// Exchange buffers.  Columns: [N][W], element b*R1 + j of column c.
template <int R1, int W, class C>
struct TwoExCol {
    C* s;  // tile + c
    __device__ __forceinline__ C* at(int b, int j) const { return s + (b * R1 + j) * W; }
};
template <int R1, class C>
struct TwoExColW {  // (width known at run time)
    C* s;
    int W;
    __device__ __forceinline__ C* at(int b, int j) const { return s + (b * R1 + j) * W; }
};
// Rows: element b*R1 + j of a pencil at b*(R1 + D) + j.  An odd distance R1 + D between the
// runs that neighbouring butterflies write keeps the writes free of bank conflicts.
template <int R1, class C>
struct TwoExRow {
    static constexpr int D = R1 % 2 == 0 ? 1 : 0;
    C* s;  // start of the pencil
    __device__ __forceinline__ C* at(int b, int j) const { return s + b * (R1 + D) + j; }
};

// The complex type of a kernel's arithmetic (packed2: paired sums).
template <bool PACKED> struct TwoComplex { using type = float2; };
template <> struct TwoComplex<true> { using type = packed2; };

// Twiddles: staged (copied to `stw`, which the barrier between the stages publishes) or as they are.
template <int N, bool STAGE, class C>
__device__ __forceinline__ const C* two_twiddles(const float2* twg, C* stw, int threads) {
    const C* tw = reinterpret_cast<const C*>(twg);
    if constexpr (STAGE) {
        for (int i = threadIdx.x; i < N; i += threads) stw[i] = tw[i];
        return stw;
    } else {
        return tw;
    }
}

// The column pass of long axes: one tile of W columns shared by a cluster of two CTAs.  CTA r takes the stage-1
// butterflies b of its half and the stage-2 butterflies k of its half; element (b, k) goes straight into the shared
// memory of the CTA that needs it (half of the stores through distributed shared memory), [b][k - its first k][column].
// Barriers: the first (arrived at entry) tells that the partner runs before anything is stored into its
// memory; the second publishes the stores.  No CTA touches its partner's memory after that, so either may
// leave, and both have read their rows of the tile before either writes (in place).
// What bounds it: the latency of a round at three or four CTAs of about 250 threads per SM, 5.0-5.5 TB/s across megabytes
// (the 16-column tile in one CTA of its own per SM: 4.4-4.9).
template <int N, bool LONG>
__global__ void __cluster_dims__(2, 1, 1)
    __launch_bounds__(croft_two_col(N, LONG).w* croft_two_col(N, LONG).t, croft_two_col(N, LONG).minb)
    croft_two_pair_kernel(const float2* in, float2* out, const __grid_constant__ PassArgs A) {
    constexpr CroftTwo K = croft_two_col(N, LONG);
    constexpr int R1 = K.r1, R2 = N / R1, T = K.t, W = K.w;
    constexpr int H1 = (R2 + 1) / 2, H2 = (R1 + 1) / 2;  // butterflies of CTA 0 in the two stages
    constexpr int Q1 = (H1 + T - 1) / T, Q2 = (H2 + T - 1) / T;
    namespace cg = cooperative_groups;
    using C = typename TwoComplex<K.packed != 0>::type;
    extern __shared__ __align__(16) float2 two_raw[];
    C* two_smem = reinterpret_cast<C*>(two_raw);
    const cg::cluster_group cluster = cg::this_cluster();
    const int r = (int)cluster.block_rank();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    pdl_allow_dependents();
    pdl_wait();
    const int c = threadIdx.x % W, lane = threadIdx.x / W;
    const long long col = (long long)col_tile(A, blockIdx.x / 2, gridDim.x / 2) * W + c;
    const bool ok = col < A.ncols;
    long long b_, m_;
    col_split(col, A, b_, m_);
    const long long base = b_ * (long long)N * A.M + m_;
    {
        const GlobalInT<C> src{reinterpret_cast<const C*>(in) + base, A.M, A.isign};
        C v[Q1][R1];
#pragma unroll
        for (int q = 0; q < Q1; ++q) {
            const int lb = lane + q * T, b = r * H1 + lb;
            if (ok && lb < H1 && b < R2) {
#pragma unroll
                for (int j = 0; j < R1; ++j) v[q][j] = src.load(b + j * R2);
            }
        }
#pragma unroll
        for (int q = 0; q < Q1; ++q) dft<R1>(v[q]);
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        C* first = (r == 0 ? two_smem : cluster.map_shared_rank(two_smem, 0)) + c;
        C* second = (r == 1 ? two_smem : cluster.map_shared_rank(two_smem, 1)) + c;
#pragma unroll
        for (int q = 0; q < Q1; ++q) {
            const int lb = lane + q * T, b = r * H1 + lb;
            if (lb < H1 && b < R2) {
#pragma unroll
                for (int j = 0; j < R1; ++j) (j < H2 ? first : second)[(b * H2 + (j < H2 ? j : j - H2)) * W] = v[q][j];
            }
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    const GlobalOutT<C> dst{reinterpret_cast<C*>(out) + base, A.M, A.isign};
    const C* tw = reinterpret_cast<const C*>(A.tw);
#pragma unroll
    for (int q = 0; q < Q2; ++q) {
        const int lk = lane + q * T, k = r * H2 + lk;
        if (lk < H2 && k < R1) {
            C v[R2];
#pragma unroll
            for (int j = 0; j < R2; ++j) v[j] = two_smem[(j * H2 + lk) * W + c];
#pragma unroll
            for (int j = 1; j < R2; ++j) v[j] = cmul(v[j], tw[j * R1 + k]);
            dft<R2>(v);
            if (ok) {
#pragma unroll
                for (int j = 0; j < R2; ++j) dst.store(k + j * R1, v[j]);
            }
        }
    }
}

// The column pass: W adjacent columns per CTA, T threads per column.  LONG: the tile for strides
// beyond kTwoLongStride (croft_two_col).
template <int N, bool LONG>
__global__ void __launch_bounds__(croft_two_col(N, LONG).w* croft_two_col(N, LONG).t, croft_two_col(N, LONG).minb)
    croft_two_col_kernel(const float2* in, float2* out, const __grid_constant__ PassArgs A) {
    constexpr CroftTwo K = croft_two_col(N, LONG);
    using C = typename TwoComplex<K.packed != 0>::type;
    extern __shared__ __align__(16) float2 two_raw[];
    C* two_smem = reinterpret_cast<C*>(two_raw);
    C* tile = two_smem + (K.stage ? croft_two_pad(N) : 0);
    pdl_allow_dependents();
    const C* tw = two_twiddles<N, K.stage != 0>(A.tw, two_smem, K.w * K.t);
    pdl_wait();
    const int c = threadIdx.x % K.w, lane = threadIdx.x / K.w;
    const long long col = (long long)col_tile(A, blockIdx.x, gridDim.x) * K.w + c;
    const bool ok = col < A.ncols;
    long long b, m;
    col_split(col, A, b, m);
    const long long base = b * (long long)N * A.M + m;
    two_pencil<N, K.r1, K.t>(GlobalInT<C>{reinterpret_cast<const C*>(in) + base, A.M, A.isign},
                             GlobalOutT<C>{reinterpret_cast<C*>(out) + base, A.M, A.isign},
                             TwoExCol<K.r1, K.w, C>{tile + c}, tw, lane, ok);
}

// The row pass: W contiguous pencils per CTA, T threads per pencil.
template <int N>
__global__ void __launch_bounds__(croft_two_row(N).w* croft_two_row(N).t, croft_two_row(N).minb)
    croft_two_row_kernel(const float2* in, float2* out, const __grid_constant__ PassArgs A) {
    constexpr CroftTwo K = croft_two_row(N);
    using C = typename TwoComplex<K.packed != 0>::type;
    extern __shared__ __align__(16) float2 two_raw[];
    C* two_smem = reinterpret_cast<C*>(two_raw);
    C* tile = two_smem + (K.stage ? croft_two_pad(N) : 0);
    pdl_allow_dependents();
    const C* tw = two_twiddles<N, K.stage != 0>(A.tw, two_smem, K.w * K.t);
    pdl_wait();
    const int c = threadIdx.x / K.t, lane = threadIdx.x % K.t;
    const long long col = (long long)blockIdx.x * K.w + c;
    const bool ok = col < A.ncols;
    const long long base = col * N;
    two_pencil<N, K.r1, K.t>(GlobalInUnitT<C>{reinterpret_cast<const C*>(in) + base, A.isign},
                             GlobalOutUnitT<C>{reinterpret_cast<C*>(out) + base, A.isign},
                             TwoExRow<K.r1, C>{tile + c * K.ld}, tw, lane, ok);
}

}  // namespace croft
