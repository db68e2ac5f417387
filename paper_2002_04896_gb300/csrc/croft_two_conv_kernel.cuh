// croft_two_conv_kernel.cuh - the fused pass of croft_exec_convolve (croft_conv_kernel.cuh: last
// forward 1D FFT, multiply by G, first backward 1D FFT on one column tile) for the lengths that
// split into two stages N = R1 * R2 (croft_two_stage_kernel.cuh).
//
// The backward transform takes the radices in the opposite order, R2 then R1: the outputs
// k + j*R1 of the forward transform's last butterfly k are then exactly the inputs of the
// backward transform's first butterfly k, so the last forward stage, the multiply and the first
// backward stage run in registers, and the column crosses shared memory twice in all:
//   forward stage 1 (radix R1)  HBM -> element b*R1 + j
//   middle, butterfly k < R1    elements k + j*R1 -> twiddles, radix R2, conj(G * .), radix R2 -> the same slots
//   backward stage 2, butterfly b < R2   elements b*R1 + j, twiddles w_N^{jb}, radix R1, conj -> y[b + j*R2]
// (the backward transform is conj o F o conj).  The middle stage works in place, so no barrier
// stands between its reads and its writes.  The three-stage kernel crossed shared memory four times with a barrier
// on either side of each; this one is bounded by the latency of its three phases at two to four CTAs per
// SM (data and G tiles) and, at 256 points and below, by instruction issue: 134M points (2.7 GB) at 256
// points 602 -> 527 us, at 512 points 755 -> 580.  Every thread copies the G values of its own middle
// butterflies to shared memory (cp.async at entry, behind the forward stage) and reads only those.
#pragma once
#include "croft_conv_kernel.cuh"
#include "croft_two_stage_kernel.cuh"

namespace croft {

// Shared memory: [twiddles when STAGE][tile: N x W complex][G tile: N x W real].
template <int N, int R1, int T, int W, bool STAGE, class C>
__device__ __forceinline__ void two_conv_body(const C* in, C* out, const float* g, const PassArgs& A) {
    constexpr int R2 = N / R1;
    constexpr int Q1 = (R2 + T - 1) / T, Q2 = (R1 + T - 1) / T;
    extern __shared__ __align__(16) float2 two_raw[];
    C* two_smem = reinterpret_cast<C*>(two_raw);
    C* tile = two_smem + (STAGE ? croft_two_pad(N) : 0);
    const int c = threadIdx.x % W, lane = threadIdx.x / W;
    float* gs = reinterpret_cast<float*>(tile + N * W) + c;
    const TwoExCol<R1, W, C> ex{tile + c};
    const long long col = (long long)blockIdx.x * W + c;
    const bool ok = col < A.ncols;
    long long b_, m_;
    col_split(col, A, b_, m_);
    const long long base = b_ * (long long)N * A.M + m_;

    pdl_allow_dependents();
    if (ok) {
#pragma unroll
        for (int q = 0; q < Q2; ++q) {
            const int k = lane + q * T;
            if (R1 % T == 0 || k < R1)
#pragma unroll
                for (int j = 0; j < R2; ++j) conv_cp_async(gs + (k + j * R1) * W, g + base + (long long)(k + j * R1) * A.M);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const C* tw = two_twiddles<N, STAGE>(A.tw, two_smem, W * T);
    pdl_wait();  // (G and the twiddles are not written by the previous pass)

    {
        const GlobalInT<C> src{in + base, A.M, 1.f};
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
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q2; ++q) {
        const int k = lane + q * T;
        if (R1 % T == 0 || k < R1) {
            C v[R2];
#pragma unroll
            for (int j = 0; j < R2; ++j) v[j] = *ex.at(j, k);
#pragma unroll
            for (int j = 1; j < R2; ++j) v[j] = cmul(v[j], tw[j * R1 + k]);
            dft<R2>(v);
#pragma unroll
            for (int j = 0; j < R2; ++j) {
                const float ga = gs[(k + j * R1) * W];
                v[j] = mkc<C>(v[j].x * ga, -(v[j].y * ga));
            }
            dft<R2>(v);
#pragma unroll
            for (int j = 0; j < R2; ++j) *ex.at(j, k) = v[j];
        }
    }
    __syncthreads();
    const GlobalOutT<C> dst{out + base, A.M, -1.f};
#pragma unroll
    for (int q = 0; q < Q1; ++q) {
        const int b = lane + q * T;
        if (R2 % T == 0 || b < R2) {
            C v[R1];
#pragma unroll
            for (int j = 0; j < R1; ++j) v[j] = *ex.at(b, j);
#pragma unroll
            for (int j = 1; j < R1; ++j) v[j] = cmul(v[j], tw[b * R1 + j]);
            dft<R1>(v);
            if (ok) {
#pragma unroll
                for (int j = 0; j < R1; ++j) dst.store(b + j * R2, v[j]);
            }
        }
    }
}

template <int N>
__global__ void __launch_bounds__(croft_two_conv(N).w* croft_two_conv(N).t, croft_two_conv(N).minb)
    croft_two_conv_kernel(const float2* in, float2* out, const float* g, const __grid_constant__ PassArgs A) {
    constexpr CroftTwo K = croft_two_conv(N);
    using C = typename TwoComplex<K.packed != 0>::type;
    two_conv_body<N, K.r1, K.t, K.w, K.stage != 0>(reinterpret_cast<const C*>(in), reinterpret_cast<C*>(out), g, A);
}

}  // namespace croft
