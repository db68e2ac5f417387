// croft_tc_two_kernel.cuh - tensor-core pass in two stages, N = 16 * R2 (32 <= N <= 512): the radix-16
// stage on the tensor cores, then one radix-R2 stage (R2 <= 32) on the CUDA cores.
//
// The radix-16 stage is croft_tc_kernel.cuh's: butterflies as rows of 128 x 32 x 32 split-operand GEMMs, operands
// staged in shared memory, one tcgen05.mma chain per 128 rows, FP32 accumulators in TMEM, tcgen05.ld back to the
// registers of the thread that owns the butterfly.  Here a thread owns up to two butterflies (Q: two groups of
// rows), so that 16 threads serve a pencil of up to 512 points and each then takes one radix-R2
// butterfly of the second stage:
//   load Q x 16 points -> split -> operand rows -> MMA -> TMEM -> registers -> exchange buffer -> radix R2 -> HBM.
//
// What bounds it: the latency of that chain at three or four 256-thread CTAs per SM (five barriers and an MMA round trip
// in it); the tensor pipe idles.  Against three stages (16, then the near-equal split of the rest: one exchange and
// two barriers more, at 32 threads per pencil) a 512^3 bf16x3 forward transform went from 1630 to 1364 us, 256^3 from 184 to 149.
// The next pass may become resident while this one drains (programmatic dependent launch).  Its CTAs hold TMEM
// while they wait for this pass to end, so no CTA of this pass may still want TMEM then: the warp that allocates
// it lets the dependents start only after it has it.  (Allowed earlier, a dependent on the same SM could take the columns that a
// CTA of this pass waits for, beside another program's kernel that holds the rest, and neither would end.)
#pragma once
#include "croft_tc_kernel.cuh"
#include "croft_two_stage_kernel.cuh"

namespace croft {

// Threads per pencil, pencils per CTA (256 threads: two 128-row groups per butterfly of a thread), butterflies per
// thread in the first stage, row pencil's length in the exchange buffer.
CROFT_HD constexpr int tc_two_threads(int n) { return n / 16 > 8 ? 16 : 8; }
CROFT_HD constexpr int tc_two_width(int n) { return 256 / tc_two_threads(n); }
CROFT_HD constexpr int tc_two_q(int n) { return (n / 16 + tc_two_threads(n) - 1) / tc_two_threads(n); }
CROFT_HD constexpr int tc_two_ld(int n) { return n / 16 * 17; }
CROFT_HD constexpr int tc_two_smem(int n, bool row) {
    const int ops = tc_two_q(n) * 256 * 128, tile = tc_two_width(n) * (row ? tc_two_ld(n) : n) * 8;
    return 4096 + (ops > tile ? ops : tile);
}
// CTAs per SM that the registers must allow: four (64) where a thread holds one butterfly of 16 points, three (80, a
// few spilled) where it holds two or a radix above 16.  512^3 with two / three: 1538 / 1394 us, 432x400x288 669 / 606;
// 256^3 with three / four 169 / 152.
CROFT_HD constexpr int tc_two_minb(int n) { return n / 16 <= 16 ? 4 : 3; }

// Paired sums (packed2) in the second stage: where they measured faster (x or z pass, us: 384 points 254 -> 250, 432 205 ->
// 197, 288 213 -> 209, 512 499 -> 487; 320 246 -> 257 the other way, the rest equal).
CROFT_HD constexpr bool tc_two_packed(int n) { return n == 288 || n == 384 || n == 432 || n == 512; }

// The y pass follows A.backwards (256^3 53.2 -> 51.2 us, 400 points 194.7 -> 190.5), but at 512 points, whose
// registers are spent: 469 -> 485 us with the choice of the tile compiled in.
//
// Shared memory: [B operand: 4 KB][A operands: Q x 256 rows of 128 bytes | exchange buffer].
template <int LAYOUT, int N, int PREC>
__global__ void __launch_bounds__(256, tc_two_minb(N)) croft_tc_two_kernel(const float2* in, float2* out,
                                                                            const __grid_constant__ PassArgs A) {
    constexpr int R2 = N / 16, T = tc_two_threads(N), W = tc_two_width(N), Q = tc_two_q(N), Q2 = 16 / T;
    constexpr int NCOLS = 64 * Q;  // 32 accumulator columns per 128 rows
    extern __shared__ __align__(16) float2 smem[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_slot;
    unsigned char* bmat = (unsigned char*)smem;
    unsigned char* ops = bmat + 4096;  // group (q, g): hi 8 KB at (2 * (2 * q + g)) * 8192, lo behind it
    const int tid = threadIdx.x, g = tid >> 7, row = tid & 127;
    // CTAs of such passes that an SM's shared memory (228 KB, 1 KB of it reserved per CTA) holds never want more than its
    // 512 columns together, whatever their lengths, so the allocation waits only for other kernels
    static_assert((tc_two_smem(N, LAYOUT == LAYOUT_ROW) + 1024) * 512 >= NCOLS * 228 * 1024, "TMEM columns per SM");
    ((uint4*)bmat)[tid] = ((const uint4*)A.tc_b)[tid];
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)), "r"(NCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        pdl_allow_dependents();  // (by this warp alone: not before the allocation)
    }

    int c, lane;
    if constexpr (LAYOUT == LAYOUT_ROW) {
        c = tid / T;
        lane = tid % T;
    } else {
        c = tid % W;
        lane = tid / W;
    }
    const long long col = (long long)(LAYOUT == LAYOUT_COL && N < 512 ? col_tile(A, blockIdx.x, gridDim.x) : blockIdx.x) * W + c;
    const bool ok = col < A.ncols;
    long long base = 0, M = 1;
    if constexpr (LAYOUT == LAYOUT_ROW) {
        base = (ok ? col : 0) * N;
    } else {
        M = A.M;
        long long b, m;
        col_split(ok ? col : 0, A, b, m);
        base = b * (long long)N * M + m;
    }
    float unscale[Q];
    pdl_wait();
    {
        const float2* p = in + base;
        float2 u[Q][16];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int b = lane + q * T;
            if (ok && b < R2) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int a = b + j * R2;
                    u[q][j] = LAYOUT == LAYOUT_ROW ? p[a] : p[(long long)a * M];
                    conj_if(u[q][j], A.isign);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) u[q][j] = make_float2(0.f, 0.f);
            }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float scale = 1.f;
            unscale[q] = 1.f;
            if constexpr (PREC == TC_FP16X3) {  // the largest component into [2^14, 2^15) (exact)
                float m = 0.f;
#pragma unroll
                for (int j = 0; j < 16; ++j) m = fmaxf(m, fmaxf(fabsf(u[q][j].x), fabsf(u[q][j].y)));
                const int sh = min(141 - (int)((__float_as_uint(m) >> 23) & 0xff), 126);
                scale = __uint_as_float((uint32_t)(sh + 127) << 23);
                unscale[q] = __uint_as_float((uint32_t)(127 - sh) << 23);
            }
            unsigned char* hi = ops + (2 * q + g) * 16384;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                uint32_t h[4], l[4];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const int k = kk * 8 + e;
                    const float x0 = ((k < 16) ? u[q][k & 15].x : u[q][k & 15].y) * scale;
                    const float x1 = ((k < 16) ? u[q][(k + 1) & 15].x : u[q][(k + 1) & 15].y) * scale;
                    tc_split2<PREC>(x0, x1, h[e / 2], l[e / 2]);
                }
                *(uint4*)(hi + tc_cm_offset(row, kk * 8)) = make_uint4(h[0], h[1], h[2], h[3]);
                *(uint4*)(hi + 8192 + tc_cm_offset(row, kk * 8)) = make_uint4(l[0], l[1], l[2], l[3]);
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;");  // the operands, for the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_slot;
    if (tid == 0) {
        const uint32_t bh = smem_addr(bmat);
#pragma unroll
        for (int gg = 0; gg < 2 * Q; ++gg) {
            const uint32_t d = tmem + 32 * gg, ah = smem_addr(ops) + gg * 16384, al = ah + 8192;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {  // K = 32 as two steps of 16
                tc_mma<PREC>(d, tc_desc(ah + ks * 256), tc_desc(bh + ks * 256), ks);
                tc_mma<PREC>(d, tc_desc(ah + ks * 256), tc_desc(bh + 2048 + ks * 256), 1);
                tc_mma<PREC>(d, tc_desc(al + ks * 256), tc_desc(bh + ks * 256), 1);
            }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(&mbar)));
    }
    // one warp waits for the commit (bounded), the others at the barrier
    if (tid < 32 && !tc_wait(smem_addr(&mbar), 0) && A.status && tid == 0) atomicExch(A.status, 5 /* CROFT_ERR_TIMEOUT */);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    // exchange buffer (over the operands, which every MMA has read): element b*16 + j of a pencil
    float2* tile = (float2*)ops;
    const TwoExCol<16, W, float2> exc{tile + c};
    const TwoExRow<16, float2> exr{tile + c * tc_two_ld(N)};
    auto at = [&](int b, int j) { return LAYOUT == LAYOUT_ROW ? exr.at(b, j) : exc.at(b, j); };
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float d[32];
        tc_ld32(tmem + 32 * (2 * q + g) + ((uint32_t)(((tid >> 5) & 3) * 32) << 16), d);
        const int b = lane + q * T;
        if (b < R2) {
#pragma unroll
            for (int j = 0; j < 16; ++j) *at(b, j) = make_float2(d[j] * unscale[q], d[16 + j] * unscale[q]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (tid < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NCOLS));
    using C = typename TwoComplex<tc_two_packed(N)>::type;
    const C* tw = reinterpret_cast<const C*>(A.tw);
    C* dst = reinterpret_cast<C*>(out) + base;
#pragma unroll
    for (int q = 0; q < Q2; ++q) {
        const int k = lane + q * T;
        C v[R2];
#pragma unroll
        for (int j = 0; j < R2; ++j) v[j] = *reinterpret_cast<const C*>(at(j, k));
#pragma unroll
        for (int j = 1; j < R2; ++j) v[j] = cmul(v[j], tw[j * 16 + k]);
        dft<R2>(v);
        if (ok) {
#pragma unroll
            for (int j = 0; j < R2; ++j) {
                conj_if(v[j], A.isign);
                const int a = k + j * 16;
                dst[LAYOUT == LAYOUT_ROW ? a : (long long)a * M] = v[j];
            }
        }
    }
}

}  // namespace croft
