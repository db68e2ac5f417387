// croft_batched_kernel.cuh - many independent 3D grids of uneven sizes in one
// persistent launch.
//
// Paper mapping: the paper transforms one grid with a fixed plan; its "option 4"
// (Sec. 5.1) is a single plan that covers many 1D FFTs at once, and its chunk
// parameter K (Sec. 5.1) trades chunk size against the number of calls.  Here
// one launch covers every pencil of every pass of every grid of a batch (e.g.
// the per-system PME meshes of an MD ensemble): the work list holds one item per
// tile (W pencils of one axis of one grid), ordered pass by pass (all z tiles,
// then all y tiles, then all x tiles), and resident CTAs pull items from a
// single atomic counter, so uneven grids balance themselves.
//
// Dependencies: the y tiles of grid g need every z tile of g finished (and the
// x tiles every y tile).  The CTA that finishes a tile bumps done[g][pass]
// after a device-scope fence; a CTA holding a dependent item waits for the
// count with a bounded spin (clock64 budget, nanosleep back-off).  Items are
// dequeued in pass order, so whatever an item waits for was dequeued earlier by
// a running CTA that never waits on a later item: the wait always ends unless
// the budget runs out, in which case the CTA records CROFT_ERR_TIMEOUT in the
// status word, stops waiting (every later wait returns at once) and the host
// reads the status (croft_plan_last_device_status).  Data written by another
// CTA in the same launch is read through L2 only (ld.global.cg).
#pragma once
#include "croft_fft_core.cuh"
#include "croft_internal.h"
#include "croft_two_stage_kernel.cuh"

namespace croft {

#define CROFT_BATCH_THREADS 256
#define CROFT_BATCH_MAX_N 128

struct BatchGrid {
    const float2* in;
    float2* out;
    long long M[3];     // element stride of the pass's axis (pass 0 = z, 1 = y, 2 = x)
    long long ncols[3]; // pencils of the pass
    int n[3];           // FFT length of the pass (1 = pass skipped)
    int W[3];           // pencils per tile
    int ntiles[3];      // tiles of the pass (0 when skipped)
    int dep[3];         // pass this pass waits for (-1: none)
    int first_pass;     // first pass that runs (reads `in`; later passes read `out`)
    int tw_off[3];      // offset of the axis' twiddle table in the pool
    CroftColDiv cdiv[3];  // col / M[pass] as a multiply-high (croft_coldiv.h; m = 0: divide)
};

struct BatchItem {
    int grid;
    int pass;
    int tile;
    int pad;
};

struct BatchArgs {
    const BatchGrid* grids;
    const BatchItem* items;
    const float2* tw_pool;
    int* queue;           // work counter of this launch
    int* done;            // [count][3] finished tiles
    int* status;          // CROFT_OK / CROFT_ERR_TIMEOUT
    long long wait_cycles;
    int item_begin;       // this launch serves items [item_begin, item_end)
    int item_end;
    int extra_wait;       // test hook: grid 0's pass-1 items wait for one tile more than exists
    int direct;           // 1: one CTA per item (item = item_begin + blockIdx.x), no counters, no waits
    float isign;
};

typedef void (*batch_tile_fn)(const BatchGrid&, int pass, int tile, const float2* tw, float2* smem, float isign);

// One pencil in two stages as two_pencil has them, the second stage's butterflies one after the other: the kernel's
// registers (80 for three CTAs per SM) hold a thread's first-stage points and little more (one launch for 96 grids
// of 64^3 513 -> 480 us, for 12 of 108^3 296 -> 280).
template <int N, int R1, int T, class Src, class Dst, class Ex>
__device__ __forceinline__ void batch_pencil(const Src& src, const Dst& dst, const Ex& ex, const typename Src::value_type* tw,
                                             int lane, bool ok) {
    using C = typename Src::value_type;
    constexpr int R2 = N / R1, Q1 = (R2 + T - 1) / T, Q2 = (R1 + T - 1) / T;
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
#pragma unroll
        for (int q = 0; q < Q1; ++q) {
            const int b = lane + q * T;
            if (R2 % T == 0 || b < R2) {
                dft<R1>(v[q]);
#pragma unroll
                for (int j = 0; j < R1; ++j) *ex.at(b, j) = v[q][j];
            }
        }
    }
    __syncthreads();
    if (!ok) return;
#pragma unroll 1
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
            for (int j = 0; j < R2; ++j) dst.store(k + j * R1, v[j]);
        }
    }
}

// One tile = W pencils of one pass of one grid, processed by the whole CTA.  Lengths with a two-stage kernel take its
// radices and sums (croft_two_batch), so a batch has the same bits whatever its schedule.  Against the general
// stages, one launch for all: batches of 90, 108 and 125 points 1.13-1.35x, most others 1.0-1.1x, 48 and 64 points
// 0.98 and 0.96, 60 points (radices 6 and 10 on 4 threads) 0.88; 96 meshes of mixed lengths 1023 -> 1005 us.
template <int LAYOUT, int N>
__device__ __noinline__ void batch_tile(const BatchGrid& G, int pass, int tile, const float2* twg, float2* smem,
                                        float isign) {
    constexpr int T = croft_threads_per_pencil(N);
    constexpr CroftTwo K = croft_two_batch(N, LAYOUT == LAYOUT_ROW);
    float2* stw = smem;
    float2* sbuf = smem + ((CROFT_BATCH_MAX_N + 1) / 2) * 2;
    const int W = G.W[pass];
    constexpr int ntw = K.r1 ? N : (croft_make_sched(N).count > 1 ? N - 1 : 0);
    for (int i = threadIdx.x; i < ntw; i += blockDim.x) stw[i] = __ldg(twg + i);
    using C = typename TwoComplex<K.packed != 0>::type;
    C* const cbuf = reinterpret_cast<C*>(sbuf);
    const C* const ctw = reinterpret_cast<const C*>(stw);
    const float2* in = (pass == G.first_pass) ? G.in : G.out;
    float2* out = G.out;
    if constexpr (LAYOUT == LAYOUT_ROW) {
        const int c = threadIdx.x / T;
        const int lane = threadIdx.x - c * T;
        const long long col = (long long)tile * W + c;
        const bool ok = c < W && col < G.ncols[pass];
        const long long base = (ok ? col : 0) * N;
        if constexpr (K.r1 != 0)
            batch_pencil<N, K.r1, T>(GlobalInCGT<C>{in + base, 1, isign},
                                     GlobalOutUnitT<C>{reinterpret_cast<C*>(out) + base, isign},
                                     TwoExRow<K.r1, C>{cbuf + c * croft_two_batch_ld(N)}, ctw, lane, ok);
        else
            fft_pencil_row<N, T>(GlobalInCG{in + base, 1, isign}, sbuf + (ok ? c : 0) * croft_row_ld_staged(N),
                                 GlobalOutUnit{out + base, isign}, stw, lane, ok);
    } else {
        const long long M = G.M[pass];
        const int c = threadIdx.x % W;
        const int lane = threadIdx.x / W;
        const long long col = (long long)tile * W + c;
        const bool ok = lane < T && col < G.ncols[pass];
        const long long cc = ok ? col : 0;
        const CroftColDiv dv = G.cdiv[pass];
        long long b, m;
        if (dv.m) {
            const unsigned q = croft_coldiv_q(dv.m, dv.s1, dv.s2, (unsigned)cc);
            b = q;
            m = (unsigned)cc - q * (unsigned)M;
        } else {
            b = cc / M;
            m = cc - b * M;
        }
        const long long base = b * (long long)N * M + m;
        if constexpr (K.r1 != 0) {
            static_assert(CROFT_BATCH_THREADS / T % 16 == 0, "W * T threads are the whole CTA: every lane is below T");
            batch_pencil<N, K.r1, T>(GlobalInCGT<C>{in + base, M, isign},
                                     GlobalOutT<C>{reinterpret_cast<C*>(out) + base, M, isign},
                                     TwoExColW<K.r1, C>{cbuf + c, W}, ctw, lane, ok);
        } else
            fft_pencil<N, T>(GlobalInCG{in + base, M, isign}, SmemCol{sbuf + c, W}, GlobalOut{out + base, M, isign}, stw,
                             lane, ok);
    }
}

}  // namespace croft
