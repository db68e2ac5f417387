// croft_plane_pass_kernel.cuh - the z and y transforms of whole yz-planes in one pass: one CTA per
// plane, the plane in its shared memory.
//
// Paper mapping: steps 1 to 5 of Sec. 4.1 (FFTs along z, the rearrangement, FFTs along y) with the
// rearrangement inside the CTA: a small grid's transform takes two launches instead of three and
// crosses the L2 twice.
//
// What bounds it: for small grids the launches (a 32^3 transform: 9.1 us of host time for three, 5.1 for
// two; on the device, in a graph, 7.5 -> 4.5 us), beyond that the instruction issue of four
// barrier-separated stages at 64 registers, 1024 threads per SM: 2.6-2.9 TB/s of the 16 bytes a point that it moves (960 planes
// of 72^2 in 27.4 us, of 96^2 in 54.0), where two axis passes in a row come to the same 2.6-3.0 TB/s of those 16
// bytes (30.4 and 48.4 us): hence the limits of croft_plane_pass_rule.
//
// Both transforms take two stages n = R1 * R2, split and summed as in the axis passes (croft_plane_axis: the same bits), every stage in place, so that a thread may take any
// number of butterflies one after the other and a barrier stands only between stages:
//   z1  butterfly b < R2 of a row reads z = b + j*R2 (j < R1) from HBM, radix R1, element (k, b)
//   z2  butterfly k < R1: elements (k, j), twiddles w_nz^{jk}, radix R2; element (k, j) is now frequency k + j*R1
//   y1  butterfly b < R2 of a column: rows b + j*R2, radix R1, output k in row b + k*R2
//   y2  butterfly k < R1: rows j + k*R2, twiddles, radix R2, frequency k + j*R1 to HBM
// Element (k, b) of a row lies in slot k*pitch + b, pitch odd; rows are an odd distance apart: the lanes of a
// warp take neighbouring rows in z2 and neighbouring z frequencies in y1 and y2 (so that the stores to
// HBM are contiguous and a warp shares its twiddles), each a walk of odd stride over the banks.
//
// The kernel is specialised on ny; the z stages are functions of their own, one per nz, called once
// per plane (20 kernels and 16 such functions instead of a kernel for every pair of lengths).
#pragma once
#include "croft_butterflies.cuh"
#include "croft_fft_core.cuh"
#include "croft_internal.h"
#include "croft_plane_pass.h"
#include "croft_two_stage_kernel.cuh"

namespace croft {

// z1 and z2 of a plane of ny rows.
template <int NZ>
__device__ __noinline__ void plane_z(const float2* in, const float2* tw, int ny, unsigned div_ny, float isign) {
    extern __shared__ __align__(16) float2 plane_raw[];
    using C = typename TwoComplex<croft_plane_axis(NZ, true).packed != 0>::type;
    C* plane_tile = reinterpret_cast<C*>(plane_raw);
    constexpr int R1 = croft_plane_r1z(NZ), R2 = NZ / R1, PITCH = croft_plane_pitch(NZ), LD = croft_plane_ld(NZ);
    for (int i = threadIdx.x; i < ny * R2; i += blockDim.x) {
        const int y = i / R2, b = i - y * R2;
        const C* src = reinterpret_cast<const C*>(in) + y * NZ + b;
        C v[R1];
#pragma unroll
        for (int j = 0; j < R1; ++j) {
            v[j] = src[j * R2];
            conj_if(v[j], isign);
        }
        dft<R1>(v);
        C* d = plane_tile + y * LD + b;
#pragma unroll
        for (int k = 0; k < R1; ++k) d[k * PITCH] = v[k];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ny * R1; i += blockDim.x) {
        const int k = (int)__umulhi((unsigned)i, div_ny), y = i - k * ny;
        C* d = plane_tile + y * LD + k * PITCH;
        C v[R2];
#pragma unroll
        for (int j = 0; j < R2; ++j) v[j] = d[j];
#pragma unroll
        for (int j = 1; j < R2; ++j) v[j] = cmul(v[j], reinterpret_cast<const C*>(tw)[j * R1 + k]);
        dft<R2>(v);
#pragma unroll
        for (int j = 0; j < R2; ++j) d[j] = v[j];
    }
}

#define CROFT_PLANE_Y_SIZES(X)                                                                                   \
    X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) X(72) X(75) X(80) X(81) X(90) X(96) X(100) X(108)      \
    X(120) X(125) X(128)
#define CROFT_PLANE_Z_SIZES(X)                                                                                   \
    X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) X(72) X(75) X(80) X(81) X(90) X(96) X(125)

template <int NY>
__global__ void __launch_bounds__(1024) croft_plane_pass_kernel(const __grid_constant__ PlanePassArgs A) {
    constexpr int R1 = croft_plane_r1y(NY), R2 = NY / R1;
    using C = typename TwoComplex<croft_plane_axis(NY, false).packed != 0>::type;
    constexpr unsigned DIV_NY = (unsigned)((0x100000000ull + NY - 1) / NY);
    extern __shared__ __align__(16) float2 plane_raw[];
    C* plane_tile = reinterpret_cast<C*>(plane_raw);
    pdl_allow_dependents();
    const int nz = A.nz, ld = A.ld;
    unsigned short* slot = reinterpret_cast<unsigned short*>(plane_tile + NY * ld);
    for (int i = threadIdx.x; i < nz; i += blockDim.x) slot[i] = (unsigned short)((i % A.r1z) * A.pitch + i / A.r1z);
    const long long base = (long long)blockIdx.x * (NY * nz);
    const float2* in = A.in + base;
    float2* out = A.out + base;
    pdl_wait();
    switch (nz) {
#define CROFT_PLANE_Z(NZ)                                                \
    case NZ: plane_z<NZ>(in, A.tw_z, NY, DIV_NY, A.isign); break;
        CROFT_PLANE_Z_SIZES(CROFT_PLANE_Z)
#undef CROFT_PLANE_Z
        default: break;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nz * R2; i += blockDim.x) {
        const int b = (int)__umulhi((unsigned)i, A.div_nz), s = slot[i - b * nz];
        C* d = plane_tile + b * ld + s;
        C v[R1];
#pragma unroll
        for (int j = 0; j < R1; ++j) v[j] = d[j * R2 * ld];
        dft<R1>(v);
#pragma unroll
        for (int k = 0; k < R1; ++k) d[k * R2 * ld] = v[k];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nz * R1; i += blockDim.x) {
        const int k = (int)__umulhi((unsigned)i, A.div_nz), kz = i - k * nz;
        const C* d = plane_tile + (k * R2) * ld + slot[kz];
        C v[R2];
#pragma unroll
        for (int j = 0; j < R2; ++j) v[j] = d[j * ld];
#pragma unroll
        for (int j = 1; j < R2; ++j) v[j] = cmul(v[j], reinterpret_cast<const C*>(A.tw_y)[j * R1 + k]);
        dft<R2>(v);
        C* o = reinterpret_cast<C*>(out) + k * nz + kz;
#pragma unroll
        for (int j = 0; j < R2; ++j) {
            conj_if(v[j], A.isign);
            o[j * R1 * nz] = v[j];
        }
    }
}

}  // namespace croft
