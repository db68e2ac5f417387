// croft_butterflies.cuh - in-register radix-R DFT butterflies (forward sign).
//
// dft<R>(v) overwrites v[0..R-1] with y[k] = sum_j v[j] exp(-2 pi i j k / R),
// output in natural order.  These are the serial 1D FFT building blocks that
// replace the FFTW codelets of the paper (Sec. 4, Sec. 5).  The backward
// transform reuses them through conj(F(conj(x))), applied at the global load
// and store of each pass.
//
// Radix 8, 9, 15 and 16 are split Cooley-Tukey (2x4, 3x3, 5x3 and 4x4) with the
// inner twiddles as compile-time constants; 3 and 5 use the symmetric cos/sin form.  The
// constants are the exact mathematical values rounded to the working precision
// (float for complex64, double for complex128).  The larger radices of the two-stage
// passes (6, 10, 12, 18 .. 32: DftSplit) take the same split with the inner twiddles
// computed at compile time.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

namespace croft {

// Complex helpers for float2 (complex64) and double2 (complex128).
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// complex64 whose sums and differences take one instruction for both parts (add and fma .f32x2 of sm_100 and later; the
// same roundings as float2's, whose products the butterflies below fuse with their sums explicitly).  Kernels that are bound by instruction issue or by the length of their
// butterflies gain a few per cent, kernels short of registers lose to the pairing: each two-stage kernel
// has the measured choice in its table (croft_two_stage.h).
struct __align__(8) packed2 {
    float x, y;
};
__device__ __forceinline__ packed2 cadd(packed2 a, packed2 b) {
    packed2 r;
    asm("{\n .reg .b64 p, q;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n add.rn.f32x2 p, p, q;\n mov.b64 {%0, %1}, p;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ packed2 csub(packed2 a, packed2 b) {
    packed2 r;
    asm("{\n .reg .b64 p, q, m;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n mov.b64 m, {%6, %6};\n fma.rn.f32x2 p, q, m, p;\n"
        " mov.b64 {%0, %1}, p;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(-1.f));
    return r;
}
__device__ __forceinline__ packed2 cmul(packed2 a, packed2 b) {
    packed2 r;
    r.x = fmaf(a.x, b.x, -a.y * b.y);
    r.y = fmaf(a.x, b.y, a.y * b.x);
    return r;
}

template <class C> struct CxScalar;
template <> struct CxScalar<packed2> { using T = float; };
template <> struct CxScalar<float2> { using T = float; };
template <> struct CxScalar<double2> { using T = double; };

template <class C> __device__ __forceinline__ C mkc(typename CxScalar<C>::T re, typename CxScalar<C>::T im) {
    C c;
    c.x = re;
    c.y = im;
    return c;
}
// a * (-i)
template <class C> __device__ __forceinline__ C mul_mi(C a) { return mkc<C>(a.y, -a.x); }
// a * (c + i s) for constants
template <class C>
__device__ __forceinline__ C mul_cs(C a, typename CxScalar<C>::T c, typename CxScalar<C>::T s) {
    return mkc<C>(fma(a.x, c, -a.y * s), fma(a.x, s, a.y * c));
}

// cos(pi/8), sin(pi/8), sqrt(2)/2, sqrt(3)/2, cos(2pi/5), cos(4pi/5), sin(2pi/5), sin(4pi/5):
// the exact values, rounded to the working precision.
#define CROFT_C8 0.92387953251128675613
#define CROFT_S8 0.38268343236508977173
#define CROFT_R2 0.70710678118654752440
#define CROFT_R3 0.86602540378443864676
#define CROFT_C51 0.30901699437494742410
#define CROFT_C52 (-0.80901699437494742410)
#define CROFT_S51 0.95105651629515357212
#define CROFT_S52 0.58778525229247312917
// cos and sin of 2 pi m / 9 (m = 1, 2, 4) and of 2 pi m / 15 (m = 1, 2, 4, 8; m = 3 and
// 6 are the radix-5 constants above), exact values rounded to the working precision.
#define CROFT_C9_1 0.7660444431189780352024
#define CROFT_S9_1 0.6427876096865393263226
#define CROFT_C9_2 0.1736481776669303488517
#define CROFT_S9_2 0.9848077530122080593667
#define CROFT_C9_4 (-0.9396926207859083840541)
#define CROFT_S9_4 0.3420201433256687330441
#define CROFT_C15_1 0.9135454576426008955021
#define CROFT_S15_1 0.4067366430758002077540
#define CROFT_C15_2 0.6691306063588582138263
#define CROFT_S15_2 0.7431448254773942350147
#define CROFT_C15_4 (-0.1045284632676534713998)
#define CROFT_S15_4 0.9945218953682733369227
#define CROFT_C15_8 (-0.9781476007338056379286)
#define CROFT_S15_8 (-0.2079116908177593371017)

template <int R, class C> __device__ __forceinline__ void dft(C* v);

template <class C> __device__ __forceinline__ void dft4(C& x0, C& x1, C& x2, C& x3) {
    C a = cadd(x0, x2), b = csub(x0, x2);
    C c = cadd(x1, x3), d = mul_mi(csub(x1, x3));
    x0 = cadd(a, c);
    x2 = csub(a, c);
    // (rotated by -i: a swap of the parts, which a pair of scalar sums has for nothing)
    x1 = mkc<C>(b.x + d.x, b.y + d.y);
    x3 = mkc<C>(b.x - d.x, b.y - d.y);
}

template <int R, class C> struct Dft;

template <class C> struct Dft<2, C> {
    __device__ __forceinline__ static void run(C* v) {
        C t = v[0];
        v[0] = cadd(t, v[1]);
        v[1] = csub(t, v[1]);
    }
};

template <class C> struct Dft<4, C> {
    __device__ __forceinline__ static void run(C* v) { dft4(v[0], v[1], v[2], v[3]); }
};

template <class C> struct Dft<8, C> {
    __device__ __forceinline__ static void run(C* v) {
        using T = typename CxScalar<C>::T;
        const T r2 = (T)CROFT_R2;
        // j = 4*j1 + j2: length-2 DFTs over j1, twiddle W8^(j2*k1), length-4 DFTs over j2.
        C a0[4], a1[4];
#pragma unroll
        for (int j2 = 0; j2 < 4; ++j2) {
            a0[j2] = cadd(v[j2], v[4 + j2]);
            a1[j2] = csub(v[j2], v[4 + j2]);
        }
        a1[1] = mul_cs(a1[1], r2, -r2);   // W8^1
        a1[2] = mul_mi(a1[2]);            // W8^2 = -i
        a1[3] = mul_cs(a1[3], -r2, -r2);  // W8^3
        dft4(a0[0], a0[1], a0[2], a0[3]);
        dft4(a1[0], a1[1], a1[2], a1[3]);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
            v[2 * k2] = a0[k2];
            v[2 * k2 + 1] = a1[k2];
        }
    }
};

template <class C> struct Dft<16, C> {
    __device__ __forceinline__ static void run(C* v) {
        using T = typename CxScalar<C>::T;
        const T c8 = (T)CROFT_C8, s8 = (T)CROFT_S8, r2 = (T)CROFT_R2;
        // j = 4*j1 + j2: length-4 DFTs over j1, twiddle W16^(j2*k1), length-4 DFTs over j2.
        C a[4][4];  // a[k1][j2]
#pragma unroll
        for (int j2 = 0; j2 < 4; ++j2) {
            C x0 = v[j2], x1 = v[4 + j2], x2 = v[8 + j2], x3 = v[12 + j2];
            dft4(x0, x1, x2, x3);
            a[0][j2] = x0;
            a[1][j2] = x1;
            a[2][j2] = x2;
            a[3][j2] = x3;
        }
        a[1][1] = mul_cs(a[1][1], c8, -s8);   // W16^1
        a[1][2] = mul_cs(a[1][2], r2, -r2);   // W16^2
        a[1][3] = mul_cs(a[1][3], s8, -c8);   // W16^3
        a[2][1] = mul_cs(a[2][1], r2, -r2);   // W16^2
        a[2][2] = mul_mi(a[2][2]);            // W16^4
        a[2][3] = mul_cs(a[2][3], -r2, -r2);  // W16^6
        a[3][1] = mul_cs(a[3][1], s8, -c8);   // W16^3
        a[3][2] = mul_cs(a[3][2], -r2, -r2);  // W16^6
        a[3][3] = mul_cs(a[3][3], -c8, s8);   // W16^9
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            dft4(a[k1][0], a[k1][1], a[k1][2], a[k1][3]);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = a[k1][k2];
        }
    }
};

template <class C> struct Dft<3, C> {
    __device__ __forceinline__ static void run(C* v) {
        using T = typename CxScalar<C>::T;
        const T r3 = (T)CROFT_R3;
        C t = cadd(v[1], v[2]);
        C d = csub(v[1], v[2]);
        C m = mkc<C>(fma((T)-0.5, t.x, v[0].x), fma((T)-0.5, t.y, v[0].y));
        v[0] = cadd(v[0], t);
        // m -+ i (sqrt3/2) d as multiply-adds, one rounding each (paired sums of the rounded products would
        // take as many instructions and round twice)
        v[1] = mkc<C>(fma(r3, d.y, m.x), fma(-r3, d.x, m.y));
        v[2] = mkc<C>(fma(-r3, d.y, m.x), fma(r3, d.x, m.y));
    }
};

template <class C> struct Dft<5, C> {
    __device__ __forceinline__ static void run(C* v) {
        using T = typename CxScalar<C>::T;
        const T c1 = (T)CROFT_C51, c2 = (T)CROFT_C52, s1 = (T)CROFT_S51, s2 = (T)CROFT_S52;
        C t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
        C d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
        C x0 = v[0];
        C a1 = mkc<C>(fma(c1, t1.x, fma(c2, t2.x, x0.x)), fma(c1, t1.y, fma(c2, t2.y, x0.y)));
        C a2 = mkc<C>(fma(c2, t1.x, fma(c1, t2.x, x0.x)), fma(c2, t1.y, fma(c1, t2.y, x0.y)));
        C b1 = mkc<C>(fma(s1, d1.x, s2 * d2.x), fma(s1, d1.y, s2 * d2.y));
        C b2 = mkc<C>(fma(s2, d1.x, -s1 * d2.x), fma(s2, d1.y, -s1 * d2.y));
        v[0] = mkc<C>(x0.x + t1.x + t2.x, x0.y + t1.y + t2.y);
        // y1 = a1 - i b1, y4 = a1 + i b1, y2 = a2 - i b2, y3 = a2 + i b2
        v[1] = mkc<C>(a1.x + b1.y, a1.y - b1.x);
        v[4] = mkc<C>(a1.x - b1.y, a1.y + b1.x);
        v[2] = mkc<C>(a2.x + b2.y, a2.y - b2.x);
        v[3] = mkc<C>(a2.x - b2.y, a2.y + b2.x);
    }
};

template <class C> struct Dft<9, C> {
    __device__ __forceinline__ static void run(C* v) {
        using T = typename CxScalar<C>::T;
        // j = 3*j1 + j2: length-3 DFTs over j1, twiddle W9^(j2*k1), length-3 DFTs over j2.
        C a[3][3];  // a[k1][j2]
#pragma unroll
        for (int j2 = 0; j2 < 3; ++j2) {
            C t[3] = {v[j2], v[3 + j2], v[6 + j2]};
            Dft<3, C>::run(t);
            a[0][j2] = t[0];
            a[1][j2] = t[1];
            a[2][j2] = t[2];
        }
        a[1][1] = mul_cs(a[1][1], (T)CROFT_C9_1, -(T)CROFT_S9_1);  // W9^1
        a[1][2] = mul_cs(a[1][2], (T)CROFT_C9_2, -(T)CROFT_S9_2);  // W9^2
        a[2][1] = mul_cs(a[2][1], (T)CROFT_C9_2, -(T)CROFT_S9_2);  // W9^2
        a[2][2] = mul_cs(a[2][2], (T)CROFT_C9_4, -(T)CROFT_S9_4);  // W9^4
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            Dft<3, C>::run(a[k1]);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = a[k1][k2];
        }
    }
};

template <class C> struct Dft<15, C> {
    __device__ __forceinline__ static void run(C* v) {
        using T = typename CxScalar<C>::T;
        // j = 3*j1 + j2 (j1 < 5, j2 < 3): length-5 DFTs over j1, twiddle W15^(j2*k1),
        // length-3 DFTs over j2; output k1 + 5*k2.
        C a[5][3];  // a[k1][j2]
#pragma unroll
        for (int j2 = 0; j2 < 3; ++j2) {
            C t[5] = {v[j2], v[3 + j2], v[6 + j2], v[9 + j2], v[12 + j2]};
            Dft<5, C>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < 5; ++k1) a[k1][j2] = t[k1];
        }
        a[1][1] = mul_cs(a[1][1], (T)CROFT_C15_1, -(T)CROFT_S15_1);  // W15^1
        a[2][1] = mul_cs(a[2][1], (T)CROFT_C15_2, -(T)CROFT_S15_2);  // W15^2
        a[3][1] = mul_cs(a[3][1], (T)CROFT_C51, -(T)CROFT_S51);      // W15^3 = W5^1
        a[4][1] = mul_cs(a[4][1], (T)CROFT_C15_4, -(T)CROFT_S15_4);  // W15^4
        a[1][2] = mul_cs(a[1][2], (T)CROFT_C15_2, -(T)CROFT_S15_2);  // W15^2
        a[2][2] = mul_cs(a[2][2], (T)CROFT_C15_4, -(T)CROFT_S15_4);  // W15^4
        a[3][2] = mul_cs(a[3][2], (T)CROFT_C52, -(T)CROFT_S52);      // W15^6 = W5^2
        a[4][2] = mul_cs(a[4][2], (T)CROFT_C15_8, -(T)CROFT_S15_8);  // W15^8
#pragma unroll
        for (int k1 = 0; k1 < 5; ++k1) {
            Dft<3, C>::run(a[k1]);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) v[k1 + 5 * k2] = a[k1][k2];
        }
    }
};

template <int R, class C> __device__ __forceinline__ void dft(C* v) { Dft<R, C>::run(v); }

// ---------------------------------------------------------------------------
// composite radices with compile-time inner twiddles
// ---------------------------------------------------------------------------

// cos(2 pi m / R) in float64 at compile time: the angle is folded into the first octant by
// integer arithmetic (exact), where 14 Taylor terms leave an error far below half a ulp.
constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double octant_sin(double x) {
    double t = x, s = x;
    for (int i = 1; i < 14; ++i) {
        t *= -x * x / ((2 * i) * (2 * i + 1));
        s += t;
    }
    return s;
}
constexpr double octant_cos(double x) {
    double t = 1, s = 1;
    for (int i = 1; i < 14; ++i) {
        t *= -x * x / ((2 * i - 1) * (2 * i));
        s += t;
    }
    return s;
}
constexpr double cos_2pi(long long m, long long R) {
    m = ((m % R) + R) % R;
    if (2 * m > R) m = R - m;
    if (4 * m > R) return -cos_2pi(R - 2 * m, 2 * R);
    if (8 * m <= R) return octant_cos(2 * kPi * (double)m / (double)R);
    return octant_sin(2 * kPi * (double)(R - 4 * m) / (double)(4 * R));
}
constexpr double sin_2pi(long long m, long long R) { return cos_2pi(4 * m - R, 4 * R); }

// f(integral_constant<int, 0>) ... f(integral_constant<int, N - 1>): a loop whose index is a constant
// expression, so that every twiddle is computed by the compiler.
template <class F, int... I>
__device__ __forceinline__ void for_each_index(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F> __device__ __forceinline__ void for_each_index(F&& f) {
    for_each_index(f, std::make_integer_sequence<int, N>{});
}

// a * exp(-2 pi i M / R)
template <int R, int M, class C> __device__ __forceinline__ C mul_root(C a) {
    using T = typename CxScalar<C>::T;
    constexpr int m = ((M % R) + R) % R;
    if constexpr (m == 0) return a;
    else if constexpr (4 * m == R) return mul_mi(a);
    else if constexpr (2 * m == R) return mkc<C>(-a.x, -a.y);
    else if constexpr (4 * m == 3 * R) return mkc<C>(-a.y, a.x);
    else {
        constexpr double c = cos_2pi(m, R), s = -sin_2pi(m, R);
        return mul_cs(a, (T)c, (T)s);
    }
}

// Radix R = A * B: j = B*j1 + j2; length-A DFTs over j1, twiddle W_R^(j2*k1), length-B DFTs over
// j2; output k1 + A*k2.
template <int A, int B, class C> struct DftSplit {
    __device__ __forceinline__ static void run(C* v) {
        C a[A][B];  // a[k1][j2]
        for_each_index<B>([&](auto j2c) {
            constexpr int j2 = decltype(j2c)::value;
            C t[A];
#pragma unroll
            for (int j1 = 0; j1 < A; ++j1) t[j1] = v[B * j1 + j2];
            Dft<A, C>::run(t);
            for_each_index<A>([&](auto k1c) {
                constexpr int k1 = decltype(k1c)::value;
                a[k1][j2] = mul_root<A * B, j2 * k1>(t[k1]);
            });
        });
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            Dft<B, C>::run(a[k1]);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = a[k1][k2];
        }
    }
};
// ---------------------------------------------------------------------------
// power-of-two radices as fused multiply-add butterflies (complex128)
// ---------------------------------------------------------------------------

// A radix-R butterfly of a stage with P > 1 needs the DFT of w^j v[j] (w = exp(-2 pi i k / (P R))).  By decimation in
// time, DFT_R = E[m] + (w W_R^m) O[m], E[m] - (w W_R^m) O[m] with E over the even j and O over the odd j, both with
// w^2 in the place of w: the stage's twiddles merge with the inner ones.  A factor is taken as
//     f = (-i)^q s (1 + i r),   q the nearest quarter turn, s = cos, r = -tan of the rest (|r| <= 1),
// (Linzer and Feig 1993 factor the rotation like this) and one radix-2 butterfly is
//     b1 = (-i)^q b (selects and sign bits),  b2 = b1 + i r b1,  a + s b2,  a - s b2:
// 6 multiply-adds whatever f, each result two roundings from its operands, against 8 instructions and three
// roundings for product, then sum and difference.  The factors of m and m + R/4 differ by -i, so R/2 factors are
// read instead of R - 1.  Radix 16 with twiddles: 192 instructions against 228, radix 8: 72 against 84.  The
// complex128 passes take these butterflies, being bound by the FP64 pipe (about 2 instructions per SM clock,
// everything else idles): 128^3 109 -> 92 us a pass, 256^3 797 -> 680; rounding error of a 128-point row 1.67e-16 ->
// 1.58e-16, of 1024 points 2.04e-16 -> 1.95e-16 (against 80 bits and more).  A stage without twiddles keeps the split butterflies: with constant factors in this form
// radix 16 would take 148 instructions instead of 168 (128^3 88 us a pass instead of 92), but its rounding error grows
// by 6 %, two rounded constants standing for every factor.
//
// Table order: level n = R, R/2, .., 2, for each the factors w^{R/n} W_n^m, m < max(1, n/4), as (s, r) with q in the
// top two bits of s, which are 0 in a number of [0.7, 1].
constexpr int fma_twiddle_offset(int R, int n) { return n == R ? 0 : fma_twiddle_offset(R, 2 * n) + (2 * n / 4 > 0 ? 2 * n / 4 : 1); }

// (-i)^q b, q in bits 31 and 30 of `q`.
__device__ __forceinline__ double2 quarter_turns(double2 b, int q) {
    const bool swap = (q & 0x40000000) != 0;
    const int fx = q & 0x80000000, fy = (q ^ (q << 1)) & 0x80000000;
    const int xh = __double2hiint(b.x), xl = __double2loint(b.x), yh = __double2hiint(b.y), yl = __double2loint(b.y);
    return make_double2(__hiloint2double((swap ? yh : xh) ^ fx, swap ? yl : xl),
                        __hiloint2double((swap ? xh : yh) ^ fy, swap ? xl : yl));
}
// a, b -> a + f b, a - f b with f = s (1 + i r) after b's quarter turns.
__device__ __forceinline__ void fma_butterfly(double2& a, double2& b, double s, double r) {
    const double2 c = make_double2(fma(-r, b.y, b.x), fma(r, b.x, b.y));
    b = make_double2(fma(-s, c.x, a.x), fma(-s, c.y, a.y));
    a = make_double2(fma(s, c.x, a.x), fma(s, c.y, a.y));
}

// The n-point level of a radix-R butterfly: v[0], v[STRIDE], .. -> out[0 .. n-1].
template <int R, int N, int STRIDE> struct FmaLevel {
    __device__ __forceinline__ static void run(const double2* v, double2* out, const double2* w) {
        double2 e[N / 2], o[N / 2];
        FmaLevel<R, N / 2, 2 * STRIDE>::run(v, e, w);
        FmaLevel<R, N / 2, 2 * STRIDE>::run(v + STRIDE, o, w);
        for_each_index<N / 2>([&](auto mc) {
            constexpr int m = decltype(mc)::value;
            constexpr bool turned = N >= 4 && m >= N / 4;  // factor of m - N/4 times -i
            const double2 f = w[fma_twiddle_offset(R, N) + (turned ? m - N / 4 : m)];
            const int hi = __double2hiint(f.x);
            double2 a = e[m], b = quarter_turns(turned ? mul_mi(o[m]) : o[m], hi);
            fma_butterfly(a, b, __hiloint2double(hi & 0x3fffffff, __double2loint(f.x)), f.y);
            out[m] = a;
            out[m + N / 2] = b;
        });
    }
};
template <int R, int STRIDE> struct FmaLevel<R, 1, STRIDE> {
    __device__ __forceinline__ static void run(const double2* v, double2* out, const double2*) { out[0] = v[0]; }
};
// v[0 .. R-1] -> the DFT of w^j v[j], f the R/2 factors.
template <int R> __device__ __forceinline__ void fma_dft(double2* v, const double2* f) {
    double2 out[R];
    FmaLevel<R, R, 1>::run(v, out, f);
#pragma unroll
    for (int j = 0; j < R; ++j) v[j] = out[j];
}

template <class C> struct Dft<6, C> : DftSplit<3, 2, C> {};
template <class C> struct Dft<10, C> : DftSplit<5, 2, C> {};
template <class C> struct Dft<12, C> : DftSplit<4, 3, C> {};
template <class C> struct Dft<18, C> : DftSplit<9, 2, C> {};
template <class C> struct Dft<20, C> : DftSplit<5, 4, C> {};
template <class C> struct Dft<24, C> : DftSplit<8, 3, C> {};
template <class C> struct Dft<25, C> : DftSplit<5, 5, C> {};
template <class C> struct Dft<27, C> : DftSplit<9, 3, C> {};
template <class C> struct Dft<30, C> : DftSplit<15, 2, C> {};
template <class C> struct Dft<32, C> : DftSplit<8, 4, C> {};

}  // namespace croft
