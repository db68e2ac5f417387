// croft_plane_pass.h - the z+y pass over whole yz-planes in shared memory
// (croft_plane_pass_kernel.cuh): which plane shapes it takes and its launch shape.
#pragma once

#include "croft_sched.h"
#include "croft_two_stage.h"

// Lengths a plane's y axis may have, and its z axis (those that croft_plane_pass_rule takes).
CROFT_HD constexpr bool croft_plane_y(int n) {
    return n == 32 || n == 36 || n == 40 || n == 45 || n == 48 || n == 50 || n == 54 || n == 60 || n == 64 || n == 72 ||
           n == 75 || n == 80 || n == 81 || n == 90 || n == 96 || n == 100 || n == 108 || n == 120 || n == 125 || n == 128;
}
CROFT_HD constexpr bool croft_plane_z(int n) { return croft_plane_y(n) && (n <= 96 || n == 125); }
// How a plane's z and y axes split, n = R1 * R2, and whether their sums are paired: as the axis passes do (32 points: their
// stages 16 and 2), so that a transform has the same bits whether z and y run as one pass or as two (per-axis timing,
// croft_exec_axes, batches).
struct CroftPlaneAxis {
    int r1, packed;
};
CROFT_HD constexpr CroftPlaneAxis croft_plane_axis(int n, bool z) {
    if (!(z ? croft_plane_z(n) : croft_plane_y(n))) return CroftPlaneAxis{0, 0};
    if (n == 32) return CroftPlaneAxis{16, 0};
    const CroftTwo k = z ? croft_two_row(n) : croft_two_col(n, false);
    return CroftPlaneAxis{k.r1, k.packed};
}
CROFT_HD constexpr int croft_plane_r1z(int nz) { return croft_plane_axis(nz, true).r1; }
CROFT_HD constexpr int croft_plane_r1y(int ny) { return croft_plane_axis(ny, false).r1; }
// Elements from one run of a z transform's second stage to the next in shared memory (odd: no bank conflicts
// between neighbouring frequencies), and from one row of the plane to the next (odd likewise).
CROFT_HD constexpr int croft_plane_pitch(int nz) { return (nz / croft_plane_r1z(nz)) | 1; }
CROFT_HD constexpr int croft_plane_ld(int nz) { return (croft_plane_r1z(nz) * croft_plane_pitch(nz)) | 1; }
// Shared memory: [plane: ny rows of ld][slot of every z frequency: nz 16-bit numbers].
CROFT_HD constexpr int croft_plane_smem(int ny, int nz) { return ny * croft_plane_ld(nz) * 8 + (nz * 2 + 15) / 16 * 16; }

// Whether a plan's transforms, or its convolutions, run the z and y axes as one pass over the nx planes, on a device of `sms`
// SMs.  A convolution gains more: it saves two of five launches, one of them between the fused pass and the next.  Measured
// over all pairs of lengths and 26 to 91 values of nx, as captured graphs and as loops of single calls, axis by axis over
// plane pass; each rule takes what is no slower either way.  Transforms: 6439 shapes as graphs 0.95 to 2.0, median 1.14, two
// below 0.97, 1637 of them as single calls 1.00 to 1.65; convolutions: 2933 shapes, graphs 0.94 to 2.1, median 1.20, three below
// 0.97, single calls 0.96 to 2.0.
//  * few planes (one CTA per plane, at most two SMs of three busy): the launch saved outweighs the stages' latency up to
//    about 2700 points (transforms: 32^3 1.68, 36^3 1.21, 48^3 1.12; not 60^3 0.88, 64^3 0.93; from 64 planes on 3600 where
//    the row pass moves least, below), for convolutions up to 3100, and 4096 from 64 planes on.  Rows of 32 points, whose
//    passes are short of work, at any plane size;
//  * many planes: the z lengths whose own row pass moves least (5.6 to 6.6 TB/s: 36, 45, 50, 54, 60, 75, 81, 125, and
//    32), from the number of planes at which each is ahead at every plane size, up to 4800 points (transforms: 300 planes of 54^2
//    1.21, 60^2 1.10; 480 of 36 x 81 1.10); in convolutions smaller planes of the other lengths too.  What is left gains
//    or loses by the number of planes that the last round of CTAs holds (transforms: 300 planes of 64^2 1.27, 600 of
//    them 0.95; 300 of 80^2 1.00, 960 of 80^2 0.95), and grids beyond 32 MB lose: two axis passes in a row read the L2.
CROFT_HD constexpr bool croft_plane_pass_rule(int nx, int ny, int nz, int sms, bool convolution) {
    if (!croft_plane_y(ny) || !croft_plane_z(nz)) return false;
    const int plane = ny * nz;
    const bool large = plane > 4800 || (long long)nx * plane > 4 * 1024 * 1024;
    if (nz == 32 && (convolution || 6 * nx < 5 * sms)) return !large;
    if (!convolution) {
        if (3 * nx <= 2 * sms) {
            if (nz == 40 || nz == 48) return plane <= (nx == 1 ? 1536 : 2304);
            if (12 * nx > 5 * sms && (nz == 36 || nz == 45 || nz == 50 || nz == 54 || nz == 81)) return plane <= 3600;
            return plane <= (nx == 1 || nz == 64 || nz == 72 ? 2304 : 2700);
        }
        if (large) return false;
        if (nz == 54 || (nz == 45 && nx > sms)) return ny >= 48 || 3 * nx >= 5 * sms;
        if (ny < 36) return false;
        if (nz == 36 || nz == 45 || nz == 60 || nz == 125) return 3 * nx >= 5 * sms;
        if (nz == 75 || nz == 81) return 5 * nx >= 13 * sms;
        if (nz == 96) return nx >= 2 * sms && nx <= 4 * sms;
        return (nz == 32 || nz == 50) && nx >= 3 * sms;
    }
    if (8 * nx <= sms) return plane <= 2700;
    if (3 * nx <= 2 * sms) {
        if (nz == 72) return plane <= 2700;
        const bool higher = nz <= 45 || nz == 50 || nz == 54 || nz == 81 || nz == 96 || nz == 125;
        return plane <= (12 * nx > 5 * sms ? 4096 : (higher ? 3700 : 3100));
    }
    if (nx <= sms) return plane <= 3100 && nz != 72 && nz != 75;
    if (large) return false;
    if (nz == 36 || nz == 45 || nz == 50 || nz == 54 || nz == 81 || nz == 125) return true;
    if (nz == 60) return plane <= 3100;
    if (nz == 75) return nx >= 2 * sms;
    if (nz == 40 || nz == 48 || nz == 96) return 2 * nx >= 3 * sms && plane <= 3100;
    return nz != 72 && 2 * nx >= 3 * sms && (nz == 90 || plane <= 3600);
}
// Threads of a plane's CTA: enough for one round of butterflies a stage where an SM holds one plane, fewer (and
// more planes at a time) where there are many.  64^3: 128 / 256 / 384 / 512 / 1024 threads 0.81 / 0.89 / 0.88 /
// 0.92 / 0.90 of the three passes' speed, 300 planes of 64^2 1.12 / 1.25 / 1.02 / 1.02 / 0.91, 4096 of 32^2
// 1.20 / 1.15 / 1.04 / 1.05 / 0.79; 960 planes of 60^2 27.0 / 23.9 / 25.6 / 26.3 / 31.2 us (measured with the splits 8*8, 10*6
// and 8*4 of these lengths).
CROFT_HD constexpr int croft_plane_threads(int nx, int ny, int nz, int sms) {
    return nx <= sms ? 512 : (nx <= 4 * sms || ny * nz > 1600 ? 256 : 128);
}
