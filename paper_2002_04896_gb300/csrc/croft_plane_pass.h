// croft_plane_pass.h - the z+y pass over whole yz-planes in shared memory
// (croft_plane_pass_kernel.cuh): which plane shapes it takes and its launch shape.
#pragma once

#include "croft_sched.h"
#include "croft_two_stage.h"

// Whether an axis of n points may be one of a plane (both radices at most 16; 125: 25).
CROFT_HD constexpr bool croft_plane_length(int n) {
    return n == 32 || n == 36 || n == 40 || n == 45 || n == 48 || n == 50 || n == 54 || n == 60 || n == 64 || n == 72 ||
           n == 75 || n == 80 || n == 81 || n == 90 || n == 96 || n == 100 || n == 108 || n == 120 || n == 125 || n == 128;
}
// How a plane's z and y axes split, n = R1 * R2, and whether their sums are paired: as the axis passes do (32 points: their
// stages 16 and 2), so that a transform has the same bits whether z and y run as one pass or as two (per-axis timing,
// croft_exec_axes, batches).
struct CroftPlaneAxis {
    int r1, packed;
};
CROFT_HD constexpr CroftPlaneAxis croft_plane_axis(int n, bool z) {
    if (!croft_plane_length(n)) return CroftPlaneAxis{0, 0};
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

// Whether a plan runs its z and y axes as one pass over the planes.  Measured in graph replays (no host time),
// three passes over plane pass + x pass: 32^3 1.71, 36^3 1.15, 48^3 1.10, 54^3 1.10, 64^3 0.92, 80^3 0.93,
// 96^3 0.94, 100^3 1.14, 108^3 0.89; 300 planes of 48^2 1.41, 54^2 1.48, 60^2 1.40, 64^2 1.25, 80^2 1.08, 90^2
// 1.20, 96^2 1.13, 100^2 1.05, 108^2 1.00, 120^2 0.96; 4 planes of 64^2 0.92, 16 of 96^2 0.69.  Launched one by
// one, a transform of up to about 64^3 points takes as long as its launches (9 us for three, 5 for two), so
// planes of up to 4096 points always take it; larger ones from about two planes per SM on (162 of 90 x 108, one
// round and a rest: a convolution takes 36.6 us against 35.3), up to 6400 points, and up to 10,000 while the grid
// stays in the L2 (z and y of 960 planes, two passes / plane pass: 72^2 30.4 / 27.4 us, 80^2 35.3 / 35.8, 96^2
// 48.4 / 54.0, 108^2 60 / 67).
CROFT_HD constexpr bool croft_plane_pass_rule(int nx, int ny, int nz) {
    return croft_plane_length(ny) && croft_plane_length(nz) &&
           (ny * nz <= 4096 || (nx >= 288 && (ny * nz <= 6400 || (ny * nz <= 10000 && nx <= 456))));
}
// Threads of a plane's CTA: enough for one round of butterflies a stage where an SM holds one plane, fewer (and
// more planes at a time) where there are many.  64^3: 128 / 256 / 384 / 512 / 1024 threads 0.81 / 0.89 / 0.88 /
// 0.92 / 0.90 of the three passes' speed, 300 planes of 64^2 1.12 / 1.25 / 1.02 / 1.02 / 0.91, 4096 of 32^2
// 1.20 / 1.15 / 1.04 / 1.05 / 0.79; 960 planes of 60^2 27.0 / 23.9 / 25.6 / 26.3 / 31.2 us.
CROFT_HD constexpr int croft_plane_threads(int nx, int ny, int nz) {
    return nx <= 152 ? 512 : (nx <= 608 || ny * nz > 1600 ? 256 : 128);
}
