// croft_two_stage.h - which passes run as two stages N = R1 * R2 (croft_two_stage_kernel.cuh) and
// with what tile, shared by the planner and the kernels.
//
// One entry per axis length, from a sweep of every split with radices of at most 32 points, the
// threads per pencil that either stage asks for, 8- to 32-column tiles, the register bounds that
// leave room for a thread's points, and both places for the twiddles, on 2.1 GB grids (CUDA
// events, median of 7): per length the fastest, spill-free where that costs less than 0.5 %.  In
// the comments: GB/s (16 bytes a point over the time) of the pass it replaces -> of this one,
// where 6700 to 7100 is a plain copy.  Lengths without an entry keep the croft_pass_kernel.cuh
// kernels: those of at most 32 points (one or two short stages there as well), the few
// without such a split (972, 1000), those beyond 1024 (radices above 32), and those where the
// other kernel is as fast (below 3 % for columns, 2 % for rows; 256-point columns 6595 against 6678).  At 128 points the
// tiles are those that are fastest on a 128^3 grid, which the L2 holds.  The figures are those of unpaired sums; paired
// ones (packed = 1) are on where a second sweep of the chosen tiles measured 0.6 % or more for them: most
// convolutions (256 points 5 %, 480 6 %), columns of 360 (4 %), 625 (11 %), 900 (10 %) points; not where the
// registers are short (480 -4 %, 432 -15 %, 1024 -5 %).
#pragma once

#include "croft_sched.h"

struct CroftTwo {
    int r1;     // first radix (0: the length has no two-stage kernel)
    int t;      // threads per pencil
    int w;      // pencils per CTA
    int minb;   // CTAs per SM that the registers must allow (launch bound)
    int stage;  // 1: twiddles copied to shared memory at entry; 0: read through L1
    int ld;     // rows: elements from one pencil to the next in shared memory; columns: 0
    int ctas;   // columns: CTAs that share a tile (2: croft_two_pair_kernel)
    int packed; // 1: sums and differences of both parts in one instruction (packed2)
};

// Column passes of more than 625 points need 80 KB and more for a 16-column tile: one CTA per SM, with nothing to
// overlap its load, compute and store.  Across megabytes two CTAs share the tile instead, three or four of
// them per SM (x pass at 2 MB strides, one CTA / two per tile: 640 points 4516 / 4922 GB/s, 729 4511 / 5378,
// 1024 4899 / 5478).  While the axis's elements lie at most this far apart 8-column tiles (64-byte row pieces) of one CTA
// are as good or better for most lengths: 1024 points across 8 / 32 / 128 / 256 KB 5450 / 5380 / 5170 / 5160 GB/s,
// against 3530 at 2 MB, where every piece lies in a page of its own.
constexpr long long kTwoLongStride = 256 * 1024;

CROFT_HD constexpr bool croft_two_split_by_stride(int n) { return n > 625; }

// x: axis of n x 512 x 512 (2 MB strides); y: of 512 x n x 512 (4 KB strides).
CROFT_HD constexpr CroftTwo croft_two_col(int n, bool long_stride) {
    switch (n) {
        case 36: return CroftTwo{9, 4, 32, 9, 1, 0, 1, 1};  // x 5597 -> 6951, y 5624 -> 7127
        case 40: return CroftTwo{10, 4, 32, 9, 1, 0, 1, 1};  // x 4473 -> 6844, y 4477 -> 7095
        case 45: return CroftTwo{9, 5, 32, 9, 0, 0, 1, 1};  // x 4369 -> 6830, y 4372 -> 7087
        case 48: return CroftTwo{8, 6, 32, 7, 0, 0, 1, 0};  // x 5438 -> 6837, y 5725 -> 7116
        case 50: return CroftTwo{10, 5, 32, 10, 1, 0, 1, 0};  // x 4220 -> 6906, y 4256 -> 7044
        case 54: return CroftTwo{9, 6, 32, 7, 1, 0, 1, 0};  // x 3934 -> 6862, y 3923 -> 7095
        case 60: return CroftTwo{6, 10, 32, 5, 1, 0, 1, 1};  // x 5654 -> 6899, y 5891 -> 7119
        case 64: return CroftTwo{8, 8, 32, 5, 0, 0, 1, 0};  // x 5773 -> 6891, y 5966 -> 7119
        case 72: return CroftTwo{12, 6, 32, 6, 1, 0, 1, 0};  // x 5471 -> 6886, y 5702 -> 7088
        case 75: return CroftTwo{15, 5, 32, 6, 0, 0, 1, 0};  // x 6175 -> 6895, y 6210 -> 7090
        case 80: return CroftTwo{16, 5, 32, 5, 0, 0, 1, 0};  // x 5714 -> 6760, y 6016 -> 7077
        case 81: return CroftTwo{9, 9, 32, 5, 1, 0, 1, 0};  // x 4598 -> 6755, y 4738 -> 7107
        case 90: return CroftTwo{15, 6, 32, 5, 1, 0, 1, 0};  // x 4182 -> 6901, y 4254 -> 7083
        case 96: return CroftTwo{16, 6, 32, 5, 0, 0, 1, 0};  // x 5595 -> 6764, y 5668 -> 7088
        case 100: return CroftTwo{10, 10, 32, 6, 1, 0, 1, 0};  // x 4258 -> 6853, y 4332 -> 7082
        case 108: return CroftTwo{12, 9, 32, 4, 1, 0, 1, 0};  // x 4231 -> 6840, y 4330 -> 7115
        case 120: return CroftTwo{15, 8, 32, 4, 1, 0, 1, 0};  // x 6244 -> 6712, y 6415 -> 7087
        case 125: return CroftTwo{25, 5, 32, 4, 0, 0, 1, 0};  // x 4437 -> 6797, y 4489 -> 7067
        case 128: return CroftTwo{16, 8, 32, 4, 1, 0, 1, 0};  // x 6360 -> 6838, y 6572 -> 7045; 128^3 18.8 -> 18.5 us
        case 135: return CroftTwo{15, 9, 32, 4, 1, 0, 1, 0};  // x 6031 -> 6753, y 6277 -> 7075
        case 144: return CroftTwo{18, 8, 32, 4, 1, 0, 1, 1};  // x 5887 -> 6882, y 6174 -> 7066
        case 150: return CroftTwo{25, 6, 32, 4, 1, 0, 1, 0};  // x 5633 -> 6814, y 5806 -> 7063
        case 160: return CroftTwo{16, 10, 32, 3, 1, 0, 1, 0};  // x 5564 -> 6798, y 5863 -> 7080
        case 162: return CroftTwo{18, 9, 32, 3, 1, 0, 1, 0};  // x 4192 -> 6646, y 4468 -> 7059
        case 180: return CroftTwo{20, 9, 32, 3, 1, 0, 1, 0};  // x 4092 -> 6748, y 4251 -> 7073
        case 192: return CroftTwo{24, 8, 32, 4, 0, 0, 1, 0};  // x 5611 -> 6855, y 5787 -> 7083
        case 200: return CroftTwo{20, 10, 32, 3, 1, 0, 1, 0};  // x 4496 -> 6675, y 4650 -> 7068
        case 216: return CroftTwo{24, 9, 32, 3, 1, 0, 1, 0};  // x 4613 -> 6720, y 4773 -> 7020
        case 225: return CroftTwo{25, 9, 32, 3, 1, 0, 1, 0};  // x 4348 -> 6716, y 4574 -> 6993
        case 240: return CroftTwo{15, 16, 16, 5, 0, 0, 1, 0};  // x 6273 -> 6514, y 6669 -> 7020
        case 243: return CroftTwo{27, 9, 16, 5, 0, 0, 1, 1};  // x 4927 -> 6350, y 4970 -> 7046
        case 250: return CroftTwo{25, 10, 32, 2, 1, 0, 1, 1};  // x 3802 -> 6312, y 3974 -> 6537
        case 270: return CroftTwo{15, 18, 16, 4, 1, 0, 1, 1};  // x 5375 -> 6210, y 5641 -> 6939
        case 288: return CroftTwo{16, 18, 16, 4, 1, 0, 1, 1};  // x 5568 -> 6348, y 5726 -> 7077
        case 300: return CroftTwo{15, 20, 16, 4, 1, 0, 1, 0};  // x 5534 -> 6240, y 5699 -> 6939
        case 320: return CroftTwo{20, 20, 16, 4, 0, 0, 1, 0};  // x 5701 -> 6269, y 5965 -> 6925
        case 324: return CroftTwo{18, 18, 16, 4, 0, 0, 1, 1};  // x 4273 -> 6061, y 4388 -> 6864
        case 360: return CroftTwo{20, 20, 16, 3, 0, 0, 1, 1};  // x 5087 -> 6069, y 5542 -> 6640
        case 375: return CroftTwo{25, 15, 16, 3, 1, 0, 1, 1};  // x 5408 -> 5927, y 5813 -> 6708
        case 384: return CroftTwo{24, 16, 16, 3, 1, 0, 1, 0};  // x 6185 -> 6353, y 6134 -> 6985
        case 400: return CroftTwo{25, 16, 16, 3, 1, 0, 1, 0};  // x 5502 -> 6266, y 6033 -> 6986
        case 405: return CroftTwo{27, 15, 16, 3, 1, 0, 1, 0};  // x 4452 -> 5787, y 4850 -> 6554
        case 432: return CroftTwo{24, 24, 16, 3, 0, 0, 1, 0};  // x 5325 -> 5925, y 5716 -> 6623
        case 450: return CroftTwo{30, 15, 16, 3, 0, 0, 1, 0};  // x 4407 -> 5725, y 4652 -> 6426
        case 480: return CroftTwo{30, 16, 16, 3, 1, 0, 1, 0};  // x 5329 -> 5798, y 5710 -> 6711
        case 486: return CroftTwo{18, 27, 16, 2, 1, 0, 1, 0};  // x 4314 -> 5664, y 4578 -> 6271
        case 500: return CroftTwo{20, 25, 16, 2, 1, 0, 1, 0};  // x 3922 -> 5552, y 4396 -> 6157
        case 512: return CroftTwo{32, 16, 16, 3, 0, 0, 1, 1};  // x 5354 -> 6177, y 5785 -> 6861
        case 540: return CroftTwo{20, 27, 16, 2, 1, 0, 1, 0};  // x 3128 -> 5772, y 5047 -> 6347
        case 576: return CroftTwo{24, 24, 16, 2, 1, 0, 1, 0};  // x 3138 -> 5920, y 4501 -> 6498
        case 600: return CroftTwo{24, 25, 16, 2, 1, 0, 1, 0};  // x 3119 -> 5916, y 4391 -> 6422
        case 625: return CroftTwo{25, 25, 16, 2, 0, 0, 1, 1};  // x 3230 -> 5440, y 4505 -> 5992
        case 640: return long_stride ? CroftTwo{20, 16, 16, 3, 0, 0, 2, 1} : CroftTwo{32, 20, 8, 3, 0, 0, 1, 1};  // x 3149 -> 4922, y 4678 -> 5892
        case 648: return CroftTwo{24, 14, 16, 4, 0, 0, 2, 1};  // x 3173 -> 5436, y 3795 -> 5946
        case 675: return long_stride ? CroftTwo{27, 14, 16, 4, 0, 0, 2, 1} : CroftTwo{25, 27, 8, 3, 0, 0, 1, 1};  // x 3141 -> 5407, y 4516 -> 5791
        case 720: return long_stride ? CroftTwo{24, 15, 16, 3, 0, 0, 2, 0} : CroftTwo{24, 30, 8, 3, 1, 0, 1, 1};  // x 3135 -> 4953, y 4850 -> 5641
        case 729: return CroftTwo{27, 14, 16, 4, 0, 0, 2, 1};  // x 3218 -> 5378, y 3879 -> 5806
        case 750: return long_stride ? CroftTwo{25, 15, 16, 3, 0, 0, 2, 1} : CroftTwo{25, 30, 8, 3, 1, 0, 1, 1};  // x 3172 -> 4784, y 4098 -> 5544
        case 768: return long_stride ? CroftTwo{24, 16, 16, 3, 0, 0, 2, 0} : CroftTwo{24, 32, 8, 3, 0, 0, 1, 1};  // x 3156 -> 5098, y 5072 -> 5535
        case 800: return long_stride ? CroftTwo{25, 16, 16, 3, 0, 0, 2, 0} : CroftTwo{25, 32, 8, 3, 0, 0, 1, 1};  // x 3146 -> 5062, y 4334 -> 5645
        case 810: return long_stride ? CroftTwo{27, 15, 16, 3, 0, 0, 2, 0} : CroftTwo{27, 30, 8, 3, 0, 0, 1, 1};  // x 3085 -> 4939, y 3688 -> 5686
        case 864: return long_stride ? CroftTwo{27, 16, 16, 3, 0, 0, 2, 0} : CroftTwo{27, 32, 8, 2, 1, 0, 1, 1};  // x 3145 -> 5238, y 4361 -> 5539
        case 900: return CroftTwo{30, 15, 16, 3, 0, 0, 2, 1};  // x 3092 -> 4970, y 3746 -> 5365
        case 960: return CroftTwo{32, 16, 16, 3, 0, 0, 2, 0};  // x 3145 -> 5177, y 4646 -> 5623
        case 1024: return CroftTwo{32, 16, 16, 3, 0, 0, 2, 0};  // x 3134 -> 5478, y 5003 -> 5884
        default: return CroftTwo{0, 0, 0, 0, 0, 0, 0, 0};
    }
}

// z axis of 512 x 512 x n.
CROFT_HD constexpr CroftTwo croft_two_row(int n) {
    switch (n) {
        case 36: return CroftTwo{6, 6, 16, 15, 0, 42, 1, 0};  // 3692 -> 6434
        case 40: return CroftTwo{8, 8, 12, 15, 0, 56, 1, 0};  // 4551 -> 6850
        case 45: return CroftTwo{9, 5, 19, 14, 0, 45, 1, 1};  // 3686 -> 5777
        case 48: return CroftTwo{8, 8, 12, 14, 0, 56, 1, 0};  // 4088 -> 6807
        case 50: return CroftTwo{10, 5, 19, 16, 0, 55, 1, 0};  // 3653 -> 5584
        case 54: return CroftTwo{9, 6, 16, 16, 0, 54, 1, 1};  // 3803 -> 6201
        case 60: return CroftTwo{6, 10, 10, 14, 0, 70, 1, 1};  // 4882 -> 6623
        case 64: return CroftTwo{8, 8, 32, 6, 1, 72, 1, 0};  // 5081 -> 7126
        case 72: return CroftTwo{8, 9, 14, 15, 1, 89, 1, 0};  // 5074 -> 6718
        case 75: return CroftTwo{15, 5, 19, 15, 0, 75, 1, 0};  // 4661 -> 5953
        case 80: return CroftTwo{8, 10, 13, 14, 0, 90, 1, 0};  // 5155 -> 6771
        case 81: return CroftTwo{9, 9, 28, 7, 1, 81, 1, 0};  // 4594 -> 6250
        case 90: return CroftTwo{9, 10, 26, 6, 1, 90, 1, 1};  // 4015 -> 6672
        case 96: return CroftTwo{8, 12, 11, 14, 0, 108, 1, 0};  // 4445 -> 6986
        case 100: return CroftTwo{10, 10, 13, 14, 0, 110, 1, 0};  // 4349 -> 6749
        case 108: return CroftTwo{12, 12, 8, 16, 0, 124, 1, 0};  // 4517 -> 6991
        case 120: return CroftTwo{12, 12, 8, 14, 0, 140, 1, 0};  // 6158 -> 6972
        case 125: return CroftTwo{5, 5, 19, 8, 0, 125, 1, 0};  // 4119 -> 5817
        case 128: return CroftTwo{16, 8, 16, 8, 0, 136, 1, 0};  // 6548 -> 7000; 128^3 18.8 -> 18.4 us
        case 135: return CroftTwo{15, 9, 28, 5, 1, 135, 1, 0};  // 5108 -> 6267
        case 144: return CroftTwo{12, 12, 21, 6, 0, 156, 1, 0};  // 6120 -> 7025
        case 150: return CroftTwo{15, 15, 6, 15, 0, 150, 1, 0};  // 4727 -> 6202
        case 160: return CroftTwo{10, 16, 6, 16, 0, 176, 1, 0};  // 5730 -> 7043
        case 162: return CroftTwo{18, 9, 14, 9, 1, 171, 1, 0};  // 4494 -> 6210
        case 180: return CroftTwo{12, 15, 17, 6, 0, 195, 1, 0};  // 4497 -> 6583
        case 192: return CroftTwo{24, 8, 12, 9, 0, 200, 1, 0};  // 6228 -> 7085
        case 200: return CroftTwo{25, 8, 12, 8, 0, 200, 1, 1};  // 5261 -> 6563
        case 216: return CroftTwo{12, 18, 5, 13, 0, 234, 1, 1};  // 5833 -> 6797
        case 225: return CroftTwo{15, 15, 6, 14, 0, 225, 1, 0};  // 5244 -> 6554
        case 240: return CroftTwo{16, 16, 8, 10, 0, 256, 1, 0};  // 5285 -> 7048
        case 243: return CroftTwo{27, 9, 28, 3, 1, 249, 1, 1};  // 5219 -> 6024
        case 250: return CroftTwo{25, 10, 13, 5, 1, 250, 1, 1};  // 4382 -> 6190
        case 256: return CroftTwo{16, 16, 16, 4, 1, 272, 1, 0};  // 6813 -> 7032
        case 270: return CroftTwo{15, 18, 5, 13, 0, 274, 1, 0};  // 5318 -> 6714
        case 288: return CroftTwo{16, 18, 7, 9, 0, 306, 1, 0};  // 5854 -> 7021
        case 300: return CroftTwo{20, 20, 6, 9, 0, 324, 1, 1};  // 5193 -> 6758
        case 320: return CroftTwo{16, 20, 6, 9, 0, 340, 1, 0};  // 6025 -> 7049
        case 324: return CroftTwo{18, 18, 7, 8, 0, 354, 1, 0};  // 4767 -> 6762
        case 360: return CroftTwo{24, 24, 4, 10, 0, 376, 1, 1};  // 5294 -> 6890
        case 375: return CroftTwo{15, 25, 4, 8, 0, 375, 1, 1};  // 5399 -> 6363
        case 384: return CroftTwo{16, 16, 8, 6, 0, 416, 1, 0};  // 6393 -> 7047
        case 400: return CroftTwo{16, 16, 6, 8, 0, 425, 1, 0};  // 6344 -> 6792
        case 405: return CroftTwo{27, 15, 17, 3, 1, 415, 1, 0};  // 5152 -> 5985
        case 432: return CroftTwo{24, 24, 4, 10, 0, 456, 1, 0};  // 6228 -> 7026
        case 450: return CroftTwo{30, 15, 6, 7, 0, 465, 1, 0};  // 4605 -> 6564
        case 480: return CroftTwo{20, 24, 5, 7, 0, 504, 1, 1};  // 6558 -> 7043
        case 486: return CroftTwo{18, 27, 5, 5, 0, 513, 1, 1};  // 4803 -> 6397
        case 500: return CroftTwo{20, 25, 5, 7, 0, 537, 1, 1};  // 4848 -> 6789
        case 512: return CroftTwo{16, 16, 8, 5, 0, 544, 1, 0};  // 6676 -> 7045
        case 540: return CroftTwo{20, 27, 5, 5, 0, 567, 1, 1};  // 4355 -> 6538
        case 576: return CroftTwo{24, 24, 4, 9, 0, 600, 1, 0};  // 5212 -> 6900
        case 600: return CroftTwo{24, 25, 5, 6, 0, 633, 1, 1};  // 4843 -> 6697
        case 625: return CroftTwo{25, 25, 5, 6, 0, 633, 1, 1};  // 4846 -> 6600
        case 640: return CroftTwo{20, 32, 3, 9, 0, 672, 1, 0};  // 5982 -> 7077
        case 648: return CroftTwo{24, 27, 4, 7, 0, 683, 1, 1};  // 5053 -> 6588
        case 675: return CroftTwo{27, 27, 4, 7, 0, 683, 1, 1};  // 4813 -> 6480
        case 720: return CroftTwo{24, 30, 3, 8, 0, 750, 1, 1};  // 5484 -> 6755
        case 729: return CroftTwo{27, 27, 4, 7, 0, 731, 1, 1};  // 4390 -> 6539
        case 750: return CroftTwo{30, 30, 3, 8, 0, 775, 1, 1};  // 4348 -> 6622
        case 768: return CroftTwo{32, 32, 3, 8, 0, 800, 1, 0};  // 5749 -> 7039
        case 800: return CroftTwo{32, 32, 3, 8, 0, 825, 1, 0};  // 5178 -> 7001
        case 810: return CroftTwo{27, 30, 3, 8, 0, 814, 1, 0};  // 4371 -> 6682
        case 864: return CroftTwo{32, 32, 3, 7, 0, 896, 1, 0};  // 5261 -> 7030
        case 900: return CroftTwo{30, 30, 3, 7, 0, 930, 1, 0};  // 4412 -> 6630
        case 960: return CroftTwo{32, 32, 3, 8, 0, 992, 1, 0};  // 6164 -> 7035
        case 1024: return CroftTwo{32, 32, 4, 5, 0, 1056, 1, 0};  // 6488 -> 7026
        default: return CroftTwo{0, 0, 0, 0, 0, 0, 0, 0};
    }
}

// The entry of a batch's pass: its grids' strides are short.
CROFT_HD constexpr CroftTwo croft_two_batch(int n, bool row) { return row ? croft_two_row(n) : croft_two_col(n, false); }
// Row pencil's length in the exchange buffer of the persistent batched kernel, whose pencils take 4 or 8 threads: the
// smallest distance at which the 16 threads of a half warp, on neighbouring pencils, meet no bank twice (one launch for 96 grids
// of 64^3, distances of the row passes / these: 490 / 480 us).
CROFT_HD constexpr int croft_two_batch_ld(int n) {
    const int r1 = croft_two_row(n).r1, step = croft_threads_per_pencil(n) == 4 ? 8 : 16;
    int ld = n / r1 * (r1 + (r1 % 2 == 0));
    while (ld % step != step / 2) ++ld;
    return ld;
}

// The fused convolution pass (croft_two_conv_kernel.cuh), x axis of n x 512 x 512; GB/s of its 20 bytes a
// point (grid in and out, G in) of the three-stage kernel it replaced -> of this one.  Chosen for the long strides
// of an x axis, the usual last axis; a 2D grid's y axis takes the same tiles.
CROFT_HD constexpr CroftTwo croft_two_conv(int n) {
    switch (n) {
        case 36: return CroftTwo{6, 6, 32, 10, 1, 0, 1, 1};  // 5120 -> 6546
        case 40: return CroftTwo{5, 8, 32, 8, 1, 0, 1, 0};  // 4876 -> 6460
        case 45: return CroftTwo{5, 9, 32, 7, 0, 0, 1, 0};  // 4602 -> 6306
        case 48: return CroftTwo{12, 4, 32, 10, 1, 0, 1, 1};  // 5120 -> 6592
        case 50: return CroftTwo{10, 10, 32, 5, 1, 0, 1, 0};  // 4129 -> 6006
        case 54: return CroftTwo{9, 9, 32, 6, 1, 0, 1, 1};  // 4189 -> 6413
        case 60: return CroftTwo{5, 5, 32, 8, 1, 0, 1, 0};  // 4800 -> 6486
        case 64: return CroftTwo{8, 8, 32, 8, 0, 0, 1, 0};  // 4814 -> 5479
        case 72: return CroftTwo{8, 9, 32, 6, 0, 0, 1, 0};  // 4496 -> 6491
        case 75: return CroftTwo{15, 5, 32, 6, 0, 0, 1, 1};  // 4915 -> 6234
        case 80: return CroftTwo{10, 10, 32, 6, 1, 0, 1, 0};  // 4995 -> 6269
        case 81: return CroftTwo{9, 9, 16, 13, 0, 0, 1, 1};  // 4822 -> 5182
        case 90: return CroftTwo{10, 9, 32, 5, 0, 0, 1, 1};  // 4189 -> 6101
        case 96: return CroftTwo{12, 8, 32, 5, 1, 0, 1, 1};  // 4551 -> 6213
        case 100: return CroftTwo{10, 10, 32, 4, 0, 0, 1, 1};  // 4129 -> 5826
        case 108: return CroftTwo{9, 9, 32, 4, 0, 0, 1, 1};  // 4320 -> 5928
        case 120: return CroftTwo{15, 8, 32, 4, 1, 0, 1, 1};  // 4954 -> 5800
        case 125: return CroftTwo{25, 5, 32, 4, 0, 0, 1, 1};  // 4324 -> 5787
        case 128: return CroftTwo{16, 8, 32, 4, 0, 0, 1, 1};  // 4819 -> 6125
        case 135: return CroftTwo{15, 9, 32, 3, 0, 0, 1, 1};  // 4488 -> 5531
        case 144: return CroftTwo{16, 9, 32, 3, 0, 0, 1, 1};  // 4666 -> 5703
        case 150: return CroftTwo{15, 10, 32, 3, 0, 0, 1, 1};  // 4364 -> 5623
        case 160: return CroftTwo{16, 10, 32, 3, 0, 0, 1, 1};  // 4357 -> 5786
        case 162: return CroftTwo{18, 9, 32, 3, 0, 0, 1, 0};  // 3840 -> 5455
        case 180: return CroftTwo{10, 10, 16, 5, 1, 0, 1, 0};  // 4151 -> 5122
        case 192: return CroftTwo{8, 8, 32, 2, 0, 0, 1, 0};  // 4551 -> 5243
        case 200: return CroftTwo{8, 8, 16, 5, 0, 0, 1, 1};  // 4063 -> 5118
        case 216: return CroftTwo{9, 9, 32, 2, 0, 0, 1, 0};  // 4254 -> 5127
        case 225: return CroftTwo{15, 15, 16, 4, 1, 0, 1, 1};  // 4299 -> 4911
        case 240: return CroftTwo{12, 12, 16, 3, 1, 0, 1, 0};  // 4690 -> 5090
        case 243: return CroftTwo{9, 9, 16, 4, 1, 0, 1, 1};  // 4290 -> 4829
        case 250: return CroftTwo{10, 10, 32, 2, 0, 0, 1, 1};  // 3404 -> 4872
        case 256: return CroftTwo{16, 16, 16, 3, 0, 0, 1, 1};  // 4458 -> 5094
        case 270: return CroftTwo{18, 18, 16, 3, 0, 0, 1, 1};  // 3456 -> 4929
        case 288: return CroftTwo{12, 12, 16, 3, 0, 0, 1, 0};  // 3723 -> 5138
        case 300: return CroftTwo{12, 12, 16, 3, 0, 0, 1, 1};  // 3623 -> 4868
        case 320: return CroftTwo{20, 20, 16, 3, 1, 0, 1, 1};  // 3562 -> 4998
        case 324: return CroftTwo{12, 12, 16, 3, 0, 0, 1, 1};  // 3560 -> 4963
        case 360: return CroftTwo{24, 24, 16, 2, 0, 0, 1, 0};  // 3777 -> 4674
        case 375: return CroftTwo{25, 25, 16, 2, 0, 0, 1, 1};  // 3582 -> 4358
        case 384: return CroftTwo{24, 24, 16, 2, 0, 0, 1, 0};  // 3855 -> 4872
        case 400: return CroftTwo{25, 25, 16, 2, 0, 0, 1, 0};  // 3821 -> 4630
        case 405: return CroftTwo{27, 27, 16, 2, 0, 0, 1, 1};  // 3716 -> 4496
        case 432: return CroftTwo{27, 27, 16, 2, 1, 0, 1, 1};  // 3908 -> 4718
        case 450: return CroftTwo{25, 18, 16, 2, 1, 0, 1, 1};  // 3282 -> 4348
        case 480: return CroftTwo{30, 16, 16, 2, 1, 0, 1, 1};  // 3913 -> 4584
        case 486: return CroftTwo{27, 27, 16, 2, 0, 0, 1, 1};  // 3232 -> 4403
        case 500: return CroftTwo{20, 25, 16, 2, 0, 0, 1, 1};  // 3026 -> 4216
        case 512: return CroftTwo{32, 16, 16, 2, 0, 0, 1, 1};  // 3552 -> 4630
        case 540: return CroftTwo{20, 27, 16, 2, 1, 0, 1, 0};  // 2999 -> 3689
        case 576: return CroftTwo{24, 24, 16, 2, 1, 0, 1, 1};  // 2949 -> 3817
        case 600: return CroftTwo{25, 25, 16, 2, 0, 0, 1, 1};  // 2699 -> 3638
        case 625: return CroftTwo{25, 25, 16, 1, 1, 0, 1, 0};  // 2716 -> 3204
        case 640: return CroftTwo{32, 32, 16, 1, 1, 0, 1, 0};  // 2801 -> 3569
        case 648: return CroftTwo{24, 27, 16, 1, 1, 0, 1, 0};  // 2751 -> 3520
        case 675: return CroftTwo{27, 27, 16, 1, 1, 0, 1, 0};  // 2789 -> 3333
        case 720: return CroftTwo{24, 30, 16, 1, 1, 0, 1, 0};  // 2864 -> 3577
        case 729: return CroftTwo{27, 27, 16, 1, 1, 0, 1, 0};  // 2732 -> 3390
        case 750: return CroftTwo{30, 30, 16, 1, 1, 0, 1, 0};  // 2747 -> 3340
        case 768: return CroftTwo{32, 32, 16, 1, 1, 0, 1, 0};  // 2819 -> 3700
        case 800: return CroftTwo{32, 32, 16, 1, 1, 0, 1, 0};  // 2672 -> 3618
        case 810: return CroftTwo{30, 30, 16, 1, 1, 0, 1, 0};  // 2665 -> 3492
        case 864: return CroftTwo{27, 32, 16, 1, 1, 0, 1, 0};  // 2761 -> 3630
        case 900: return CroftTwo{30, 30, 16, 1, 1, 0, 1, 0};  // 2672 -> 3482
        case 960: return CroftTwo{32, 32, 16, 1, 1, 0, 1, 0};  // 2465 -> 3645
        case 1024: return CroftTwo{32, 32, 16, 1, 0, 0, 1, 0};  // 2532 -> 3715
        default: return CroftTwo{0, 0, 0, 0, 0, 0, 0, 0};
    }
}
CROFT_HD constexpr int croft_two_conv_smem(const CroftTwo& k, int n) { return ((k.stage ? (n + 1) / 2 * 2 : 0) + k.w * n) * 8 + k.w * n * 4; }

// Shared memory: [twiddles when staged][tile].
CROFT_HD constexpr int croft_two_pad(int n) { return (n + 1) / 2 * 2; }
CROFT_HD constexpr int croft_two_smem(const CroftTwo& k, int n, bool row) {
    if (k.ctas == 2) return n / k.r1 * ((k.r1 + 1) / 2) * k.w * 8;
    return ((k.stage ? croft_two_pad(n) : 0) + k.w * (row ? k.ld : n)) * 8;
}
