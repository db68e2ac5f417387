// croft_two.cu - instantiates the two-stage pass kernels (croft_two_stage_kernel.cuh).
// Compiled once per group of axis lengths (-DCROFT_TWO_GROUP=0..3).
#include "croft_sizes.h"
#include "croft_two_stage_kernel.cuh"

#ifndef CROFT_TWO_GROUP
#error "compile with -DCROFT_TWO_GROUP=<0..3>"
#endif

#define CROFT_CAT_(a, b) a##b
#define CROFT_CAT(a, b) CROFT_CAT_(a, b)

namespace croft {

template <int N, bool LONG>
static pass_fn two_col_at() {
    if constexpr (croft_two_col(N, LONG).ctas == 2) return croft_two_pair_kernel<N, LONG>;
    else if constexpr (croft_two_col(N, LONG).r1 != 0) return croft_two_col_kernel<N, LONG>;
    else return nullptr;
}
template <int N>
static pass_fn two_col(bool long_stride) {
    if constexpr (croft_two_split_by_stride(N)) {
        if (long_stride) return two_col_at<N, true>();
    }
    return two_col_at<N, false>();
}

template <int N>
static pass_fn two_row() {
    if constexpr (croft_two_row(N).r1 != 0) return croft_two_row_kernel<N>;
    else return nullptr;
}

pass_fn CROFT_CAT(lookup_two_kernel_group_, CROFT_TWO_GROUP)(int layout, int n, bool long_stride) {
#define CROFT_TWO_CASE(N) \
    case N: return layout == LAYOUT_ROW ? two_row<N>() : two_col<N>(long_stride);
    switch (n) {
        CROFT_CAT(CROFT_SIZES_, CROFT_TWO_GROUP)(CROFT_TWO_CASE)
        default: return nullptr;
    }
#undef CROFT_TWO_CASE
}

}  // namespace croft
