// k_sh_row.cu -- launches of the FP32 spot kernel with a warp per subaperture (k_sh_row.cuh), one
// wavefront per subaperture; k_sh_row_slices.cu holds its per-slice variant.
#include "k_sh_row.cuh"

namespace gbwfs {

cudaError_t row_slices_launch_shape(const ShArgs &a, LaunchShape *out);

bool sh_row_supported(int n, int N) { return n >= 3 && n <= 16 && N <= 32; }

cudaError_t row_launch_shape(const ShArgs &a, LaunchShape *out) {
    if (a.slice_opd_stride > 0) return row_slices_launch_shape(a, out);
    // Three CTAs per SM for n <= 10 (80 registers), two above.  A 32-point launch whose warps all fit at
    // two CTAs waits for its slowest chain instead of the pipes: it takes 128 registers, without spills
    // (one LGS of 30 x 30, n = 10, three layers: frame 24.7 -> 18.5 us; 20 x 20: 16.5 and 16.4 us).
    return row_sizes(a, [&](auto s) {
        using S = decltype(s);
        if constexpr (S::cN == 32)
            if (a.total <= kRowWave2) return row_shape_k<S::n, S::cN, S::cnd, false, 2>(a, out);
        return row_shape_k<S::n, S::cN, S::cnd, false, S::n <= 10 ? 3 : 2>(a, out);
    });
}

}  // namespace gbwfs
