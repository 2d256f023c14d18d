// k_sh_row_slices.cu -- launches of the FP32 spot kernel with a warp per subaperture (k_sh_row.cuh) in the
// LGS per-slice model, after a projection of every (WFS, slice) pair.
#include "k_sh_row.cuh"

namespace gbwfs {

cudaError_t row_slices_launch_shape(const ShArgs &a, LaunchShape *out) {
    // A warp runs its slices one after the other, so it is the latency of a slice that counts: 128
    // registers and two CTAs per SM, or three for n <= 10 where all subapertures then fit at once and
    // would not at two (n = 10, N = 32, 8 slices, spot kernel: 2,828 subapertures 66.3 us at two, 53.7 at
    // three; 1,976: 35.8 and 41.0; 3,852: 66.7 and 94.6; 10,048: 132 and 145 us).
    return row_sizes(a, [&](auto s) {
        using S = decltype(s);
        if constexpr (S::n <= 10)
            if (a.total > kRowWave2 && a.total <= kRowWave3) return row_shape_k<S::n, S::cN, S::cnd, true, 3>(a, out);
        return row_shape_k<S::n, S::cN, S::cnd, true, 2>(a, out);
    });
}

}  // namespace gbwfs
