// self_project.cuh -- one subaperture's OPD straight from the screens, for spot kernels that project
// their own subapertures (Sec. 4 "Open Loop generation"; the arithmetic of the projection kernels:
// layer offsets in FP64, bilinear samples summed over the layers in order, then the uplink tilt).
#pragma once
#include "internal.h"
#include "proj_math.cuh"

namespace gbwfs {

// The geometric term of sodium slice sl in the LGS per-slice model, 1/2 |x - r_L|^2 k_s relative to
// the subaperture centre r_b: k_s ((x - r_b).(r_b - r_L) + 1/2 |x - r_b|^2).
struct SliceTerm {
    float ebx = 0.0f, eby = 0.0f, dxp = 0.0f, c0 = 0.0f;
    __device__ __forceinline__ SliceTerm() {}
    __device__ __forceinline__ SliceTerm(const InstDesc &I, const WfsDesc &W, int v, int n) {
        const int id = __ldg(W.subap + v), sy = id / W.n_sub, sx = id - sy * W.n_sub;
        const float half = 0.5f * (float)(W.n_sub * n - 1);
        c0 = 0.5f * (float)(n - 1);
        dxp = (float)(W.pupil_dx_over_ds * I.ds);
        ebx = ((float)(sx * n) + c0 - half) * dxp - (float)W.launch_x;
        eby = ((float)(sy * n) + c0 - half) * dxp - (float)W.launch_y;
    }
    __device__ __forceinline__ float at(float ks, int p, int q) const {
        const float ux = ((float)q - c0) * dxp, uy = ((float)p - c0) * dxp;
        return ks * fmaf(ux, ebx, fmaf(uy, eby, 0.5f * fmaf(ux, ux, uy * uy)));
    }
};

// The OPD of subaperture v into so[n * n] (shared by the team's threads tid = 0 .. team - 1; the
// caller synchronises), also written to D.opd for slice 0.  lo: the layers' offsets.  A slice sees
// the layers through its own cone (the scale); the offsets are shared.  The geometric term of a
// slice is not added.
__device__ __forceinline__ void self_project(const ShArgs &a, const WfsDesc &W, const InstDesc &I, const InstDyn &D,
                                             const SliceDesc *SD, int sl, int v, int n, const LayerOffs *lo, int tid,
                                             int team, float *so) {
    const int L = proj_layers(I, D), nn = n * n;
    const int S = I.S;
    const bool pow2 = (S & (S - 1)) == 0;
    const int id = __ldg(W.subap + v), sy = id / W.n_sub, sx = id - sy * W.n_sub;
    const float half = 0.5f * (float)(W.n_sub * n - 1);
    float *out = D.opd + W.opd_off + (size_t)v * nn;
    for (int i = tid; i < nn; i += team) {
        const int pp = i / n, qq = i - pp * n;
        const float xr = (float)(sx * n + qq) - half, yr = (float)(sy * n + pp) - half;
        float acc = 0.0f;
        for (int l = 0; l < L; ++l) {
            const LayerOffs L0 = lo[l];
            const float ch = SD ? SD->c[sl][l].x : L0.c, cl = SD ? SD->c[sl][l].y : L0.cl;
            int ou, ov, i0, i1, j0, j1;
            float fx, gy;
            screen_offset(ch, cl, L0.fu, xr, ou, fx);
            screen_offset(ch, cl, L0.fv, yr, ov, gy);
            wrap_pair(L0.bu + ou, S, pow2, i0, i1);
            wrap_pair(L0.bv + ov, S, pow2, j0, j1);
            if (!guard(i0 >= 0 && i1 < S && i1 >= 0 && j0 >= 0 && j1 < S && j1 >= 0 && i0 < S && j0 < S, a.status))
                continue;
            const float *scr = layer_screen(I, D, l);
            const float *r0 = scr + (size_t)j0 * S, *r1 = scr + (size_t)j1 * S;
            const float s00 = __ldg(r0 + i0), s01 = __ldg(r0 + i1);
            const float s10 = __ldg(r1 + i0), s11 = __ldg(r1 + i1);
            const float top = fmaf(fx, s01 - s00, s00);
            const float bot = fmaf(fx, s11 - s10, s10);
            acc += fmaf(gy, bot - top, top);
        }
        if (W.uplink) acc += fmaf(W.uplink->x, xr, W.uplink->y * yr);
        if (sl == 0) out[i] = acc;
        so[i] = acc;
    }
}

}  // namespace gbwfs
