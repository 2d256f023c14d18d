// spot_tail.cuh -- the stages of the 32-point tensor-core spot kernels that follow the first
// transfer-domain stage, on the CUDA cores, for one subaperture owned by one warp
// (Sec. 4 LGS SH: elongation by the sodium kernel, binning, noise-added image,
// centroid), and the noise pass's noise and centroid.  The FP32 kernel with a warp per
// subaperture takes the small helpers only (packed arithmetic, warp sums).
//
//   M[dy][dx] = Kt[dy][dx] sum_k Ga(dy, k) T[k][dx]       (k = lane: a 32-point DFT)
//   Q[iy][dx] = sum_dy G(dy, iy) M[dy][dx]                 (an nd-point DFT over dy)
//   B[iy][ix] = Re sum_dx Q[iy][dx] G[dx][ix]              (lane = iy, column half)
// with Ga(dy, k) = exp(+2 pi i (k - cN) dy / N) = ph(dy) w^(k dy), w = exp(2 pi i / N),
// ph(dy) = exp(-2 pi i cN dy / N), and G(dy, i) = sum_{r<b} exp(-2 pi i (b i + r - cN) dy / N)
// (conjugated for dy < 0).  The sum over k is a DFT of each column across the lanes: radix 2,
// decimation in frequency, one shuffle per stage and component; lane i ends with frequency
// bitrev5(i).  Kt carries 1/N^2 and the Hermitian weight c_dx, so B is the binned elongated
// spot.  Since N = b nd, G(dy, i) = h(dy) v^(i dy) with h(dy) = sum_{r<b} exp(-2 pi i (r - cN)
// dy / N) and v = exp(-2 pi i / nd): Q is the nd-point DFT of m[j] = sum_{dy = j mod nd} h(dy)
// M[dy][dx].  The lanes i and i ^ 1 hold the frequencies f and f + 16 (the same j, since
// nd = 16), so one shuffle folds them, and the positions p = i >> 1 hold j = bitrev4(p): a
// decimation-in-time DFT across the positions ends with Q[p] in natural order, the even lane
// of each pair working the first column pairs and the odd lane the rest.  The lane pair then swaps
// its halves, so that both lanes hold row p of Q, and the even lane forms the columns ix < nd/2 of
// B, the odd lane their mirrors nd - 1 - ix: G(dx, nd-1-ix) = conj G(dx, ix), so every lane
// multiplies by the same numbers, which come from the kernel's parameters (the constant port) and
// not from shared memory.  Then E = photons fill B / sum B, C = Poisson(E) + ron z (or E), and the
// centre of gravity.
#pragma once
#include "internal.h"
#include "noise.cuh"

namespace gbwfs {
namespace tail {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr int kFftTable = 11 * 32;  // float2: five stages of twiddles, ph h(dy), four more stages, ph* h(dy)

// Per-lane DFT constants: entry s * 32 + lane (s < 5, span h = 16 >> s) is 1 for the upper
// lane of a butterfly and w^((lane mod h) 16 / h) for the lower; entry 5 * 32 + lane is
// ph(dy) h(dy) = sum_{r<2} exp(-2 pi i r dy / 32) of the lane's output frequency dy when
// |dy| < n, else 0; entry (6 + s) * 32 + lane (s < 4, span q = 2^s in positions p = lane >> 1)
// is 1 for the upper position of a butterfly and exp(-2 pi i (p mod q) / 2q) for the lower; entry
// 10 * 32 + lane is ph(dy)* h(dy) = sum_{r<2} exp(-2 pi i (r + 1) dy / 32) for |dy| < n, else 0.
// Call from every thread of the block.
template <int n>
__device__ __forceinline__ void fill_fft_table(float2 *tab, int tid, int nthreads) {
    for (int i = tid; i < kFftTable; i += nthreads) {
        const int st = i >> 5, l = i & 31;
        float sn = 0.0f, cs = 1.0f;
        if (st < 5) {
            const int h = 16 >> st;
            if (l & h) sincospif((float)((l & (h - 1)) * (16 / h)) / 16.0f, &sn, &cs);
        } else if (st == 5) {
            const int f = (int)(__brev((unsigned)l) >> 27), dy = f < 16 ? f : f - 32;
            if (dy > -n && dy < n) {
                sincospif((float)(-dy) / 16.0f, &sn, &cs);  // exp(-2 pi i dy / 32)
                cs += 1.0f;
            } else {
                cs = 0.0f;
            }
        } else if (st < 10) {
            const int q = 1 << (st - 6), p = l >> 1;
            if (p & q) sincospif((float)(-(p & (q - 1))) / (float)q, &sn, &cs);
        } else {
            const int f = (int)(__brev((unsigned)l) >> 27), dy = f < 16 ? f : f - 32;
            cs = 0.0f;
            if (dy > -n && dy < n) {
                float s1, c1, s2, c2;
                sincospif((float)(-dy) / 16.0f, &s1, &c1);
                sincospif((float)(-2 * dy) / 16.0f, &s2, &c2);
                sn = s1 + s2;
                cs = c1 + c2;
            }
        }
        tab[i] = make_float2(cs, sn);
    }
}

// Packed FP32x2 arithmetic (one instruction for two lanes of values, each rounded as the scalar
// operation): the column pairs (dx, dx + 1) of the tail travel together.
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// K~ of a subaperture (column pairs first, so that a warp's read is contiguous) for this lane's
// frequency: the entries its share of the elongation stage takes (rows past the band read the nearest
// row and are multiplied by zero).
template <int n>
__device__ __forceinline__ void load_ktil(const float2 *kt, int lane, float4 (&kq)[n / 2]) {
    const int f = (int)(__brev((unsigned)lane) >> 27), dy = f < 16 ? f : f - 32;
    const int dyi = min(max(dy + n - 1, 0), 2 * n - 2);
    const float4 *src = reinterpret_cast<const float4 *>(kt) + dyi;
#pragma unroll
    for (int c = 0; c < n / 2; ++c) kq[c] = __ldg(src + c * (2 * n - 1));
}

constexpr int kBScratch = 272;  // floats: the 16 x 16 image, its lower half 16 words off

// The first part of the elongation stage.  T: this lane's row k = lane of the first stage (T[k][dx],
// dx < n); on return Tr[c], Ti[c] are the parts of sum_k w^(k dy) T[k][dx] for the lane's frequency dy
// and the columns dx = 2c, 2c + 1.  fft: the table above.
template <int n>
__device__ __forceinline__ void lane_dft(const float2 (&T)[n], const float2 *fft, int lane, float2 (&Tr)[n / 2],
                                         float2 (&Ti)[n / 2]) {
    constexpr int P = n / 2;
    static_assert(n <= 16, "frequencies |dy| < n must be distinct modulo 32");
    static_assert(n % 2 == 0, "columns travel in pairs");
    // columns as pairs: Tr[c] = (re 2c, re 2c+1), Ti[c] = (im 2c, im 2c+1)
#pragma unroll
    for (int c = 0; c < P; ++c) {
        Tr[c] = make_float2(T[2 * c].x, T[2 * c + 1].x);
        Ti[c] = make_float2(T[2 * c].y, T[2 * c + 1].y);
    }
    // M: DFT over the lanes, five radix-2 stages
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int h = 16 >> st;
        const float2 sg = dup2((lane & h) ? -1.0f : 1.0f);
        const float2 tw = fft[st * 32 + lane];
        const float2 twx = dup2(tw.x), twy = dup2(tw.y), ntwy = dup2(-tw.y);
#pragma unroll
        for (int c = 0; c < P; ++c) {
            const float2 tr = make_float2(__shfl_xor_sync(0xffffffffu, Tr[c].x, h),
                                          __shfl_xor_sync(0xffffffffu, Tr[c].y, h));
            const float2 ti = make_float2(__shfl_xor_sync(0xffffffffu, Ti[c].x, h),
                                          __shfl_xor_sync(0xffffffffu, Ti[c].y, h));
            const float2 sr = fma2(sg, Tr[c], tr), si = fma2(sg, Ti[c], ti);
            Tr[c] = fma2(si, ntwy, mul2(sr, twx));
            Ti[c] = fma2(si, twx, mul2(sr, twy));
        }
    }
}

// The rest, from lane_dft's Tr, Ti (consumed).  ph: the lane's entry 5 of the table; with Ti negated and
// entry 10 instead, the stage takes the conjugate of the spot's transfer-domain image, which is that
// of the spot mirrored about its centre: the spot of the negated wavefront.  kq: load_ktil.  Gc:
// uniform G for ix < nd/2, entry ix (n/2) + c holds the columns dx = 2c, 2c + 1 as (re, re, -im, -im)
// (ShArgs::Gc).  Bs is per-warp scratch (kBScratch floats, 16-byte aligned).
// On return Bv[j] = B[half * nd/2 + j][ix] for lane = half * 16 + ix.
template <int n, int nd>
__device__ __forceinline__ void lgs_binned(float2 (&Tr)[n / 2], float2 (&Ti)[n / 2], const float2 ph, float *Bs,
                                           const float2 *fft, const float4 *Gc, const float4 (&kq)[n / 2], int lane,
                                           float (&Bv)[nd / 2]) {
    constexpr int P = n / 2, PH = (P + 1) / 2;
    static_assert(nd == 16, "the detector tile maps to 16 lanes x 2 half-warps");
    // h(dy) M[dy] for the lane's frequency (zero outside the band |dy| < n, through the table),
    // then folded with the lane holding dy -/+ 16
    {
        const float2 phx = dup2(ph.x), phy = dup2(ph.y), nphy = dup2(-ph.y);
#pragma unroll
        for (int c = 0; c < P; ++c) {
            const float2 xr = fma2(Ti[c], nphy, mul2(Tr[c], phx));
            const float2 xi = fma2(Ti[c], phx, mul2(Tr[c], phy));
            const float2 kr = make_float2(kq[c].x, kq[c].z), ki = make_float2(kq[c].y, kq[c].w);
            const float2 mr = fma2(xi, make_float2(-ki.x, -ki.y), mul2(xr, kr));
            const float2 mi = fma2(xi, kr, mul2(xr, ki));
            Tr[c] = __fadd2_rn(mr, make_float2(__shfl_xor_sync(0xffffffffu, mr.x, 1),
                                               __shfl_xor_sync(0xffffffffu, mr.y, 1)));
            Ti[c] = __fadd2_rn(mi, make_float2(__shfl_xor_sync(0xffffffffu, mi.x, 1),
                                               __shfl_xor_sync(0xffffffffu, mi.y, 1)));
        }
    }
    // Q: a 16-point DFT across the positions p = lane >> 1 (input bit-reversed, output in
    // natural order), four radix-2 decimation-in-time stages; the even lane of a position
    // takes the column pairs [0, PH), the odd lane the rest
    const int par = lane & 1;
    float2 Wr[PH], Wi[PH];
#pragma unroll
    for (int j = 0; j < PH; ++j) {
        const int c1 = PH + j;
        const float2 zr = c1 < P ? Tr[c1 < P ? c1 : 0] : make_float2(0.0f, 0.0f);
        const float2 zi = c1 < P ? Ti[c1 < P ? c1 : 0] : make_float2(0.0f, 0.0f);
        Wr[j] = par ? zr : Tr[j];
        Wi[j] = par ? zi : Ti[j];
    }
#pragma unroll
    for (int st = 0; st < 4; ++st) {
        const int q = 1 << st;
        const float2 sg = dup2(((lane >> 1) & q) ? -1.0f : 1.0f);
        const float2 tw = fft[(6 + st) * 32 + lane];
        const float2 twx = dup2(tw.x), twy = dup2(tw.y), ntwy = dup2(-tw.y);
#pragma unroll
        for (int j = 0; j < PH; ++j) {
            // the lower position's value times its twiddle; then upper = own + partner's,
            // lower = partner's - own
            float2 vr = Wr[j], vi = Wi[j];
            if (st > 0) {  // the first stage's twiddles are all 1
                vr = fma2(Wi[j], ntwy, mul2(Wr[j], twx));
                vi = fma2(Wi[j], twx, mul2(Wr[j], twy));
            }
            const float2 pr = make_float2(__shfl_xor_sync(0xffffffffu, vr.x, 2 * q),
                                          __shfl_xor_sync(0xffffffffu, vr.y, 2 * q));
            const float2 pi = make_float2(__shfl_xor_sync(0xffffffffu, vi.x, 2 * q),
                                          __shfl_xor_sync(0xffffffffu, vi.y, 2 * q));
            Wr[j] = fma2(sg, vr, pr);
            Wi[j] = fma2(sg, vi, pi);
        }
    }
    // row iy = lane >> 1 of Q in both lanes of the pair; the odd lane's columns are mirrored, which
    // changes the sign of Im G: taken into Im Q
    const float2 sgn = dup2(par ? -1.0f : 1.0f);
    float2 qr[P], qi[P];
    {
        float2 pr[PH], pi[PH];
#pragma unroll
        for (int j = 0; j < PH; ++j) {
            Wi[j] = mul2(Wi[j], sgn);
            pr[j] = make_float2(__shfl_xor_sync(0xffffffffu, Wr[j].x, 1), __shfl_xor_sync(0xffffffffu, Wr[j].y, 1));
            pi[j] = make_float2(__shfl_xor_sync(0xffffffffu, Wi[j].x, 1), __shfl_xor_sync(0xffffffffu, Wi[j].y, 1));
        }
#pragma unroll
        for (int c = 0; c < P; ++c) {
            const int j = c < PH ? c : c - PH;
            const bool mine = c < PH ? !par : par;
            qr[c] = make_float2(mine ? Wr[j].x : pr[j].x, mine ? Wr[j].y : pr[j].y);
            qi[c] = make_float2(mine ? Wi[j].x : -pi[j].x, mine ? Wi[j].y : -pi[j].y);
        }
    }
    // B[iy][ix] = Re sum_dx Q[iy][dx] G[dx][ix], even and odd columns dx summed apart
    float bt[nd / 2];
#pragma unroll
    for (int j = 0; j < nd / 2; ++j) {
        float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int c = 0; c < P; ++c) {
            const float4 g = Gc[j * P + c];
            s = fma2(qr[c], make_float2(g.x, g.y), fma2(qi[c], make_float2(g.z, g.w), s));
        }
        bt[j] = s.x + s.y;
    }
    // to lane = (row half, column): 16-byte words w of row iy at w ^ (bit 1 of iy), so that neither
    // side meets a bank twice
    const int iy = lane >> 1, sw = (iy >> 1) & 1;
    float *row = Bs + iy * nd + (iy >= 8 ? 16 : 0);
    __syncwarp();  // earlier reads of the scratch by other lanes are done
    float4 *row4 = reinterpret_cast<float4 *>(row);
    if (par) {
        row4[3 ^ sw] = make_float4(bt[3], bt[2], bt[1], bt[0]);
        row4[2 ^ sw] = make_float4(bt[7], bt[6], bt[5], bt[4]);
    } else {
        row4[0 ^ sw] = make_float4(bt[0], bt[1], bt[2], bt[3]);
        row4[1 ^ sw] = make_float4(bt[4], bt[5], bt[6], bt[7]);
    }
    __syncwarp();
    const int ix = lane & 15, half = lane >> 4;
#pragma unroll
    for (int j = 0; j < nd / 2; ++j) {
        const int y = half * (nd / 2) + j;
        Bv[j] = Bs[y * nd + half * 16 + ((((ix >> 2) ^ ((y >> 1) & 1)) << 2) | (ix & 3))];
    }
}

// NGS: b x b binning of the spot image rows Iw ([32][33] floats).
template <int nd>
__device__ __forceinline__ void ngs_binned(const float *Iw, int lane, float (&Bv)[nd / 2]) {
    constexpr int N = 32, b = N / nd;
    const int ix = lane & 15, half = lane >> 4;
#pragma unroll
    for (int j = 0; j < nd / 2; ++j) {
        const int iy = half * (nd / 2) + j;
        float s = 0.0f;
        if (ix < nd) {
#pragma unroll
            for (int r = 0; r < b; ++r)
#pragma unroll
                for (int c = 0; c < b; ++c) s += Iw[(b * iy + r) * (N + 1) + b * ix + c];
        }
        Bv[j] = s;
    }
}

// Photometry: ev[j] = E of detector row half * nd/2 + j, column ix (lane = half * 16 + ix),
// E = photons fill B / sum B.
template <int nd>
__device__ __forceinline__ void expected(const float (&Bv)[nd / 2], const WfsDesc &W, int v, int lane,
                                         float (&ev)[nd / 2]) {
    constexpr int J = nd / 2;
    const int ix = lane & 15;
    float sb = 0.0f;
    if (ix < nd) {
#pragma unroll
        for (int j = 0; j < J; ++j) sb += Bv[j];
    }
    sb = warp_sum(sb);
    const float scale = sb > 0.0f ? W.photons * __ldg(W.fill + v) / sb : 0.0f;
#pragma unroll
    for (int j = 0; j < J; ++j) ev[j] = scale * Bv[j];
}

// Stores E of subaperture v to D.st_E (when given).
template <int nd>
__device__ __forceinline__ void store_expected(const float (&ev)[nd / 2], const WfsDesc &W, const InstDyn &D,
                                               int v, int lane) {
    constexpr int nd2 = nd * nd, J = nd / 2;
    const int ix = lane & 15, half = lane >> 4;
    if (!D.st_E || ix >= nd) return;
    float *st_E = D.st_E + W.det_off + (size_t)v * nd2;
#pragma unroll
    for (int j = 0; j < J; ++j) st_E[(half * J + j) * nd + ix] = ev[j];
}

// The detector row of a lane's slot j in the noise pass.  Without noise, the layout of expected().
// With noise, slots m and m + nd/4 (searched together) hold neighbouring rows, and the two
// half-warps take rows mirrored about the centre, so that the rows a warp searches together are
// about as bright: its search lasts as long as its brightest pixel's.
template <int nd>
__device__ __forceinline__ int noise_row(int j, int half, bool noise) {
    constexpr int J = nd / 2;
    if (!noise) return half * J + j;
    const int r = 2 * (j & (J / 2 - 1)) + j / (J / 2);
    return half ? nd - 1 - r : r;
}

// Noise and the centroid of subaperture v of WFS W from its expected image ev (row noise_row of
// slot j); lane 0 writes the slopes.  rk2: fill_recip_pairs.  One generator block per pixel pair;
// each exchange between the lane pair is followed by both pixels' inversion searches, and the rare
// pixels with E >= 16 go last through one PTRS call site.  Call from the whole warp.
template <int nd>
__device__ __forceinline__ void noise_centroid(const float (&ev)[nd / 2], const WfsDesc &W, const InstDyn &D,
                                               uint64_t seed, int v, int lane, const float4 *rk2) {
    constexpr int nd2 = nd * nd, J = nd / 2;
    static_assert(nd == 16, "pixel pairs are the lane pairs (ix, ix + 1) of a 16-lane row");
    const int ix = lane & 15, half = lane >> 4;
    const bool noise = D.noise != 0;
    const float cd = 0.5f * (float)(nd - 1);
    const uint32_t tlo = (uint32_t)__double_as_longlong(D.t);
    const uint32_t thi = (uint32_t)((unsigned long long)__double_as_longlong(D.t) >> 32);
    float *st_C = D.st_C ? D.st_C + W.det_off + (size_t)v * nd2 : nullptr;
    float sc = 0.0f, sx = 0.0f, sy = 0.0f;
    float cv[J];
    if (noise) {
        // Pixel pairs (2m, 2m + 1) are the lanes (ix, ix + 1) of one row: the even lane forms the
        // pair blocks of its first J/2 slots, the odd lane those of its last J/2, and each hands
        // its partner that pixel's deviate and uniform; slots m and m + J/2 are then sampled
        // together.
        const uint32_t pix0 = (uint32_t)(v * nd2 + ix);
        const int par = ix & 1;
        uint32_t big = 0;
        float z[J];
#pragma unroll
        for (int m = 0; m < J / 2; ++m) {
            const uint32_t pix = pix0 + (uint32_t)(nd * (par ? noise_row<nd>(m + J / 2, half, true)
                                                             : noise_row<nd>(m, half, true)));
            const uint4 r = pair_stream(seed, pix, (uint32_t)W.gs_index, tlo, thi).block(0);
            float ze, zd;
            box_muller_pair(r.x, r.y, ze, zd);
            const float zr = __shfl_xor_sync(0xffffffffu, par ? ze : zd, 1);
            const float ur = __shfl_xor_sync(0xffffffffu, philox_unit(par ? r.z : r.w), 1);
            const float zo = par ? zd : ze, uo = philox_unit(par ? r.w : r.z);
            z[m] = par ? zr : zo;
            z[m + J / 2] = par ? zo : zr;
            const float ea = ev[m], eb = ev[m + J / 2];
            if (ea >= 16.0f) big |= 1u << m;
            if (eb >= 16.0f) big |= 1u << (m + J / 2);
            const float2 e = make_float2(inversion_mean(ea), inversion_mean(eb));
            int ka, kb;
            poisson_inversion_pair(e, make_float2(par ? ur : uo, par ? uo : ur),
                                   make_float2(expf(-e.x), expf(-e.y)), rk2, ka, kb);
            cv[m] = (float)ka + W.read_noise * z[m];
            cv[m + J / 2] = (float)kb + W.read_noise * z[m + J / 2];
        }
        while (big) {  // PTRS: one call site, rare
            const int j = __ffs(big) - 1;
            big &= big - 1;
            float e = 0.0f, zj = 0.0f;
#pragma unroll
            for (int jj = 0; jj < J; ++jj)
                if (jj == j) {
                    e = ev[jj];
                    zj = z[jj];
                }
            const PairStream q = pair_stream(seed, pix0 + (uint32_t)(nd * noise_row<nd>(j, half, true)),
                                             (uint32_t)W.gs_index, tlo, thi);
            const float c = (float)poisson_ptrs(e, q, par) + W.read_noise * zj;
#pragma unroll
            for (int jj = 0; jj < J; ++jj)
                if (jj == j) cv[jj] = c;
        }
    } else {
#pragma unroll
        for (int j = 0; j < J; ++j) cv[j] = ev[j];
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int iy = noise_row<nd>(j, half, noise), o = iy * nd + ix;
        if (st_C) st_C[o] = cv[j];
        sc += cv[j];
        sx = fmaf((float)ix - cd, cv[j], sx);
        sy = fmaf((float)iy - cd, cv[j], sy);
    }
    sc = warp_sum(sc);
    sx = warp_sum(sx);
    sy = warp_sum(sy);
    if (lane == 0) {
        const bool ok = sc > 0.0f;
        float *sl = D.slopes + W.slope_off;
        sl[2 * v] = ok ? sx / sc : 0.0f;
        sl[2 * v + 1] = ok ? sy / sc : 0.0f;
    }
}

// Photometry, then the centroid of the expected image in place (a measurement without noise); with
// split, the expected image is stored and the noise kernel completes the measurement.  slopes: the
// WFS's.  The sums of the centroid run in noise_centroid's order.  Without noise the image would only
// travel to the noise kernel and back: 16 us of a noise-free ELT frame; a calibration's chunk of 64
// measurements 857 + 148 us -> 869 us in place.
template <int nd>
__device__ __forceinline__ void finish(const float (&Bv)[nd / 2], const WfsDesc &W, const InstDyn &D, int v,
                                       int lane, bool split, float *slopes) {
    constexpr int nd2 = nd * nd, J = nd / 2;
    const int ix = lane & 15, half = lane >> 4;
    float ev[J];
    expected<nd>(Bv, W, v, lane, ev);
    store_expected<nd>(ev, W, D, v, lane);
    if (split) return;
    const float cd = 0.5f * (float)(nd - 1);
    float *st_C = D.st_C ? D.st_C + W.det_off + (size_t)v * nd2 : nullptr;
    float sc = 0.0f, sx = 0.0f, sy = 0.0f;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int iy = half * J + j;
        if (st_C) st_C[iy * nd + ix] = ev[j];
        sc += ev[j];
        sx = fmaf((float)ix - cd, ev[j], sx);
        sy = fmaf((float)iy - cd, ev[j], sy);
    }
    sc = warp_sum(sc);
    sx = warp_sum(sx);
    sy = warp_sum(sy);
    if (lane == 0) {
        const bool ok = sc > 0.0f;
        slopes[2 * v] = ok ? sx / sc : 0.0f;
        slopes[2 * v + 1] = ok ? sy / sc : 0.0f;
    }
}

// The centroid of a binned image without noise and without stage outputs (the push-pull pairs), from the
// differences of pixels mirrored about the centre: d = B[iy][ix] - B[iy][nd-1-ix] and e likewise down the
// columns, so that the sums' roundings are those of the small differences and not of the pixels: the two
// slopes of a pair share what comes before, and would not average it out as two measurements do.  RMS
// error against 64 bits, FP16S, 80 x 80, n = 10: 3.79e-6 of the rows' RMS for two measurements, 3.82e-6 for
// a pair by finish()'s sums, 3.02e-6 by these; 64 modes of it (BF16X3) 1,236 -> 1,191 us.
template <int nd>
__device__ __forceinline__ void centroid(const float (&Bv)[nd / 2], const WfsDesc &W, int v, int lane, float *slopes) {
    constexpr int J = nd / 2;
    static_assert(nd == 16, "columns mirror within 16 lanes, rows across the half-warps");
    const int ix = lane & 15, half = lane >> 4;
    const float cd = 0.5f * (float)(nd - 1);
    float sc = 0.0f, sx = 0.0f, sy = 0.0f;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        sc += Bv[j];
        sx += Bv[j] - __shfl_xor_sync(0xffffffffu, Bv[j], 15);
        sy = fmaf((float)(half * J + j) - cd, Bv[j] - __shfl_xor_sync(0xffffffffu, Bv[J - 1 - j], 16), sy);
    }
    // every pair is counted from both of its ends
    sx = 0.5f * warp_sum(((float)ix - cd) * sx);
    sc = warp_sum(sc);
    sy = 0.5f * warp_sum(sy);
    if (lane == 0) {
        const bool ok = sc > 0.0f && W.photons * __ldg(W.fill + v) > 0.0f;
        slopes[2 * v] = ok ? sx / sc : 0.0f;
        slopes[2 * v + 1] = ok ? sy / sc : 0.0f;
    }
}

}  // namespace tail
}  // namespace gbwfs
