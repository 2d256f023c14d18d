// k_sh_row.cuh -- the plain-FP32 spot kernel of the geometries with N <= 32 DFT points and n <= 16
// pupil pixels per subaperture (Sec. 4 "LGS Shack Hartmann wavefront sensor"): one warp per
// subaperture, lane k owns DFT row k.
//
// The stages are those of k_sh.cu (spot, elongation through the transfer function, binning,
// photometry, noise, centroid), with every centred DFT folded about its centre: a centred matrix has
// F[k][n-1-p] = F[N-1-k][p] = conj F[k][p], so with S = x[p] + x[n-1-p] and D = x[p] - x[n-1-p]
//     sum_p F[k][p] x[p]     = sum_{p < n/2} Re F S + i Im F D = a + b,
//     sum_p F[N-1-k][p] x[p] = a - b,
// i.e. two real products per element of each half in place of four per element of the whole, and
// two outputs for one pass over the inputs.  A middle element is its own mirror: S = x, Im F = 0.
// The four dense stages of a subaperture then cost a quarter of the multiplications:
//   U = F X            lane k: row k of U from the folded pixel rows (shared memory, broadcast)
//   Y = U F^T, |Y|^2   columns m and N-1-m together from the row's folded U (registers)
//   T = I Ga^T         the two intensities folded straight into the row's transform (registers)
//   A = Ga T           dy and -dy together, T's rows folded in shared memory
//   M = K~ A, Q = G^T M   rows iy and nd-1-iy together, M's rows folded
//   B = Re Q G         columns ix and nd-1-ix together
// All products are packed FP32x2 (a scalar factor for both halves costs nothing extra; splitting the
// sums over pairs of summands instead, to avoid it, was slower: 125 against 107 us).
//
// Bound: shared-memory wavefronts (80 % of the pipe) and latency (53 % issue at 24 warps per SM; 2,143
// warp instructions per 32-point LGS subaperture); launches of one wave wait for their chains.  The
// slices have instances of their own: in one body the plain path paid for them with registers (2,377
// instructions, 100 bytes of spills) and a slice for its geometry and samples.  Measured, spot
// kernel alone: ELT frame (27,792 LGS subapertures, n = 10, N = 32) 125.5 us with a kernel of its own for
// N = 32 (row pairs, column quadruples), 107.5 with slices in one body, 97.8 now; 5,056 subapertures of
// n = 6, N = 24 76, 22.1 and 21.4 us, 2 LGS + 1 NGS of 37 x 37, n = 9, N = 21 38.2, 20.7 and 18.2 us and
// 316 NGS subapertures of n = 8, N = 16 with noise 19.5, 16.8 and 15.2 us (the first of each: the
// generic kernel, which forms one output per lane and reads both operands of every product from shared
// memory).  With 8 slices: the ELT frame 398.7 us by the N = 32 kernel, 408 in one body, 334 now; one LGS
// of 30 x 30, n = 10, 35.8, 42.4 and 25.7 us.  The noise runs in place (ELT frame 127.8 us with it: less
// than a pass of its own at 47 us).
#include <mutex>

#include "internal.h"
#include "noise.cuh"
#include "self_project.cuh"
#include "spot_tail.cuh"

namespace gbwfs {

namespace {

using tail::dup2;
using tail::fma2;
using tail::warp_sum;

// Shared memory of a launch: the geometry's folded tables, then one scratch per warp (bytes, all
// 16-byte aligned).
struct RowSmem {
    int F, Y, T, M, Q, B, rk;  // tables
    int warp0, warp_bytes;     // first warp's scratch, size of one
    int r2, lo;                // within a warp's scratch: second region, layer offsets
    int total;
};

// Lanes of the elongation stages: column dx = lane mod n, group g = lane / n < row_groups(n); a group
// owns row_span(n) consecutive rows dy.
__host__ __device__ constexpr int row_groups(int n) { return 32 / n; }
__host__ __device__ constexpr int row_span(int n) { return ((n + row_groups(n) - 1) / row_groups(n) + 1) & ~1; }
// Rows iy of Q per lane and pass.
constexpr int kQRows = 4;

__host__ __device__ constexpr RowSmem row_smem(int n, int N, int nd, int warps, bool project) {
    const int H = (n + 1) / 2, H2 = (H + 1) & ~1, hN = (N + 1) / 2, hd = (nd + 1) / 2, nT = n | 1;
    const int mrows = row_groups(n) * row_span(n), qrows = (hd + kQRows - 1) / kQRows * kQRows;
    RowSmem s{};
    int o = 0;
    s.F = o;   // [H][N] Re F[k][p] for k < N/2, Im F[N-1-k][p] from there on
    o += (H * N * 4 + 15) & ~15;
    s.Y = o;   // [hN][H2] complex: F[m][q]
    o += hN * H2 * 8;
    s.T = o;   // [hN][H] (re, re, im, im) of Ga[dx][m], Ga[dx + 1][m] (zero past n)
    o += hN * H * 16;
    s.M = o;   // [hN][mrows] complex: Ga[dy][k] (zero past n)
    o += hN * mrows * 8;
    s.Q = o;   // [n][qrows] complex: G[dy][iy] (zero past nd/2)
    o += n * qrows * 8;
    s.B = o;   // [2H][hd] complex: G[dx][ix] (zero past n)
    o += H * hd * 16;
    s.rk = o;  // RN(1/k) for the Poisson searches
    o += kRecipTable / 2 * 16;
    s.warp0 = o;
    // first region: the folded field, then an NGS's spot rows, or the folded T, then Q
    int r1 = 2 * H * H * 16;
    const int rows = (N * (N + 1) * 4 + 15) & ~15, ts = hN * nT * 16, q = nd * H * 16;
    r1 = r1 > rows ? r1 : rows;
    r1 = r1 > ts ? r1 : ts;
    r1 = r1 > q ? r1 : q;
    // second region: a self-projected OPD, then the folded M, then the binned image
    int r2 = n * nT * 16;
    const int so = (n * n * 4 + 15) & ~15, b = (nd * nd * 4 + 15) & ~15;
    r2 = r2 > so ? r2 : so;
    r2 = r2 > b ? r2 : b;
    s.r2 = r1;
    s.lo = r1 + r2;
    s.warp_bytes = r1 + r2 + (project ? ((int)(sizeof(LayerOffs) * kMaxProjLayers) + 15) & ~15 : 0);
    s.total = o + warps * s.warp_bytes;
    return s;
}

}  // namespace

// cN, cnd: the DFT and detector sizes where they are compiled in (the configured geometries: the
// table and scratch offsets are then constants), else 0.  kSl: the LGS per-slice model on projected
// slices (ShArgs::slice_opd_stride); else one wavefront, projected before or, with ShArgs::project, here.
// kCtas: CTAs of eight warps the registers are budgeted for (row_shape).
template <int n, int cN, int cnd, bool kSl, int kCtas>
__global__ void __launch_bounds__(256, kCtas) k_sh_row(const __grid_constant__ ShArgs a) {
    constexpr int H = (n + 1) / 2, H2 = (H + 1) & ~1, C = 2 * H, nT = n | 1, nn = n * n;
    constexpr int G = row_groups(n), R = row_span(n), MR = G * R;
    const int N = cN ? cN : a.N, nd = cnd ? cnd : a.nd;
    const int hN = (N + 1) >> 1, hd = (nd + 1) >> 1, nd2 = nd * nd, QR = (hd + kQRows - 1) / kQRows * kQRows;
    // N a multiple of 4: the columns m and m + N/2 fold once more in T (Ga[d][m + N/2] = (-1)^d Ga[d][m])
    constexpr bool kQuad = cN > 0 && cN % 4 == 0;
    constexpr int kUnroll = kSl ? 8 : 2;  // of that loop: a slice's chains are what its warp waits for (n = 10: 91 -> 83 us)
    extern __shared__ __align__(16) unsigned char row_sm[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const RowSmem L = row_smem(n, N, nd, nw, a.project != 0);
    float *tF = reinterpret_cast<float *>(row_sm + L.F);
    float2 *tYe = reinterpret_cast<float2 *>(row_sm + L.Y), *tMe = reinterpret_cast<float2 *>(row_sm + L.M);
    float2 *tQe = reinterpret_cast<float2 *>(row_sm + L.Q), *tB = reinterpret_cast<float2 *>(row_sm + L.B);
    float *tTe = reinterpret_cast<float *>(row_sm + L.T);
    float4 *rk2 = reinterpret_cast<float4 *>(row_sm + L.rk);
    const float4 *tY = reinterpret_cast<const float4 *>(tYe), *tT = reinterpret_cast<const float4 *>(tTe);
    const float4 *tM = reinterpret_cast<const float4 *>(tMe), *tQ = reinterpret_cast<const float4 *>(tQe);
    // global tables: F[q * N + m] = F[m][q], Ga[d * N + k], G[d * nd + i]
    const float2 zero = make_float2(0.0f, 0.0f);
    for (int i = threadIdx.x; i < H * N; i += blockDim.x) {
        const int p = i / N, k = i - p * N;
        tF[i] = k < hN ? a.F[i].x : a.F[p * N + N - 1 - k].y;
    }
    for (int i = threadIdx.x; i < H2 * hN; i += blockDim.x) {
        const int m = i / H2, q = i - m * H2;
        tYe[i] = q < H ? a.F[q * N + m] : zero;
    }
    for (int i = threadIdx.x; i < C * hN; i += blockDim.x) {
        const int m = i / C, d = i - m * C;
        const float2 g = d < n ? a.Ga[d * N + m] : zero;
        float *e = tTe + 4 * (m * H + (d >> 1)) + (d & 1);
        e[0] = g.x;
        e[2] = g.y;
    }
    for (int i = threadIdx.x; i < MR * hN; i += blockDim.x) {
        const int k = i / MR, d = i - k * MR;
        tMe[i] = d < n ? a.Ga[d * N + k] : zero;
    }
    for (int i = threadIdx.x; i < n * QR; i += blockDim.x) {
        const int d = i / QR, x = i - d * QR;
        tQe[i] = x < hd ? a.G[d * nd + x] : zero;
    }
    for (int i = threadIdx.x; i < C * hd; i += blockDim.x) {
        const int d = i / hd, x = i - d * hd;
        tB[i] = d < n ? a.G[d * nd + x] : zero;
    }
    fill_recip_pairs(rk2, threadIdx.x, blockDim.x);
    __syncthreads();
    wait_prior_grid();

    unsigned char *scratch = row_sm + L.warp0 + wib * L.warp_bytes;
    float4 *X4 = reinterpret_cast<float4 *>(scratch), *TS = X4;  // first region
    float2 *Qs = reinterpret_cast<float2 *>(scratch);
    float *Iw = reinterpret_cast<float *>(scratch);
    float4 *MS = reinterpret_cast<float4 *>(scratch + L.r2);  // second region
    float *B = reinterpret_cast<float *>(MS), *so = B;
    LayerOffs *lo = reinterpret_cast<LayerOffs *>(scratch + L.lo);
    // the mirror row N - 1 - k; the lanes k < N/2 form the half sum over S, the mirror lanes that over D
    const int mirror = lane < N ? N - 1 - lane : lane;
    const bool own = mirror == lane, lower = lane < hN;
    const int dx = lane % n, grp = lane / n;
    const float cd = 0.5f * (float)(nd - 1);
    const int rcp_nd = (65536 + nd - 1) / nd;  // o / nd = o rcp >> 16 for o < nd^2 <= 1024

    // Work split: warp i starts with subaperture i; with a.work and more subapertures than warps,
    // lane 0 draws one ticket per subaperture (issued at the top, used at the bottom).
    const int nwarps = gridDim.x * nw;
    const bool tickets = a.work && a.total > nwarps;
    for (int g = blockIdx.x * nw + wib; g < a.total;) {
        int ticket = 0;
        if (tickets && lane == 0) ticket = atomicAdd(a.work, 1);
        const WfsDesc &W = a.wfs[find_wfs(a.wfs, a.n_wfs, g)];
        const InstDyn &D = a.dyn[W.inst];
        const int v = g - W.subap_begin;
        __syncwarp();
        if (guard(v >= 0 && v < W.n_valid, a.status)) {  // uniform over the warp
            const bool lgs = W.is_lgs != 0;
            // LGS per-slice model: one wavefront and one DFT per sodium slice, the weighted spots
            // summed (their transform is linear, so T adds up instead); a natural star has one
            const SliceDesc *SD = kSl ? W.slices : nullptr;
            const int n_sl = SD ? SD->n : 1;
            const InstDesc &I = a.inst[W.inst];
            if (!kSl && a.project) {
                for (int l = lane; l < proj_layers(I, D); l += 32) lo[l] = layer_offsets(I, W, D.t, l);
                __syncwarp();
            }
            const uint32_t *mk = W.mask + (size_t)v * a.mask_words;
            float *stI = D.st_I && lane < N ? D.st_I + W.int_off + (size_t)v * (N * N) + lane * N : nullptr;
            // the lane's samples: elements i = lane + 32 m of the folded field, pixel (p, q) and its mirror
            // (n - 1 - p, q); unlit where either is missing
            constexpr int kF = (H * C + 31) / 32;
            // slices: the samples a slice ahead and their geometric terms kept, where the registers hold them
            // (n <= 12; with n = 16 the spills cost more: 223 against 250 us for 6,456 subapertures of 8 slices)
            constexpr bool kAhead = kSl && kF <= 3;
            const float *opd = D.opd + W.opd_off + (size_t)v * nn;
            float oa[kF], ob[kF], ref;
            bool la[kF], lb[kF];
            struct Pixel {
                int p, q;      // the pixel, or (0, 0)
                int mp, mq;    // its mirror, or (0, 0)
                bool in, two;  // whether there is one
            };
            auto pixel = [&](int m) {
                const int i = lane + 32 * m, p = i / C, q = i - p * C;
                Pixel x;
                x.in = p < H && q < n;
                x.two = x.in && p != n - 1 - p;
                x.p = x.in ? p : 0;
                x.q = x.in ? q : 0;
                x.mp = x.two ? n - 1 - p : 0;
                x.mq = x.two ? q : 0;
                return x;
            };
            auto load = [&](const float *o) {
                ref = __ldg(o);
#pragma unroll
                for (int m = 0; m < kF; ++m) {
                    const Pixel x = pixel(m);
                    oa[m] = __ldg(o + x.p * n + x.q);
                    ob[m] = __ldg(o + x.mp * n + x.mq);
                }
            };
            // the slices' geometric terms of the lane's samples, and of the reference's
            float ga[kF], gb[kF], gr = 0.0f;
            SliceTerm term;
            if (SD) term = SliceTerm(I, W, v, n);
            if (kAhead) {
                load(opd);
                gr = term.at(1.0f, 0, 0);
#pragma unroll
                for (int m = 0; m < kF; ++m) {
                    const Pixel x = pixel(m);
                    ga[m] = term.at(1.0f, x.p, x.q);
                    gb[m] = term.at(1.0f, x.mp, x.mq);
                }
            }
#pragma unroll
            for (int m = 0; m < kF; ++m) {
                const Pixel x = pixel(m);
                const int ia = x.p * n + x.q, ib = x.mp * n + x.mq;
                la[m] = x.in && ((__ldg(mk + (ia >> 5)) >> (ia & 31)) & 1u);
                lb[m] = x.two && ((__ldg(mk + (ib >> 5)) >> (ib & 31)) & 1u);
            }
            float2 T[C];  // column pairs: T[2c] = (re, re), T[2c + 1] = (im, im) of columns (2c, 2c + 1)
#pragma unroll
            for (int d = 0; d < C; ++d) T[d] = make_float2(0.0f, 0.0f);
            for (int sl = 0; sl < n_sl; ++sl) {
                // field, piston-free, folded about the middle row: entry [p][q / 2] holds
                // S = X[p] + X[n-1-p] and D = X[p] - X[n-1-p] of the columns (q, q + 1) as
                // (re, re, im, im); a column past n is zero
                if (kSl) {
                    const float ks = SD ? SD->k[sl] : 0.0f;
                    if (!kAhead) load(opd + (size_t)sl * a.slice_opd_stride);
                    ref = fmaf(ks, kAhead ? gr : term.at(1.0f, 0, 0), ref);
#pragma unroll
                    for (int m = 0; m < kF; ++m) {
                        const Pixel x = pixel(m);
                        oa[m] = fmaf(ks, kAhead ? ga[m] : term.at(1.0f, x.p, x.q), oa[m]);
                        ob[m] = fmaf(ks, kAhead ? gb[m] : term.at(1.0f, x.mp, x.mq), ob[m]);
                    }
                } else if (a.project) {
                    self_project(a, W, I, D, nullptr, 0, v, n, lo, lane, 32, so);
                    __syncwarp();
                    ref = so[0];
#pragma unroll
                    for (int m = 0; m < kF; ++m) {
                        const Pixel x = pixel(m);
                        oa[m] = so[x.p * n + x.q];
                        ob[m] = so[x.mp * n + x.mq];
                    }
                } else {
                    load(opd);
                }
#pragma unroll
                for (int m = 0; m < kF; ++m) {
                    const int i = lane + 32 * m, p = i / C, q = i - p * C;
                    if (p < H) {
                        float sa, ca, sb, cb;
                        field_phasor(W.k_phase * (oa[m] - ref), sa, ca);
                        field_phasor(W.k_phase * (ob[m] - ref), sb, cb);
                        ca = la[m] ? ca : 0.0f;
                        sa = la[m] ? sa : 0.0f;
                        cb = lb[m] ? cb : 0.0f;
                        sb = lb[m] ? sb : 0.0f;
                        float *e = reinterpret_cast<float *>(X4 + p * H + (q >> 1)) + (q & 1);
                        e[0] = ca + cb;
                        e[2] = sa + sb;
                        e[4 * H * H] = sb - sa;
                        e[4 * H * H + 2] = ca - cb;
                    }
                }
                if (kAhead && sl + 1 < n_sl) load(opd + (size_t)(sl + 1) * a.slice_opd_stride);  // ahead of its use
                __syncwarp();
                // U[k][q], column pairs: the lane's half sum, then U[k] = a + b for k < N/2 and
                // U[N-1-k] = a - b after one exchange (the middle row of an odd N has b = 0)
                float2 ur[H], ui[H];
#pragma unroll
                for (int c = 0; c < H; ++c) ur[c] = ui[c] = make_float2(0.0f, 0.0f);
                {
                    const float4 *V = X4 + (lower ? 0 : H * H);
                    const float *fk = tF + min(lane, N - 1);
#pragma unroll
                    for (int j = 0; j < H; ++j) {
                        const float2 f = dup2(fk[j * N]);
#pragma unroll
                        for (int c = 0; c < H; ++c) {
                            const float4 x = V[j * H + c];
                            ur[c] = fma2(f, make_float2(x.x, x.y), ur[c]);
                            ui[c] = fma2(f, make_float2(x.z, x.w), ui[c]);
                        }
                    }
                    const float2 sg = dup2(lower ? 1.0f : -1.0f), keep = dup2(own ? 0.0f : 1.0f);
#pragma unroll
                    for (int c = 0; c < H; ++c) {
                        const float2 pr = make_float2(__shfl_sync(0xffffffffu, ur[c].x, mirror),
                                                      __shfl_sync(0xffffffffu, ur[c].y, mirror));
                        const float2 pi = make_float2(__shfl_sync(0xffffffffu, ui[c].x, mirror),
                                                      __shfl_sync(0xffffffffu, ui[c].y, mirror));
                        ur[c] = fma2(sg, ur[c], tail::mul2(keep, pr));
                        ui[c] = fma2(sg, ui[c], tail::mul2(keep, pi));
                    }
                }
                // the row folded about the middle column: S = (re, im), i D = (-im, re)
                float2 SS[H], DD[H];
                {
                    auto u = [&](int q) {
                        return make_float2((q & 1) ? ur[q >> 1].y : ur[q >> 1].x, (q & 1) ? ui[q >> 1].y : ui[q >> 1].x);
                    };
#pragma unroll
                    for (int q = 0; q < H; ++q) {
                        const float2 x = u(q), y = n - 1 - q == q ? zero : u(n - 1 - q);
                        SS[q] = make_float2(x.x + y.x, x.y + y.y);
                        DD[q] = make_float2(y.y - x.y, x.x - y.x);
                    }
                }
                const float wsl = SD ? SD->w[sl] : 1.0f;
                // the intensities of columns m and N - 1 - m (the middle column alone: 0 for the other)
                auto pair_intensity = [&](int m, float &i0, float &i1) {
                    float2 s = zero, d = zero;
#pragma unroll
                    for (int q = 0; q < H; q += 2) {
                        const float4 f = tY[(m * H2 + q) >> 1];
                        s = fma2(dup2(f.x), SS[q], s);
                        d = fma2(dup2(f.y), DD[q], d);
                        if (q + 1 < H) {
                            s = fma2(dup2(f.z), SS[q + 1], s);
                            d = fma2(dup2(f.w), DD[q + 1], d);
                        }
                    }
                    const float2 y0 = __fadd2_rn(s, d), y1 = make_float2(s.x - d.x, s.y - d.y);
                    i0 = fmaf(y0.x, y0.x, y0.y * y0.y);
                    i1 = 2 * m + 1 == N ? 0.0f : fmaf(y1.x, y1.x, y1.y * y1.y);
                    if (SD) {
                        i0 *= wsl;
                        i1 *= wsl;
                    }
                    if (stI) {
                        stI[m] = sl == 0 ? i0 : stI[m] + i0;
                        if (2 * m + 1 != N) stI[N - 1 - m] = sl == 0 ? i1 : stI[N - 1 - m] + i1;
                    }
                };
                if (lgs) {
                    // columns (dx, dx + 1) together: re += re Ga (I0 + I1), im += im Ga (I0 - I1)
                    if constexpr (kQuad) {
#pragma unroll kUnroll
                        for (int m = 0; m < cN / 4; ++m) {
                            float i0, i1, i2, i3;  // columns m, N-1-m, N/2-1-m, N/2+m
                            pair_intensity(m, i0, i1);
                            pair_intensity(cN / 2 - 1 - m, i2, i3);
                            const float p = i0 + i1, q = i2 + i3, r = i0 - i1, t = i3 - i2;
                            const float2 ps = make_float2(p + q, p - q), ms = make_float2(r + t, r - t);
#pragma unroll
                            for (int c = 0; c < H; ++c) {
                                const float4 ga = tT[m * H + c];
                                T[2 * c] = fma2(ps, make_float2(ga.x, ga.y), T[2 * c]);
                                T[2 * c + 1] = fma2(ms, make_float2(ga.z, ga.w), T[2 * c + 1]);
                            }
                        }
                    } else {
#pragma unroll 2
                        for (int m = 0; m < hN; ++m) {
                            float i0, i1;
                            pair_intensity(m, i0, i1);
                            const float2 ps = dup2(i0 + i1), ms = dup2(i0 - i1);
#pragma unroll
                            for (int c = 0; c < H; ++c) {
                                const float4 ga = tT[m * H + c];
                                T[2 * c] = fma2(ps, make_float2(ga.x, ga.y), T[2 * c]);
                                T[2 * c + 1] = fma2(ms, make_float2(ga.z, ga.w), T[2 * c + 1]);
                            }
                        }
                    }
                } else {
                    __syncwarp();  // the field's last readers are done: the rows alias it
#pragma unroll 2
                    for (int m = 0; m < hN; ++m) {
                        float i0, i1;
                        pair_intensity(m, i0, i1);
                        if (lane < N) {
                            Iw[lane * (N + 1) + m] = i0;
                            if (2 * m + 1 != N) Iw[lane * (N + 1) + N - 1 - m] = i1;
                        }
                    }
                }
                __syncwarp();  // the field and a self-projected OPD are rewritten by the next slice
            }
            if (lgs) {
                // K~ of this lane's outputs, in flight during the first stage
                const float2 *kt = W.ktil + (size_t)v * (2 * n - 1) * n;
                float2 kp[R], km[R];
                int dy[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    dy[r] = min(grp * R + r, n - 1);
                    kp[r] = __ldg(kt + (n - 1 + dy[r]) * n + dx);
                    km[r] = __ldg(kt + (n - 1 - dy[r]) * n + dx);
                }
                // T's rows k and N - 1 - k folded: lane k < N/2 stores S and D
                // as (S.re, S.im, -D.im, D.re)
#pragma unroll
                for (int d = 0; d < n; ++d) {
                    const float tx = (d & 1) ? T[d & ~1].y : T[d & ~1].x, ty = (d & 1) ? T[d | 1].y : T[d | 1].x;
                    const float px = __shfl_sync(0xffffffffu, tx, mirror);
                    const float py = __shfl_sync(0xffffffffu, ty, mirror);
                    const float mx = own ? 0.0f : px, my = own ? 0.0f : py;
                    if (lower) TS[lane * nT + d] = make_float4(tx + mx, ty + my, my - ty, tx - mx);
                }
                __syncwarp();
                // A[+-dy][dx], then M = K~ A folded: S = M[dy] + M[-dy], i D (dy = 0: S = M)
                float2 a1[R], a2[R];
#pragma unroll
                for (int r = 0; r < R; ++r) a1[r] = a2[r] = zero;
                const float4 *tMg = tM + min(grp, G - 1) * (R / 2);
#pragma unroll 2
                for (int k = 0; k < hN; ++k) {
                    const float4 t = TS[k * nT + dx];
#pragma unroll
                    for (int r = 0; r < R; r += 2) {
                        const float4 ga = tMg[k * (MR / 2) + r / 2];
                        a1[r] = fma2(dup2(ga.x), make_float2(t.x, t.y), a1[r]);
                        a2[r] = fma2(dup2(ga.y), make_float2(t.z, t.w), a2[r]);
                        a1[r + 1] = fma2(dup2(ga.z), make_float2(t.x, t.y), a1[r + 1]);
                        a2[r + 1] = fma2(dup2(ga.w), make_float2(t.z, t.w), a2[r + 1]);
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float2 p = __fadd2_rn(a1[r], a2[r]), q = make_float2(a1[r].x - a2[r].x, a1[r].y - a2[r].y);
                    const float2 mp = make_float2(fmaf(p.x, kp[r].x, -p.y * kp[r].y), fmaf(p.x, kp[r].y, p.y * kp[r].x));
                    float2 mm = make_float2(fmaf(q.x, km[r].x, -q.y * km[r].y), fmaf(q.x, km[r].y, q.y * km[r].x));
                    if (dy[r] == 0) mm = zero;
                    if (grp < G && grp * R + r < n)
                        MS[dy[r] * nT + dx] = make_float4(mp.x + mm.x, mp.y + mm.y, mm.y - mp.y, mp.x - mm.x);
                }
                __syncwarp();
                // Q[iy][dx] and Q[nd-1-iy][dx] (dy = 0 has Im G = 0, so its D does not matter)
                for (int b = grp * kQRows; b < hd && grp < G; b += G * kQRows) {
                    float2 q1[kQRows], q2[kQRows];
#pragma unroll
                    for (int i = 0; i < kQRows; ++i) q1[i] = q2[i] = zero;
#pragma unroll
                    for (int y = 0; y < n; ++y) {
                        const float4 m = MS[y * nT + dx];
#pragma unroll
                        for (int i = 0; i < kQRows; i += 2) {
                            const float4 ga = tQ[(y * QR + b + i) >> 1];
                            q1[i] = fma2(dup2(ga.x), make_float2(m.x, m.y), q1[i]);
                            q2[i] = fma2(dup2(ga.y), make_float2(m.z, m.w), q2[i]);
                            q1[i + 1] = fma2(dup2(ga.z), make_float2(m.x, m.y), q1[i + 1]);
                            q2[i + 1] = fma2(dup2(ga.w), make_float2(m.z, m.w), q2[i + 1]);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < kQRows; ++i)
                        if (b + i < hd) {
                            Qs[(b + i) * C + dx] = __fadd2_rn(q1[i], q2[i]);
                            Qs[(nd - 1 - b - i) * C + dx] = make_float2(q1[i].x - q2[i].x, q1[i].y - q2[i].y);
                        }
                }
                if (n != C)
                    for (int i = lane; i < nd; i += 32) Qs[i * C + n] = make_float2(0.0f, 0.0f);
                __syncwarp();
                // B[iy][ix] and B[iy][nd-1-ix]
                const int gb = lane / hd, ix = lane - gb * hd, GB = 32 / hd;
                if (gb < GB) {
                    float2 gc[C];
#pragma unroll
                    for (int d = 0; d < C; ++d) gc[d] = tB[d * hd + ix];
                    const float4 *Q4 = reinterpret_cast<const float4 *>(Qs);
#pragma unroll 2
                    for (int iy = gb; iy < nd; iy += GB) {
                        float2 s = make_float2(0.0f, 0.0f), t = s;
#pragma unroll
                        for (int c = 0; c < H; ++c) {
                            const float4 q = Q4[iy * H + c];
                            s = fma2(make_float2(q.x, q.y), gc[2 * c], s);
                            t = fma2(make_float2(q.z, q.w), gc[2 * c + 1], t);
                        }
                        s = __fadd2_rn(s, t);
                        B[iy * nd + ix] = s.x - s.y;
                        B[iy * nd + nd - 1 - ix] = s.x + s.y;
                    }
                }
            } else {
                const int b = N / nd;
                for (int o = lane; o < nd2; o += 32) {
                    const int iy = (o * rcp_nd) >> 16, ix = o - iy * nd;
                    float s = 0.0f;
                    for (int r = 0; r < b; ++r)
                        for (int c = 0; c < b; ++c) s += Iw[(b * iy + r) * (N + 1) + b * ix + c];
                    B[o] = s;
                }
            }
            __syncwarp();
            // photometry
            float sb = 0.0f;
            for (int o = lane; o < nd2; o += 32) sb += B[o];
            sb = warp_sum(sb);
            const float scale = sb > 0.0f ? W.photons * __ldg(W.fill + v) / sb : 0.0f;
            float *st_E = D.st_E ? D.st_E + W.det_off + (size_t)v * nd2 : nullptr;
            if (st_E)
                for (int o = lane; o < nd2; o += 32) st_E[o] = scale * B[o];
            {
                float *st_C = D.st_C ? D.st_C + W.det_off + (size_t)v * nd2 : nullptr;
                float sc = 0.0f, sx = 0.0f, sy = 0.0f;
                auto add = [&](int o, float c) {
                    const int iy = (o * rcp_nd) >> 16, ix = o - iy * nd;
                    if (st_C) st_C[o] = c;
                    sc += c;
                    sx = fmaf((float)ix - cd, c, sx);
                    sy = fmaf((float)iy - cd, c, sy);
                };
                if (D.noise) {
                    // pixel pairs of the generator (counted over the sensor's pixels): a pair at
                    // either end of the image may have only one pixel in it
                    const uint32_t base = (uint32_t)v * (uint32_t)nd2;
                    const uint32_t tlo = (uint32_t)__double_as_longlong(D.t);
                    const uint32_t thi = (uint32_t)((unsigned long long)__double_as_longlong(D.t) >> 32);
                    const int odd = (int)(base & 1u), pairs = (nd2 + odd + 1) >> 1;
                    for (int j0 = 0; j0 < pairs; j0 += 32) {
                        const int oe = 2 * (j0 + lane) - odd, oo = oe + 1;
                        const bool ine = oe >= 0 && oe < nd2, ino = oo < nd2;
                        const float ee = ine ? scale * B[oe] : 0.0f, eo = ino ? scale * B[oo] : 0.0f;
                        float ce, co;
                        noise_pair(ee, eo, W.read_noise, I.seed, base + (uint32_t)(ine ? oe : oo), (uint32_t)W.gs_index,
                                   tlo, thi, rk2, ce, co);
                        if (ine) add(oe, ce);
                        if (ino) add(oo, co);
                    }
                } else {
                    for (int o = lane; o < nd2; o += 32) add(o, scale * B[o]);
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
        }
        g = tickets ? nwarps + __shfl_sync(0xffffffffu, ticket, 0) : g + nwarps;
    }
    if (tickets) {
        // every ticket of this CTA was drawn before the barrier; the last CTA to get here leaves
        // the counters at zero for the next launch
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(a.work + 1, 1) == (int)gridDim.x - 1) {
                a.work[0] = 0;
                a.work[1] = 0;
            }
        }
    }
}

namespace {

constexpr int kRowMaxSmem = 200 * 1024;

template <int n, int cN, int cnd, bool kSl, int kCtas>
cudaError_t row_shape_k(const ShArgs &a, LaunchShape *out) {
    const void *f = (const void *)k_sh_row<n, cN, cnd, kSl, kCtas>;
    // per device, once: the dynamic shared-memory limit (process-wide, so never lowered) and the
    // register count
    static std::mutex mu;
    static int regs[64] = {};
    int dev = 0, r = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev < 0 || dev >= 64 || !regs[dev]) {
            cudaFuncAttributes fa;
            if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowMaxSmem)) != cudaSuccess ||
                (e = cudaFuncGetAttributes(&fa, f)) != cudaSuccess)
                return e;
            r = fa.numRegs;
            if (dev >= 0 && dev < 64) regs[dev] = r;
        } else {
            r = regs[dev];
        }
    }
    // warps per CTA: eight, or fewer where the subapertures would not reach every SM twice
    int warps = a.cta_warps == 4 || a.cta_warps == 8 ? a.cta_warps : 8;
    if (!a.cta_warps) {
        const int spread = (a.total + 2 * 152 - 1) / (2 * 152);
        warps = spread < 8 ? (spread < 1 ? 1 : spread) : 8;
    }
    const int smem = row_smem(n, a.N, a.nd, warps, a.project != 0).total;
    int per_sm = 65536 / (((r + 7) & ~7) * 32 * warps);
    per_sm = min(per_sm, 227 * 1024 / (smem + 1024));
    per_sm = max(1, min(per_sm, 64 / warps));
    const int cap = a.grid_cap > 0 ? a.grid_cap : 152 * per_sm;
    out->func = f;
    out->grid = dim3(max(1, min((a.total + warps - 1) / warps, cap)));
    out->block = dim3(32 * warps);
    out->smem = smem;
    return cudaSuccess;
}

// The sizes of a launch as a type: the instance compiled for them is f(RowSize<...>).
template <int n_, int cN_ = 0, int cnd_ = 0>
struct RowSize {
    static constexpr int n = n_, cN = cN_, cnd = cnd_;
};

template <typename F>
cudaError_t row_sizes(const ShArgs &a, F f) {
    if (a.n == 8 && a.N == 16 && a.nd == 8) return f(RowSize<8, 16, 8>{});
    if (a.n == 6 && a.N == 24 && a.nd == 12) return f(RowSize<6, 24, 12>{});
    if (a.n == 8 && a.N == 32 && a.nd == 16) return f(RowSize<8, 32, 16>{});
    if (a.n == 10 && a.N == 32 && a.nd == 16) return f(RowSize<10, 32, 16>{});
    switch (a.n) {
        case 3: return f(RowSize<3>{});
        case 4: return f(RowSize<4>{});
        case 5: return f(RowSize<5>{});
        case 6: return f(RowSize<6>{});
        case 7: return f(RowSize<7>{});
        case 8: return f(RowSize<8>{});
        case 9: return f(RowSize<9>{});
        case 10: return f(RowSize<10>{});
        case 11: return f(RowSize<11>{});
        case 12: return f(RowSize<12>{});
        case 13: return f(RowSize<13>{});
        case 14: return f(RowSize<14>{});
        case 15: return f(RowSize<15>{});
        case 16: return f(RowSize<16>{});
        default: return cudaErrorInvalidValue;
    }
}

// Subapertures of one wave: a warp each on 152 SMs, at two and three CTAs of eight warps per SM.
constexpr int kRowWave2 = 152 * 16, kRowWave3 = 152 * 24;

}  // namespace
}  // namespace gbwfs
