// k_project.cu -- the layered frozen-flow projection (Sec. 4 "Open Loop generation": each layer's
// screen shifted for the star's direction and the wind, shrunk by the LGS cone c = 1 - h / range, and
// the layers summed by bilinear interpolation).
//
// A warp owns a block: up to 64 consecutive pupil columns of a run of subapertures by up to 11 pupil
// rows of one subaperture row; lane i takes the columns i and i + 32.  Per layer, the box of screen
// pixels that the block's taps touch (at most 68 x 12) is copied to one of the warp's own two slots by
// cp.async, a layer ahead of the interpolation; nothing but the warp itself waits for it, so the
// warps of an SM run out of step and cover each other's copies.  The geometry of all of a block's
// boxes is formed at its start, a layer per lane.  Going down a column, pupil row p + 1 falls on the
// same screen row pair as row p or one row lower (the cone factor is at most one for a tiled WFS), so
// a row's lower interpolated tap pair is the next row's upper pair; the two columns travel as packed
// FP32x2 operations.
//
// A WFS whose pupil samples the screens more coarsely than one screen pixel, a sodium slice below a
// layer, and every WFS of the allocation-free entry point, is projected by direct gathers
// (proj_direct.cuh), 32 blocks of 2 x 2 pixels a warp.  Every form does the same per-tap arithmetic in
// the same order: the same OPD.
//
// Bound: issue and latency (48 % issue at 15 warps per SM), and at the start of a launch the instruction
// fetches and the dependent loads of the first blocks: the rare copies are kept out of line for that
// (with them inlined, 45 -> 49 us).  Measured against boxes of up to 400 columns moved by bulk copies of
// two producer warps to eight consumer warps of a CTA (library events, L2 flushed): ELT frame 44.6 -> 37
// us, 48 (LGS, slice) pairs of it 235 -> 207 us, 316 subapertures on one layer 15.0 -> 12.5 us; an uneven
// batch of 64 frames 477 -> 430 us.  Slower: 64 measurements on one layer 96.5 -> 102 us (nothing to copy
// ahead), 3 sensors of 37 x 37, n = 9, on five layers 15.4 -> 16.7 us.  Three slots, 24 warps per SM, and
// preparing a block while the one before it runs gained nothing.
#include <algorithm>
#include <mutex>

#include "internal.h"
#include "proj_direct.cuh"
#include "proj_math.cuh"

namespace gbwfs {

namespace {

constexpr int kProjWarps = 8;
constexpr int kProjThreads = 32 * kProjWarps;
constexpr int kProjCtas = 2;                    // CTAs per SM
constexpr int kBlockCols = 64;                  // pupil columns of a block
constexpr int kBlockRows = 11;                  // most pupil rows of a block
// A box has at most np + 1 rows and ncol + 4 columns (c <= 1: the taps' extent, the bilinear neighbour
// and up to three columns for the 16-byte alignment); one more of each where c = 1 up to rounding.
constexpr int kBoxCols = kBlockCols + 8;
constexpr int kPitch = 4 * kBoxCols;            // bytes of a box row
constexpr int kSlots = 2;
constexpr int kRowPitch = kBlockRows + 1;       // row table of a layer
constexpr int kOffsTable = 512;                 // (WFS, layer) offsets a CTA keeps for its whole launch

// The rows of a block: n pupil rows in equal parts of at most kBlockRows.
__host__ __device__ inline int block_rows(int n) {
    const int parts = (n + kBlockRows - 1) / kBlockRows;
    return (n + parts - 1) / parts;
}

// One layer of a warp's block.
struct __align__(16) LayerBox {
    float c, cl, fu, fv;
    const float *src;  // the box's first element in the screen
    int bx0, by0;      // the box's first column and row, as offsets from the layer base
    const float *scr;  // the layer
    int cs, rs;        // the box's first screen column (a multiple of 4 but for kUnaligned) and row
    int mode;          // kInside, kEdge, kUnaligned, or kNone
    int cols, rows;    // its extent (kEdge, kUnaligned)
    int pad;
};
// How a box is copied: by 16-byte words with the block's fixed extent; the same word by word across
// the periodic screen's edges; element by element (rows without 16-byte alignment); not at all (the
// taps do not fit, which does not happen: reported).
enum { kInside = 0, kEdge = 1, kUnaligned = 2, kNone = 3 };

// i in (-S, 2 S) wrapped into [0, S).
__device__ __forceinline__ int wrap_once(int i, int S) {
    i += i < 0 ? S : 0;
    return i - (i >= S ? S : 0);
}

__device__ __forceinline__ void copy16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// Shared memory of a CTA (bytes): per warp kSlots boxes of box_rows rows, the row tables and the
// geometry of the layers' boxes; then the launch's layer offsets, when they fit.
struct ProjSmem {
    int box, rows, geo, warp, tab, total;
};
__host__ __device__ inline ProjSmem proj_smem(int box_rows, int max_layers, int n_wfs) {
    ProjSmem s;
    s.box = box_rows * kPitch;
    s.rows = kSlots * s.box;
    s.geo = s.rows + max_layers * kRowPitch * (int)sizeof(float2);
    s.warp = box_rows > 0 ? s.geo + max_layers * (int)sizeof(LayerBox) : 0;
    s.tab = kProjWarps * s.warp;
    const int entries = n_wfs * max_layers <= kOffsTable ? n_wfs * max_layers : kProjWarps * max_layers;
    s.total = s.tab + ((entries * (int)sizeof(LayerOffs) + 15) & ~15);
    return s;
}

// Bilinear taps of two columns (a, b) on the box row at byte offset off, interpolated across with the
// columns' fractions (x - y as fma(y, -1, x): the rounded difference).
__device__ __forceinline__ float2 lerp_at(const char *pa, const char *pb, int off, float2 fx) {
    const float *ra = reinterpret_cast<const float *>(pa + off), *rb = reinterpret_cast<const float *>(pb + off);
    const float2 s0 = make_float2(ra[0], rb[0]), s1 = make_float2(ra[1], rb[1]);
    return __ffma2_rn(fx, __ffma2_rn(s0, make_float2(-1.0f, -1.0f), s1), s0);
}

// R pupil rows whose box rows step by 0 or 1: straight-line code, so that the taps of later rows load
// while earlier rows are interpolated.  A step of 0 keeps the row pair (its lower pair is recomputed
// from the same taps: the same value).  rows[i]: byte offset of the lower box row (int bits), fraction.
template <int R>
__device__ __forceinline__ void rows_unit(float2 (&acc)[kBlockRows], const float2 *rows, const char *pa, const char *pb,
                                          float2 fx) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    float2 rp[R];
#pragma unroll
    for (int i = 0; i < R; ++i) rp[i] = rows[i];
    int prev = __float_as_int(rp[0].x);
    float2 top = lerp_at(pa, pb, prev - kPitch, fx);
    float2 bot = lerp_at(pa, pb, prev, fx);
    acc[0] = __fadd2_rn(acc[0], __ffma2_rn(make_float2(rp[0].y, rp[0].y), __ffma2_rn(top, m1, bot), top));
#pragma unroll
    for (int i = 1; i < R; ++i) {
        const int off = __float_as_int(rp[i].x);
        const float2 nb = lerp_at(pa, pb, off, fx);
        const bool same = off == prev;
        top = make_float2(same ? top.x : bot.x, same ? top.y : bot.y);
        bot = nb;
        prev = off;
        acc[i] = __fadd2_rn(acc[i], __ffma2_rn(make_float2(rp[i].y, rp[i].y), __ffma2_rn(top, m1, bot), top));
    }
}

// The copy of a box across the periodic screen's edges (word by word) or of rows without 16-byte
// alignment (element by element: every box of a screen whose side is no multiple of 4 or whose address is
// off).  A lane keeps its columns, wrapped once, and goes down the rows.  Out of line: the kernel's code
// stays short for the boxes that are copied as they lie.  ELT frame, screens one float off 16 bytes:
// 110.8 us with a division and two remainders per element -> 48.8 us (35.7 us for aligned screens); with
// boxes across the edges 39.6 -> 37.0 us.
__device__ __noinline__ void copy_box_slow(const LayerBox *b, uint32_t dst, int S, int lane) {
    const float *scr = b->scr;
    const int cs = b->cs, n_rows = b->rows;
    // cs + c wrapped (cs < S, c < kBoxCols); a remainder only on screens narrower than a box.  Loops in its
    // place made the kernel's own code slower: 48 (LGS, slice) pairs 204.9 -> 207.1 us.
    auto column = [&](int c) {
        c += cs;
        return c < S ? c : c - S < S ? c - S : c % S;
    };
    int row = b->rs;  // in [0, S)
    if (b->mode == kEdge) {
        const int w4 = b->cols >> 2, word = lane & 15;
        const int c = column(4 * word);
        const bool on = word < w4;
        row += lane >> 4;
        for (int r = lane >> 4; r < n_rows; r += 2, row += 2) {  // half a warp per row
            if (row >= S) row %= S;
            if (on) copy16(dst + r * kPitch + 16 * word, scr + (size_t)row * S + c);
        }
        // the words past the sixteenth, one or two a row
        const int more = w4 - 16;
        if (lane < n_rows * more) {
            const int r = more == 2 ? lane >> 1 : lane, w = 16 + (more == 2 ? lane & 1 : 0);
            row = b->rs + r;
            if (row >= S) row %= S;
            copy16(dst + r * kPitch + 16 * w, scr + (size_t)row * S + column(4 * w));
        }
    } else {
        const int c0 = column(lane), c1 = column(lane + 32), c2 = column(lane + 64);
        const bool on0 = lane < b->cols, on1 = lane + 32 < b->cols, on2 = lane + 64 < b->cols;
        for (int r = 0; r < n_rows; ++r) {
            const float *src = scr + (size_t)row * S;
            const uint32_t d = dst + r * kPitch + 4 * lane;
            if (on0) copy4(d, src + c0);
            if (on1) copy4(d + 128, src + c1);
            if (on2) copy4(d + 256, src + c2);
            row = row + 1 == S ? 0 : row + 1;
        }
    }
}
static_assert(kBoxCols <= 72 && 2 * (kBlockRows + 2) <= 32, "at most two words past the sixteenth, a lane each");

// A warp's block seg (of W.segs) of a tiled WFS.
__device__ __forceinline__ void project_block(const ProjArgs &a, const ProjSmem &L, const WfsDesc &W, const InstDesc &I,
                                              const InstDyn &D, const LayerOffs *wt, int seg, char *scratch, int lane) {
    const int4 sg = __ldg(W.segs + seg);
    // sg: subaperture row | first pupil row << 16, first valid index and column of the run,
    // first pupil column of the block within the run | columns << 24
    const int n = W.n, sy = sg.x & 0xFFFF, p0 = sg.x >> 16, col0 = sg.w & 0xFFFFFF, ncol = sg.w >> 24;
    const int np = min(block_rows(n), n - p0);
    const int S = I.S, layers = proj_layers(I, D), n_scr = I.n_layers;
    const float half = 0.5f * (float)(W.n_sub * n - 1);
    const float x_first = (float)(sg.z * n + col0) - half, y_first = (float)(sy * n + p0) - half;
    LayerBox *geo = reinterpret_cast<LayerBox *>(scratch + L.geo);
    // 16-byte words and rows of a box copied by words
    const int words = (ncol + 7) >> 2, box_rows = np + 1;
    bool unit = true;  // every layer's box rows step by 0 or 1 from one pupil row to the next
    for (int l = lane; l < layers; l += 32) {
        const LayerOffs o = wt[l];
        LayerBox b;
        b.scr = l < n_scr ? D.screens + (size_t)l * S * S : D.dm + (size_t)(l - n_scr) * S * S;
        b.c = o.c;
        b.cl = o.cl;
        b.fu = o.fu;
        b.fv = o.fv;
        int c0, c1, r0, r1;
        float f, f0;
        screen_offset(o.c, o.cl, o.fu, x_first, c0, f);
        screen_offset(o.c, o.cl, o.fu, x_first + (float)(ncol - 1), c1, f);
        screen_offset(o.c, o.cl, o.fv, y_first, r0, f0);
        screen_offset(o.c, o.cl, o.fv, y_first + (float)(np - 1), r1, f);
        // a step of 2 needs c = 1 up to rounding and a row on a screen row up to rounding
        unit = unit && (o.c < 0.999999f || (f0 > 1e-4f && f0 < 0.9999f));
        const bool vec = (S & 3) == 0 && (reinterpret_cast<uintptr_t>(b.scr) & 15) == 0;
        // |c x / ds| < S (checked at creation), and the base is in [0, S)
        const int cs = wrap_once(o.bu + c0, S), al = vec ? cs & 3 : 0;
        b.cs = cs - al;
        b.rs = wrap_once(o.bv + r0, S);
        b.src = b.scr + (size_t)b.rs * S + b.cs;
        b.bx0 = c0 - al;
        b.by0 = r0;
        b.cols = (c1 - c0 + 2 + al + 3) & ~3;
        b.rows = r1 - r0 + 2;
        const bool fits = c1 >= c0 && r1 >= r0 && b.cols <= kBoxCols && b.rows * kPitch <= L.box;
        b.mode = !fits ? kNone
                 : !vec ? kUnaligned
                 : b.cs + 4 * words <= S && b.rs + box_rows <= S && b.cols <= 4 * words && b.rows <= box_rows ? kInside
                                                                                                        : kEdge;
        if (!fits && a.status) atomicCAS(a.status, 0, 6 /* WFS_EUNSUPPORTED */);
        geo[l] = b;
    }
    unit = __all_sync(0xffffffffu, unit);
    __syncwarp();

    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(scratch);
    // half a warp per box row: word lane mod 16 of rows half + 2 i; then the rows' last words, a row
    // per lane (and half)
    const int word = lane & 15, hrow = lane >> 4;
    const bool word_on = word < words, tail_on = words > 16 && lane < box_rows;
    auto copy_box = [&](int l, int slot) {
        const LayerBox &b = geo[l];
        const uint32_t dst = ring + (uint32_t)(slot * L.box);
        const int mode = b.mode;
        if (mode == kInside) {
            const float *src = b.src;
            const float *sw = src + hrow * S + 4 * word;
            const uint32_t dw = dst + hrow * kPitch + 16 * word;
#pragma unroll
            for (int i = 0; i < (kBlockRows + 2) / 2; ++i)
                if (word_on && 2 * i + hrow < box_rows) copy16(dw + 2 * i * kPitch, sw + (size_t)(2 * i) * S);
            if (tail_on) copy16(dst + lane * kPitch + 256, src + (size_t)lane * S + 64);
        } else if (mode != kNone) {
            copy_box_slow(&b, dst, S, lane);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    const float xa = x_first + (float)lane, xb = xa + 32.0f;
    float2 acc[kBlockRows];
#pragma unroll
    for (int i = 0; i < kBlockRows; ++i) acc[i] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int l = 0; l < kSlots - 1; ++l) {
        if (l < layers) copy_box(l, l);
        else asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // every layer's row table while the first boxes travel, a (layer, row) per lane: byte offset of the
    // lower box row, fraction
    float2 *rows = reinterpret_cast<float2 *>(scratch + L.rows);
    {
        const int per = 32 / np, l0 = lane / np, p = lane - l0 * np;
        const float y = y_first + (float)p;
        for (int l = l0; l < layers && l0 < per; l += per) {
            const LayerBox &b = geo[l];
            int off;
            float fr;
            screen_offset(b.c, b.cl, b.fv, y, off, fr);
            const int br = min(max(off - b.by0, 0), b.rows - 2);
            rows[l * kRowPitch + p] = make_float2(__int_as_float((br + 1) * kPitch), fr);
        }
    }
    int slot = 0;
    for (int l = 0; l < layers; ++l) {
        // the slot of layer l + kSlots - 1 was read for the layer before l (a warp barrier ago)
        const int ahead = slot == 0 ? kSlots - 1 : slot - 1;
        if (l + kSlots - 1 < layers) copy_box(l + kSlots - 1, ahead);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        const LayerBox &b = geo[l];
        int oa, ob;
        float2 fx;
        screen_offset(b.c, b.cl, b.fu, xa, oa, fx.x);
        screen_offset(b.c, b.cl, b.fu, xb, ob, fx.y);
        guard(lane >= ncol || (oa - b.bx0 >= 0 && oa - b.bx0 + 1 < b.cols), a.status);
        // columns kept inside the box (those past the block's are computed and dropped)
        const int ca = min(max(oa - b.bx0, 0), kBoxCols - 2), cb = min(max(ob - b.bx0, 0), kBoxCols - 2);
        const bool fits = b.mode != kNone;
        const char *box = scratch + slot * L.box;
        const char *pa = box + 4 * ca, *pb = box + 4 * cb;
        const float2 *rt = rows + l * kRowPitch;
        asm volatile("cp.async.wait_group %0;" ::"n"(kSlots - 1) : "memory");
        __syncwarp();  // every lane's copies of layer l, and the row tables
        if (fits && unit) {
            switch (np) {
#define GBWFS_ROWS_CASE(R) \
    case R: rows_unit<R>(acc, rt, pa, pb, fx); break;
                GBWFS_ROWS_CASE(1) GBWFS_ROWS_CASE(2) GBWFS_ROWS_CASE(3) GBWFS_ROWS_CASE(4)
                GBWFS_ROWS_CASE(5) GBWFS_ROWS_CASE(6) GBWFS_ROWS_CASE(7) GBWFS_ROWS_CASE(8)
                GBWFS_ROWS_CASE(9) GBWFS_ROWS_CASE(10) GBWFS_ROWS_CASE(11)
#undef GBWFS_ROWS_CASE
                default: break;
            }
        } else if (fits) {
            const float2 m1 = make_float2(-1.0f, -1.0f);
#pragma unroll
            for (int i = 0; i < kBlockRows; ++i)
                if (i < np) {
                    const float2 rp = rt[i];
                    const int o = __float_as_int(rp.x);
                    const float2 top = lerp_at(pa, pb, o - kPitch, fx), bot = lerp_at(pa, pb, o, fx);
                    acc[i] = __fadd2_rn(acc[i], __ffma2_rn(make_float2(rp.y, rp.y), __ffma2_rn(top, m1, bot), top));
                }
        }
        __syncwarp();  // the slot may be refilled
        slot = slot == kSlots - 1 ? 0 : slot + 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    // the uplink tip-tilt as a plane over the pupil (zero when off); the uplink kernel may still be
    // running (programmatic dependent launch): wait for it first
    float2 up = make_float2(0.0f, 0.0f);
    if (W.uplink) {
        wait_prior_grid();
        up = *W.uplink;
    }
    float *opd = D.opd + W.opd_off + (size_t)sg.y * n * n;
    const int ta = col0 + lane, tb = ta + 32, va = ta / n, vb = tb / n;
    float *da = opd + (size_t)va * n * n + (ta - va * n), *db = opd + (size_t)vb * n * n + (tb - vb * n);
    const bool on_a = lane < ncol, on_b = lane + 32 < ncol;
    da += p0 * n;
    db += p0 * n;
    const bool tilt = W.uplink != nullptr;
#pragma unroll
    for (int i = 0; i < kBlockRows; ++i)
        if (i < np) {
            if (tilt) {
                const float y = y_first + (float)i;
                acc[i].x += fmaf(up.x, xa, up.y * y);
                acc[i].y += fmaf(up.x, xb, up.y * y);
            }
            if (on_a) da[i * n] = acc[i].x;
            if (on_b) db[i * n] = acc[i].y;
        }
}

}  // namespace

// Blocks 0 .. n_blocks of this launch.  Each warp starts with a block of its own; with a.work the
// grid holds only as many CTAs as fit at once and each warp draws its next block from the ticket
// counter (issued at the top, consumed after the block), so CTAs that start late take fewer
// blocks and no partial last wave is left; the last CTA to finish resets the counter.
__global__ void __launch_bounds__(kProjThreads, kProjCtas) k_project(const __grid_constant__ ProjArgs a) {
    allow_dependent_grid();  // every CTA of this grid is resident or done: the spot kernel may start
    extern __shared__ __align__(16) char psm[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const ProjSmem L = proj_smem(a.box_rows, a.max_layers, a.n_wfs);
    LayerOffs *tab = reinterpret_cast<LayerOffs *>(psm + L.tab);
    // the layer offsets of every (WFS, layer) of this launch, once per CTA, when they fit; else a
    // warp forms those of its block's WFS
    const bool all_offs = a.n_wfs * a.max_layers <= kOffsTable;
    if (all_offs) {
        for (int i = threadIdx.x; i < a.n_wfs * a.max_layers; i += blockDim.x) {
            const int w = i / a.max_layers, l = i - w * a.max_layers;
            const WfsDesc &W = a.wfs[w];
            const InstDesc &I = a.inst[W.inst];
            if (l < proj_layers(I, a.dyn[W.inst])) tab[i] = layer_offsets(I, W, a.dyn[W.inst].t, l);
        }
        __syncthreads();
    }
    char *scratch = psm + wib * L.warp;
    const int nwarps = gridDim.x * kProjWarps;
    int last = -1;
    // consecutive blocks go to different CTAs, so that a launch of few blocks reaches every SM
    for (int blk = wib * gridDim.x + blockIdx.x; blk < a.n_blocks;) {
        int ticket = 0;
        if (a.work && lane == 0) ticket = atomicAdd(a.work, 1);
        // the WFS owning this block: last entry whose first block of the kind is <= bid
        const bool part = blk >= a.n_full;
        const int bid = part ? blk - a.n_full + a.part_base : blk + a.block_base;
        int lo = 0, hi = a.n_wfs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(part ? &a.wfs[mid].proj_part_begin : &a.wfs[mid].proj_block_begin) <= bid) lo = mid;
            else hi = mid - 1;
        }
        const WfsDesc &W = a.wfs[lo];
        const InstDesc &I = a.inst[W.inst];
        const InstDyn &D = a.dyn[W.inst];
        const LayerOffs *wt = all_offs ? tab + lo * a.max_layers : tab + wib * a.max_layers;
        if (!all_offs && lo != last) {
            __syncwarp();  // earlier reads of the warp's offsets are done
            for (int l = lane; l < proj_layers(I, D); l += 32) tab[wib * a.max_layers + l] = layer_offsets(I, W, D.t, l);
            last = lo;
            __syncwarp();
        }
        const int seg = part ? W.n_full + bid - W.proj_part_begin : bid - W.proj_block_begin;
        if (W.tiled && a.box_rows > 0) project_block(a, L, W, I, D, wt, seg, scratch, lane);
        else project_direct<32>(a, W, I, D, wt, seg, lane);
        __syncwarp();
        blk = a.work ? nwarps + __shfl_sync(0xffffffffu, ticket, 0) : blk + nwarps;
    }
    if (a.work) {
        __syncthreads();  // every warp of the CTA has drawn past the end
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(a.work + 1, 1) == (int)gridDim.x - 1) {
                a.work[0] = 0;
                a.work[1] = 0;
            }
        }
    }
}

ProjRange project_blocks(const WfsDesc &d) {
    if (d.tiled) return {d.n_full, d.n_segs - d.n_full};
    const int nb = (d.n + 1) / 2;
    return {(d.n_valid * nb * nb + 31) / 32, 0};
}

void place_blocks(WfsDesc &d, ProjRange &r) {
    const ProjRange n = project_blocks(d);
    d.proj_block_begin = r.full;
    d.proj_part_begin = r.part;
    r.full += n.full;
    r.part += n.part;
}

int project_box_rows(const WfsDesc &d) { return d.tiled ? block_rows(d.n) + 2 : 0; }

int build_segments(const std::vector<int32_t> &ids, int n_sub, int n, std::vector<int4> &segs) {
    segs.clear();
    const int R = block_rows(n);
    for (size_t v = 0; v < ids.size();) {
        const int sy = ids[v] / n_sub, sx = ids[v] - sy * n_sub;
        size_t e = v + 1;  // the run of consecutive valid subapertures of this row
        while (e < ids.size() && ids[e] == ids[e - 1] + 1 && ids[e] / n_sub == sy) ++e;
        const int cols = (int)(e - v) * n;
        for (int c = 0; c < cols; c += kBlockCols)
            for (int p = 0; p < n; p += R)
                segs.push_back(make_int4(sy | p << 16, (int)v, sx, c | std::min(kBlockCols, cols - c) << 24));
        v = e;
    }
    std::stable_sort(segs.begin(), segs.end(), [](const int4 &x, const int4 &y) { return x.w >> 24 > y.w >> 24; });
    int full = 0;
    while (full < (int)segs.size() && segs[full].w >> 24 == kBlockCols) ++full;
    return full;
}

cudaError_t launch_project(const ProjArgs &a, ProjRange blocks, cudaStream_t s, bool after_uplink) {
    if (blocks.full + blocks.part <= 0) return cudaSuccess;
    LaunchShape sh;
    cudaError_t e = project_launch_shape(a, blocks, &sh);
    if (e != cudaSuccess) return e;
    // beside the uplink kernel's few CTAs, whose FP64 sums the launch ends up waiting for: whole CTAs of
    // blocks rather than a block on every SM (two LGS of 22 x 22, n = 10, four layers, uplink on: 36.9 us
    // spread, 30.7 us packed; 33.5 and 33.1 us for 7 x 7, n = 16)
    if (after_uplink) sh.grid.x = std::min(sh.grid.x, (unsigned)(blocks.full + blocks.part + kProjWarps - 1) / kProjWarps);
    ProjArgs b = a;
    b.n_full = blocks.full;
    b.n_blocks = blocks.full + blocks.part;
    void *args[] = {(void *)&b};
    if (!after_uplink) return cudaLaunchKernel(sh.func, sh.grid, sh.block, args, sh.smem, s);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = sh.grid;
    cfg.blockDim = sh.block;
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, sh.func, args);
}

cudaError_t project_launch_shape(const ProjArgs &a, ProjRange blocks, LaunchShape *out) {
    const int total_blocks = blocks.full + blocks.part;
    const int smem = proj_smem(a.box_rows, a.max_layers, a.n_wfs).total;
    // the dynamic shared-memory limit is process-wide: set once per device, to the most a CTA may have
    static std::mutex m;
    static bool set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lk(m);
        if (dev < 0 || dev >= 64 || !set[dev]) {
            if ((e = cudaFuncSetAttribute(k_project, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)) != cudaSuccess)
                return e;
            if (dev >= 0 && dev < 64) set[dev] = true;
        }
    }
    int grid = std::max(1, (total_blocks + kProjWarps - 1) / kProjWarps);
    if (total_blocks < 152 * kProjWarps) grid = std::min(std::max(total_blocks, 1), 152);  // every SM
    if (a.work) {
        // resident CTAs: two per SM where shared memory allows
        const int per_sm = std::max(1, std::min(kProjCtas, 227 * 1024 / (smem + 1024)));
        grid = std::min(grid, 152 * per_sm);
    }
    out->func = (const void *)k_project;
    out->grid = dim3(grid);
    out->block = dim3(kProjThreads);
    out->smem = smem;
    return cudaSuccess;
}

}  // namespace gbwfs
