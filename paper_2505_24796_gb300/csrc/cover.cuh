// cover.cuh -- device helpers of the sorting stage shared by its two forms: block scans, depth keys and
// the Gaussian-tile coverage test.
#pragma once

#include "common.cuh"

namespace tcgs {
namespace {

// Exclusive scan over a block of NT threads; returns the thread's exclusive prefix and the total.
template <typename T, int NT>
__device__ __forceinline__ T block_exclusive_scan(T x, T* warp_sums, T& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T v = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    if (warp == 0) {
        constexpr int NW = NT / 32;
        T w = lane < NW ? warp_sums[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < NW) warp_sums[lane] = w;
    }
    __syncthreads();
    T before = warp > 0 ? warp_sums[warp - 1] : T(0);
    total = warp_sums[NT / 32 - 1];
    __syncthreads();
    return before + v - x;
}

__device__ __forceinline__ uint32_t orderable_bits(float f) {
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Exact tile coverage (tcgs_bin_sort_exact): Gaussian g reaches tile t when the least value of its
// conic form over t's 16 x 16 box of pixel centres, in tile-local coordinates, is at most its reach
// limit (the TC renderer's block-mark limit, whose boxes lie inside the tile's).  Per warp, the 32
// Gaussians' parameters are staged in shared memory once; every splat then reads its Gaussian's.
struct Cover {
    float mx, my, a, b, c, ia, ic, lim;
};

__device__ __forceinline__ Cover cover_of(const float* __restrict__ mean2d, const float* __restrict__ conic,
                                          const float* __restrict__ opacity, uint32_t g) {
    Cover v;
    const float2 m = reinterpret_cast<const float2*>(mean2d)[g];
    v.mx = m.x; v.my = m.y;
    v.a = conic[3 * g]; v.b = conic[3 * g + 1]; v.c = conic[3 * g + 2];
    v.lim = reach_limit(__logf(opacity[g]));
    v.ia = __fdividef(1.f, v.a);
    v.ic = __fdividef(1.f, v.c);
    return v;
}

// Gaussian v reaches the tile whose centre is at tile-local offset (lx, ly) from its mean when the
// least value of its conic form over the tile's 16 x 16 pixel-centre box is within its reach limit.
__device__ __forceinline__ bool tile_reached(const Cover& v, float lx, float ly) {
    constexpr float h = 0.5f * (kTile - 1);
    return v.lim >= 0.f && min_q_box_facing(lx, ly, v.a, v.b, v.c, v.ia, v.ic, -h, h, -h, h) <= v.lim;
}

// ---- exact coverage by tile rows
//
// In one row of tiles the tiles a Gaussian reaches form an interval: their pixel-centre boxes span
// the same band of rows, and a box meets the convex region {q <= lim} exactly when its x-range meets
// the region's shadow on the x axis within that band.  So each (Gaussian, tile row) is one unit of
// work: the shadow's ends come from the ellipse in closed form, and the per-tile test (tile_reached)
// fixes the end tiles that the closed form leaves in doubt.  row_span keeps the run from the first to the last
// tile so found, and scans the rows of degenerate conics; row_tiles leaves every tile in doubt to the caller's
// tests, so that the tiles are those that the per-tile test keeps, also where FP32 ties at the reach limit
// make it keep a row in parts.

// Extent of the reach ellipse {q <= lim} about the mean: half-widths W (x) and H (y), the y offset s
// of its leftmost point (the rightmost one is at -s), and det = ac - b^2.  W < 0: scan the row.
struct Reach {
    float W, H, s, det;
};

__device__ __forceinline__ Reach reach_of(const Cover& v) {
    Reach e;
    e.det = __fsub_rn(__fmul_rn(v.a, v.c), __fmul_rn(v.b, v.b));
    e.W = -1.f;
    e.H = e.s = 0.f;
    if (!(e.det > 0.f) || !(v.lim >= 0.f)) return e;
    const float idet = __frcp_rn(e.det);
    const float W = __fsqrt_rn(__fmul_rn(__fmul_rn(v.lim, v.c), idet));
    const float H = __fsqrt_rn(__fmul_rn(__fmul_rn(v.lim, v.a), idet));
    if (!(W < 1e30f) || !(H < 1e30f)) return e;
    e.W = W;
    e.H = H;
    e.s = __fmul_rn(__fmul_rn(v.b, W), v.ic);
    return e;
}

__device__ __forceinline__ int clamp_tile(float f, int lo, int hi) {
    return (int)fminf(fmaxf(f, (float)lo), (float)hi);   // NaN -> lo
}

// Tiles [L, R] (empty when L > R) of rectangle columns [x0, x1] in tile row ty that Gaussian v reaches.
__device__ int2 row_span(const Cover& v, const Reach& e, int ty, int x0, int x1) {
    const int2 none = make_int2(1, 0);
    if (!(v.lim >= 0.f)) return none;
    const float ly = v.my - (float)(ty * kTile + kTile / 2);
    auto test = [&](int tx) { return tile_reached(v, v.mx - (float)(tx * kTile + kTile / 2), ly); };
    auto scan = [&]() {
        int L = x0;
        while (L <= x1 && !test(L)) ++L;
        if (L > x1) return none;
        int R = x1;
        while (R > L && !test(R)) --R;
        return make_int2(L, R);
    };
    if (e.W < 0.f || x1 - x0 < 3) return scan();
    // the shadow [xa, xb] of the ellipse on the x axis within the row's band of pixel centres
    const float yl = __fsub_rn((float)(ty * kTile) + 0.5f, v.my), yh = __fadd_rn(yl, 15.f);
    float Lf = 1.f, Rf = 0.f;   // empty unless the band meets the ellipse
    float xa_ = 0.f, xb_ = 0.f, rl_ = 0.f, rr_ = 0.f;
    if (!(yl > e.H || yh < -e.H)) {
        const float alim = __fmul_rn(v.a, v.lim);
        const float dl = fminf(yh, fmaxf(yl, e.s)), dr = fminf(yh, fmaxf(yl, -e.s));
        const float rl = __fsqrt_rn(fmaxf(0.f, __fsub_rn(alim, __fmul_rn(e.det, __fmul_rn(dl, dl)))));
        const float rr = __fsqrt_rn(fmaxf(0.f, __fsub_rn(alim, __fmul_rn(e.det, __fmul_rn(dr, dr)))));
        const float xa = __fmul_rn(__fsub_rn(__fmul_rn(-v.b, dl), rl), v.ia);
        const float xb = __fmul_rn(__fadd_rn(__fmul_rn(-v.b, dr), rr), v.ia);
        xa_ = xa; xb_ = xb; rl_ = rl; rr_ = rr;
        // tiles whose box [16 tx + 0.5, 16 tx + 15.5] meets [mx + xa, mx + xb]
        Lf = ceilf(__fmul_rn(__fsub_rn(__fadd_rn(v.mx, xa), 15.5f), 1.f / kTile));
        Rf = floorf(__fmul_rn(__fsub_rn(__fadd_rn(v.mx, xb), 0.5f), 1.f / kTile));
    }
    if (!(Lf <= Rf) || Rf < (float)x0 || Lf > (float)x1) {
        // no shadow in the rectangle: probe the tile holding the point of least q in the band (the
        // least of the minima over x, (det / a) dy^2, is at the dy nearest to 0), grow from there
        const float dyc = fminf(yh, fmaxf(yl, 0.f));
        const float xc = __fadd_rn(v.mx, __fmul_rn(__fmul_rn(-v.b, dyc), v.ia));
        const int c = clamp_tile(floorf(__fmul_rn(xc, 1.f / kTile)), x0, x1);
        if (!test(c)) return none;
        int L = c, R = c;
        while (L > x0 && test(L - 1)) --L;
        while (R < x1 && test(R + 1)) ++R;
        return make_int2(L, R);
    }
    int L = clamp_tile(Lf, x0, x1), R = clamp_tile(Rf, x0, x1);
    // Ends that need no test.  Along y = dl (dr) the form is lim - 2 r e + a e^2 at a distance e inside the
    // shadow's end (r = rl or rr, half its slope there), so the end tile passes when that is below lim at
    // the point of its box nearest to the minimum; by convexity it is at least lim + 2 r g over the band at a
    // distance g outside, where the outer neighbour's box begins.  Both must clear a bound on the roundings
    // of this code and of the test (1e-5 of the sum of magnitudes, 168 times 2^-24, and of the positions).  The
    // four tests it saves were most of a row: the runs of 605M splats at 3840 x 2160 take 1.48 ms, against
    // 1.82 ms with every end tested.
    const float X = fmaxf(fabsf(xa_), fabsf(xb_)) + 16.f, Y = fmaxf(fabsf(yl), fabsf(yh));
    const float slack0 = 1e-5f * (v.a * X * X + v.c * Y * Y), slack1 = 1e-5f * (fabsf(v.mx) + X);
    auto sure = [&](float r, float far, bool clamped) {   // far: from the end to the far side of the end tile's box
        const float e = fminf(fmaxf(r * v.ia, far - 15.f), far), s = slack0 + slack1 * r;
        return far >= 0.f && e * (2.f * r - v.a * e) > s && (clamped || 2.f * r * (16.f - far) > s);
    };
    const bool sure_l = sure(rl_, (float)(L * kTile) + 15.5f - (v.mx + xa_), (float)L > Lf);
    const bool sure_r = sure(rr_, (v.mx + xb_) - ((float)(R * kTile) + 0.5f), (float)R < Rf);
    if (sure_l && sure_r && L <= R) return make_int2(L, R);
    if (sure_l) {
    } else if (test(L)) {
        while (L > x0 && test(L - 1)) --L;
    } else {
        int k = L + 1;
        while (k <= R && !test(k)) ++k;
        if (k > R) return scan();
        L = k;
    }
    if (sure_r) {
    } else if (test(R)) {
        while (R < x1 && test(R + 1)) ++R;
    } else {
        int k = R - 1;
        while (k > L && !test(k)) --k;
        R = k;
    }
    return make_int2(L, R);
}

// The shadow [xa, xb] of the ellipse on the x axis within tile row ty's band [yl, yh] of pixel centres, relative to
// the mean (in: the band meets the ellipse); rl and rr: half the slope of the form across its ends, at the offsets
// dl and dr where the ellipse reaches furthest inside the band.  (As row_span forms it.)
struct Shadow {
    float yl, yh, xa, xb, rl, rr;
    bool in;
};

__device__ __forceinline__ Shadow shadow_of(const Cover& v, const Reach& e, int ty) {
    Shadow h;
    h.yl = __fsub_rn((float)(ty * kTile) + 0.5f, v.my);
    h.yh = __fadd_rn(h.yl, 15.f);
    h.xa = h.xb = h.rl = h.rr = 0.f;
    h.in = !(h.yl > e.H || h.yh < -e.H);
    if (h.in) {
        const float alim = __fmul_rn(v.a, v.lim);
        const float dl = fminf(h.yh, fmaxf(h.yl, e.s)), dr = fminf(h.yh, fmaxf(h.yl, -e.s));
        h.rl = __fsqrt_rn(fmaxf(0.f, __fsub_rn(alim, __fmul_rn(e.det, __fmul_rn(dl, dl)))));
        h.rr = __fsqrt_rn(fmaxf(0.f, __fsub_rn(alim, __fmul_rn(e.det, __fmul_rn(dr, dr)))));
        h.xa = __fmul_rn(__fsub_rn(__fmul_rn(-v.b, dl), h.rl), v.ia);
        h.xb = __fmul_rn(__fadd_rn(__fmul_rn(-v.b, dr), h.rr), v.ia);
    }
    return h;
}

// First and last tile whose box [16 tx + 0.5, 16 tx + 15.5] meets [mx + xa, mx + xb].
__device__ __forceinline__ float first_met(const Cover& v, float xa) {
    return ceilf(__fmul_rn(__fsub_rn(__fadd_rn(v.mx, xa), 15.5f), 1.f / kTile));
}
__device__ __forceinline__ float last_met(const Cover& v, float xb) {
    return floorf(__fmul_rn(__fsub_rn(__fadd_rn(v.mx, xb), 0.5f), 1.f / kTile));
}

// Bound on the relative error of Reach.s: that of the determinant is 1.2e-7 ac / det, of which the ellipse's width
// takes half; infinite where the terms of higher order would count.
__device__ __forceinline__ float turn_error(const Cover& v) {
    const float rel = 2e-7f * __fdividef(v.a * v.c, __fsub_rn(__fmul_rn(v.a, v.c), __fmul_rn(v.b, v.b)));
    return rel >= 0.f && rel < 0.2f ? rel : __int_as_float(0x7f800000);
}

// What the closed form must clear before a tile needs no test.  Along y = dl (dr) the form is lim - 2 r e + a e^2
// at a distance e inside the shadow's end, so the end tile passes when that is below lim at the point of its
// box nearest to the minimum; at a distance g outside, where the outer neighbour's box begins, it is at
// least lim + 2 (r - |b| d) g - c d^2 over the band, d being the error of dl.  Both are compared with a bound on the roundings
// of this code and of the test: 1e-5 of the sum of magnitudes (168 times 2^-24) and of the positions.
struct Slack {
    float form, pos, turn;   // of the form, of a position, of half a slope (|b| d)
    __device__ __forceinline__ float at(float r) const { return form + pos * r; }
    __device__ __forceinline__ float slope(float r) const { return r - turn; }   // at most 0: nothing is known
};

__device__ __forceinline__ Slack slack_of(const Cover& v, float rel, const Shadow& h, float X) {
    const float Y = fmaxf(fabsf(h.yl), fabsf(h.yh)), d = rel * Y;
    Slack s;
    s.form = 1e-5f * (v.a * X * X + v.c * Y * Y) + v.c * d * d;
    s.pos = 1e-5f * (fabsf(v.mx) + X);
    s.turn = fabsf(v.b) * d;
    return s;
}

// far: from the shadow's end to the far side of the end tile's box.  clamped: the rectangle ends at that tile.
__device__ __forceinline__ bool end_sure(const Cover& v, const Slack& s, float r, float far, bool clamped) {
    const float e = fminf(fmaxf(r * v.ia, far - 15.f), far);
    return far >= 0.f && e * (2.f * r - v.a * e) > s.at(r) && (clamped || 2.f * s.slope(r) * (16.f - far) > s.at(r));
}

// The tiles of rectangle columns [x0, x1] in tile row ty that tile_reached admits one by one, rounding included:
// sure, exactly [lo, hi] (none when lo > hi); else some of [lo, hi], which the caller tests.  The form is
// convex, so a row whose ends clear the slack of the whole rectangle (that of the largest offsets in it) has no
// tile inside that fails and none outside that passes.  Needles, whose form cancels, do not clear it.
struct RowTiles {
    int lo, hi;
    bool sure;
};

__device__ RowTiles row_tiles(const Cover& v, const Reach& e, float rel, int ty, int x0, int x1) {
    const RowTiles none{1, 0, true}, all{x0, x1, false};
    if (!(v.ia < 1e30f) || !(v.ic < 1e30f)) return all;
    const Shadow h = shadow_of(v, e, ty);
    const float Xl = v.mx - (float)(x0 * kTile), Xr = (float)((x1 + 1) * kTile) - v.mx;
    const Slack s = slack_of(v, rel, h, fmaxf(fabsf(Xl), fabsf(Xr)));
    if (!h.in) {   // the least q of the band, (det / a) dy^2, against the limit
        const float dy = fminf(h.yh, fmaxf(h.yl, 0.f));
        return e.det * v.ia * dy * dy > v.lim + s.form ? none : all;
    }
    const float Lf = first_met(v, h.xa), Rf = last_met(v, h.xb);
    if (Rf < (float)x0)
        return 2.f * s.slope(h.rr) * ((float)(x0 * kTile) + 0.5f - (v.mx + h.xb)) > s.at(h.rr) ? none : all;
    if (Lf > (float)x1)
        return 2.f * s.slope(h.rl) * ((v.mx + h.xa) - ((float)(x1 * kTile) + 15.5f)) > s.at(h.rl) ? none : all;
    if (!(Lf <= Rf)) return all;
    const int L = clamp_tile(Lf, x0, x1), R = clamp_tile(Rf, x0, x1);
    if (end_sure(v, s, h.rl, (float)(L * kTile) + 15.5f - (v.mx + h.xa), (float)L > Lf) &&
        end_sure(v, s, h.rr, (v.mx + h.xb) - ((float)(R * kTile) + 0.5f), (float)R < Rf))
        return RowTiles{L, R, true};
    // no tile passes beyond a distance of s.at / (2 s.slope) from the ends
    const float ul = 2.f * s.slope(h.rl), ur = 2.f * s.slope(h.rr);
    RowTiles t = all;
    if (s.at(h.rl) < 1e6f * ul) t.lo = clamp_tile(first_met(v, h.xa - __fdividef(s.at(h.rl), ul)) - 1.f, x0, x1);
    if (s.at(h.rr) < 1e6f * ur) t.hi = clamp_tile(last_met(v, h.xb + __fdividef(s.at(h.rr), ur)) + 1.f, x0, x1);
    return t;
}

// Gaussians whose rectangle is at least this many tiles wide are covered by rows; the narrower ones
// tile by tile (for them a row costs about as many box tests as it has tiles, plus the row's own
// bookkeeping).
constexpr int kRowMinWidth = 6;
// With a splat capacity of at least this many splats per Gaussian, wide Gaussians' rows are kept from the first
// to the last reached tile (row_span), else tile by tile.
constexpr int kRowsCapacityPerGaussian = 32;

}  // namespace
}  // namespace tcgs
