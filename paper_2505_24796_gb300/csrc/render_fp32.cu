// render_fp32.cu -- conditional alpha-blending on CUDA cores (Algorithm 1, Eq. 4-6): the FP32 forward
// and the backward replay.
#include <type_traits>

#include "common.cuh"
#include "pairs.cuh"

namespace tcgs {
namespace {

struct FwdParams {
    DevCamera cam;
    const uint32_t* ranges;
    const uint32_t* order;   // nullable: the tile of each CTA
    const uint32_t* ids;
    const float* mean2d;
    const float* conic;
    const float* opacity;
    const float* rgb;
    float bg[3];
    float alpha_max;
    int early_cull;
    float* img;
    float* T_final;
    uint32_t* n_contrib;
    uint32_t* stats;
};

// Forward: one CTA of 128 threads per tile, two pixels a thread, each warp an 8 x 8 pixel block.  The tile's
// sorted list is taken in batches of kFwdBatch fragments, each thread staging one and testing it against the
// four blocks; a warp then walks its block's fragments four at a time (independent exponentials, then
// Algorithm 1 in order, by selects).
//
// What bounds it: instruction issue.  Hence the packed arithmetic (one issue slot for the thread's two
// pixels) and the block test, which leaves out only what no pixel of the block can blend: q, the
// fragment's conic form, is at least its minimum over the block's pixel centres, and alpha >= 1/255 needs
// q <= the reach limit.  Both are compared with a slack for the rounding of q here and in the exponent
// (kQSlack of the sum of magnitudes of its terms); conics that are not safely positive definite, and
// values too large for the bound, are walked everywhere.  1024 x 512, 250k Gaussians of small footprints: 230 us
// with every entry at every pixel, 133 us so, 98 us with the tiles longest first.  Without the tests (kCull false)
// a warp skips the blend of a group that none of its pixels passes: 1920 x 1080, 1M Gaussians in 3-sigma lists
// 932 -> 818 us (one pixel a thread 842; with EarlyCull, which then skips the exponentials, 704 and here 889).
constexpr int kFwdThreads = kPairThreads;
constexpr int kFwdWarps = kFwdThreads / 32;
constexpr int kFwdBatch = kFwdThreads;
constexpr int kFwdGroup = 4;
constexpr float kQSlack = 2e-6f;   // about 17 roundings

// The block tests' limit on q for a Gaussian at (x, y) from the tile's centre, the same in the forward and the
// backward: negative when no pixel blends it, infinite when the test must not be used.
__device__ __forceinline__ float fp32_limit(float x, float y, float a, float b, float c, float o, float lno) {
    const float inf = __int_as_float(0x7f800000);
    const float X = fabsf(x) + 0.5f * kTile, Y = fabsf(y) + 0.5f * kTile;
    const float M = a * X * X + 2.f * fabsf(b) * X * Y + c * Y * Y;
    if (!(a > 0.f && c > 0.f && a * c - b * b > 1e-5f * (a * c) && M < kHuge && o < kHuge)) return inf;
    const float lim = reach_limit(lno);
    return lim >= 0.f ? lim + kQSlack * M : -1.f;
}

template <bool kEarly, bool kStats, bool kCull>
__global__ void __launch_bounds__(kFwdThreads, 7) k_render_fp32(FwdParams p) {
    __shared__ PairRec s_f[2][kFwdBatch + 1];                    // the last record is blended by no pixel
    __shared__ uint32_t s_mark[2][kFwdWarps + 1][kFwdBatch / 32];   // per block: fragments to walk; last: odd colours
    __shared__ __align__(4) uint8_t s_list[kFwdWarps][kFwdBatch + kFwdGroup];
    const long long t_start = kStats ? clock64() : 0;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int tile = p.order ? (int)p.order[blockIdx.x] : (int)blockIdx.x;
    if (tile < 0 || tile >= p.cam.grid_w * p.cam.grid_h) return;   // never index past the grid
    const int tx = tile % p.cam.grid_w, ty = tile / p.cam.grid_w;
    const PairPixels q = pair_pixels(warp, lane);
    const float cx = (float)(tx * kTile + kTile / 2), cy = (float)(ty * kTile + kTile / 2);
    const uint32_t start = p.ranges[2 * tile], stop = p.ranges[2 * tile + 1];
    const uint32_t len = stop > start ? stop - start : 0u;   // an inverted range is an empty list
    const float amax = p.alpha_max, inf = __int_as_float(0x7f800000);
    const int px_i = tx * kTile + q.lx, py_i = ty * kTile + q.ly;
    const bool in0 = px_i < p.cam.width && py_i < p.cam.height, in1 = px_i < p.cam.width && py_i + 4 < p.cam.height;
    const f32x2 npx = pack2f(-(px_i + 0.5f), -(px_i + 0.5f)), npy = pack2f(-(py_i + 0.5f), -(py_i + 4 + 0.5f));
    f32x2 T = pack2f(1.f, 1.f), C0 = 0ull, C1 = 0ull, C2 = 0ull;   // C: minus the colour
    float thr0 = in0 ? -kCullAlpha : -inf, thr1 = in1 ? -kCullAlpha : -inf;   // -alpha blends at or below; -inf: ended
    uint32_t last0 = 0, last1 = 0, n_eval0 = len, n_eval1 = len, n_blend0 = 0, n_blend1 = 0, slots = 0, walked = 0;

    // thread t's fragment of the next batch, in registers during the walk of the current one
    float mx = 0.f, my = 0.f, a = 0.f, b = 0.f, c = 0.f, o = 0.f, r = 0.f, g = 0.f, bl = 0.f;
    uint32_t id = t < len ? p.ids[start + t] : 0u;
    auto fetch = [&](uint32_t i) {   // fragment i, whose id is known; the id of the batch after
        if (i < len) {
            const float2 m = reinterpret_cast<const float2*>(p.mean2d)[id];
            mx = m.x; my = m.y;
            a = p.conic[3 * (size_t)id]; b = p.conic[3 * (size_t)id + 1]; c = p.conic[3 * (size_t)id + 2];
            o = p.opacity[id];
            r = p.rgb[3 * (size_t)id]; g = p.rgb[3 * (size_t)id + 1]; bl = p.rgb[3 * (size_t)id + 2];
        }
        if (i + kFwdBatch < len) id = p.ids[start + i + kFwdBatch];
    };
    auto stage = [&](uint32_t i, int buf) {
        bool hit[kFwdWarps + 1] = {};
        if (i < len) {
            const float lno = __logf(o);
            s_f[buf][t] = pair_rec(mx, my, a, b, c, o, r, g, bl, lno);
            hit[kFwdWarps] = !(fabsf(r) + fabsf(g) + fabsf(bl) < kHuge);
            const float lx = mx - cx, ly = my - cy;
            const float lim = kCull ? fp32_limit(lx, ly, a, b, c, o, lno) : inf;
            if (lim >= 0.f) {
                const float ia = __fdividef(1.f, a), ic = __fdividef(1.f, c);
#pragma unroll
                for (int k = 0; k < kFwdWarps; ++k) {
                    const float x0 = 8.f * (k & 1) - 7.5f, y0 = 8.f * (k >> 1) - 7.5f;
                    hit[k] = lim == inf || min_q_box_facing(lx, ly, a, b, c, ia, ic, x0, x0 + 7.f, y0, y0 + 7.f) <= lim;
                }
            }
        }
#pragma unroll
        for (int k = 0; k <= kFwdWarps; ++k) {
            const uint32_t m = __ballot_sync(0xffffffffu, hit[k]);
            if (lane == 0) s_mark[buf][k][warp] = m;
        }
    };
    if (t < 2) s_f[t][kFwdBatch] = pair_rec(0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
    if (len) {
        fetch(t);
        stage(t, 0);
        fetch(kFwdBatch + t);
    }
    bool more = __syncthreads_or(in0 || in1);
    for (uint32_t b0 = 0, buf = 0; b0 < len && more; b0 += kFwdBatch, buf ^= 1u) {
        bool strict = false;
        uint32_t n = 0;
#pragma unroll
        for (int k = 0; k < kFwdBatch / 32; ++k) {
            const uint32_t m = s_mark[buf][warp][k];
            strict = strict || s_mark[buf][kFwdWarps][k];
            if ((m >> lane) & 1u) s_list[warp][n + __popc(m & ((1u << lane) - 1u))] = (uint8_t)(32 * k + lane);
            n += __popc(m);
        }
        if (lane < kFwdGroup) s_list[warp][n + lane] = (uint8_t)kFwdBatch;   // pads the last group
        __syncwarp();
        for (uint32_t at = 0; at < n; at += kFwdGroup) {
            if (__all_sync(0xffffffffu, fmaxf(thr0, thr1) == -inf)) break;
            if (kStats) slots += 64u * (n - at < (uint32_t)kFwdGroup ? n - at : (uint32_t)kFwdGroup);
            const uint32_t four = *reinterpret_cast<const uint32_t*>(&s_list[warp][at]);
            float n0[kFwdGroup], n1[kFwdGroup];   // minus the alphas
#pragma unroll
            for (int f = 0; f < kFwdGroup; ++f) {
                const PairRec& rec = s_f[buf][(four >> (8 * f)) & 0xFFu];
                const ulonglong2 xa = rec.q[0], bc = rec.q[1], yo = rec.q[2];
                const f32x2 pw = pair_power(xa.y, bc.x, bc.y, add2(xa.x, npx), add2(yo.x, npy));
                const f32x2 raw = mul2(yo.y, pack2f(expf(lo2(pw)), expf(hi2(pw))));
                n0[f] = fmaxf(-amax, lo2(raw));
                n1[f] = fmaxf(-amax, hi2(raw));
                if (kEarly) {   // Sec. 4.1
                    const float lno = rec.lno();
                    if (lo2(pw) + lno < kBetaCull) n0[f] = 0.f;
                    if (hi2(pw) + lno < kBetaCull) n1[f] = 0.f;
                }
            }
            if (!kCull) {   // without block tests most groups are blended nowhere in the block
                bool any = false;
#pragma unroll
                for (int f = 0; f < kFwdGroup; ++f) any = any || n0[f] <= thr0 || n1[f] <= thr1;
                if (!__any_sync(0xffffffffu, any)) continue;
            }
#pragma unroll
            for (int f = 0; f < kFwdGroup; ++f) {
                const uint32_t j = (four >> (8 * f)) & 0xFFu;
                const uint32_t pos = b0 + j + 1u;
                const bool pass0 = n0[f] <= thr0, pass1 = n1[f] <= thr1;                // Eq. (5)
                const f32x2 na = pack2f(pass0 ? n0[f] : 0.f, pass1 ? n1[f] : 0.f);
                const f32x2 Tn = fma2(na, T, T);                                        // T - alpha T
                f32x2 wn = mul2(na, T);
                const bool end0 = lo2(Tn) < kTmin, end1 = hi2(Tn) < kTmin;              // Algorithm 1: terminate
                wn = pack2f(end0 ? 0.f : lo2(wn), end1 ? 0.f : hi2(wn));
                T = pack2f(end0 ? lo2(T) : lo2(Tn), end1 ? hi2(T) : hi2(Tn));
                thr0 = end0 ? -inf : thr0;
                thr1 = end1 ? -inf : thr1;
                last0 = pass0 && !end0 ? pos : last0;
                last1 = pass1 && !end1 ? pos : last1;
                f32x2 cr = s_f[buf][j].q[3].x, cg = s_f[buf][j].q[3].y, cb = s_f[buf][j].q[4].x;
                if (strict) {   // 0 times an infinity or a NaN would reach pixels that do not blend it
                    cr = where2(wn, cr);
                    cg = where2(wn, cg);
                    cb = where2(wn, cb);
                }
                C0 = fma2(cr, wn, C0);
                C1 = fma2(cg, wn, C1);
                C2 = fma2(cb, wn, C2);
                if (kStats) {
                    n_eval0 = end0 ? pos : n_eval0;
                    n_eval1 = end1 ? pos : n_eval1;
                    n_blend0 += pass0 && !end0;
                    n_blend1 += pass1 && !end1;
                }
            }
        }
        walked = b0 + kFwdBatch < len ? b0 + kFwdBatch : len;
        if (b0 + kFwdBatch < len) {
            stage(b0 + kFwdBatch + t, (int)(buf ^ 1u));
            fetch(b0 + 2 * kFwdBatch + t);
        }
        // one barrier a batch: batch k walked and its buffer free, batch k + 1 staged
        more = __syncthreads_or(fmaxf(thr0, thr1) > -inf);
    }
    const size_t plane = (size_t)p.cam.width * p.cam.height;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (k == 0 ? !in0 : !in1) continue;
        const size_t pix = (size_t)(py_i + 4 * k) * p.cam.width + px_i;
        const float Tk = k ? hi2(T) : lo2(T);
        p.img[pix] = fmaf(Tk, p.bg[0], -(k ? hi2(C0) : lo2(C0)));
        p.img[plane + pix] = fmaf(Tk, p.bg[1], -(k ? hi2(C1) : lo2(C1)));
        p.img[2 * plane + pix] = fmaf(Tk, p.bg[2], -(k ? hi2(C2) : lo2(C2)));
        p.T_final[pix] = Tk;
        p.n_contrib[pix] = k ? last1 : last0;
    }
    if (kStats) {
        __shared__ unsigned long long s_acc[3];
        if (t < 3) s_acc[t] = 0ull;
        __syncthreads();
        if (in0) {
            atomicAdd(&s_acc[0], (unsigned long long)n_blend0);
            atomicAdd(&s_acc[1], (unsigned long long)(n_eval0 - n_blend0));
        }
        if (in1) {
            atomicAdd(&s_acc[0], (unsigned long long)n_blend1);
            atomicAdd(&s_acc[1], (unsigned long long)(n_eval1 - n_blend1));
        }
        if (lane == 0) atomicAdd(&s_acc[2], (unsigned long long)slots);
        __syncthreads();
        if (t == 0) {
            uint32_t* st = p.stats + 8 * tile;
            atomicAdd(&st[0], (uint32_t)s_acc[0]);
            atomicAdd(&st[1], (uint32_t)s_acc[1]);
            atomicAdd(&st[2], (uint32_t)s_acc[2]);
            atomicAdd(&st[3], len);
            atomicAdd(&st[4], walked);
            atomicAdd(&st[5], (uint32_t)((clock64() - t_start) >> 6));
        }
    }
}

// ---------------------------------------------------------------- backward
//
// One CTA of 128 threads per tile, two pixels a thread, each warp an 8 x 8 pixel block.  Each pixel replays
// its fragments 0 .. n_contrib-1 front to back with the forward's FP32 alpha arithmetic (pair_power), so T_j
// matches the FP32 forward bit for bit; the colour blended after fragment j is img - bg T_final - (prefix up
// to j).
//
// What bounds it: instruction issue (the replay and the sums over a warp's pixels; memory is idle).
// Hence
//   - the two pixels of a thread go through packed FP32 instructions (fma.rn.f32x2 and its kin: one issue
//     slot for two IEEE results), from operands staged twice over in shared memory;
//   - a warp replays only the fragments that the forward's block test admits (fp32_limit: with the bare reach limit,
//     needles whose form cancels were blended by the forward and left out here), listed per batch of
//     kBwdBatch fragments, four at a time: the exponentials of four fragments are independent, and
//     their sums share the warp reduction: two transposing levels leave each quarter of the warp with one
//     fragment's nine sums over eight lanes, three more finish them (37 shuffles for four fragments; 14
//     each one by one);
//   - the block adds its warps' sums once per batch of 128, a thread per fragment (slots that no warp replayed
//     are not read), and issues one atomic per parameter.
// Four blocks of 128 threads an SM (128 registers; five blocks spill, and with two fragments' exponentials at a time
// are slower).  1024 x 512, 250k Gaussians: 403 us one fragment at a time, 263 us so, 193 us with the tiles
// longest first; 1280 x 720, 500k wide ones: 315 and 236 us; 1920 x 1080, 1M: 732 and 583 us (515 longest first).
// The sums over a tile are formed in a fixed order (a thread's two pixels, the butterfly's levels 16 .. 1,
// the warps): only the order of the tiles' atomics differs between runs.

struct BwdParams {
    DevCamera cam;
    const uint32_t* ranges;
    const uint32_t* order;   // nullable: the tile of each CTA
    const uint32_t* ids;
    const float* mean2d;
    const float* conic;
    const float* opacity;
    const float* rgb;
    float bg[3];
    float alpha_max;
    int early_cull;
    const float* img;
    const float* T_final;
    const uint32_t* n_contrib;
    const float* dL_dimg;
    float* dmean2d;
    float* dconic;
    float* dopacity;
    float* drgb;
};

constexpr int kBwdThreads = kPairThreads;
constexpr int kBwdWarps = kBwdThreads / 32;
constexpr int kBwdBatch = kBwdThreads;   // fragments staged at a time, one a thread
constexpr int kBwdGroup = 4;             // fragments replayed together: one per 8 lanes of the reduction
constexpr int kBwdParams = 9;            // dmean2d (2), dconic (3), dopacity, drgb (3), up to constant factors

template <bool kEarly>
__global__ void __launch_bounds__(kBwdThreads, 4) k_render_bwd(BwdParams p) {
    __shared__ PairRec s_f[kBwdBatch + 1];                             // the last record contributes nothing
    __shared__ float s_part[kBwdWarps][kBwdBatch + 1][kBwdParams];
    __shared__ uint32_t s_mark[2][kBwdWarps][kBwdBatch / 32];          // per block: fragments to replay
    __shared__ __align__(4) uint8_t s_list[kBwdWarps][kBwdBatch + kBwdGroup];
    __shared__ uint32_t s_max;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int tile = p.order ? (int)p.order[blockIdx.x] : (int)blockIdx.x;
    if (tile < 0 || tile >= p.cam.grid_w * p.cam.grid_h) return;   // never index past the grid
    const int tx = tile % p.cam.grid_w, ty = tile / p.cam.grid_w;
    const PairPixels q = pair_pixels(warp, lane);
    const float cx = (float)(tx * kTile + kTile / 2), cy = (float)(ty * kTile + kTile / 2);
    const uint32_t start = p.ranges[2 * tile], stop = p.ranges[2 * tile + 1];
    if (stop <= start) return;   // an empty list (an inverted range is one): no gradient
    const uint32_t end = stop;
    const float amax = p.alpha_max, inf = __int_as_float(0x7f800000);

    // per pixel: n_contrib, -dL/dimg, T_final, the colour still to come, the replayed T
    uint32_t nc[2] = {0u, 0u};
    float ng[3][2] = {}, R_[3][2] = {}, Tf_[2] = {1.f, 1.f};
    const float bg0 = p.bg[0], bg1 = p.bg[1], bg2 = p.bg[2];
    const bool has_bg = bg0 != 0.f || bg1 != 0.f || bg2 != 0.f;   // a NaN counts
    const int px_i = tx * kTile + q.lx;
    const float px = px_i + 0.5f;
    const size_t plane = (size_t)p.cam.width * p.cam.height;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int py_i = ty * kTile + q.ly + 4 * k;
        if (px_i < p.cam.width && py_i < p.cam.height) {
            const size_t pix = (size_t)py_i * p.cam.width + px_i;
            nc[k] = p.n_contrib[pix];
            Tf_[k] = p.T_final[pix];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                ng[c][k] = -p.dL_dimg[c * plane + pix];
                R_[c][k] = fmaf(-Tf_[k], p.bg[c], p.img[c * plane + pix]);
            }
        }
    }
    const f32x2 npx = pack2f(-px, -px);
    const f32x2 npy = pack2f(-(ty * kTile + q.ly + 0.5f), -(ty * kTile + q.ly + 4 + 0.5f));
    const f32x2 ng0 = pack2f(ng[0][0], ng[0][1]), ng1 = pack2f(ng[1][0], ng[1][1]), ng2 = pack2f(ng[2][0], ng[2][1]);
    const f32x2 one = pack2f(1.f, 1.f), Tf = pack2f(Tf_[0], Tf_[1]);
    f32x2 R0 = pack2f(R_[0][0], R_[0][1]), R1 = pack2f(R_[1][0], R_[1][1]), R2 = pack2f(R_[2][0], R_[2][1]), T = one;
    bool odd_pixel = false;   // values that 0 must not multiply
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < 2; ++k) odd_pixel = odd_pixel || !(fabsf(ng[c][k]) + fabsf(R_[c][k]) < kHuge);

    const uint32_t warp_nc = __reduce_max_sync(0xffffffffu, nc[0] > nc[1] ? nc[0] : nc[1]);
    if (t == 0) {
        s_max = 0u;
        s_f[kBwdBatch] = pair_rec(0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    if (lane == 0) atomicMax(&s_max, warp_nc);
    __syncthreads();
    const uint32_t span = s_max;
    uint32_t g_next = start + t < end ? p.ids[start + t] : 0u;
    for (uint32_t b0 = 0, par = 0; b0 < span; b0 += kBwdBatch, par ^= 1u) {
        // thread t stages fragment t of the batch and tests it against the four blocks
        const uint32_t g = g_next;
        const bool valid = b0 + t < end - start && b0 + t < span;
        bool near_[kBwdWarps] = {}, odd = odd_pixel;
        if (valid) {
            const float2 m = reinterpret_cast<const float2*>(p.mean2d)[g];
            const float a = p.conic[3 * (size_t)g], b = p.conic[3 * (size_t)g + 1], c = p.conic[3 * (size_t)g + 2], o = p.opacity[g];
            const float lno = __logf(o), lim = fp32_limit(m.x - cx, m.y - cy, a, b, c, o, lno);
            const float r = p.rgb[3 * (size_t)g], gr = p.rgb[3 * (size_t)g + 1], bl = p.rgb[3 * (size_t)g + 2];
            s_f[t] = pair_rec(m.x, m.y, a, b, c, o, r, gr, bl, lno);
            odd = odd || !(fabsf(r) + fabsf(gr) + fabsf(bl) < kHuge) || !(fabsf(a) + fabsf(b) + fabsf(c) < kHuge) ||
                  !(fabsf(m.x) + fabsf(m.y) < kHuge);
            if (lim >= 0.f) {
                const float ia = __fdividef(1.f, a), ic = __fdividef(1.f, c);
#pragma unroll
                for (int k = 0; k < kBwdWarps; ++k) {
                    const float x0 = 8.f * (k & 1) - 7.5f, y0 = 8.f * (k >> 1) - 7.5f;
                    near_[k] = lim == inf || min_q_box_facing(m.x - cx, m.y - cy, a, b, c, ia, ic, x0, x0 + 7.f, y0, y0 + 7.f) <= lim;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kBwdWarps; ++k) {
            const uint32_t m = __ballot_sync(0xffffffffu, near_[k]);
            if (lane == 0) s_mark[par][k][warp] = m;
        }
        const uint32_t i_next = start + b0 + kBwdBatch + t;
        if (i_next < end) g_next = p.ids[i_next];
        const bool strict = __syncthreads_or(odd);
        // this warp's fragments: marked, and in some pixel's replay range
        uint32_t n = 0;
#pragma unroll
        for (int k = 0; k < kBwdBatch / 32; ++k) {
            const uint32_t first = b0 + 32 * k;
            const uint32_t in = warp_nc <= first ? 0u : (warp_nc - first >= 32u ? 0xFFFFFFFFu : (1u << (warp_nc - first)) - 1u);
            const uint32_t m = s_mark[par][warp][k] & in;
            if (lane == 0) s_mark[par][warp][k] = m;
            if ((m >> lane) & 1u) s_list[warp][n + __popc(m & ((1u << lane) - 1u))] = (uint8_t)(32 * k + lane);
            n += __popc(m);
        }
        if (lane < kBwdGroup) s_list[warp][n + lane] = (uint8_t)kBwdBatch;   // pads the last group
        __syncwarp();
        // two copies of the replay: the masks that odd values need cost 5% in one (1024 x 512, 250k Gaussians: 307 and
        // 278 us)
        auto replay = [&](auto odd_values) {
            constexpr bool kStrict = decltype(odd_values)::value;
            for (uint32_t at = 0; at < n; at += kBwdGroup) {
                const uint32_t four = *reinterpret_cast<const uint32_t*>(&s_list[warp][at]);
                // alphas of the four fragments (negated; 0: the pixel does not blend it), exp(power) (0: or with a
                // clamped alpha), dx, dy
                f32x2 na[kBwdGroup], G[kBwdGroup], dx[kBwdGroup], dy[kBwdGroup];
                bool any = false;
#pragma unroll
                for (int f = 0; f < kBwdGroup; ++f) {
                    const uint32_t j = (four >> (8 * f)) & 0xFFu;
                    const PairRec& r = s_f[j];
                    const ulonglong2 xa = r.q[0], bc = r.q[1], yo = r.q[2];
                    dx[f] = add2(xa.x, npx);
                    dy[f] = add2(yo.x, npy);
                    const f32x2 pw = pair_power(xa.y, bc.x, bc.y, dx[f], dy[f]);
                    const float G0 = expf(lo2(pw)), G1 = expf(hi2(pw));
                    const f32x2 raw = mul2(yo.y, pack2f(G0, G1));   // -o exp(power)
                    const float a0 = fmaxf(-amax, lo2(raw)), a1 = fmaxf(-amax, hi2(raw));
                    bool in0 = a0 <= -kCullAlpha && b0 + j < nc[0], in1 = a1 <= -kCullAlpha && b0 + j < nc[1];
                    if (kEarly) {   // the forward's test
                        const float lno = r.lno();
                        in0 = in0 && !(lo2(pw) + lno < kBetaCull);
                        in1 = in1 && !(hi2(pw) + lno < kBetaCull);
                    }
                    any = any || in0 || in1;
                    na[f] = pack2f(in0 ? a0 : 0.f, in1 ? a1 : 0.f);
                    G[f] = pack2f(in0 && lo2(raw) >= -amax ? G0 : 0.f, in1 && hi2(raw) >= -amax ? G1 : 0.f);
                }
                const bool u16 = lane & 16, u8 = lane & 8, u4 = lane & 4, u2 = lane & 2, u1 = lane & 1;
                const uint32_t jl = (four >> ((u16 ? 8 : 0) + (u8 ? 16 : 0))) & 0xFFu;   // this quarter's fragment
                float* part = s_part[warp][jl];
                if (!__any_sync(0xffffffffu, any)) {
                    part[lane & 7] = 0.f;
                    part[8] = 0.f;
                    continue;
                }
                float z[2][kBwdParams];
#pragma unroll
                for (int f = 0; f < kBwdGroup; f += 2) {
                    float v[2][kBwdParams];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const f32x2 na_f = na[f + e], G_f = G[f + e];
                        f32x2 dx_f = dx[f + e], dy_f = dy[f + e];
                        const PairRec& r = s_f[(four >> (8 * (f + e))) & 0xFFu];
                        f32x2 cr = r.q[3].x, cg = r.q[3].y, cb = r.q[4].x, h0 = ng0, h1 = ng1, h2 = ng2;
                        if (kStrict) {   // 0 times an infinity or a NaN would reach what does not blend it
                            cr = where2(na_f, cr); cg = where2(na_f, cg); cb = where2(na_f, cb);
                            h0 = where2(na_f, h0); h1 = where2(na_f, h1); h2 = where2(na_f, h2);
                        }
                        const f32x2 wn = mul2(na_f, T);   // -alpha T
                        R0 = fma2(cr, wn, R0);
                        R1 = fma2(cg, wn, R1);
                        R2 = fma2(cb, wn, R2);
                        // -1 / (1 - alpha): the approximate reciprocal (1 ulp) and one Newton-Raphson step, which
                        // squares its error: within an ulp, the rounding of the step's last operation
                        const f32x2 om = add2(one, na_f);
                        const f32x2 r0 = pack2f(rcp_approx(-lo2(om)), rcp_approx(-hi2(om)));
                        const f32x2 nia = fma2(fma2(om, r0, one), r0, r0);
                        f32x2 X0 = R0, X1 = R1, X2 = R2;
                        if (has_bg) {
                            X0 = fma2(Tf, pack2f(bg0, bg0), R0);
                            X1 = fma2(Tf, pack2f(bg1, bg1), R1);
                            X2 = fma2(Tf, pack2f(bg2, bg2), R2);
                        }
                        // -dL/dalpha = -g (c T - (R + T_final bg) / (1 - alpha))
                        const f32x2 A0 = fma2(cr, T, mul2(X0, nia)), A1 = fma2(cg, T, mul2(X1, nia)), A2 = fma2(cb, T, mul2(X2, nia));
                        const f32x2 nd_all = fma2(h2, A2, fma2(h0, A0, mul2(h1, A1)));
                        const f32x2 nd = where2(G_f, nd_all);
                        const f32x2 d = mul2(nd, na_f);   // dL/dpower
                        const f32x2 bx = mul2(r.q[1].x, dx_f), cy = mul2(r.q[1].y, dy_f);
                        f32x2 m0 = fma2(r.q[1].x, dy_f, mul2(r.q[0].y, dx_f));   // -(a dx + b dy)
                        f32x2 m1 = pack2f(__fadd_rn(lo2(bx), lo2(cy)), __fadd_rn(hi2(bx), hi2(cy)));   // -(b dx + c dy)
                        if (kStrict) {   // nor may the geometry's, where d is 0
                            m0 = where2(G_f, m0); m1 = where2(G_f, m1);
                            dx_f = where2(G_f, dx_f); dy_f = where2(G_f, dy_f);
                        }
                        const f32x2 ddx = mul2(d, dx_f), ddy = mul2(d, dy_f);
                        v[e][0] = dot2(d, m0);
                        v[e][1] = dot2(d, m1);
                        v[e][2] = dot2(ddx, dx_f);
                        v[e][3] = dot2(ddx, dy_f);
                        v[e][4] = dot2(ddy, dy_f);
                        v[e][5] = dot2(nd, G_f);
                        v[e][6] = dot2(wn, h0);
                        v[e][7] = dot2(wn, h1);
                        v[e][8] = dot2(wn, h2);
                        T = fma2(na_f, T, T);
                    }
#pragma unroll
                    for (int k = 0; k < kBwdParams; ++k) z[f / 2][k] = exchange(v[0][k], v[1][k], u16, 16);
                }
                float y[kBwdParams];
#pragma unroll
                for (int k = 0; k < kBwdParams; ++k) y[k] = exchange(z[0][k], z[1][k], u8, 8);
                // value 4 bit2 + 2 bit1 + bit0 of the first eight ends in each lane of the quarter, the ninth in all
                const float e0 = exchange(y[0], y[4], u4, 4), e1 = exchange(y[1], y[5], u4, 4);
                const float e2 = exchange(y[2], y[6], u4, 4), e3 = exchange(y[3], y[7], u4, 4);
                const float k0 = exchange(e0, e2, u2, 2), k1 = exchange(e1, e3, u2, 2);
                const float mine = exchange(k0, k1, u1, 1);
                float ninth = y[8];
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) ninth += __shfl_xor_sync(0xffffffffu, ninth, o);
                part[lane & 7] = mine;
                if ((lane & 7) == 0) part[8] = ninth;
            }
        };
        if (strict) replay(std::true_type{}); else replay(std::false_type{});
        __syncthreads();
        // thread t adds the warps' sums of fragment t
        float s[kBwdParams] = {};
        bool used = false;
#pragma unroll
        for (int w = 0; w < kBwdWarps; ++w) {
            if ((s_mark[par][w][warp] >> lane) & 1u) {
                used = true;
#pragma unroll
                for (int k = 0; k < kBwdParams; ++k) s[k] += s_part[w][t][k];
            }
        }
        if (used) {
            const float scale[kBwdParams] = {1.f, 1.f, -0.5f, -1.f, -0.5f, -1.f, 1.f, 1.f, 1.f};
            float* dst[kBwdParams] = {p.dmean2d + 2 * (size_t)g, p.dmean2d + 2 * (size_t)g + 1, p.dconic + 3 * (size_t)g,
                                      p.dconic + 3 * (size_t)g + 1, p.dconic + 3 * (size_t)g + 2, p.dopacity + g,
                                      p.drgb + 3 * (size_t)g, p.drgb + 3 * (size_t)g + 1, p.drgb + 3 * (size_t)g + 2};
#pragma unroll
            for (int k = 0; k < kBwdParams; ++k)
                if (s[k] != 0.f) atomicAdd(dst[k], scale[k] * s[k]);
        }
    }
}

}  // namespace
}  // namespace tcgs

namespace tcgs {
tcgs_status launch_render_fp32(const tcgs_camera* cam, const tcgs_render_opts* opts, const uint32_t* tile_ranges,
                               const uint32_t* ids_sorted, const float* mean2d, const float* conic,
                               const float* opacity, const float* rgb, const float* bg3, float* img, float* T_final,
                               uint32_t* n_contrib, const uint32_t* order, cudaStream_t s) {
    FwdParams p;
    p.cam = make_dev_camera(*cam);
    p.ranges = tile_ranges; p.order = order; p.ids = ids_sorted; p.mean2d = mean2d; p.conic = conic; p.opacity = opacity;
    p.rgb = rgb;
    for (int i = 0; i < 3; ++i) p.bg[i] = bg3 ? bg3[i] : 0.f;
    p.alpha_max = opts->alpha_max;
    p.early_cull = opts->early_cull;
    p.img = img; p.T_final = T_final; p.n_contrib = n_contrib; p.stats = opts->tile_stats;
    int tiles = p.cam.grid_w * p.cam.grid_h;
    auto launch = [&](auto kern) { kern<<<tiles, kFwdThreads, 0, s>>>(p); };
    if (opts->tile_cull) {
        if (p.early_cull) p.stats ? launch(k_render_fp32<true, true, true>) : launch(k_render_fp32<true, false, true>);
        else p.stats ? launch(k_render_fp32<false, true, true>) : launch(k_render_fp32<false, false, true>);
    } else {
        if (p.early_cull) p.stats ? launch(k_render_fp32<true, true, false>) : launch(k_render_fp32<true, false, false>);
        else p.stats ? launch(k_render_fp32<false, true, false>) : launch(k_render_fp32<false, false, false>);
    }
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}
}  // namespace tcgs

extern "C" tcgs_status tcgs_render_bwd_ordered(const tcgs_camera* cam, const tcgs_render_opts* opts,
                                               const uint32_t* tile_order, const uint32_t* tile_ranges,
                                               const uint32_t* ids_sorted, const float* mean2d, const float* conic,
                                               const float* opacity, const float* rgb, const float* bg3,
                                               const float* img, const float* T_final, const uint32_t* n_contrib,
                                               const float* dL_dimg, float* dmean2d, float* dconic,
                                               float* dopacity, float* drgb, tcgs_stream stream) {
    using namespace tcgs;
    if (!valid_camera(cam) || !opts || !tile_ranges || !ids_sorted || !mean2d || !conic || !opacity || !rgb ||
        !img || !T_final || !n_contrib || !dL_dimg || !dmean2d || !dconic || !dopacity || !drgb)
        return TCGS_ERR_INVALID;
    if (!(opts->alpha_max > 0.f && opts->alpha_max <= 1.f)) return TCGS_ERR_INVALID;
    if (opts->alpha_max >= 1.f) return TCGS_ERR_INVALID;  // 1 / (1 - alpha) must stay finite
    if (reinterpret_cast<uintptr_t>(mean2d) & 7) return TCGS_ERR_INVALID;
    BwdParams p;
    p.cam = make_dev_camera(*cam);
    p.ranges = tile_ranges; p.order = tile_order; p.ids = ids_sorted; p.mean2d = mean2d; p.conic = conic; p.opacity = opacity;
    p.rgb = rgb;
    for (int i = 0; i < 3; ++i) p.bg[i] = bg3 ? bg3[i] : 0.f;
    p.alpha_max = opts->alpha_max;
    p.early_cull = opts->early_cull;
    p.img = img; p.T_final = T_final; p.n_contrib = n_contrib; p.dL_dimg = dL_dimg;
    p.dmean2d = dmean2d; p.dconic = dconic; p.dopacity = dopacity; p.drgb = drgb;
    int tiles = p.cam.grid_w * p.cam.grid_h;
    if (p.early_cull) k_render_bwd<true><<<tiles, kBwdThreads, 0, (cudaStream_t)stream>>>(p);
    else k_render_bwd<false><<<tiles, kBwdThreads, 0, (cudaStream_t)stream>>>(p);
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}

extern "C" tcgs_status tcgs_render_bwd(const tcgs_camera* cam, const tcgs_render_opts* opts,
                                       const uint32_t* tile_ranges, const uint32_t* ids_sorted, const float* mean2d,
                                       const float* conic, const float* opacity, const float* rgb, const float* bg3,
                                       const float* img, const float* T_final, const uint32_t* n_contrib,
                                       const float* dL_dimg, float* dmean2d, float* dconic, float* dopacity,
                                       float* drgb, tcgs_stream stream) {
    return tcgs_render_bwd_ordered(cam, opts, nullptr, tile_ranges, ids_sorted, mean2d, conic, opacity, rgb, bg3, img,
                                   T_final, n_contrib, dL_dimg, dmean2d, dconic, dopacity, drgb, stream);
}
