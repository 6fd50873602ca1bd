// sched.cu -- the learned tile-cost model that orders the batched renderer's work queue.
//
// Not part of the paper: TC-GS accelerates each tile's alpha-blending; a multi-view batch still
// finishes with its most expensive tiles, whose cost (list entries walked until every pixel has
// terminated) is not the list length.  A small MLP (8 -> 32 -> 32 -> 1, FP16 weights and
// activations, FP32 accumulation) predicts log(tile cost) from cheap per-tile statistics; the
// queue is ordered longest-predicted first.  Its training data are the per-tile costs the
// renderer itself records (tile_stats).
//
// Kernels: per-tile features, feature normaliser, MLP forward, MLP backward
// (mean squared error), Adam.  The ordering sort lives with the radix sort in binsort.cu.
#include <mutex>

#include "common.cuh"
#include "f32x2.cuh"

namespace tcgs {
namespace {

constexpr int kIn = TCGS_MLP_IN, kHid = TCGS_MLP_HIDDEN;
// parameter layout (float32 masters): W1[kHid][kIn], b1[kHid], W2[kHid][kHid], b2[kHid], W3[kHid], b3
constexpr int kW1 = 0, kB1 = kW1 + kHid * kIn, kW2 = kB1 + kHid, kB2 = kW2 + kHid * kHid, kW3 = kB2 + kHid,
              kB3 = kW3 + kHid, kParams = kB3 + 1;
static_assert(kParams == TCGS_MLP_PARAMS, "parameter layout");

__device__ __forceinline__ float h16(float x) { return __half2float(__float2half_rn(x)); }

// ---------------------------------------------------------------- features

constexpr int kFewTilesPerSm = 4;
constexpr int kWarpTiles = 8;   // tiles a block where each has a warp

// NT threads per tile, kTiles tiles a block (several only with a warp each).  Bound by the latency of two dependent
// gathers (id, then the Gaussian's values from L2), so a thread has kDeep entries in flight, and where the view has few
// tiles a tile gets many threads: 16 views of 320 x 240 (300 tiles each, about 8000 entries a tile) took 8.13 ms
// with one warp a tile and one entry in flight and take 0.75 ms, bound by the gathers' requests (seven a list
// entry, 32 lines each).  Where the tiles' warps fill the chip, a warp each is faster than a block of 128
// (3840 x 2160, 1M small footprints: 69 and 159 us; 1920 x 1080, 300k wide ones: 496 and 648 us): nothing waits on
// barriers, and the lists that neighbouring tiles share are walked at the same time.
template <int NT, int kTiles, bool kPairs>
__global__ void __launch_bounds__(NT * kTiles) k_tile_features(DevCamera cam, const uint32_t* __restrict__ ranges,
                                                      const uint32_t* __restrict__ ids,
                                                      const float* __restrict__ mean2d,
                                                      const float* __restrict__ conic,
                                                      const float* __restrict__ opacity,
                                                      const float* __restrict__ depth,
                                                      const int32_t* __restrict__ radius, float* __restrict__ feat) {
    constexpr int kSums = 6, kDeep = 4;   // entries a thread has in flight
    __shared__ float s_sum[NT / 32][kSums];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile = kTiles == 1 ? blockIdx.x : blockIdx.x * kTiles + warp, tid = kTiles == 1 ? threadIdx.x : lane;
    if (kTiles > 1 && tile >= cam.grid_w * cam.grid_h) return;
    const int tx = tile % cam.grid_w, ty = tile / cam.grid_w;
    const float x0 = (float)(kTile * tx), y0 = (float)(kTile * ty);
    const uint32_t start = ranges[2 * tile], end = ranges[2 * tile + 1];
    const uint32_t len = end > start ? end - start : 0u;   // an inverted range is an empty list
    float so = 0.f, mo = 0.f, dmin = 3.0e38f, dmax = -3.0e38f, sdet = 0.f, cov = 0.f;
    for (uint32_t k0 = tid; k0 < len; k0 += kDeep * NT) {
        uint32_t g[kDeep];
        bool in[kDeep];
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            in[u] = k0 + u * NT < len;
            g[u] = ids[start + (in[u] ? k0 + u * NT : k0)];
        }
        float o[kDeep], d[kDeep], a[kDeep], b[kDeep], c[kDeep], r[kDeep];
        float2 m[kDeep];
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            o[u] = opacity[g[u]];
            d[u] = depth[g[u]];
            if (kPairs) {   // 8 bytes at the multiple of 8 inside the conic, and the other 4
                const bool odd = g[u] & 1u;
                const float* q = conic + 3 * (size_t)g[u];
                const float2 two = *reinterpret_cast<const float2*>(q + (odd ? 1 : 0));
                const float other = q[odd ? 0 : 2];
                a[u] = odd ? other : two.x;
                b[u] = odd ? two.x : two.y;
                c[u] = odd ? two.y : other;
            } else {
                a[u] = conic[3 * (size_t)g[u]]; b[u] = conic[3 * (size_t)g[u] + 1]; c[u] = conic[3 * (size_t)g[u] + 2];
            }
            m[u] = reinterpret_cast<const float2*>(mean2d)[g[u]];
            r[u] = (float)radius[g[u]];
        }
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            if (!in[u]) continue;
            so += o[u];
            mo = fmaxf(mo, o[u]);
            dmin = fminf(dmin, d[u]);
            dmax = fmaxf(dmax, d[u]);
            sdet += __logf(fmaxf(a[u] * c[u] - b[u] * b[u], 1e-30f));
            const float ox = fmaxf(0.f, fminf(m[u].x + r[u], x0 + kTile) - fmaxf(m[u].x - r[u], x0));
            const float oy = fmaxf(0.f, fminf(m[u].y + r[u], y0 + kTile) - fmaxf(m[u].y - r[u], y0));
            cov += ox * oy * (1.f / (kTile * kTile));
        }
    }
    auto over_warp = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            so += __shfl_xor_sync(0xffffffffu, so, o);
            mo = fmaxf(mo, __shfl_xor_sync(0xffffffffu, mo, o));
            dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
            dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
            sdet += __shfl_xor_sync(0xffffffffu, sdet, o);
            cov += __shfl_xor_sync(0xffffffffu, cov, o);
        }
    };
    over_warp();
    if (NT > 32) {
        if (lane == 0) {
            const float v[kSums] = {so, mo, dmin, dmax, sdet, cov};
#pragma unroll
            for (int k = 0; k < kSums; ++k) s_sum[warp][k] = v[k];
        }
        __syncthreads();
        if (warp > 0) return;
        const bool in = lane < NT / 32;
        so = in ? s_sum[lane][0] : 0.f;
        mo = in ? s_sum[lane][1] : 0.f;
        dmin = in ? s_sum[lane][2] : 3.0e38f;
        dmax = in ? s_sum[lane][3] : -3.0e38f;
        sdet = in ? s_sum[lane][4] : 0.f;
        cov = in ? s_sum[lane][5] : 0.f;
        over_warp();
    }
    if (lane == 0) {
        const float n = (float)len;
        const float inv = n > 0.f ? 1.f / n : 0.f;
        const int w_in = min(kTile, cam.width - kTile * tx), h_in = min(kTile, cam.height - kTile * ty);
        float* f = feat + (size_t)tile * kIn;
        f[0] = log1pf(n);
        f[1] = so * inv;
        f[2] = mo;
        f[3] = n > 0.f ? log1pf(dmax - dmin) : 0.f;
        f[4] = sdet * inv;
        f[5] = log1pf(cov);
        f[6] = logf((float)cam.width * (float)cam.height);
        f[7] = (float)(w_in * h_in) * (1.f / (kTile * kTile));
    }
}

// norm[0..7] = mean, norm[8..15] = 1 / max(std, 1e-6) of each feature column (FP64 sums)
__global__ void __launch_bounds__(1024) k_feature_norm(const float* __restrict__ x, int n, float* __restrict__ norm) {
    __shared__ double s1[kIn][32], s2[kIn][32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    double a[kIn], b[kIn];
#pragma unroll
    for (int k = 0; k < kIn; ++k) a[k] = b[k] = 0.0;
    for (int i = t; i < n; i += blockDim.x)
#pragma unroll
        for (int k = 0; k < kIn; ++k) {
            const double v = x[(size_t)i * kIn + k];
            a[k] += v;
            b[k] += v * v;
        }
#pragma unroll
    for (int k = 0; k < kIn; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            a[k] += __shfl_xor_sync(0xffffffffu, a[k], o);
            b[k] += __shfl_xor_sync(0xffffffffu, b[k], o);
        }
        if (lane == 0) { s1[k][warp] = a[k]; s2[k][warp] = b[k]; }
    }
    __syncthreads();
    if (t < kIn) {
        double A = 0.0, B = 0.0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) { A += s1[t][w]; B += s2[t][w]; }
        const double mean = n > 0 ? A / n : 0.0;
        const double var = n > 0 ? B / n - mean * mean : 0.0;
        const double sd = var > 1e-12 ? sqrt(var) : 1e-6;
        norm[t] = (float)mean;
        norm[kIn + t] = (float)(1.0 / sd);
    }
}

// ---------------------------------------------------------------- MLP

// One item a thread.  The weights lie in shared memory with the outputs of a layer side by side, so that
// one 16-byte broadcast read feeds two packed FP32 operations (fma.rn.f32x2: two outputs of the same
// input); every output's sum keeps the order bias, inputs 0 .. 31.  Read one weight at a time (and, in the
// forward, lifted out of a loop over items into spilled registers) the two kernels took 122 us forward
// and 129 us backward for 56,048 items; they take 8 and 28 us.
struct __align__(16) MlpWeights {   // FP16-rounded
    float w1[kIn][kHid], b1[kHid];  // [input][output]
    float w2[kHid][kHid + 4], b2[kHid];
    float w3[kHid];
    float b3, norm[2 * kIn], pad[3];
};

// 128 threads; every load is in flight before the first store (one at a time, their latencies were 4 us of
// either kernel).
constexpr int kMlpThreads = 128;

__device__ __forceinline__ void load_weights(const float* __restrict__ params, const float* __restrict__ norm,
                                             MlpWeights& w) {
    constexpr int kEach = (kParams + kMlpThreads - 1) / kMlpThreads;
    float v[kEach], nm = 0.f;
#pragma unroll
    for (int q = 0; q < kEach; ++q) {
        const int i = q * kMlpThreads + threadIdx.x;
        v[q] = i < kParams ? params[i] : 0.f;
    }
    if (threadIdx.x < 2 * kIn) nm = norm[threadIdx.x];
#pragma unroll
    for (int q = 0; q < kEach; ++q) {
        const int i = q * kMlpThreads + threadIdx.x;
        const float x = h16(v[q]);
        if (i < kB1) w.w1[i % kIn][i / kIn] = x;
        else if (i < kW2) w.b1[i - kB1] = x;
        else if (i < kB2) w.w2[(i - kW2) % kHid][(i - kW2) / kHid] = x;
        else if (i < kW3) w.b2[i - kB2] = x;
        else if (i < kB3) w.w3[i - kW3] = x;
        else if (i == kB3) w.b3 = x;
    }
    if (threadIdx.x < 2 * kIn) w.norm[threadIdx.x] = nm;
}

// acc[0 .. 31] += in * row[0 .. 31], two outputs an operation.
__device__ __forceinline__ void add_row(f32x2 (&acc)[kHid / 2], const float* row, float in) {
    const f32x2 v = pack2f(in, in);
#pragma unroll
    for (int q = 0; q < kHid / 4; ++q) {
        const ulonglong2 w = reinterpret_cast<const ulonglong2*>(row)[q];
        acc[2 * q] = fma2(w.x, v, acc[2 * q]);
        acc[2 * q + 1] = fma2(w.y, v, acc[2 * q + 1]);
    }
}

__device__ __forceinline__ void load_row(f32x2 (&acc)[kHid / 2], const float* row) {
#pragma unroll
    for (int q = 0; q < kHid / 4; ++q) {
        const ulonglong2 w = reinterpret_cast<const ulonglong2*>(row)[q];
        acc[2 * q] = w.x;
        acc[2 * q + 1] = w.y;
    }
}

__device__ __forceinline__ void relu_h16(const f32x2 (&acc)[kHid / 2], float* h) {
#pragma unroll
    for (int q = 0; q < kHid / 2; ++q) {
        h[2 * q] = h16(fmaxf(lo2(acc[q]), 0.f));
        h[2 * q + 1] = h16(fmaxf(hi2(acc[q]), 0.f));
    }
}

// forward of one item; keeps the FP16-rounded input and hidden activations
__device__ __forceinline__ float mlp_forward(const MlpWeights& w, const float* __restrict__ xi, float* xh, float* h1,
                                             float* h2) {
#pragma unroll
    for (int k = 0; k < kIn; ++k) xh[k] = h16((xi[k] - w.norm[k]) * w.norm[kIn + k]);
    f32x2 acc[kHid / 2];
    load_row(acc, w.b1);
#pragma unroll
    for (int k = 0; k < kIn; ++k) add_row(acc, w.w1[k], xh[k]);
    relu_h16(acc, h1);
    load_row(acc, w.b2);
#pragma unroll
    for (int k = 0; k < kHid; ++k) add_row(acc, w.w2[k], h1[k]);
    relu_h16(acc, h2);
    float y = w.b3;
#pragma unroll
    for (int k = 0; k < kHid; ++k) y = fmaf(w.w3[k], h2[k], y);
    return y;
}

__global__ void __launch_bounds__(kMlpThreads) k_mlp_fwd(const float* __restrict__ params, const float* __restrict__ norm,
                                                 const float* __restrict__ x, int n, float* __restrict__ y) {
    __shared__ MlpWeights w;
    load_weights(params, norm, w);
    __syncthreads();
    const int i = blockIdx.x * 128 + threadIdx.x;   // no loop: the compiler would lift the weights out of it, into spills
    if (i >= n) return;
    float xh[kIn], h1[kHid], h2[kHid];
    y[i] = mlp_forward(w, x + (size_t)i * kIn, xh, h1, h2);
}

// Backward of L = (1/n) sum (y - t)^2 for a block of kBwdItems items, one a thread: the deltas are formed in
// registers and kept in shared memory with the activations (in FP16, which holds them exactly); the block
// then sums every parameter's gradient over its items, each thread a 4 x 2 piece of W2's, two of W1's and
// one of the rest, and adds it to `grad` with one atomic each.  61 KB a block: 3 blocks an SM, so that
// 58,000 items are one wave.
constexpr int kBwdItems = kMlpThreads;

struct __align__(16) MlpBwdSmem {
    MlpWeights w;
    float w2[kHid][kHid + 4];              // [output][input], for the deltas
    float d1[kBwdItems][kHid + 4], d2[kBwdItems][kHid + 4], dy[kBwdItems];
    __half xh[kBwdItems][kIn], h1[kBwdItems][kHid + 8], h2[kBwdItems][kHid + 8];
};

__device__ __forceinline__ void store_halves(__half* dst, const float* v, int n) {   // n a multiple of 8
#pragma unroll
    for (int q = 0; q < n / 8; ++q) {
        uint32_t u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            u[k] = (uint32_t)__half_as_ushort(__float2half_rn(v[8 * q + 2 * k])) |
                   (uint32_t)__half_as_ushort(__float2half_rn(v[8 * q + 2 * k + 1])) << 16;
        reinterpret_cast<uint4*>(dst)[q] = make_uint4(u[0], u[1], u[2], u[3]);
    }
}

__device__ __forceinline__ f32x2 two_halves(const __half* p) {   // 4-byte aligned
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(p));
    return pack2f(v.x, v.y);
}

__global__ void __launch_bounds__(kBwdItems) k_mlp_bwd(const float* __restrict__ params, const float* __restrict__ norm,
                                                       const float* __restrict__ x, const float* __restrict__ target,
                                                       int n, float* __restrict__ grad, float* __restrict__ loss) {
    extern __shared__ __align__(16) uint8_t smem[];
    MlpBwdSmem& s = *reinterpret_cast<MlpBwdSmem*>(smem);
    load_weights(params, norm, s.w);
    __syncthreads();
    const int t = threadIdx.x;
#pragma unroll
    for (int q = 0; q < kHid * kHid / kBwdItems; ++q) {   // the weights by output, from those by input
        const int i = q * kBwdItems + t;
        s.w2[i / kHid][i % kHid] = s.w.w2[i % kHid][i / kHid];
    }
    __syncthreads();
    const int i = blockIdx.x * kBwdItems + t;
    float se = 0.f;
    if (i < n) {
        float xh[kIn], h1[kHid], h2[kHid];
        const float y = mlp_forward(s.w, x + (size_t)i * kIn, xh, h1, h2);
        const float e = y - target[i];
        se = e * e;
        const float dy = 2.f * e / (float)n;
        store_halves(s.xh[t], xh, kIn);
        store_halves(s.h1[t], h1, kHid);
        store_halves(s.h2[t], h2, kHid);
        s.dy[t] = dy;
        f32x2 acc[kHid / 2];
#pragma unroll
        for (int k = 0; k < kHid / 2; ++k) acc[k] = 0ull;
#pragma unroll
        for (int j = 0; j < kHid; ++j) {
            const float d2 = h2[j] > 0.f ? dy * s.w.w3[j] : 0.f;
            s.d2[t][j] = d2;
            add_row(acc, s.w2[j], d2);
        }
#pragma unroll
        for (int k = 0; k < kHid / 2; ++k) {
            s.d1[t][2 * k] = h1[2 * k] > 0.f ? lo2(acc[k]) : 0.f;
            s.d1[t][2 * k + 1] = h1[2 * k + 1] > 0.f ? hi2(acc[k]) : 0.f;
        }
    }
    __syncthreads();
    const int items = min(kBwdItems, n - (int)blockIdx.x * kBwdItems);
    const int j2 = (t >> 4) * 4, k2 = (t & 15) * 2;   // W2[j2 .. j2 + 3][k2, k2 + 1]
    const int j1 = t >> 2, k1 = (t & 3) * 2;          // W1[j1][k1, k1 + 1]
    const int warp = t >> 5, lane = t & 31;           // warp 0: b1, 1: b2, 2: W3, 3 (lane 0): b3
    f32x2 g2[4] = {0ull, 0ull, 0ull, 0ull}, g1 = 0ull;
    float g0 = 0.f;
#pragma unroll 4
    for (int it = 0; it < items; ++it) {
        const float4 d2 = *reinterpret_cast<const float4*>(&s.d2[it][j2]);
        const f32x2 h = two_halves(&s.h1[it][k2]);
        g2[0] = fma2(pack2f(d2.x, d2.x), h, g2[0]);
        g2[1] = fma2(pack2f(d2.y, d2.y), h, g2[1]);
        g2[2] = fma2(pack2f(d2.z, d2.z), h, g2[2]);
        g2[3] = fma2(pack2f(d2.w, d2.w), h, g2[3]);
        const float d1 = s.d1[it][j1];
        g1 = fma2(pack2f(d1, d1), two_halves(&s.xh[it][k1]), g1);
        if (warp == 0) g0 += s.d1[it][lane];
        else if (warp == 1) g0 += s.d2[it][lane];
        else if (warp == 2) g0 = fmaf(s.dy[it], __half2float(s.h2[it][lane]), g0);
        else g0 += s.dy[it];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        atomicAdd(&grad[kW2 + (j2 + k) * kHid + k2], lo2(g2[k]));
        atomicAdd(&grad[kW2 + (j2 + k) * kHid + k2 + 1], hi2(g2[k]));
    }
    atomicAdd(&grad[kW1 + j1 * kIn + k1], lo2(g1));
    atomicAdd(&grad[kW1 + j1 * kIn + k1 + 1], hi2(g1));
    if (warp < 3) atomicAdd(&grad[(warp == 0 ? kB1 : (warp == 1 ? kB2 : kW3)) + lane], g0);
    else if (lane == 0) atomicAdd(&grad[kB3], g0);
    if (loss) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
        if ((t & 31) == 0) atomicAdd(loss, se / (float)n);
    }
}

__global__ void k_adam(float* __restrict__ params, float* __restrict__ m, float* __restrict__ v,
                       float* __restrict__ grad, int n, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = grad[i];
    grad[i] = 0.f;   // consumed: the next backward accumulates into a zeroed buffer
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace
}  // namespace tcgs

extern "C" tcgs_status tcgs_tile_features(const tcgs_camera* cam, const uint32_t* tile_ranges,
                                          const uint32_t* ids_sorted, const float* mean2d, const float* conic,
                                          const float* opacity, const float* depth, const int32_t* radius,
                                          float* features, tcgs_stream stream) {
    using namespace tcgs;
    if (!valid_camera(cam) || !tile_ranges || !ids_sorted || !mean2d || !conic || !opacity || !depth || !radius ||
        !features || (reinterpret_cast<uintptr_t>(mean2d) & 7))
        return TCGS_ERR_INVALID;
    const DevCamera dc = make_dev_camera(*cam);
    const int tiles = dc.grid_w * dc.grid_h;
    // a view of few tiles leaves most of the chip idle unless each tile gets many warps
    DeviceInfo d;
    const int sms = current_device_info(&d) ? d.sms : 128;
    const bool pairs = (reinterpret_cast<uintptr_t>(conic) & 7) == 0;
    auto launch = [&](auto kern, int threads, int per_block) {
        const int blocks = tiles / per_block + (tiles % per_block != 0);
        kern<<<blocks, threads, 0, (cudaStream_t)stream>>>(dc, tile_ranges, ids_sorted, mean2d, conic, opacity, depth, radius,
                                                           features);
    };
    if (tiles <= kFewTilesPerSm * sms)
        pairs ? launch(k_tile_features<512, 1, true>, 512, 1) : launch(k_tile_features<512, 1, false>, 512, 1);
    else
        pairs ? launch(k_tile_features<32, kWarpTiles, true>, 32 * kWarpTiles, kWarpTiles)
              : launch(k_tile_features<32, kWarpTiles, false>, 32 * kWarpTiles, kWarpTiles);
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}

extern "C" tcgs_status tcgs_feature_norm(const float* x, int32_t n, float* norm, tcgs_stream stream) {
    using namespace tcgs;
    if (n < 0 || !norm || (n > 0 && !x)) return TCGS_ERR_INVALID;
    k_feature_norm<<<1, 1024, 0, (cudaStream_t)stream>>>(x, n, norm);
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}

extern "C" tcgs_status tcgs_mlp_fwd(const float* params, const float* norm, const float* x, int32_t n, float* y,
                                    tcgs_stream stream) {
    using namespace tcgs;
    if (n < 0 || !params || !norm || (n > 0 && (!x || !y))) return TCGS_ERR_INVALID;
    if (n == 0) return TCGS_OK;
    const int blocks = n / 128 + (n % 128 != 0);
    k_mlp_fwd<<<blocks, 128, 0, (cudaStream_t)stream>>>(params, norm, x, n, y);
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}

extern "C" tcgs_status tcgs_mlp_bwd(const float* params, const float* norm, const float* x, const float* target,
                                    int32_t n, float* grad, float* loss, tcgs_stream stream) {
    using namespace tcgs;
    if (n < 0 || !params || !norm || !grad || (n > 0 && (!x || !target))) return TCGS_ERR_INVALID;
    if (n == 0) return TCGS_OK;
    {
        static std::mutex mu;
        static bool raised[kMaxDevices] = {};   // the shared memory limit, per device
        DeviceInfo d;
        if (!current_device_info(&d)) return TCGS_ERR_CUDA;
        std::lock_guard<std::mutex> lock(mu);
        if (!raised[d.device]) {
            if (cudaFuncSetAttribute(k_mlp_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpBwdSmem)) !=
                cudaSuccess)
                return TCGS_ERR_CUDA;
            raised[d.device] = true;
        }
    }
    k_mlp_bwd<<<n / kBwdItems + (n % kBwdItems != 0), kBwdItems, sizeof(MlpBwdSmem), (cudaStream_t)stream>>>(
        params, norm, x, target, n, grad, loss);
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}

extern "C" tcgs_status tcgs_adam_step(float* params, float* m, float* v, float* grad, int32_t n_params,
                                      float lr, float beta1, float beta2, float eps, int32_t step,
                                      tcgs_stream stream) {
    using namespace tcgs;
    if (n_params < 0 || step < 1 || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) ||
        (n_params > 0 && (!params || !m || !v || !grad)))
        return TCGS_ERR_INVALID;
    if (n_params == 0) return TCGS_OK;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    k_adam<<<(n_params + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, m, v, grad, n_params, lr, beta1, beta2,
                                                                    eps, c1, c2);
    count_launches(1);
    TCGS_CHECK_LAUNCH();
    return TCGS_OK;
}
