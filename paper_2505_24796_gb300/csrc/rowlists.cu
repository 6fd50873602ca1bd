// rowlists.cu -- the sorting stage by tile-row lists (Sec. 3.1, Eq. 3): from the depth order of the
// Gaussians to the depth-ordered list of every tile.
//
// A Gaussian's tiles in one row of tiles are consecutive, so the unit that is sorted is not the splat
// (Gaussian, tile) but the run (Gaussian, tile row, first and last column): a stable counting sort of
// the runs by row gives every row's runs in depth order, and a second one, per row, expands them into
// the columns they span.  Neither sorts by comparing or ranking digits of splats: inside a block of
// runs, the runs that cover a column are one bit each of a (column x run) bit matrix, and a run's rank
// in the column is the number of bits before its own.
//   1. spans    256 Gaussians a block, in depth order: their runs (4 bytes each) and runs per row;
//   2. offsets  per row, the exclusive prefix of the blocks' counts; N and the capacity check;
//   3. scatter  the runs to their rows (id 4 bytes, columns 2 bytes);
//   4. counts   chunks of kChunk runs of a row: how many cover each column;
//   5. offsets  per (row, column), the exclusive prefix over the row's chunks, and the tile's length;
//   6. expand   each chunk writes its ids to the columns' lists; the tile ranges.
// Bytes from the depth order to the lists: 24 per run and 4 per splat, against 36 to 52 per splat for
// radix passes over the splats (binsort.cu, which sorts grids beyond 256 x 256 tiles).  From the depth order
// on, radix passes and row lists: 605M splats at 3840 x 2160 8.9 and 4.7 ms, 11.6M at 1280 x 720 0.36 and
// 0.19 ms, 2.0M at 1920 x 1080 0.15 and 0.13 ms.
// No block waits on another block; every launch is a programmatic dependent one.
#include "rowlists.cuh"

#include <mutex>

#include "cover.cuh"

namespace tcgs {
namespace {

constexpr int kRowThreads = 256;             // also the Gaussians of a span block and the columns or rows of a scan
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kChunk = 512;                  // runs expanded together: 16 words of the bit matrix per column
constexpr int kChunkWords = kChunk / 32;
constexpr uint32_t kFiveBlocksFrom = 10;      // span blocks an SM
constexpr uint32_t kOneTest = 1u << 16;      // a row to test, beside the runs that a round of spans has so far
constexpr int kSpanBuffer = 3072;            // runs of a span block kept in shared memory (more: evaluated twice)
constexpr int kScatterStage = 4096;          // runs regrouped by row at a time
constexpr int kExpandStage = 3584;           // ids regrouped by column at a time (4 expand blocks an SM up to 256 columns)
static_assert(kRowThreads == kRowListsMaxGrid && kChunk <= kExpandStage && kRowThreads <= kScatterStage,
              "a thread per row or column; a column of a chunk, or a row of a block, fits the stage");
static_assert(kRowThreads * (kRowMinWidth / 2) < kOneTest, "the runs of a round's narrow and decided rows");

// Counters zeroed by k_row_keys.
struct RowCounters {
    unsigned long long runs;      // runs reserved so far
    unsigned long long splats;    // N
    uint32_t n_ok;                // N, or 0 when it exceeds the capacity
    uint32_t pad;
    uint32_t row_runs[kRowListsMaxGrid];    // runs of each row
    uint32_t row_splats[kRowListsMaxGrid];  // splats of each row
};

struct RowScratch {
    RowCounters* ctr;
    uint32_t* block_base;    // per span block: its first run in `runs`
    uint32_t* block_count;   // and their number; bit 31: some row of a Gaussian has several runs
    uint32_t* tile_count;    // per tile
    uint32_t* m1;            // [row][span block]: counts, then offsets inside the row
    uint32_t* run_id;        // runs by row, in depth order: Gaussian
    uint16_t* run_span;      // and first | last << 8 column
    uint32_t* runs;          // runs by span block: owner | row << 8 | first << 16 | last << 24
    uint32_t* m2;            // [chunk][column]: counts, then offsets inside the tile (over `runs`)
    size_t bytes;
};

RowScratch row_scratch(char* base, int64_t P, int64_t cap) {
    RowScratch w;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base ? base + off : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    const size_t nb = (size_t)(P + kRowThreads - 1) / kRowThreads;
    const size_t runs = (size_t)cap;   // N <= cap splats make at most cap runs
    w.ctr = (RowCounters*)take(sizeof(RowCounters));
    w.block_base = (uint32_t*)take(4 * nb);
    w.block_count = (uint32_t*)take(4 * nb);
    w.tile_count = (uint32_t*)take(4 * (size_t)kRowListsMaxGrid * kRowListsMaxGrid);
    w.m1 = (uint32_t*)take(4 * nb * kRowListsMaxGrid);
    w.run_id = (uint32_t*)take(4 * runs);
    w.run_span = (uint16_t*)take(2 * runs);
    // the runs by span block end with the scatter, the chunk counts begin after it: one region
    const size_t m2 = 4 * (size_t)kRowListsMaxGrid * (runs / kChunk + kRowListsMaxGrid);
    w.runs = (uint32_t*)take(4 * runs > m2 ? 4 * runs : m2);
    w.m2 = w.runs;
    w.bytes = off;
    return w;
}

__global__ void __launch_bounds__(kRowThreads) k_row_keys(uint32_t P, const float* __restrict__ depth,
                                                          const int32_t* __restrict__ radius,
                                                          uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                          uint32_t* __restrict__ ranges, uint32_t n_range_words,
                                                          uint32_t* __restrict__ digit_total0,
                                                          uint32_t* __restrict__ counters) {
    pdl_wait();
    const uint32_t i = blockIdx.x * kRowThreads + threadIdx.x;
    if (blockIdx.x == 0) {
        digit_total0[threadIdx.x] = 0u;
        for (uint32_t k = threadIdx.x; k < sizeof(RowCounters) / 4; k += kRowThreads) counters[k] = 0u;
    }
    if (i < n_range_words) ranges[i] = 0u;
    if (i < P) {
        keys[i] = radius[i] > 0 ? orderable_bits(depth[i]) : 0xFFFFFFFFu;
        vals[i] = i;
    }
}

// Runs of reached tiles of a wide Gaussian whose conic is not positive definite, every tile of columns
// [x0, x1] of row ty tested: one run from the first to the last reached tile with `fill`, else every
// maximal run.  Returns their number, adds their length to `len`, and stores those below `most` to
// dst (null: none).  Out of line: counting and storing then take the same decisions.
__device__ __noinline__ uint32_t tested_runs(const Cover& v, int ty, int x0, int x1, bool fill, uint32_t head,
                                             uint32_t* dst, uint32_t most, uint32_t& len) {
    const float ly = v.my - (float)(ty * kTile + kTile / 2);
    uint32_t n = 0;
    int first = -1, last = -1;
    for (int tx = x0; tx <= x1 + 1; ++tx) {
        const bool in = tx <= x1 && tile_reached(v, v.mx - (float)(tx * kTile + kTile / 2), ly);
        if (in) {
            if (first < 0) first = tx;
            last = tx;
        }
        if (first >= 0 && (tx > x1 || (!in && !fill))) {
            if (dst && n < most) dst[n] = head | (uint32_t)first << 16 | (uint32_t)last << 24;
            len += (uint32_t)(last - first + 1);
            ++n;
            first = -1;
        }
    }
    return n;
}

// 1. Runs of 256 consecutive Gaussians of the depth order.  A row of a rectangle is one unit of work,
// dealt out over the block's threads (owner by binary search over the prefix of the row counts), so that
// a Gaussian with hundreds of rows is spread over the block; the rounds' runs are packed in unit order,
// which keeps the depth order inside every row.  A block reserves its slice of `runs` with one atomic
// once it knows its size (slices in any order: the offsets find them by block), from shared memory;
// a block with more than kSpanBuffer runs evaluates them a second time instead.
// EXACT: RowLists.exact.  TILES: exact without fill_rows, every tile kept or left out as the per-tile test decides: a wide
// row is taken from the closed form where that decides every tile of it (row_tiles), else the block's warps test it, 32
// tiles at a time.  20,000 needles of 20 to 300 pixels in 170,000 Gaussians sort in 0.40 ms (3.55 ms by radix passes
// that test every tile; 0.25 ms, with a tile in 10^6 kept or left out otherwise, when the rows' ends alone are
// tested; 1.45 ms with a lane a row, where one needle across the view was the tail of its block).
// kBlocks: five blocks an SM need 48 registers, where the compiler takes 53 and four: the sorting stage of 211,000
// Gaussians at 1743 x 1004 is 5% slower with five (a chain's loads are not all in flight), of 1M at 1920 x 1080 3%
// faster; they meet at about kFiveBlocksFrom blocks an SM.  With the better one the 1237 x 701 and 1920 x 1080 frames
// take what they take when the ends alone are tested, within 0.5%.
// fill_rows is read where it is always set: as a constant it has the compiler contract row_span's tests
// otherwise, which moves FP32 ties.
// An instance of its own: in one kernel with row_span both take more registers (605M splats at 3840 x 2160:
// 1.51 -> 1.59 ms).
template <bool EXACT, bool TILES, int kBlocks = 0>
__global__ void __launch_bounds__(kRowThreads, kBlocks) k_row_spans(DevCamera cam, uint32_t P,
                                                           const uint32_t* __restrict__ order,
                                                           const float* __restrict__ mean2d,
                                                           const int32_t* __restrict__ radius,
                                                           const float* __restrict__ conic,
                                                           const float* __restrict__ opacity, int fill_rows,
                                                           unsigned long long run_cap, uint32_t nb, RowScratch w) {
    pdl_wait();
    __shared__ Cover s_cv[EXACT ? kRowThreads : 1];
    __shared__ uint32_t s_pre[kRowThreads];    // exclusive prefix of the row counts
    __shared__ uint32_t s_rect[kRowThreads];   // x0 | x1 << 8 | y0 << 16
    __shared__ uint32_t s_rows[kRowThreads];   // runs per tile row
    __shared__ uint32_t s_buf[kSpanBuffer];
    __shared__ uint32_t s_ws[kRowWarps];
    __shared__ unsigned long long s_len, s_base;
    __shared__ uint32_t s_multi;
    // TILES: the rows to test, their threads, and each thread's row's bits, [32 tiles][thread]
    __shared__ uint32_t s_task[TILES ? kRowThreads : 1];
    __shared__ uint8_t s_thread[TILES ? kRowThreads : 1];
    extern __shared__ uint32_t s_mask[];
    const int t = threadIdx.x;
    const uint32_t i = blockIdx.x * kRowThreads + t;
    uint32_t rows = 0, rect = 0;
    Cover cv{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, -1.f};
    if (i < P) {
        const uint32_t g = order[i];
        const float2 m = reinterpret_cast<const float2*>(mean2d)[g];
        const Rect rc = tile_rect(m.x, m.y, radius[g], cam.grid_w, cam.grid_h);
        if (rect_count(rc)) {
            if (EXACT) cv = cover_of(mean2d, conic, opacity, g);
            if (!EXACT || cv.lim >= 0.f) {
                rows = (uint32_t)(rc.y1 - rc.y0 + 1);
                rect = (uint32_t)rc.x0 | (uint32_t)rc.x1 << 8 | (uint32_t)rc.y0 << 16;
            }
        }
    }
    uint32_t total_rows;
    s_pre[t] = block_exclusive_scan<uint32_t, kRowThreads>(rows, s_ws, total_rows);
    s_rect[t] = rect;
    s_rows[t] = 0u;
    if (EXACT) s_cv[t] = cv;
    if (t == 0) {
        s_len = 0ull;
        s_multi = 0u;
    }
    __syncthreads();
    uint32_t n_out = 0;
    unsigned long long len_sum = 0;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {   // one copy of the code: the second evaluation decides as the first
        n_out = 0;
        for (uint32_t r0 = 0; r0 < total_rows; r0 += kRowThreads) {
            const uint32_t rr = r0 + (uint32_t)t;
            const bool active = rr < total_rows;
            uint32_t owner = 0, n = 0, len = 0, reached = 0;   // reached: a narrow row's tiles, one bit each
            int ty = 0, x0 = 0, x1 = 0, L = 0, R = -1;
            bool tested = false;
            if (active) {
#pragma unroll
                for (int step = kRowThreads / 2; step > 0; step >>= 1)
                    if (s_pre[owner + step] <= rr) owner += step;
                const uint32_t rc = s_rect[owner];
                x0 = (int)(rc & 0xFFu);
                x1 = (int)((rc >> 8) & 0xFFu);
                ty = (int)((rc >> 16) & 0xFFu) + (int)(rr - s_pre[owner]);
                if (!EXACT) {
                    L = x0; R = x1;
                } else if (x1 - x0 + 1 < kRowMinWidth) {   // tile by tile
                    const Cover& v = s_cv[owner];
                    const float ly = v.my - (float)(ty * kTile + kTile / 2);
                    for (int tx = x0; tx <= x1; ++tx)
                        if (tile_reached(v, v.mx - (float)(tx * kTile + kTile / 2), ly)) reached |= 1u << (tx - x0);
                    if (reached) {
                        L = x0 + __ffs(reached) - 1;
                        R = x0 + 31 - __clz(reached);
                        len = __popc(reached);
                        n = __popc(reached & ~(reached << 1));
                    }
                } else {
                    const Cover& v = s_cv[owner];
                    const Reach e = reach_of(v);
                    tested = e.W < 0.f;
                    if constexpr (TILES) {
                        if (!tested) {
                            const RowTiles q = row_tiles(v, e, turn_error(v), ty, x0, x1);
                            x0 = L = q.lo; x1 = R = q.hi;
                            tested = !q.sure;
                        }
                    } else if (tested) {
                        n = tested_runs(v, ty, x0, x1, fill_rows != 0, 0u, nullptr, 0u, len);
                    } else {   // positive definite: the row's ends in closed form
                        const int2 sp = row_span(v, e, ty, x0, x1);
                        L = sp.x; R = sp.y;
                    }
                }
                if (n == 0 && L <= R && !tested) {
                    n = 1;
                    len = (uint32_t)(R - L + 1);
                }
            }
            uint32_t round_n;
            uint32_t at = block_exclusive_scan<uint32_t, kRowThreads>(TILES && tested ? kOneTest : n, s_ws, round_n);
            if constexpr (TILES) {
                if (round_n >= kOneTest) {   // uniform: some rows are to be tested
                    if (tested) {
                        s_task[at / kOneTest] = owner | (uint32_t)ty << 8 | (uint32_t)x0 << 16 | (uint32_t)x1 << 24;
                        s_thread[at / kOneTest] = (uint8_t)t;
                    }
                    __syncthreads();
                    for (uint32_t k = t >> 5; k < round_n / kOneTest; k += kRowWarps) {
                        const uint32_t job = s_task[k], j = s_thread[k];
                        const Cover& v = s_cv[job & 0xFFu];
                        const int end = (int)(job >> 24);
                        const float ly = v.my - (float)((int)((job >> 8) & 0xFFu) * kTile + kTile / 2);
                        for (int b0 = (int)((job >> 16) & 0xFFu), q = 0; b0 <= end; b0 += 32, ++q) {
                            const int tx = b0 + (t & 31);
                            const uint32_t m = __ballot_sync(
                                0xffffffffu, tx <= end && tile_reached(v, v.mx - (float)(tx * kTile + kTile / 2), ly));
                            if ((t & 31) == 0) s_mask[q * kRowThreads + j] = m;
                        }
                    }
                    __syncthreads();
                    if (tested) {
                        uint32_t carry = 0u;
                        for (int q = 0; 32 * q <= x1 - x0; ++q) {
                            const uint32_t m = s_mask[q * kRowThreads + t];
                            n += __popc(m & ~(m << 1 | carry));
                            len += __popc(m);
                            carry = m >> 31;
                        }
                    }
                    at = block_exclusive_scan<uint32_t, kRowThreads>(n, s_ws, round_n);
                }
            }
            at += n_out;
            const uint32_t head = owner | (uint32_t)ty << 8;
            if (pass == 0) {
                if (n) atomicAdd(&s_rows[ty], n);
                if (n > 1) s_multi = 0x80000000u;
                len_sum += len;
            }
            uint32_t* dst = pass == 0 ? s_buf + at : w.runs + s_base + at;
            const uint32_t most = pass == 0 ? (at < (uint32_t)kSpanBuffer ? (uint32_t)kSpanBuffer - at : 0u) : n;
            if (TILES && tested) {
                uint32_t k = 0;
                int open = -1;   // the run that has begun
                auto emit = [&](int first, int last) {
                    if (k < most) dst[k] = head | (uint32_t)first << 16 | (uint32_t)last << 24;
                    ++k;
                };
                for (int b0 = x0, q = 0; b0 <= x1; b0 += 32, ++q) {
                    uint32_t m = s_mask[q * kRowThreads + t];
                    if (open >= 0 && !(m & 1u)) {   // it ended with the 32 tiles before
                        emit(open, b0 - 1);
                        open = -1;
                    }
                    while (m) {
                        const int f = __ffs(m) - 1;
                        const uint32_t gap = ~(m >> f);
                        const int end = f + (gap ? __ffs(gap) - 1 : 32);
                        const int first = f == 0 && open >= 0 ? open : b0 + f;
                        if (end == 32) {   // it may go on
                            open = first;
                            break;
                        }
                        emit(first, b0 + end - 1);
                        open = -1;
                        m &= 0xFFFFFFFFu << end;
                    }
                }
                if (open >= 0) emit(open, x1);
            } else if (EXACT && tested) {
                tested_runs(s_cv[owner], ty, x0, x1, fill_rows != 0, head, dst, most, len);
            } else if (n == 1) {
                if (most) dst[0] = head | (uint32_t)L << 16 | (uint32_t)R << 24;
            } else if (EXACT) {
                for (uint32_t k = 0; k < n; ++k) {   // a narrow row reached in parts
                    const int f = __ffs(reached) - 1, e = __ffs(~(reached >> f)) - 1;
                    if (k < most) dst[k] = head | (uint32_t)(x0 + f) << 16 | (uint32_t)(x0 + f + e - 1) << 24;
                    reached &= ~(((1u << e) - 1u) << f);
                }
            }
            n_out += round_n;
        }
        if (pass == 1) break;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) len_sum += __shfl_xor_sync(0xffffffffu, len_sum, o);
        if ((t & 31) == 0 && len_sum) atomicAdd(&s_len, len_sum);
        __syncthreads();
        if (t == 0) {
            unsigned long long base = 0;
            if (n_out) {
                base = atomicAdd(&w.ctr->runs, (unsigned long long)n_out);
                atomicAdd(&w.ctr->splats, s_len);
            }
            s_base = base;
            w.block_base[blockIdx.x] = (uint32_t)base;
            w.block_count[blockIdx.x] = n_out | s_multi;
        }
        if (t < cam.grid_h) w.m1[(size_t)t * nb + blockIdx.x] = s_rows[t];
        __syncthreads();
        if (s_base + n_out > run_cap) break;   // then N exceeds the capacity too: nothing is placed
        if (n_out <= (uint32_t)kSpanBuffer) {
            for (uint32_t k = t; k < n_out; k += kRowThreads) w.runs[s_base + k] = s_buf[k];
            break;
        }
    }
}

// 2. Block r: the exclusive prefix of row r's counts over the span blocks (in place), and the row's
// total.  Block 0 also settles N, the status and the count that the following kernels go by.
constexpr int kScanThreads = 1024;

__global__ void __launch_bounds__(kScanThreads) k_row_offsets(uint32_t nb, long long capacity,
                                                              int64_t* __restrict__ n_splats,
                                                              int32_t* __restrict__ status, RowScratch w) {
    pdl_trigger();
    pdl_wait();
    constexpr uint32_t kPer = 4;
    __shared__ uint32_t ws[kScanThreads / 32];
    uint32_t* row = w.m1 + (size_t)blockIdx.x * nb;
    uint32_t run = 0;
    for (uint32_t b0 = 0; b0 < nb; b0 += kScanThreads * kPer) {
        const uint32_t b = b0 + threadIdx.x * kPer;
        uint32_t x[kPer], sum = 0;
#pragma unroll
        for (uint32_t k = 0; k < kPer; ++k) {
            x[k] = b + k < nb ? row[b + k] : 0u;
            sum += x[k];
        }
        uint32_t total;
        uint32_t at = run + block_exclusive_scan<uint32_t, kScanThreads>(sum, ws, total);
#pragma unroll
        for (uint32_t k = 0; k < kPer; ++k) {
            if (b + k < nb) row[b + k] = at;
            at += x[k];
        }
        run += total;
    }
    if (threadIdx.x == 0) {
        w.ctr->row_runs[blockIdx.x] = run;
        if (blockIdx.x == 0) {
            const unsigned long long n = w.ctr->splats;
            const bool ok = n <= (unsigned long long)capacity;
            *n_splats = (int64_t)n;
            *status = ok ? TCGS_OK : TCGS_ERR_CAPACITY;
            w.ctr->n_ok = ok ? (uint32_t)n : 0u;
        }
    }
}

// The largest k in [0, 256) with table[k] <= x (table ascending, table[0] <= x).
__device__ __forceinline__ uint32_t last_at_most(const uint32_t* table, uint32_t x) {
    uint32_t k = 0;
#pragma unroll
    for (uint32_t step = 128; step > 0; step >>= 1)
        if (table[k + step] <= x) k += step;
    return k;
}

// The end of the longest span of columns (rows) from c0 on whose items fit `most` (at least one column).
__device__ __forceinline__ uint32_t window_end(const uint32_t* start, uint32_t c0, uint32_t n, uint32_t most) {
    uint32_t lo = c0 + 1, hi = n;   // start[c] is the first item of column c, start[n] their number
    while (lo < hi) {
        const uint32_t m = (lo + hi + 1) >> 1;
        if (start[m] - start[c0] <= most) lo = m; else hi = m - 1;
    }
    return lo;
}

// 3. Span block b's runs to their rows.  Bit `owner` of row r's 256-bit set marks a run, so a run's rank
// in the block's part of its row is the number of set bits below its own; the runs are regrouped by row
// in shared memory (row windows of at most kScatterStage runs) and written out run by run, so that each
// row's part is one contiguous write.
__global__ void __launch_bounds__(kRowThreads) k_row_scatter(uint32_t P, const uint32_t* __restrict__ order, int grid_h,
                                                             uint32_t nb, RowScratch w) {
    pdl_wait();
    constexpr int kWords = kRowThreads / 32, kStride = kWords + 1;
    __shared__ uint32_t s_bits[kRowThreads * kStride];
    __shared__ uint16_t s_before[kRowThreads * kStride];   // set bits in the row's earlier words
    __shared__ uint32_t s_start[kRowThreads + 1];          // first item of each row among the block's runs
    __shared__ uint32_t s_delta[kRowThreads];              // global position minus that
    __shared__ uint32_t s_g[kRowThreads];
    __shared__ uint32_t s_stage[kScatterStage];
    __shared__ uint32_t s_ws[kRowWarps];
    if (w.ctr->n_ok == 0u) return;
    const uint32_t b = blockIdx.x, cnt = w.block_count[b];
    const uint32_t n = cnt & 0x7FFFFFFFu;
    if (n == 0u) return;
    const int t = threadIdx.x;
    const uint32_t* runs = w.runs + w.block_base[b];
    s_g[t] = b * kRowThreads + t < P ? order[b * kRowThreads + t] : 0u;
    uint32_t tot;
    const uint32_t row_base = block_exclusive_scan<uint32_t, kRowThreads>(t < grid_h ? w.ctr->row_runs[t] : 0u, s_ws, tot);
    const uint32_t to = row_base + (t < grid_h ? w.m1[(size_t)t * nb + b] : 0u);
    if (cnt >> 31) {   // several runs in a row of one Gaussian (never with a positive definite conic): owner by owner
        s_delta[t] = to;
        __syncthreads();
        for (uint32_t o = 0; o < (uint32_t)kRowThreads; ++o) {
            for (uint32_t k = t; k < n; k += kRowThreads) {
                const uint32_t r = runs[k];
                if ((r & 0xFFu) != o) continue;
                const uint32_t pos = atomicAdd(&s_delta[(r >> 8) & 0xFFu], 1u);
                w.run_id[pos] = s_g[o];
                w.run_span[pos] = (uint16_t)(r >> 16);
            }
            __syncthreads();
        }
        return;
    }
    for (int k = t; k < kRowThreads * kStride; k += kRowThreads) s_bits[k] = 0u;
    __syncthreads();
    for (uint32_t k = t; k < n; k += kRowThreads) {
        const uint32_t r = runs[k], o = r & 0xFFu;
        atomicOr(&s_bits[((r >> 8) & 0xFFu) * kStride + (o >> 5)], 1u << (o & 31u));
    }
    __syncthreads();
    uint32_t in_row = 0;
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
        s_before[t * kStride + k] = (uint16_t)in_row;
        in_row += __popc(s_bits[t * kStride + k]);
    }
    const uint32_t start = block_exclusive_scan<uint32_t, kRowThreads>(in_row, s_ws, tot);
    s_start[t] = start;
    s_delta[t] = to - start;
    if (t == 0) s_start[kRowThreads] = tot;
    __syncthreads();
    for (uint32_t c0 = 0; c0 < (uint32_t)kRowThreads;) {   // uniform over the block
        const uint32_t c1 = window_end(s_start, c0, kRowThreads, kScatterStage);
        const uint32_t first = s_start[c0], items = s_start[c1] - first;
        for (uint32_t k = t; k < n; k += kRowThreads) {
            const uint32_t r = runs[k], row = (r >> 8) & 0xFFu, o = r & 0xFFu;
            if (row < c0 || row >= c1) continue;
            const uint32_t at = row * kStride + (o >> 5);
            s_stage[s_start[row] - first + s_before[at] + __popc(s_bits[at] & ((1u << (o & 31u)) - 1u))] = r;
        }
        __syncthreads();
        for (uint32_t k = t; k < items; k += kRowThreads) {
            const uint32_t r = s_stage[k], pos = s_delta[(r >> 8) & 0xFFu] + first + k;
            w.run_id[pos] = s_g[r & 0xFFu];
            w.run_span[pos] = (uint16_t)(r >> 16);
        }
        __syncthreads();
        c0 = c1;
    }
}

// First run and first chunk of every row, and the number of chunks (256 threads; ends in a barrier).
struct RowTable {
    uint32_t run[kRowListsMaxGrid + 1];
    uint32_t chunk[kRowListsMaxGrid + 1];
};

__device__ __forceinline__ void build_row_table(RowTable& tab, const RowScratch& w, int grid_h, uint32_t* ws) {
    const int t = threadIdx.x;
    const uint32_t n = t < grid_h ? w.ctr->row_runs[t] : 0u;
    uint32_t total;
    tab.run[t] = block_exclusive_scan<uint32_t, kRowThreads>(n, ws, total);
    if (t == 0) tab.run[kRowListsMaxGrid] = total;
    tab.chunk[t] = block_exclusive_scan<uint32_t, kRowThreads>(n / kChunk + (n % kChunk != 0u), ws, total);
    if (t == 0) tab.chunk[kRowListsMaxGrid] = total;
    __syncthreads();
}

// The row of a chunk: the last row with chunk[row] <= c (a row with chunks: empty ones share their successor's).
__device__ __forceinline__ uint32_t chunk_row(const RowTable& tab, uint32_t c, uint32_t& first, uint32_t& n) {
    const uint32_t row = last_at_most(tab.chunk, c);
    first = tab.run[row] + (c - tab.chunk[row]) * kChunk;
    n = tab.run[row + 1] - first;
    n = n < (uint32_t)kChunk ? n : (uint32_t)kChunk;
    return row;
}

// 4. Runs of a chunk that cover each column: +1 at the first column, -1 after the last, summed.
__global__ void __launch_bounds__(kRowThreads) k_col_counts(int grid_w, int grid_h, RowScratch w) {
    pdl_trigger();
    pdl_wait();
    __shared__ RowTable s_tab;
    __shared__ uint32_t s_d[kRowListsMaxGrid + 1];
    __shared__ uint32_t s_ws[kRowWarps];
    if (w.ctr->n_ok == 0u) return;
    const int t = threadIdx.x;
    build_row_table(s_tab, w, grid_h, s_ws);
    const uint32_t chunks = s_tab.chunk[kRowListsMaxGrid];
    for (uint32_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        uint32_t first, n;
        chunk_row(s_tab, c, first, n);
        s_d[t] = 0u;
        __syncthreads();
        for (uint32_t k = t; k < n; k += kRowThreads) {
            const uint32_t sp = w.run_span[first + k];
            atomicAdd(&s_d[sp & 0xFFu], 1u);
            atomicAdd(&s_d[(sp >> 8) + 1u], 0xFFFFFFFFu);   // the word past the last column takes what is not needed
        }
        __syncthreads();
        const uint32_t d = s_d[t];
        uint32_t total;
        const uint32_t covering = block_exclusive_scan<uint32_t, kRowThreads>(d, s_ws, total) + d;
        if (t < grid_w) w.m2[(size_t)c * grid_w + t] = covering;
    }
}

// 5. Block (row, 32 columns): the exclusive prefix of the columns' counts over the row's chunks (in
// place; each warp sums, then rewrites, its part of the chunks), the tiles' lengths and the row's.  Bound by
// the latency of a warp's walk down its chunks in the longest row, hence 32 warps (605M splats at 3840 x 2160:
// 498 us with 8 warps, 293 us).
constexpr int kColThreads = 1024;
constexpr int kColWarps = kColThreads / 32;

__global__ void __launch_bounds__(kColThreads) k_col_offsets(int grid_w, RowScratch w) {
    pdl_trigger();
    pdl_wait();
    __shared__ uint32_t s_sum[kColWarps][32];
    __shared__ uint32_t s_ws[kColWarps];
    if (w.ctr->n_ok == 0u) return;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t row = blockIdx.x, col = blockIdx.y * 32u + lane;
    const uint32_t r = (uint32_t)t < row ? w.ctr->row_runs[t] : 0u;
    uint32_t chunk0;
    block_exclusive_scan<uint32_t, kColThreads>(r / kChunk + (r % kChunk != 0u), s_ws, chunk0);
    const uint32_t n = w.ctr->row_runs[row], chunks = n / kChunk + (n % kChunk != 0u);
    const uint32_t per = (chunks + kColWarps - 1) / kColWarps;
    const uint32_t lo = min((uint32_t)warp * per, chunks), hi = min(lo + per, chunks);
    const bool in = col < (uint32_t)grid_w;
    uint32_t* m = w.m2 + (size_t)chunk0 * grid_w + (in ? col : 0u);
    uint32_t sum = 0;
    if (in) {
#pragma unroll 8
        for (uint32_t c = lo; c < hi; ++c) sum += m[(size_t)c * grid_w];
    }
    s_sum[warp][lane] = sum;
    __syncthreads();
    uint32_t run = 0, total = 0;
#pragma unroll
    for (int k = 0; k < kColWarps; ++k) {
        run += k < warp ? s_sum[k][lane] : 0u;
        total += s_sum[k][lane];
    }
    if (in) {
#pragma unroll 8
        for (uint32_t c = lo; c < hi; ++c) {
            const uint32_t x = m[(size_t)c * grid_w];
            m[(size_t)c * grid_w] = run;
            run += x;
        }
    }
    if (warp == 0) {
        if (in) w.tile_count[row * (uint32_t)grid_w + col] = total;
        uint32_t all = in ? total : 0u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
        if (lane == 0 && all) atomicAdd(&w.ctr->row_splats[row], all);
    }
}

// 6. The ids of a chunk's runs to the lists of the columns they span.  Bit k of column x's set marks that
// run k covers it; a run's place in column x's part of the chunk is the number of set bits below its
// own.  The ids are regrouped by column in shared memory (column windows of at most kExpandStage ids)
// and written out in that order, so that each list's part is one contiguous write.
// Bound by latency (barriers, shared-memory round trips, the loads of a chunk) at 24 warps an SM, so
// shared memory is sized by the columns there are (4 blocks an SM, 5 up to 176 columns, instead of 3) and
// the next chunk's runs are loaded while the current one is regrouped (2.3M splats at 1920 x 1080: 37 -> 26 us,
// 605M at 3840 x 2160: 2.73 -> 2.46 ms).  A run's columns dealt to several lanes, and the sets formed by a
// prefix XOR of two toggles a run instead of one atomic a column, both measured slower.
struct ExpandSmem {
    RowTable tab;
    uint32_t row_base[kRowListsMaxGrid + 1];        // first splat of each row
    uint32_t start[kRowListsMaxGrid + 1];           // first id of each column among the chunk's
    uint32_t delta[kRowListsMaxGrid];               // global position minus that
    uint32_t stage[kExpandStage];
    uint8_t stage_col[kExpandStage];
    uint32_t ws[kRowWarps];
    // then, each [word][column]: the sets' bits, and the place of the word's first run in the chunk's ids
};

constexpr int kExpandBlocks = 5;

inline size_t expand_smem_bytes(int grid_w) { return sizeof(ExpandSmem) + 2 * 4 * (size_t)kChunkWords * grid_w; }

__global__ void __launch_bounds__(kRowThreads, kExpandBlocks) k_row_expand(int grid_w, int grid_h, uint32_t* __restrict__ ids_sorted,
                                                            uint32_t* __restrict__ ranges, RowScratch w) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t smem[];
    ExpandSmem& s = *reinterpret_cast<ExpandSmem*>(smem);
    if (w.ctr->n_ok == 0u) return;
    const int t = threadIdx.x;
    build_row_table(s.tab, w, grid_h, s.ws);
    uint32_t tot;
    s.row_base[t] = block_exclusive_scan<uint32_t, kRowThreads>(t < grid_h ? w.ctr->row_splats[t] : 0u, s.ws, tot);
    __syncthreads();
    const uint32_t chunks = s.tab.chunk[kRowListsMaxGrid];
    const uint32_t below = (1u << (t & 31)) - 1u;
    uint32_t* const bits = reinterpret_cast<uint32_t*>(smem + sizeof(ExpandSmem));
    uint32_t* const before = bits + kChunkWords * grid_w;
    uint32_t at_row = 0xFFFFFFFFu, list = 0;   // list: first splat of column t of the row
    constexpr int kEach = kChunk / kRowThreads;
    uint32_t next_row, next_id[kEach], next_sp[kEach];   // the next chunk's runs of this thread; an empty span: none
    auto fetch = [&](uint32_t c) {
        uint32_t first, n;
        next_row = chunk_row(s.tab, c, first, n);
#pragma unroll
        for (int q = 0; q < kEach; ++q) {
            const uint32_t k = (uint32_t)(q * kRowThreads + t);
            next_id[q] = 0u;
            next_sp[q] = 1u;   // first 1, last 0
            if (k < n) {
                next_sp[q] = w.run_span[first + k];
                next_id[q] = w.run_id[first + k];
            }
        }
    };
    if (blockIdx.x < chunks) fetch(blockIdx.x);
    for (uint32_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        const uint32_t row = next_row;
        uint32_t id[kEach], x0[kEach], x1[kEach];
#pragma unroll
        for (int q = 0; q < kEach; ++q) {
            id[q] = next_id[q];
            x0[q] = next_sp[q] & 0xFFu;
            x1[q] = next_sp[q] >> 8;
        }
        const uint32_t in_tile = t < grid_w ? w.m2[(size_t)c * grid_w + t] : 0u;
        for (int k = t; k < kChunkWords * grid_w; k += kRowThreads) bits[k] = 0u;
        if (row != at_row) {
            const uint32_t len = t < grid_w ? w.tile_count[row * (uint32_t)grid_w + t] : 0u;
            list = s.row_base[row] + block_exclusive_scan<uint32_t, kRowThreads>(len, s.ws, tot);
            at_row = row;
            if (c == s.tab.chunk[row] && t < grid_w && len) {   // the row's first chunk: its tiles' ranges
                ranges[2 * (row * (uint32_t)grid_w + t)] = list;
                ranges[2 * (row * (uint32_t)grid_w + t) + 1] = list + len;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kEach; ++q) {
            uint32_t* word = bits + (uint32_t)((q * kRowThreads + t) >> 5) * (uint32_t)grid_w;
            for (uint32_t x = x0[q]; x <= x1[q]; ++x) atomicOr(&word[x], 1u << (t & 31));
        }
        if (c + gridDim.x < chunks) fetch(c + gridDim.x);
        __syncthreads();
        uint32_t len = 0;
        if (t < grid_w) {
#pragma unroll
            for (int g = 0; g < kChunkWords; ++g) len += __popc(bits[g * grid_w + t]);
        }
        const uint32_t start = block_exclusive_scan<uint32_t, kRowThreads>(len, s.ws, tot);
        s.start[t] = start;
        if (t == 0) s.start[kRowListsMaxGrid] = tot;
        if (t < grid_w) {
            s.delta[t] = list + in_tile - start;
            uint32_t run = start;
#pragma unroll
            for (int g = 0; g < kChunkWords; ++g) {
                before[g * grid_w + t] = run;
                run += __popc(bits[g * grid_w + t]);
            }
        }
        __syncthreads();
        for (uint32_t c0 = 0; c0 < (uint32_t)grid_w;) {   // uniform over the block
            const uint32_t c1 = window_end(s.start, c0, (uint32_t)grid_w, kExpandStage);
            const uint32_t base = s.start[c0], items = s.start[c1] - base;
#pragma unroll
            for (int q = 0; q < kEach; ++q) {
                const uint32_t at = (uint32_t)(q * kRowThreads + t) >> 5;
                const uint32_t lo = x0[q] > c0 ? x0[q] : c0, hi = x1[q] < c1 - 1 ? x1[q] : c1 - 1;
                if (x0[q] <= x1[q])
                    for (uint32_t x = lo; x <= hi; ++x) {
                        const uint32_t k = at * (uint32_t)grid_w + x;
                        const uint32_t p = before[k] - base + __popc(bits[k] & below);
                        s.stage[p] = id[q];
                        s.stage_col[p] = (uint8_t)x;
                    }
            }
            __syncthreads();
            for (uint32_t k = t; k < items; k += kRowThreads)
                ids_sorted[s.delta[s.stage_col[k]] + base + k] = s.stage[k];
            __syncthreads();
            c0 = c1;
        }
    }
}

// Blocks of a persistent kernel resident at once on the current device, looked up once per device (and
// number of columns, on which the expansion's shared memory depends).
template <typename K>
int resident_blocks(K kern, int threads, size_t smem, size_t max_smem, int (&cached)[kMaxDevices]) {
    static std::mutex mu;
    DeviceInfo d;
    if (!current_device_info(&d)) return 256;
    std::lock_guard<std::mutex> lock(mu);
    if (cached[d.device] == 0) {
        if (max_smem) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        cached[d.device] = d.sms * (per_sm > 0 ? per_sm : 1);
    }
    return cached[d.device];
}

}  // namespace

size_t row_lists_scratch_bytes(int64_t P, int64_t capacity) { return row_scratch(nullptr, P, capacity).bytes; }

void launch_row_keys(const RowLists& a, const float* depth, uint32_t* keys, uint32_t* vals, uint32_t* digit_total0,
                     cudaStream_t s) {
    const RowScratch w = row_scratch(a.scratch, a.P, a.capacity);
    const uint32_t words = 2u * (uint32_t)(a.cam.grid_w * a.cam.grid_h);
    const uint32_t n = a.P > words ? a.P : words;
    launch_pdl(k_row_keys, (n + kRowThreads - 1) / kRowThreads, kRowThreads, 0, s, a.P, depth, a.radius, keys, vals,
               a.ranges, words, digit_total0, (uint32_t*)w.ctr);
    count_launches(1);
}

void launch_row_lists(const RowLists& a, cudaStream_t s) {
    const RowScratch w = row_scratch(a.scratch, a.P, a.capacity);
    const uint32_t nb = (a.P + kRowThreads - 1) / kRowThreads;
    const int gw = a.cam.grid_w, gh = a.cam.grid_h;
    const bool tiles = a.exact && !a.fill_rows;
    DeviceInfo d;
    const bool five = current_device_info(&d) && nb > kFiveBlocksFrom * (uint32_t)d.sms;
    auto spans = !a.exact ? k_row_spans<false, false> : a.fill_rows ? k_row_spans<true, false>
                          : five ? k_row_spans<true, true, 5> : k_row_spans<true, true>;
    launch_pdl(spans, nb, kRowThreads, tiles ? 4 * kRowThreads * ((gw + 31) / 32) : 0, s, a.cam, a.P, a.order, a.mean2d,
               a.radius, a.conic, a.opacity, (int)a.fill_rows, (unsigned long long)a.capacity, nb, w);
    launch_pdl(k_row_offsets, gh, kScanThreads, 0, s, nb, (long long)a.capacity, a.n_splats, a.status, w);
    count_launches(2);
    if (a.capacity == 0) return;   // N and the status are settled; there is nothing to place
    launch_pdl(k_row_scatter, nb, kRowThreads, 0, s, a.P, a.order, gh, nb, w);
    // at most capacity / kChunk + grid_h chunks
    static int count_blocks[kMaxDevices] = {}, expand_blocks[kRowListsMaxGrid + 1][kMaxDevices] = {};
    const size_t smem = expand_smem_bytes(gw);
    const int64_t chunks = a.capacity / kChunk + gh;
    const int64_t cb = resident_blocks(k_col_counts, kRowThreads, 0, 0, count_blocks);
    const int64_t eb = resident_blocks(k_row_expand, kRowThreads, smem, expand_smem_bytes(kRowListsMaxGrid), expand_blocks[gw]);
    launch_pdl(k_col_counts, (int)(chunks < cb ? chunks : cb), kRowThreads, 0, s, gw, gh, w);
    launch_pdl(k_col_offsets, dim3(gh, (gw + 31) / 32), kColThreads, 0, s, gw, w);
    launch_pdl(k_row_expand, (int)(chunks < eb ? chunks : eb), kRowThreads, smem, s, gw, gh, a.ids_sorted,
               a.ranges, w);
    count_launches(4);
}

}  // namespace tcgs
