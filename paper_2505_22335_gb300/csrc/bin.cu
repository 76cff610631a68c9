// Tile lists straight from the depth-ordered Gaussian-views: which Gaussians
// each 16x16 tile blends, in depth order, each list cut after its first `cap`
// entries.  No (tile, Gaussian) instance is written that no list keeps.
//
// The views' Gaussians come in depth order, N per view; a view's are cut into
// nb runs of `run`.
//  1. k_bin_count: one CTA per run counts the instances per tile.  A Gaussian
//     covers an interval of columns in each of its tile rows (packed spans,
//     tiles.cuh), so a row adds +1 and -1 at the interval's ends in shared
//     memory and a scan along the rows gives the counts: two shared atomics a
//     row instead of one per instance.
//  2. k_bin_prefix: per tile, the exclusive prefix of the counts over the runs;
//     k_bin_ranges: the kept [start, end) of every tile.
//  3. k_bin_fill: one CTA per run again.  A run none of whose tiles still has
//     room leaves at once, and so does a window of 32 Gaussians: with the
//     default cap most of a dense scene is only looked at (1M Gaussians, 8 x
//     640x480: 9.4M entries kept of 53.3M instances).  A window's (Gaussian,
//     row) pairs are spread over the CTA's lanes; every pair sets its
//     Gaussian's bit in a mask word per tile, and after a barrier the bits
//     below its own in a tile's mask are the Gaussian's rank there, so all
//     entries are written in depth order without any sorting.
// Bound by instruction issue and barriers in the fill (2 instructions a cycle
// and SM) and by the gather of 16-byte spans in depth order (one 32-byte sector
// each), not by the lists' bytes.  Measured at 8M Gaussian-views: 8 x 640x480
// (53.3M instances, 9.4M kept) count 0.11, prefix and ranges 0.02, fill
// 0.25 ms, where writing every instance and a bucket sort by tile took 0.47 +
// 0.65 and the offsets scan 0.13 ms; 8 x 1280x720 (110.9M, 28.0M kept) 0.20 +
// 0.76 ms against 1.47 (instances) + 2.01 (radix sort) + 0.34 (ranges) ms.
// Tried and not kept for the fill: one warp filtering the run's Gaussians per
// tile row (0.40 ms at 640x480), a thread walking its own Gaussian's tiles
// (one large Gaussian holds up its warp: 1.97 ms at 1280x720), all warps on
// one 32-Gaussian window at a time (0.70 ms, barrier latency).
#include <algorithm>

#include "common.cuh"
#include "list_rules.cuh"
#include "tiles.cuh"

namespace ups {

namespace {

constexpr int kBinThreads = 256;
constexpr int kBinWarps = kBinThreads / 32;

// The runs of a view: its first (nearest) nb1 * r1 Gaussians in runs of r1, the
// others in runs of r2.  The nearest Gaussians are the largest and fill most of
// the lists' room, so that long runs there would leave a few CTAs working alone
// (one 2048-Gaussian run of a 1280x720 view took 600 us); far away long runs
// keep the count matrix small.
struct Runs {
    int N, r1, nb1, r2, nb;
    __host__ __device__ int beg(int b) const { return b < nb1 ? b * r1 : nb1 * r1 + (b - nb1) * r2; }
    __host__ __device__ int end(int b) const { return beg(b + 1) < N ? beg(b + 1) : N; }
};

// counts of run blockIdx.x of view blockIdx.y: cnt[nb * tile_base + run * tiles + tile]
__global__ void __launch_bounds__(kBinThreads) k_bin_count(ViewTable vt, float alpha_min, Runs runs,
                                                           const uint32_t *__restrict__ sorted_gv,
                                                           const uint4 *__restrict__ span,
                                                           const uint4 *__restrict__ more,
                                                           const float4 *__restrict__ xyzo,
                                                           const float4 *__restrict__ conic,
                                                           uint32_t *__restrict__ cnt) {
    extern __shared__ int diff[];  // [tiles_y][tiles_x + 1]
    const DevView &cam = vt.v[blockIdx.y];
    const int tx = cam.tiles_x, ty = cam.tiles_y, ld = tx + 1, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < ld * ty; i += kBinThreads) diff[i] = 0;
    __syncthreads();
    const int beg = runs.beg(blockIdx.x), end = runs.end(blockIdx.x);
    const uint32_t *sg = sorted_gv + (size_t)blockIdx.y * runs.N;
    constexpr int U = 4;  // gathers in flight per thread
    for (int i0 = beg + threadIdx.x; i0 < end; i0 += U * kBinThreads) {
        uint32_t gv[U];
        uint4 s[U];
#pragma unroll
        for (int u = 0; u < U; ++u) gv[u] = i0 + u * kBinThreads < end ? sg[i0 + u * kBinThreads] : 0xffffffffu;
#pragma unroll
        for (int u = 0; u < U; ++u)
            s[u] = of_view(gv[u], blockIdx.y, runs.N) ? span[gv[u]] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < U; ++u)
            each_row(s[u], gv[u], more, xyzo, conic, alpha_min, cam, [&](int r, int c0, int c1) {
                atomicAdd(&diff[r * ld + c0], 1);
                atomicAdd(&diff[r * ld + c1 + 1], -1);
            });
    }
    __syncthreads();
    uint32_t *out = cnt + (size_t)runs.nb * cam.tile_base + (size_t)blockIdx.x * (tx * ty);
    for (int r = threadIdx.x >> 5; r < ty; r += kBinWarps) {
        int carry = 0;
        for (int c0 = 0; c0 < tx; c0 += 32) {
            const int c = c0 + lane;
            int x = c < tx ? diff[r * ld + c] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (c < tx) out[r * tx + c] = (uint32_t)(carry + x);
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
    }
}

// cnt -> exclusive prefix over the runs (in place), tot[tile] = sum.  A CTA
// takes 32 tiles of view blockIdx.y, a warp a contiguous part of the runs.
constexpr int kPrefWarps = 16;
__global__ void __launch_bounds__(32 * kPrefWarps) k_bin_prefix(ViewTable vt, int nb, uint32_t *__restrict__ cnt,
                                                                uint32_t *__restrict__ tot) {
    __shared__ uint32_t part[kPrefWarps][32];
    const DevView &cam = vt.v[blockIdx.y];
    const int tiles = cam.tiles_x * cam.tiles_y;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t = blockIdx.x * 32 + lane;
    if ((int)blockIdx.x * 32 >= tiles) return;
    const bool in = t < tiles;
    const int per = (nb + kPrefWarps - 1) / kPrefWarps, b0 = min(nb, w * per), b1 = min(nb, b0 + per);
    uint32_t *col = cnt + (size_t)nb * cam.tile_base + (in ? t : 0);
    uint32_t s = 0;
    if (in)
#pragma unroll 8
        for (int b = b0; b < b1; ++b) s += col[(size_t)b * tiles];
    part[w][lane] = s;
    __syncthreads();
    uint32_t at = 0, all = 0;
#pragma unroll
    for (int i = 0; i < kPrefWarps; ++i) {
        const uint32_t p = part[i][lane];
        at += i < w ? p : 0u;
        all += p;
    }
    if (!in) return;
    if (w == 0) tot[cam.tile_base + t] = all;
    for (int b8 = b0; b8 < b1; b8 += 8) {
        uint32_t x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = b8 + i < b1 ? col[(size_t)(b8 + i) * tiles] : 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (b8 + i < b1) {
                col[(size_t)(b8 + i) * tiles] = at;
                at += x[i];
            }
    }
}

// ranges[d] = the kept [start, start + min(tot[d], cap)) of every tile (clamped
// to the list buffer's n entries); bit d of trunc is set when tot[d] > cap.
// One CTA, kRangeItems consecutive tiles a thread and step.
constexpr int kRangeThreads = 1024, kRangeItems = 8;
__global__ void __launch_bounds__(kRangeThreads) k_bin_ranges(const uint32_t *__restrict__ tot, int tiles, uint32_t cap,
                                                              uint32_t n, uint2 *__restrict__ ranges,
                                                              uint32_t *__restrict__ trunc,
                                                              const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    __shared__ uint32_t wsum[kRangeThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t carry = 0;
    for (int d0 = 0; d0 < tiles; d0 += kRangeThreads * kRangeItems) {
        const int d = d0 + tid * kRangeItems;
        uint32_t kept[kRangeItems], sum = 0, over = 0;
#pragma unroll
        for (int i = 0; i < kRangeItems; ++i) kept[i] = d + i < tiles ? tot[d + i] : 0u;
#pragma unroll
        for (int i = 0; i < kRangeItems; ++i) {
            over |= (kept[i] > cap ? 1u : 0u) << i;
            kept[i] = min(kept[i], cap);
            sum += kept[i];
        }
        // four threads hold the 32 bits of one word of trunc
        uint32_t word = over << (kRangeItems * (lane & 3));
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, o);
        if ((lane & 3) == 0 && d < tiles) trunc[d >> 5] = word;
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        const uint32_t x = wsum[lane];
        uint32_t wi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        uint32_t at = carry + __shfl_sync(0xffffffffu, wi - x, w) + incl - sum;
        carry += __shfl_sync(0xffffffffu, wi, 31);
#pragma unroll
        for (int i = 0; i < kRangeItems; ++i) {
            if (d + i < tiles) ranges[d + i] = make_uint2(min(at, n), min(at + kept[i], n));
            at += kept[i];
        }
    }
}

// Queue entries of one step of the fill: 256 tile rows of up to 16 columns each
// (a step is cut to the rows that fit; a row has at most 1024 columns).
constexpr int kQueue = 4096;
constexpr int kCand = 3 * kBinThreads;  // candidate Gaussians waiting

// exclusive prefix of x over the CTA; ws: kBinWarps words.  Syncs before it
// writes ws and after.
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t *ws) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int i = 0; i < kBinWarps; ++i) before += i < w ? ws[i] : 0u;
    return before + incl - x;
}

// shared bytes of k_bin_fill: queue, candidates, a slot and a mask word per
// tile; capped: live bits and their summed-area table
struct FillShape {
    int tiles, live_words, sat;  // largest of the views (of their bands)
};
template <bool CAPPED>
size_t fill_smem(const FillShape &f) {
    return (size_t)(kQueue + kCand) * 4 + (size_t)f.tiles * (sizeof(Slot<CAPPED>) + 4) +
           (CAPPED ? (size_t)f.live_words * 4 + (size_t)f.sat * 2 : 0);
}

// BANDS: grid.x is views x bands; a CTA fills the tiles of one band of its view's rows,
// ceil(tiles_y / bands) rows each (the last ones may have none).  See plan_of.
template <bool CAPPED, bool BANDS>
__global__ void __launch_bounds__(kBinThreads) k_bin_fill(ViewTable vt, float alpha_min, Runs runs,
                                                          const uint32_t *__restrict__ sorted_gv,
                                                          const uint4 *__restrict__ span,
                                                          const uint4 *__restrict__ more,
                                                          const float4 *__restrict__ xyzo,
                                                          const float4 *__restrict__ conic,
                                                          const uint32_t *__restrict__ prior,
                                                          const uint32_t *__restrict__ tot,
                                                          const uint2 *__restrict__ ranges, uint32_t n,
                                                          uint32_t *__restrict__ lists, const int *__restrict__ gate,
                                                          int bands) {
    if (gate && *gate == 0) return;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ uint32_t wsum[2 * kBinWarps];
    __shared__ int s_first[kBinThreads + 1];      // rows of the step's candidates before each
    __shared__ uint32_t s_head[kBinThreads];      // their span heads
    __shared__ uint32_t s_woff[kBinWarps], s_end[2];  // first queue entry of each window; end, last window
    __shared__ int s_first_window;
    // runs along grid.y: the nearest runs of every view, which hold most of the
    // entries, start first
    const int view = BANDS ? blockIdx.x / bands : blockIdx.x;
    const DevView &cam = vt.v[view];
    // rows and tiles of the band, counted from its first row b0 and first tile t0
    const int per_band = BANDS ? (cam.tiles_y + bands - 1) / bands : cam.tiles_y;
    const int b0 = BANDS ? ((int)blockIdx.x - view * bands) * per_band : 0;
    const int tx = cam.tiles_x, ty = BANDS ? min(per_band, cam.tiles_y - b0) : cam.tiles_y, tiles = tx * ty;
    const int t0 = cam.tile_base + b0 * tx;
    if (BANDS && ty <= 0) return;
    const int lw = (tx + 31) >> 5;  // words of a row's live bits
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t lt_mask = (1u << lane) - 1u;
    uint32_t *queue = reinterpret_cast<uint32_t *>(sm);  // [kQueue] tile << 8 | candidate of the step
    uint32_t *cand = queue + kQueue;                     // [kCand] Gaussian-views
    Slot<CAPPED> *slot = reinterpret_cast<Slot<CAPPED> *>(cand + kCand);
    uint32_t *mask = reinterpret_cast<uint32_t *>(slot + tiles);  // Gaussians of the window on each tile
    uint32_t *live = mask + tiles;  // capped: a bit per column of each row, set while the tile has room
    uint16_t *sat = reinterpret_cast<uint16_t *>(live + lw * ty);  // capped: [ty + 1][tx + 1] live tiles above and left
    // the tiles' slots before this run; leave if none takes anything from it
    {
        const int all = tx * cam.tiles_y;  // of the view
        const uint32_t *pr = prior + (size_t)runs.nb * cam.tile_base + (size_t)blockIdx.y * all + b0 * tx;
        const uint32_t *pn = (int)blockIdx.y == runs.nb - 1 ? tot + t0 : pr + all;
        bool any = false;
        if constexpr (CAPPED) {
            for (int i = tid; i < lw * ty; i += kBinThreads) live[i] = 0u;
            __syncthreads();
        }
        for (int t = tid; t < tiles; t += kBinThreads) {
            const uint2 r = ranges[t0 + t];
            const uint32_t p = pr[t];
            const uint32_t at = r.x + min(p, r.y - r.x);
            const bool takes = pn[t] > p && at < r.y;
            any = any || takes;
            slot[t].next = at;
            mask[t] = 0u;
            if constexpr (CAPPED) {
                slot[t].stop = r.y;
                if (takes) {
                    const int row = t / tx, x = t - row * tx;
                    atomicOr(&live[row * lw + (x >> 5)], 1u << (x & 31));
                }
            }
        }
        if (!__syncthreads_or(any)) return;
    }
    if constexpr (CAPPED) {
        for (int i = tid; i < (ty + 1) * (tx + 1); i += kBinThreads) {
            const int r = i / (tx + 1), x = i - r * (tx + 1);  // live tiles of row r - 1 left of column x
            uint32_t c = 0;
            if (r > 0) {
                const uint32_t *row = live + (r - 1) * lw;
                for (int k = 0; k < x >> 5; ++k) c += __popc(row[k]);
                if (x & 31) c += __popc(row[x >> 5] & ((1u << (x & 31)) - 1u));
            }
            sat[i] = (uint16_t)c;
        }
        __syncthreads();
        for (int x = tid; x <= tx; x += kBinThreads) {
            uint32_t c = 0;
            for (int r = 1; r <= ty; ++r) {
                c += sat[r * (tx + 1) + x];
                sat[r * (tx + 1) + x] = (uint16_t)c;
            }
        }
    }
    const int beg = runs.beg(blockIdx.y), cnt = runs.end(blockIdx.y) - beg;
    const uint32_t *sg = sorted_gv + (size_t)view * runs.N + beg;
    // bits of word i of row r's live tiles inside columns [c0, c1]
    auto live_word = [&](const RowItem &t, int i) {
        uint32_t b = live[t.r * lw + i];
        if (i == t.c0 >> 5) b &= 0xffffffffu << (t.c0 & 31);
        if (i == t.c1 >> 5) b &= 0xffffffffu >> (31 - (t.c1 & 31));
        return b;
    };
    // entries of a row item: the tiles it meets that have room
    auto entries = [&](const RowItem &t) {
        if constexpr (CAPPED) {
            uint32_t c = 0;
            for (int i = t.c0 >> 5; i <= t.c1 >> 5; ++i) c += __popc(live_word(t, i));
            return c;
        } else {
            return (uint32_t)(t.c1 - t.c0 + 1);
        }
    };
    auto filled = [&](int tile) {  // the tile took its last entry
        const int row = tile / tx, x = tile - row * tx;
        atomicAnd(&live[row * lw + (x >> 5)], ~(1u << (x & 31)));
    };
    int nc = 0;  // candidates waiting (the same in every thread)
    for (int pos = 0;;) {
        // candidates: the next Gaussians whose box holds a tile with room
        while (nc < kBinThreads && pos < cnt) {
            __syncthreads();
            uint32_t gv[2], hits[2];
            bool hit[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = pos + u * kBinThreads + tid;
                gv[u] = i < cnt ? sg[i] : 0xffffffffu;
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                hit[u] = false;
                if (of_view(gv[u], view, runs.N)) {
                    const uint4 s = span[gv[u]];
                    const int nr = (int)span_rows(s.x), x0 = (int)(s.x & 1023u), y0 = (int)((s.x >> 10) & 1023u);
                    // rows [ya, yb) of the band
                    const int y1 = nr == (int)kSpanTall ? (int)(s.z >> 16) + 1 : y0 + nr;
                    const int ya = BANDS ? max(y0 - b0, 0) : y0, yb = BANDS ? min(y1 - b0, ty) : y1;
                    hit[u] = nr && (!BANDS || ya < yb);
                    if constexpr (CAPPED) {
                        const uint32_t wide = s.x >> 25;
                        const int x1 = wide == kSpanWide ? tx : x0 + (int)wide + 1;
                        const int a = ya * (tx + 1), b = yb * (tx + 1);
                        hit[u] = hit[u] &&
                                 (int)sat[b + x1] - (int)sat[b + x0] - (int)sat[a + x1] + (int)sat[a + x0] > 0;
                    }
                }
                hits[u] = __ballot_sync(0xffffffffu, hit[u]);
                if (lane == 0) wsum[u * kBinWarps + w] = __popc(hits[u]);
            }
            __syncthreads();
            int at[2] = {nc, nc};
#pragma unroll
            for (int i = 0; i < 2 * kBinWarps; ++i) {
                const int c = (int)wsum[i];
                at[0] += i < w ? c : 0;
                at[1] += i < kBinWarps + w ? c : 0;
                nc += c;
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (hit[u]) cand[at[u] + __popc(hits[u] & lt_mask)] = gv[u];
            pos += 2 * kBinThreads;
        }
        __syncthreads();
        if (nc == 0) break;
        // the first 256 candidates' rows (in the band: one at least), numbered through
        const int m = min(nc, kBinThreads);
        const uint4 s4 = tid < m ? span[cand[tid]] : make_uint4(0u, 0u, 0u, 0u);
        int nr = (int)span_rows(s4.x);
        if (nr == (int)kSpanTall) nr = (int)(s4.z >> 16) - (int)(s4.y >> 16) + 1;
        if (BANDS && tid < m) {
            const int y0 = (int)((s4.x >> 10) & 1023u);
            nr = min(y0 + nr, b0 + ty) - max(y0, b0);
        }
        const uint32_t first = block_scan((uint32_t)nr, wsum);
        s_first[tid] = (int)first;
        s_head[tid] = s4.x;
        if (tid == kBinThreads - 1) s_first[kBinThreads] = (int)first + nr;
        __syncthreads();
        const int rows = s_first[kBinThreads];
        for (int i0 = 0; i0 < rows;) {
            // a thread a row: the candidate L it belongs to, its entries
            const int i = i0 + tid;
            const bool in = i < rows;
            int L = 0;
#pragma unroll
            for (int step = kBinThreads / 2; step >= 1; step >>= 1)
                if (s_first[L + step] <= i) L += step;
            RowItem t{0, 1, 0};
            if (in) {
                const uint32_t head = s_head[L];
                const int skip = BANDS ? max(b0 - (int)((head >> 10) & 1023u), 0) : 0;  // rows above the band
                t = row_item(cand[L], head, i - s_first[L] + skip, span, more, xyzo, conic, alpha_min, cam);
                t.r -= b0;
            }
            const uint32_t c = t.c0 <= t.c1 ? entries(t) : 0u;
            uint32_t o = block_scan(c, wsum);
            // rows whose entries fit the queue (all but the last few of a step, if any are left)
            const bool fits = in && o + c <= (uint32_t)kQueue;
            const int taken = __syncthreads_count(fits);
            if (tid == taken - 1) {
                s_end[0] = o + c;
                s_end[1] = (uint32_t)L >> 5;
            }
            if (tid == 0) s_first_window = L >> 5;
            if (fits) {
                if (i == max(i0, s_first[L & ~31])) s_woff[L >> 5] = o;
                if (c) {
                    const uint32_t row = (uint32_t)(t.r * tx);
                    if constexpr (CAPPED) {
                        for (int k = t.c0 >> 5; k <= t.c1 >> 5; ++k)
                            for (uint32_t l = live_word(t, k); l; l &= l - 1)
                                queue[o++] = (row + 32 * k + __ffs(l) - 1) << 8 | (uint32_t)L;
                    } else {
                        for (int x = t.c0; x <= t.c1; ++x) queue[o++] = (row + x) << 8 | (uint32_t)L;
                    }
                }
            }
            i0 += taken;
            __syncthreads();
            const uint32_t end = s_end[0];
            const int wlast = (int)s_end[1];
            for (int k = s_first_window; k <= wlast; ++k) {
                // window k: 32 candidates, one mask bit each
                const uint32_t a = s_woff[k], b = k == wlast ? end : s_woff[k + 1];
                if (a == b) continue;
                for (uint32_t j = a + tid; j < b; j += kBinThreads) {
                    const uint32_t e = queue[j];
                    atomicOr(&mask[e >> 8], 1u << (e & 31u));
                }
                __syncthreads();
                for (uint32_t j = a + tid; j < b; j += kBinThreads) {
                    const uint32_t e = queue[j];
                    const Slot<CAPPED> sl = slot[e >> 8];
                    const uint32_t at = sl.next + __popc(mask[e >> 8] & ((1u << (e & 31u)) - 1u));
                    if (sl.fits(at, n)) lists[at] = cand[e & 255u];
                }
                __syncthreads();
                // the first Gaussian of each tile moves its slot on and clears its mask
                for (uint32_t j = a + tid; j < b; j += kBinThreads) {
                    const uint32_t e = queue[j];
                    const uint32_t bits = mask[e >> 8];
                    if ((bits & ((1u << (e & 31u)) - 1u)) || !bits) continue;
                    Slot<CAPPED> &sl = slot[e >> 8];
                    sl.next += __popc(bits);
                    mask[e >> 8] = 0u;
                    if (!sl.room()) filled((int)(e >> 8));
                }
                __syncthreads();
            }
            __syncthreads();
        }
        // the candidates left move to the front
        uint32_t keep[kCand / kBinThreads];
#pragma unroll
        for (int u = 0; u < kCand / kBinThreads; ++u)
            keep[u] = m + u * kBinThreads + tid < nc ? cand[m + u * kBinThreads + tid] : 0u;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kCand / kBinThreads; ++u)
            if (m + u * kBinThreads + tid < nc) cand[u * kBinThreads + tid] = keep[u];
        nc -= m;
    }
}

struct Plan {
    Runs runs;
    int bands, most_tiles;  // of the fill; tiles of the largest view
    FillShape fill;
    size_t count_smem;
};

// A view of more than kBandless tiles is filled in bands of about kBandTiles: the state
// of its tiles (14 bytes each) would take most of an SM's shared memory, or more than
// there is, and leave it one CTA.  One view of 2560x1440 (14,400 tiles): 300k Gaussians
// (13.8M instances) lists 0.27 ms and 1.12 the frame, where one band with the ends of the
// lists read from global memory took 0.59 and writing and bucket sorting every instance
// 1.11 (2.10); 1M small faint ones (4.8M instances) 0.33 against 0.67 and 0.41.
constexpr int kBandless = 8191, kBandTiles = 4096;
// tile sides are at most this (16,384 pixels)
constexpr int kMaxSide = 1024;

// Runs of 512 for the nearest eighth of a view and 4096 behind it; a batch with
// fewer than four runs of 2048 an SM takes short ones throughout, down to 128
// until every SM has four.
Plan plan_of(const ViewTable &vt, int N, int num_sms) {
    Plan p{};
    Runs &r = p.runs;
    const size_t total = (size_t)N * vt.n, want = (size_t)num_sms * 4;
    r.N = N;
    r.r1 = 512;
    while (r.r1 > 128 && total / r.r1 < want) r.r1 >>= 1;
    r.r2 = total / 2048 < want ? r.r1 : 4096;
    while (N / r.r2 > 30000) r.r1 <<= 1, r.r2 <<= 1;  // runs lie along grid.y
    r.nb1 = r.r1 == r.r2 ? 0 : N / 8 / r.r1;
    r.nb = r.nb1 + (N - r.nb1 * r.r1 + r.r2 - 1) / r.r2;
    for (int v = 0; v < vt.n; ++v) p.most_tiles = std::max(p.most_tiles, vt.v[v].tiles_x * vt.v[v].tiles_y);
    p.bands = p.most_tiles <= kBandless ? 1 : (p.most_tiles + kBandTiles - 1) / kBandTiles;
    for (int v = 0; v < vt.n; ++v) {
        const DevView &c = vt.v[v];
        const int rows = (c.tiles_y + p.bands - 1) / p.bands;
        p.fill.tiles = std::max(p.fill.tiles, c.tiles_x * rows);
        p.fill.live_words = std::max(p.fill.live_words, (c.tiles_x + 31) / 32 * rows);
        p.fill.sat = std::max(p.fill.sat, (c.tiles_x + 1) * (rows + 1));
        p.count_smem = std::max(p.count_smem, (size_t)(c.tiles_x + 1) * c.tiles_y * sizeof(int));
    }
    return p;
}

// The largest shape of a view or band (a band's last row may pass kBandTiles, but not
// kBandless), at most kMaxSide tiles a side.
constexpr FillShape kMaxFill{kBandless, kBandless / 32 + kMaxSide, kBandless + 2 * kMaxSide + 1};
constexpr size_t kMaxCountSmem = (size_t)(kMaxBinTiles + kMaxSide) * sizeof(int);

template <bool CAPPED, bool BANDS>
cudaError_t launch_fill(const ViewTable &vt, float alpha_min, const Plan &p, const uint32_t *sorted_gv,
                        const uint4 *span, const uint4 *more, const float4 *xyzo, const float4 *conic,
                        const uint32_t *cnt, const uint32_t *tot, const uint2 *ranges, uint32_t n, uint32_t *lists,
                        const int *gate, cudaStream_t st) {
    const cudaError_t e = allow_smem(k_bin_fill<CAPPED, BANDS>, fill_smem<CAPPED>(kMaxFill));
    if (e != cudaSuccess) return e;
    k_bin_fill<CAPPED, BANDS><<<dim3(vt.n * p.bands, p.runs.nb), kBinThreads, fill_smem<CAPPED>(p.fill), st>>>(
        vt, alpha_min, p.runs, sorted_gv, span, more, xyzo, conic, cnt, tot, ranges, n, lists, gate, p.bands);
    return cudaGetLastError();
}

}  // namespace

bool bin_supported(const ViewTable &vt) {
    for (int v = 0; v < vt.n; ++v)
        if (vt.v[v].tiles_x * vt.v[v].tiles_y > kMaxBinTiles) return false;
    return true;
}

size_t bin_scratch_bytes(const ViewTable &vt, int N, int num_sms) {
    const Plan p = plan_of(vt, N, num_sms);
    return ((size_t)p.runs.nb + 1) * vt.total_tiles * sizeof(uint32_t);
}

cudaError_t bin_count(const ViewTable &vt, float alpha_min, int N, const uint32_t *sorted_gv, const uint4 *span,
                      const uint4 *more, const float4 *xyzo, const float4 *conic, void *scratch, int num_sms, cudaStream_t st) {
    const Plan p = plan_of(vt, N, num_sms);
    uint32_t *tot = static_cast<uint32_t *>(scratch), *cnt = tot + vt.total_tiles;
    cudaError_t e = allow_smem(k_bin_count, kMaxCountSmem);
    if (e != cudaSuccess) return e;
    k_bin_count<<<dim3(p.runs.nb, vt.n), kBinThreads, p.count_smem, st>>>(vt, alpha_min, p.runs, sorted_gv, span,
                                                                     more, xyzo, conic, cnt);
    k_bin_prefix<<<dim3((p.most_tiles + 31) / 32, vt.n), 32 * kPrefWarps, 0, st>>>(vt, p.runs.nb, cnt, tot);
    return cudaGetLastError();
}

cudaError_t bin_lists(const ViewTable &vt, float alpha_min, int N, const uint32_t *sorted_gv, const uint4 *span,
                      const uint4 *more, const float4 *xyzo, const float4 *conic, void *scratch, uint32_t cap, uint32_t n, uint2 *ranges,
                      uint32_t *trunc, uint32_t *lists, int num_sms, cudaStream_t st, const int *gate) {
    const Plan p = plan_of(vt, N, num_sms);
    uint32_t *tot = static_cast<uint32_t *>(scratch), *cnt = tot + vt.total_tiles;
    k_bin_ranges<<<1, kRangeThreads, 0, st>>>(tot, vt.total_tiles, cap, n, ranges, trunc, gate);
    if (n == 0) return cudaGetLastError();
    const auto fill = cap == kNoListCap ? (p.bands > 1 ? launch_fill<false, true> : launch_fill<false, false>)
                                        : (p.bands > 1 ? launch_fill<true, true> : launch_fill<true, false>);
    return fill(vt, alpha_min, p, sorted_gv, span, more, xyzo, conic, cnt, tot, ranges, n, lists, gate, st);
}

namespace {
__global__ void k_keys_from_ranges(const uint2 *__restrict__ ranges, uint32_t *__restrict__ keys) {
    const uint2 r = ranges[blockIdx.x];
    for (uint32_t i = r.x + threadIdx.x; i < r.y; i += blockDim.x) keys[i] = blockIdx.x;
}
}  // namespace

cudaError_t keys_from_ranges(const uint2 *ranges, int nbins, uint32_t *keys, cudaStream_t st) {
    if (nbins <= 0) return cudaSuccess;
    k_keys_from_ranges<<<nbins, 256, 0, st>>>(ranges, keys);
    return cudaGetLastError();
}

}  // namespace ups
