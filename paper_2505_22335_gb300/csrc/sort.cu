// Stable LSD radix sort of (key, value) pairs and exclusive scans, written for
// this library (no CUB).  Orders the Gaussian-views by (view, depth); for views
// too large for the row-wise tile lists (bin.cu) also the tile instances by
// (view, tile), which together give the (view, tile, depth, id) order.
//
// One pass of the instance sort = histogram kernel (per-block digit counts,
// digit-major layout) + exclusive scan of the counts + scatter kernel (stable
// block-local ranking by ballots, then a scatter to the scanned offsets).  The
// order of the Gaussian-views (sorted_order) takes one kernel a pass: see below.
#include <algorithm>
#include <utility>

#include "common.cuh"

namespace ups {

namespace {

constexpr int kThreads = 256;
constexpr int kBins = 256;  // 8-bit digits
constexpr int kWarps = kThreads / 32;

// Items per thread: 8 keeps the scatter kernel near 50 registers (five
// 256-thread blocks per SM hide the latency of its ranking loop) and the
// block tile staged in shared memory under 48 KB.
template <class K> struct Radix {
    static constexpr int items = 8;
    static constexpr int tile = kThreads * items;
};

// 256-wide exclusive scan across the block (one value per thread).
__device__ __forceinline__ uint32_t scan256(uint32_t x, uint32_t *warp_tot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) before += ww < w ? warp_tot[ww] : 0u;
    return before + incl - x;
}

template <class K>
__global__ void __launch_bounds__(kThreads) k_radix_hist(const K *__restrict__ keys, size_t n,
                                                         int shift, uint32_t *__restrict__ hist,
                                                         int nblocks) {
    constexpr int TILE = Radix<K>::tile;
    __shared__ uint32_t h[kWarps][kBins];
    const int tid = threadIdx.x, w = tid >> 5;
    for (int i = tid; i < kWarps * kBins; i += kThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * TILE;
#pragma unroll 4
    for (int i = tid; i < TILE; i += kThreads) {
        size_t idx = base + i;
        if (idx < n) {
            uint32_t d = (uint32_t)(keys[idx] >> shift) & (kBins - 1);
            atomicAdd(&h[w][d], 1u);
        }
    }
    __syncthreads();
    uint32_t s = 0;
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) s += h[ww][tid];
    hist[(size_t)tid * nblocks + blockIdx.x] = s;
}

// Stable scatter of one block tile: ballot-based ranking inside each warp,
// then the tile is reordered by digit in shared memory and written out in
// order, so consecutive threads store consecutive addresses of a bucket.
template <class K>
__global__ void __launch_bounds__(kThreads) k_radix_scatter(
    const K *__restrict__ kin, const uint32_t *__restrict__ vin, K *__restrict__ kout,
    uint32_t *__restrict__ vout, size_t n, int shift, const uint32_t *__restrict__ offs,
    int nblocks) {
    constexpr int ITEMS = Radix<K>::items, TILE = Radix<K>::tile;
    __shared__ uint32_t wcnt[kWarps][kBins];
    __shared__ uint32_t dstart[kBins];
    __shared__ uint32_t gbase[kBins];
    __shared__ uint32_t wtot[kWarps];
    __shared__ K skey[TILE];
    __shared__ uint32_t sval[TILE];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    for (int i = tid; i < kWarps * kBins; i += kThreads) (&wcnt[0][0])[i] = 0;
    __syncthreads();
    const uint32_t lt_mask = (1u << lane) - 1u;
    const size_t tile_base = (size_t)blockIdx.x * TILE;
    const size_t base = tile_base + (size_t)w * (32 * ITEMS);
    K key[ITEMS];
    uint32_t val[ITEMS];
    uint32_t rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        size_t idx = base + (size_t)j * 32 + lane;
        bool valid = idx < n;
        uint32_t d = kBins;  // sentinel for out-of-range lanes
        if (valid) {
            key[j] = kin[idx];
            val[j] = vin[idx];
            d = (uint32_t)(key[j] >> shift) & (kBins - 1);
        }
        uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            uint32_t bit = (d >> b) & 1u;
            uint32_t bb = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bb : ~bb;
        }
        uint32_t lt = __popc(peers & lt_mask);
        uint32_t prior = valid ? wcnt[w][d] : 0u;
        __syncwarp();
        if (valid && lt == 0) wcnt[w][d] = prior + __popc(peers);
        __syncwarp();
        rank[j] = prior + lt;
    }
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) {
        uint32_t c = wcnt[ww][tid];
        wcnt[ww][tid] = run;
        run += c;
    }
    dstart[tid] = scan256(run, wtot);
    gbase[tid] = offs[(size_t)tid * nblocks + blockIdx.x];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        size_t idx = base + (size_t)j * 32 + lane;
        if (idx < n) {
            uint32_t d = (uint32_t)(key[j] >> shift) & (kBins - 1);
            uint32_t lpos = dstart[d] + wcnt[w][d] + rank[j];
            skey[lpos] = key[j];
            sval[lpos] = val[j];
        }
    }
    __syncthreads();
    const int nvalid = (int)min((size_t)TILE, n - tile_base);
    for (int i = tid; i < nvalid; i += kThreads) {
        K k = skey[i];
        uint32_t d = (uint32_t)(k >> shift) & (kBins - 1);
        uint32_t pos = gbase[d] + (uint32_t)i - dstart[d];
        kout[pos] = k;
        vout[pos] = sval[i];
    }
}

// ---------------------------------------------------------------------------
// exclusive scan (3 kernels: block sums, scan of block sums, apply)
// ---------------------------------------------------------------------------

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class T>
__device__ T block_exclusive_scan(T x, T *total) {
    __shared__ T warp_sums[kScanThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[w] = incl;
    __syncthreads();
    if (w == 0) {
        T s = lane < kScanThreads / 32 ? warp_sums[lane] : T(0);
        T si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += y;
        }
        if (lane < kScanThreads / 32) warp_sums[lane] = si - s;
        if (lane == kScanThreads / 32 - 1) *total = si;
    }
    __syncthreads();
    T r = warp_sums[w] + incl - x;
    __syncthreads();
    return r;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const uint32_t *__restrict__ in,
                                                              size_t n, T *__restrict__ partial) {
    __shared__ T tot;
    const size_t base = (size_t)blockIdx.x * kScanTile;
    T s = 0;
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
        size_t idx = base + i;
        if (idx < n) s += in[idx];
    }
    block_exclusive_scan<T>(s, &tot);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) k_scan_partials(T *partial, int nb) {
    __shared__ T tot;
    T carry = 0;
    for (int b0 = 0; b0 < nb; b0 += kScanThreads) {
        int i = b0 + threadIdx.x;
        T x = i < nb ? partial[i] : T(0);
        T ex = block_exclusive_scan<T>(x, &tot);
        if (i < nb) partial[i] = carry + ex;
        carry += tot;
        __syncthreads();
    }
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const uint32_t *in, T *out, size_t n,
                                                             const T *__restrict__ partial,
                                                             int write_total) {
    __shared__ uint32_t tile[kScanTile];
    __shared__ T tot;
    const size_t base = (size_t)blockIdx.x * kScanTile;
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
        size_t idx = base + i;
        tile[i] = idx < n ? in[idx] : 0u;
    }
    __syncthreads();
    T loc[kScanItems];
    T s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        loc[j] = s;
        s += tile[threadIdx.x * kScanItems + j];
    }
    T ex = block_exclusive_scan<T>(s, &tot) + partial[blockIdx.x];
    __syncthreads();
    // write back through shared memory for coalesced stores
    T *otile = reinterpret_cast<T *>(tile);  // reuse only when T fits
    if (sizeof(T) == sizeof(uint32_t)) {
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) otile[threadIdx.x * kScanItems + j] = ex + loc[j];
        __syncthreads();
        for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
            size_t idx = base + i;
            if (idx < n) out[idx] = otile[i];
        }
    } else {
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            size_t idx = base + threadIdx.x * kScanItems + j;
            if (idx < n) out[idx] = ex + loc[j];
        }
    }
    if (write_total && base <= n - 1 && n - 1 < base + kScanTile) {
        if (threadIdx.x == (int)((n - 1 - base) / kScanItems)) {
            int j = (int)((n - 1 - base) % kScanItems);
            // total = exclusive prefix of the last element + its value
            out[n] = ex + loc[j] + (T)in[n - 1];
        }
    }
}

template <class T>
cudaError_t scan_impl(const uint32_t *in, T *out, size_t n, void *scratch, int write_total,
                      cudaStream_t st) {
    if (n == 0) {
        if (write_total) return cudaMemsetAsync(out, 0, sizeof(T), st);
        return cudaSuccess;
    }
    int nb = (int)((n + kScanTile - 1) / kScanTile);
    T *partial = static_cast<T *>(scratch);
    k_scan_reduce<T><<<nb, kScanThreads, 0, st>>>(in, n, partial);
    k_scan_partials<T><<<1, kScanThreads, 0, st>>>(partial, nb);
    k_scan_apply<T><<<nb, kScanThreads, 0, st>>>(in, out, n, partial, write_total);
    return cudaGetLastError();
}

template <class K>
cudaError_t radix_impl(K **key_io, K **key_alt, uint32_t **val_io, uint32_t **val_alt, size_t n,
                       int end_bit, SortScratch &s, cudaStream_t st) {
    if (n <= 1 || end_bit <= 0) return cudaSuccess;
    int nblocks = (int)((n + Radix<K>::tile - 1) / Radix<K>::tile);
    size_t hist_n = (size_t)kBins * nblocks;
    size_t need = hist_n * sizeof(uint32_t) + scan_scratch_bytes(hist_n);
    cudaError_t e = s.hist.reserve(need);
    if (e != cudaSuccess) return e;
    uint32_t *hist = s.hist.as<uint32_t>();
    void *scr = reinterpret_cast<char *>(s.hist.ptr) + ((hist_n * sizeof(uint32_t) + 255) & ~size_t(255));
    for (int shift = 0; shift < end_bit; shift += 8) {
        k_radix_hist<K><<<nblocks, kThreads, 0, st>>>(*key_io, n, shift, hist, nblocks);
        e = scan_impl<uint32_t>(hist, hist, hist_n, scr, 0, st);
        if (e != cudaSuccess) return e;
        k_radix_scatter<K><<<nblocks, kThreads, 0, st>>>(*key_io, *val_io, *key_alt, *val_alt, n,
                                                         shift, hist, nblocks);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        K *tk = *key_io;
        *key_io = *key_alt;
        *key_alt = tk;
        uint32_t *tv = *val_io;
        *val_io = *val_alt;
        *val_alt = tv;
    }
    return cudaSuccess;
}

// Same passes as radix_impl, with the histogram and scan scratch supplied by
// the caller instead of a growable buffer.
template <class K>
cudaError_t radix_fixed(K **key_io, K **key_alt, uint32_t **val_io, uint32_t **val_alt, size_t n,
                        int end_bit, void *scratch, size_t scratch_bytes, cudaStream_t st) {
    if (n <= 1 || end_bit <= 0) return cudaSuccess;
    int nblocks = (int)((n + Radix<K>::tile - 1) / Radix<K>::tile);
    size_t hist_n = (size_t)kBins * nblocks;
    size_t hist_bytes = (hist_n * sizeof(uint32_t) + 255) & ~size_t(255);
    if (hist_bytes + scan_scratch_bytes(hist_n) > scratch_bytes) return cudaErrorInvalidValue;
    uint32_t *hist = static_cast<uint32_t *>(scratch);
    void *scr = static_cast<char *>(scratch) + hist_bytes;
    for (int shift = 0; shift < end_bit; shift += 8) {
        k_radix_hist<K><<<nblocks, kThreads, 0, st>>>(*key_io, n, shift, hist, nblocks);
        cudaError_t e = scan_impl<uint32_t>(hist, hist, hist_n, scr, 0, st);
        if (e != cudaSuccess) return e;
        k_radix_scatter<K><<<nblocks, kThreads, 0, st>>>(*key_io, *val_io, *key_alt, *val_alt, n,
                                                         shift, hist, nblocks);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        K *tk = *key_io;
        *key_io = *key_alt;
        *key_alt = tk;
        uint32_t *tv = *val_io;
        *val_io = *val_alt;
        *val_alt = tv;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// order of n keys: one kernel per 8-bit pass
// ---------------------------------------------------------------------------
//
// k_order_hist counts every digit of all passes in one read of the keys.  A
// pass is then one kernel (k_order_pass): a CTA takes the next tile of the
// input (a ticket, so that every earlier tile is already running or done),
// ranks its items by ballots, publishes its 256 digit counts and finds the
// items before it by walking back over the earlier tiles' published counts until
// one holds its inclusive sum (the "decoupled look-back" of Merrill and Garland's
// single-pass prefix scan, 2016, applied to digit counts as in Adinets and Merrill's
// Onesweep, 2022).  Every wait on a published count is bounded: a
// wait that runs out sets *err and ends the CTA (its consumers take no id on trust:
// list_rules.cuh, k_gather_counts and k_emit).  The first pass makes up the values (the positions) and the last
// one writes no keys.  Held by the ranking's ballots and the walk back, not by
// its 16 bytes an item and pass: 8M keys 0.32 to 0.35 ms (0.38 with a histogram,
// three scan kernels and a scatter a pass), 100k keys 47 us (130), where the 20
// launches were the cost.  Tiles of 2048, 2560 and 3072 keys at 8M: 0.35, 0.33,
// 0.32 ms.
//
// Up to kSmallOrder keys are sorted by one CTA in shared memory instead: below
// that size a launch costs more than a pass (2,000 keys: 18 us against 95).

constexpr int kOrderPasses = 5;  // at most 40 key bits
constexpr int kOrderPolls = 1 << 22;
constexpr int kSmallThreads = 512, kSmallWarps = kSmallThreads / 32, kSmallItems = 8;
constexpr int kSmallOrder = kSmallThreads * kSmallItems;

// Scratch of one order: digit counts and a ticket per pass, then the tiles'
// published counts (value | state << 62) of every pass.  Cleared before use.
struct OrderHead {
    uint32_t hist[kOrderPasses][kBins];
    uint32_t ticket[kOrderPasses];
    uint32_t pad[3];
};
constexpr unsigned long long kStateMask = (1ull << 62) - 1, kStateSum = 1ull << 62, kStateAll = 2ull << 62;

__device__ __forceinline__ unsigned long long state_load(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void state_store(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <class K>
__global__ void __launch_bounds__(kThreads) k_order_hist(const K *__restrict__ keys, size_t n, int passes,
                                                         OrderHead *__restrict__ head) {
    __shared__ uint32_t h[kOrderPasses][kBins];
    for (int i = threadIdx.x; i < passes * kBins; i += kThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    constexpr int U = 16 / sizeof(K);  // keys per 16-byte load
    const size_t nv = n / U, step = (size_t)gridDim.x * kThreads, t = (size_t)blockIdx.x * kThreads + threadIdx.x;
    auto count = [&](K k) {
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(uint32_t)(k >> (8 * p)) & (kBins - 1)], 1u);
    };
    for (size_t i = t; i < nv; i += step) {
        const uint4 v = reinterpret_cast<const uint4 *>(keys)[i];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if constexpr (sizeof(K) == 4)
                count(w[u]);
            else
                count((K)w[2 * u] | (K)w[2 * u + 1] << 32);
        }
    }
    for (size_t i = nv * U + t; i < n; i += step) count(keys[i]);
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kBins; i += kThreads) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&head->hist[0][0] + i, c);
    }
}

// Ranks a warp's items (item j of lane l is its 32 j + l-th) among the earlier
// items of the warp with the same digit; cnt: the warp's 256 digit counters,
// zero before, the digit totals after.
template <class K, int ITEMS>
__device__ __forceinline__ void warp_rank(const K (&key)[ITEMS], int shift, int valid, uint32_t *cnt,
                                          uint32_t (&rank)[ITEMS]) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool in = 32 * j + lane < valid;
        const uint32_t d = (uint32_t)(key[j] >> shift) & (kBins - 1);
        uint32_t peers = __ballot_sync(0xffffffffu, in);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t bit = (d >> b) & 1u;
            const uint32_t bb = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bb : ~bb;
        }
        const uint32_t lt = __popc(peers & lt_mask);
        const uint32_t prior = in ? cnt[d] : 0u;
        __syncwarp();
        if (in && lt == 0) cnt[d] = prior + __popc(peers);
        __syncwarp();
        rank[j] = prior + lt;
    }
}

template <class K, int ITEMS>
__global__ void __launch_bounds__(kThreads, 4) k_order_pass(const K *__restrict__ kin, const uint32_t *__restrict__ vin,
                                                         K *__restrict__ kout, uint32_t *__restrict__ vout, size_t n,
                                                         int pass, OrderHead *__restrict__ head,
                                                         unsigned long long *__restrict__ state,
                                                         int *__restrict__ err) {
    constexpr int TILE = kThreads * ITEMS;
    __shared__ uint32_t wcnt[kWarps][kBins];
    __shared__ uint32_t dstart[kBins], gbase[kBins], wtot[kWarps], wtot2[kWarps];
    __shared__ uint32_t s_tile;
    __shared__ K skey[TILE];
    __shared__ uint32_t sval[TILE];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, shift = 8 * pass;
    if (tid == 0) s_tile = atomicAdd(&head->ticket[pass], 1u);
    for (int i = tid; i < kWarps * kBins; i += kThreads) (&wcnt[0][0])[i] = 0;
    __syncthreads();
    const size_t tile = s_tile, tile_base = tile * TILE;
    const size_t base = tile_base + (size_t)w * (32 * ITEMS) + lane;
    const int nvalid = (int)min((size_t)TILE, n - tile_base);
    const int wvalid = min(max(nvalid - w * 32 * ITEMS, 0), 32 * ITEMS);
    K key[ITEMS];
    uint32_t val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool in = 32 * j + lane < wvalid;
        key[j] = in ? kin[base + 32 * j] : K(0);
        val[j] = !in ? 0u : vin ? vin[base + 32 * j] : (uint32_t)(base + 32 * j);
    }
    warp_rank<K, ITEMS>(key, shift, wvalid, wcnt[w], rank);
    __syncthreads();
    // digit tid: the warps' offsets inside the tile, then the tiles before this one
    uint32_t run = 0;
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) {
        const uint32_t c = wcnt[ww][tid];
        wcnt[ww][tid] = run;
        run += c;
    }
    unsigned long long *mine = state + tile * kBins + tid;
    state_store(mine, (tile == 0 ? kStateAll : kStateSum) | run);
    dstart[tid] = scan256(run, wtot);
    const uint32_t digit0 = scan256(head->hist[pass][tid], wtot2);
    unsigned long long before = 0;
    bool lost = false;
    if (tile > 0) {
        int polls = 0;
        for (const unsigned long long *p = mine - kBins;;) {
            const unsigned long long v = state_load(p);
            if (v == 0) {
                if (++polls > kOrderPolls) {
                    lost = true;
                    break;
                }
                continue;
            }
            before += v & kStateMask;
            if (v >= kStateAll) break;
            p -= kBins;  // tile 0 publishes its inclusive count: the walk ends there
        }
        if (!lost) state_store(mine, kStateAll | (before + run));
    }
    if (lost) *err = 1;
    gbase[tid] = digit0 + (uint32_t)before;
    if (__syncthreads_or(lost)) return;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        if (32 * j + lane < wvalid) {
            const uint32_t d = (uint32_t)(key[j] >> shift) & (kBins - 1);
            const uint32_t at = dstart[d] + wcnt[w][d] + rank[j];
            skey[at] = key[j];
            sval[at] = val[j];
        }
    }
    __syncthreads();
    for (int i = tid; i < nvalid; i += kThreads) {
        const K k = skey[i];
        const uint32_t d = (uint32_t)(k >> shift) & (kBins - 1);
        const uint32_t at = gbase[d] + (uint32_t)i - dstart[d];
        if (at >= n) continue;  // only after an earlier pass lost a wait
        if (kout) kout[at] = k;
        vout[at] = sval[i];
    }
}

template <class K>
__global__ void __launch_bounds__(kSmallThreads) k_order_small(const K *__restrict__ keys, int n, int passes,
                                                               uint32_t *__restrict__ vout) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    K *skey = reinterpret_cast<K *>(small_smem);                       // [kSmallOrder]
    uint32_t *sval = reinterpret_cast<uint32_t *>(skey + kSmallOrder);  // [kSmallOrder]
    uint32_t *wcnt = sval + kSmallOrder;                               // [kSmallWarps][kBins]
    __shared__ uint32_t dstart[kBins], wtot[kSmallWarps];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int first = w * 32 * kSmallItems + lane, valid = min(max(n - w * 32 * kSmallItems, 0), 32 * kSmallItems);
    K key[kSmallItems];
    uint32_t val[kSmallItems], rank[kSmallItems];
#pragma unroll
    for (int j = 0; j < kSmallItems; ++j) {
        key[j] = 32 * j + lane < valid ? keys[first + 32 * j] : K(0);
        val[j] = (uint32_t)(first + 32 * j);
    }
    for (int p = 0; p < passes; ++p) {
        for (int i = tid; i < kSmallWarps * kBins; i += kSmallThreads) wcnt[i] = 0;
        __syncthreads();
        warp_rank<K, kSmallItems>(key, 8 * p, valid, wcnt + w * kBins, rank);
        __syncthreads();
        uint32_t run = 0;
        if (tid < kBins)
#pragma unroll
            for (int ww = 0; ww < kSmallWarps; ++ww) {
                const uint32_t c = wcnt[ww * kBins + tid];
                wcnt[ww * kBins + tid] = run;
                run += c;
            }
        uint32_t incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wtot[w] = incl;
        __syncthreads();
        if (tid < kBins) {
            uint32_t before = 0;
#pragma unroll
            for (int ww = 0; ww < kBins / 32; ++ww) before += ww < w ? wtot[ww] : 0u;
            dstart[tid] = before + incl - run;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSmallItems; ++j)
            if (32 * j + lane < valid) {
                const uint32_t d = (uint32_t)(key[j] >> (8 * p)) & (kBins - 1);
                const uint32_t at = dstart[d] + wcnt[w * kBins + d] + rank[j];
                skey[at] = key[j];
                sval[at] = val[j];
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSmallItems; ++j)
            if (32 * j + lane < valid) {
                key[j] = skey[first + 32 * j];
                val[j] = sval[first + 32 * j];
            }
    }
#pragma unroll
    for (int j = 0; j < kSmallItems; ++j)
        if (32 * j + lane < valid) vout[first + 32 * j] = val[j];
}

template <class K, int ITEMS>
cudaError_t order_passes(K *key, K *key_alt, uint32_t *val, uint32_t *val_alt, size_t n, int passes, SortScratch &s,
                         int num_sms, int *err, uint32_t **sorted, int *launches, cudaStream_t st) {
    const size_t tiles = (n + kThreads * ITEMS - 1) / (kThreads * ITEMS);
    const size_t bytes = sizeof(OrderHead) + (size_t)passes * tiles * kBins * sizeof(unsigned long long);
    cudaError_t e = s.hist.reserve(bytes);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(s.hist.ptr, 0, bytes, st)) != cudaSuccess) return e;
    OrderHead *head = s.hist.as<OrderHead>();
    unsigned long long *state = reinterpret_cast<unsigned long long *>(head + 1);
    const int blocks = (int)std::min<size_t>((n + kThreads * 16 - 1) / (kThreads * 16), (size_t)num_sms * 8);
    k_order_hist<K><<<blocks, kThreads, 0, st>>>(key, n, passes, head);
    const uint32_t *vin = nullptr;  // the first pass: positions
    for (int p = 0; p < passes; ++p) {
        k_order_pass<K, ITEMS><<<(unsigned)tiles, kThreads, 0, st>>>(key, vin, p + 1 < passes ? key_alt : nullptr, val, n,
                                                                    p, head, state + (size_t)p * tiles * kBins, err);
        std::swap(key, key_alt);
        vin = val;
        std::swap(val, val_alt);
    }
    *sorted = val_alt;
    *launches = passes + 1;
    return cudaGetLastError();
}

// Tiles of 2048 keys until four tiles of 4096 an SM are there (64-bit keys: always,
// shared memory).
template <class K>
cudaError_t order_impl(K *key, K *key_alt, uint32_t *val, uint32_t *val_alt, size_t n, int end_bit, SortScratch &s,
                       int num_sms, int *err, uint32_t **sorted, int *launches, cudaStream_t st) {
    *sorted = val;
    *launches = 0;
    if (n == 0) return cudaSuccess;
    const int passes = (end_bit + 7) / 8;
    if (passes > kOrderPasses || n > (size_t)INT32_MAX) return cudaErrorInvalidValue;
    if (n <= (size_t)kSmallOrder) {
        constexpr int smem = kSmallOrder * (sizeof(K) + 4) + kSmallWarps * kBins * 4;
        const cudaError_t e = allow_smem(k_order_small<K>, smem);
        if (e != cudaSuccess) return e;
        k_order_small<K><<<1, kSmallThreads, smem, st>>>(key, (int)n, passes, val);
        *launches = 1;
        return cudaGetLastError();
    }
    if (sizeof(K) == 4 && n >= (size_t)num_sms * 4 * kThreads * 16)
        return order_passes<K, sizeof(K) == 4 ? 16 : 8>(key, key_alt, val, val_alt, n, passes, s, num_sms, err, sorted,
                                                       launches, st);
    return order_passes<K, 8>(key, key_alt, val, val_alt, n, passes, s, num_sms, err, sorted, launches, st);
}

}  // namespace

cudaError_t radix_sort_u32_fixed(uint32_t **key_io, uint32_t **key_alt, uint32_t **val_io,
                                 uint32_t **val_alt, size_t n, int end_bit, void *scratch,
                                 size_t scratch_bytes, cudaStream_t st) {
    return radix_fixed<uint32_t>(key_io, key_alt, val_io, val_alt, n, end_bit, scratch,
                                 scratch_bytes, st);
}

cudaError_t radix_sort_u64_fixed(uint64_t **key_io, uint64_t **key_alt, uint32_t **val_io,
                                 uint32_t **val_alt, size_t n, int end_bit, void *scratch,
                                 size_t scratch_bytes, cudaStream_t st) {
    return radix_fixed<uint64_t>(key_io, key_alt, val_io, val_alt, n, end_bit, scratch,
                                 scratch_bytes, st);
}

size_t scan_scratch_bytes(size_t n) {
    size_t nb = (n + kScanTile - 1) / kScanTile + 1;
    return 256 + nb * sizeof(uint64_t);
}

cudaError_t radix_sort_u32(uint32_t **key_io, uint32_t **key_alt, uint32_t **val_io,
                           uint32_t **val_alt, size_t n, int end_bit, SortScratch &s,
                           cudaStream_t st) {
    return radix_impl<uint32_t>(key_io, key_alt, val_io, val_alt, n, end_bit, s, st);
}

cudaError_t sorted_order_u32(uint32_t *key, uint32_t *key_alt, uint32_t *val, uint32_t *val_alt, size_t n, int end_bit,
                             SortScratch &s, int num_sms, int *err, uint32_t **sorted, int *launches,
                             cudaStream_t st) {
    return order_impl<uint32_t>(key, key_alt, val, val_alt, n, end_bit, s, num_sms, err, sorted, launches, st);
}

cudaError_t sorted_order_u64(uint64_t *key, uint64_t *key_alt, uint32_t *val, uint32_t *val_alt, size_t n, int end_bit,
                             SortScratch &s, int num_sms, int *err, uint32_t **sorted, int *launches,
                             cudaStream_t st) {
    return order_impl<uint64_t>(key, key_alt, val, val_alt, n, end_bit, s, num_sms, err, sorted, launches, st);
}

cudaError_t exclusive_scan_u32_u64(const uint32_t *in, uint64_t *out, size_t n, void *scratch,
                                   cudaStream_t st) {
    return scan_impl<uint64_t>(in, out, n, scratch, 1, st);
}

}  // namespace ups
