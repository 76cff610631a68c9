// EWA projection of 3D Gaussians (Eq. 1-2), depth keys, packed tile spans, tile-
// instance emission and tile ranges (for views too large for the row-wise lists), and the projection backward into mean, scale,
// rotation and SE(3) pose gradients.
//
// One thread per Gaussian-view; attributes are read as float4 records.
#include <algorithm>

#include "common.cuh"
#include "tiles.cuh"

namespace ups {

namespace {

struct Geo {
    float p[3];       // camera-space mean
    float W[9];       // rotation of T_cw
    float Rq[9];      // rotation of the normalised quaternion
    float qn[4], qinv;  // normalised quaternion and 1/|q|
    float s[3];
    float T[6];       // J W (2x3)
    float Sig[6];     // world covariance (xx, xy, xz, yy, yz, zz)
    float A, B, C;    // Sigma' (with dilation)
};

__device__ __forceinline__ void quat_rot(const float q[4], float R[9]) {
    float w = q[0], x = q[1], y = q[2], z = q[3];
    R[0] = 1.f - 2.f * (y * y + z * z);
    R[1] = 2.f * (x * y - w * z);
    R[2] = 2.f * (x * z + w * y);
    R[3] = 2.f * (x * y + w * z);
    R[4] = 1.f - 2.f * (x * x + z * z);
    R[5] = 2.f * (y * z - w * x);
    R[6] = 2.f * (x * z - w * y);
    R[7] = 2.f * (y * z + w * x);
    R[8] = 1.f - 2.f * (x * x + y * y);
}

// camera-space mean; returns validity (near plane, frustum guard, opacity)
__device__ __forceinline__ bool camera_point(const DevView &cam, const BlendParams &bp, float4 m,
                                             float p[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
        p[i] = fmaf(cam.R[3 * i], m.x, fmaf(cam.R[3 * i + 1], m.y, fmaf(cam.R[3 * i + 2], m.z, cam.t[i])));
    if (!(p[2] > bp.near_z)) return false;
    if (fabsf(p[0] / p[2]) > cam.limx || fabsf(p[1] / p[2]) > cam.limy) return false;
    return m.w >= bp.alpha_min;
}

// Sigma = R S S^T R^T, Sigma' = (J W) Sigma (J W)^T + dilation I
__device__ __forceinline__ void covariance(const DevView &cam, const BlendParams &bp, float4 sc,
                                           float4 q, Geo &G) {
    float qs = sqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
    G.qinv = 1.f / qs;
    G.qn[0] = q.x * G.qinv;
    G.qn[1] = q.y * G.qinv;
    G.qn[2] = q.z * G.qinv;
    G.qn[3] = q.w * G.qinv;
    quat_rot(G.qn, G.Rq);
    G.s[0] = sc.x;
    G.s[1] = sc.y;
    G.s[2] = sc.z;
    float M[9];  // R S
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) M[3 * i + j] = G.Rq[3 * i + j] * G.s[j];
    G.Sig[0] = M[0] * M[0] + M[1] * M[1] + M[2] * M[2];
    G.Sig[1] = M[0] * M[3] + M[1] * M[4] + M[2] * M[5];
    G.Sig[2] = M[0] * M[6] + M[1] * M[7] + M[2] * M[8];
    G.Sig[3] = M[3] * M[3] + M[4] * M[4] + M[5] * M[5];
    G.Sig[4] = M[3] * M[6] + M[4] * M[7] + M[5] * M[8];
    G.Sig[5] = M[6] * M[6] + M[7] * M[7] + M[8] * M[8];
#pragma unroll
    for (int i = 0; i < 9; ++i) G.W[i] = cam.R[i];
    float iz = 1.f / G.p[2];
    float j00 = cam.fx * iz, j02 = -cam.fx * G.p[0] * iz * iz;
    float j11 = cam.fy * iz, j12 = -cam.fy * G.p[1] * iz * iz;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        G.T[j] = j00 * G.W[j] + j02 * G.W[6 + j];
        G.T[3 + j] = j11 * G.W[3 + j] + j12 * G.W[6 + j];
    }
    const float *S = G.Sig;
    // rows of T times Sigma
    float t0[3], t1[3];
    t0[0] = G.T[0] * S[0] + G.T[1] * S[1] + G.T[2] * S[2];
    t0[1] = G.T[0] * S[1] + G.T[1] * S[3] + G.T[2] * S[4];
    t0[2] = G.T[0] * S[2] + G.T[1] * S[4] + G.T[2] * S[5];
    t1[0] = G.T[3] * S[0] + G.T[4] * S[1] + G.T[5] * S[2];
    t1[1] = G.T[3] * S[1] + G.T[4] * S[3] + G.T[5] * S[4];
    t1[2] = G.T[3] * S[2] + G.T[4] * S[4] + G.T[5] * S[5];
    G.A = t0[0] * G.T[0] + t0[1] * G.T[1] + t0[2] * G.T[2] + bp.dilation;
    G.B = t0[0] * G.T[3] + t0[1] * G.T[4] + t0[2] * G.T[5];
    G.C = t1[0] * G.T[3] + t1[1] * G.T[4] + t1[2] * G.T[5] + bp.dilation;
}

// One Gaussian-view per thread: projection, depth key and tile rectangle; then
// the tiles it meets, row by row.  A Gaussian meets 1 to over 20 tile rows, and
// a row costs two square roots and a division, so the rows are spread over the
// warp: lane i of a step takes the i-th (Gaussian, row) of the warp and reads
// that Gaussian's ellipse by shuffle (issue-bound: 78 % issue active; the
// per-thread loop ran with 17 of 32 lanes on and took 0.33 ms for 8M Gaussian-
// views at 640x480 and 0.44 at 1280x720 with the packed spans, this form 0.29
// and 0.34; without spans the loop took 0.24 and 0.30).  Row codes are collected in shared memory and
// packed by the owning thread (span and more may be null: counts only).
constexpr int kProjThreads = 256;

__global__ void __launch_bounds__(kProjThreads) k_project(
    ViewTable vt, BlendParams bp, int N, const float4 *__restrict__ mean_op,
    const float4 *__restrict__ scale, const float4 *__restrict__ quat, float4 *__restrict__ xyzo,
    float4 *__restrict__ conic, uint2 *__restrict__ rect, uint32_t *__restrict__ count,
    uint64_t *__restrict__ dkey, uint32_t *__restrict__ dval, uint32_t *__restrict__ dkey32, int vbits32,
    uint4 *__restrict__ span, uint4 *__restrict__ more, unsigned long long *__restrict__ n_inst) {
    __shared__ uint16_t s_code[kSpanRows][kProjThreads];  // columns after x0 | count << 8
    __shared__ uint32_t s_cnt[kProjThreads];              // tiles met in rows that have no code
    __shared__ uint8_t s_own[kProjThreads];               // a warp's lanes that have rows, in order
    __shared__ uint32_t s_wide[kProjThreads / 32];        // lanes with a row that does not fit a code
    __shared__ uint32_t wsum[kProjThreads / 32];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int v = blockIdx.y, gi = blockIdx.x * kProjThreads + tid, gv = v * N + gi;
    const bool in = gi < N;
    const DevView &cam = vt.v[v];
    uint2 rc = make_uint2(0u, 0u);
    float4 xo = make_float4(0.f, 0.f, 0.f, 0.f), cn = xo;
    Ellipse e{};
    int nrow = 0;
    float z = 0.f;
    if (in) {
        int gs = cam.set * N + gi;
        float4 m = mean_op[gs];
        Geo G;
        bool ok = camera_point(cam, bp, m, G.p);
        z = G.p[2];
        xo = make_float4(0.f, 0.f, G.p[2], m.w);
        if (ok) {
            covariance(cam, bp, scale[gs], quat[gs], G);
            float det = G.A * G.C - G.B * G.B;
            float idet = 1.f / det;
            cn = make_float4(G.C * idet, -G.B * idet, G.A * idet, 0.f);
            float iz = 1.f / G.p[2];
            float u = fmaf(cam.fx * G.p[0], iz, cam.cx);
            float vv = fmaf(cam.fy * G.p[1], iz, cam.cy);
            xo.x = u;
            xo.y = vv;
            // bounding box of the ellipse o exp(-q/2) >= alpha_min, with the
            // margin of the tile decisions
            float k2 = 2.f * logf(m.w / bp.alpha_min) * (1.f + kMarginQ);
            float rx = sqrtf(k2 * G.A) + kMarginPx, ry = sqrtf(k2 * G.C) + kMarginPx;
            float xlo = fmaxf(u - rx, 0.f), xhi = fminf(u + rx, (float)(cam.W - 1));
            float ylo = fmaxf(vv - ry, 0.f), yhi = fminf(vv + ry, (float)(cam.H - 1));
            if (xlo <= xhi && ylo <= yhi) {
                int x0 = (int)floorf(xlo * (1.f / kTile)), x1 = (int)floorf(xhi * (1.f / kTile));
                int y0 = (int)floorf(ylo * (1.f / kTile)), y1 = (int)floorf(yhi * (1.f / kTile));
                e = ellipse_of(xo, cn, bp.alpha_min);
                rc = make_uint2((uint32_t)x0 | ((uint32_t)y0 << 16), (uint32_t)x1 | ((uint32_t)y1 << 16));
                nrow = y1 - y0 + 1;
            }
        }
        xyzo[gv] = xo;
        conic[gv] = cn;
        rect[gv] = rc;
    }
    s_cnt[tid] = 0u;
    if (lane == 0) s_wide[wid] = 0u;
    int incl = nrow;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += y;
    }
    const int rows = __shfl_sync(full, incl, 31), first = incl - nrow;
    const uint32_t some = __ballot_sync(full, nrow > 0);
    if (nrow > 0) s_own[(wid << 5) + __popc(some & ((1u << lane) - 1u))] = (uint8_t)lane;
    __syncwarp();
    int before = 0;  // owners whose rows start before the step
    for (int b = 0; b < rows; b += 32) {
        const int i = b + lane;
        // the owner of row i: the last whose rows start at or before it
        const uint32_t starts =
            __reduce_or_sync(full, nrow > 0 && first >= b && first < b + 32 ? 1u << (first - b) : 0u);
        const int L = s_own[(wid << 5) + before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1];
        before += __popc(starts);
        Ellipse t;
        t.u = __shfl_sync(full, e.u, L);
        t.v = __shfl_sync(full, e.v, L);
        t.a = __shfl_sync(full, e.a, L);
        t.b = __shfl_sync(full, e.b, L);
        t.k2 = __shfl_sync(full, e.k2, L);
        t.detc = __shfl_sync(full, e.detc, L);
        t.ry = __shfl_sync(full, e.ry, L);
        t.dyr = __shfl_sync(full, e.dyr, L);
        t.ia = __shfl_sync(full, e.ia, L);
        const uint32_t r0 = __shfl_sync(full, rc.x, L), r1 = __shfl_sync(full, rc.y, L);
        const int k = i - __shfl_sync(full, first, L);
        if (i < rows) {
            const int x0 = r0 & 0xffff, x1 = r1 & 0xffff;
            const int2 cc = row_cols(t, (int)(r0 >> 16) + k, cam.W, cam.H, x0, x1);
            const int off = cc.x - x0, len = cc.x <= cc.y ? cc.y - cc.x + 1 : 0;
            const bool coded = k < kSpanRows && off <= 255 && len <= 255;
            if (k < kSpanRows) s_code[k][(wid << 5) + L] = coded && len ? (uint16_t)(off | (len << 8)) : (uint16_t)0;
            if (len && !coded) {
                atomicAdd(&s_cnt[(wid << 5) + L], (uint32_t)len);
                if (k < kSpanRows) atomicOr(&s_wide[wid], 1u << L);
            }
        }
    }
    __syncwarp();
    uint32_t cnt = s_cnt[tid];
    uint32_t pair[kSpanRows / 2];  // two rows a word
#pragma unroll
    for (int k = 0; k < kSpanRows; k += 2) {
        pair[k / 2] = 0u;
        if (k >= nrow) continue;
        const uint32_t lo = s_code[k][tid], hi = k + 1 < nrow ? s_code[k + 1][tid] : 0u;
        pair[k / 2] = lo | (hi << 16);
        cnt += (lo >> 8) + (hi >> 8);
    }
    if (in) {
        count[gv] = cnt;
        if (span) {
            const uint32_t head = (rc.x & 1023u) | ((rc.x >> 16 & 1023u) << 10) |
                                  (min((rc.y & 0xffffu) - (rc.x & 0xffffu), kSpanWide) << 25);
            uint4 s = make_uint4(0u, 0u, 0u, 0u);
            if (cnt && (nrow > kSpanRows || (s_wide[wid] >> lane & 1u))) {
                s = make_uint4(head | (kSpanTall << 20), rc.x, rc.y, 0u);
            } else if (cnt) {
                s = make_uint4(head | ((uint32_t)nrow << 20), pair[0], pair[1], pair[2]);
                uint4 *m = more + (size_t)kSpanMore * gv;
                if (nrow > kSpanRows1) m[0] = make_uint4(pair[3], pair[4], pair[5], pair[6]);
                if (nrow > kSpanRows1 + 8) m[1] = make_uint4(pair[7], pair[8], pair[9], pair[10]);
            }
            span[gv] = s;
        }
        if (vbits32 < 0) {
            uint32_t zb = cnt ? __float_as_uint(z) : 0xffffffffu;
            dkey[gv] = ((uint64_t)v << 32) | zb;
        } else {
            // 32-bit key: view in the top vbits32 bits, float bits of z above
            // 0.125 m below (exact while z < 2^(32 - vbits32) ulps above 0.125 m;
            // larger depths saturate and fall back to id order)
            const uint32_t zmask = vbits32 == 0 ? 0xffffffffu : (0xffffffffu >> vbits32);
            uint32_t zf = zmask;
            if (cnt) zf = min(__float_as_uint(z) - 0x3e000000u, zmask);
            dkey32[gv] = (vbits32 == 0 ? 0u : ((uint32_t)v << (32 - vbits32))) | zf;
        }
        if (dval) dval[gv] = (uint32_t)gv;
    }
    if (!n_inst) return;
    // tile instances for the host's total: one atomic a block, spread over
    // kInstCounters addresses so that 31,250 blocks (8M Gaussian-views) do not
    // queue up at one
    const uint32_t ws = __reduce_add_sync(full, cnt);
    if (lane == 0) wsum[wid] = ws;
    __syncthreads();
    if (tid == 0) {
        unsigned long long s = 0;
        for (int w = 0; w < kProjThreads / 32; ++w) s += wsum[w];
        if (s) atomicAdd(n_inst + (blockIdx.x + blockIdx.y) % kInstCounters, s);
    }
}

__global__ void k_gather_counts(const uint32_t *__restrict__ sorted_gv,
                                const uint32_t *__restrict__ count, uint32_t *__restrict__ out,
                                int total) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < total) out[s] = count[min(sorted_gv[s], (uint32_t)total - 1u)];
}

// Instances of 32 consecutive depth-ordered Gaussian-views are written by one
// warp: the warp walks its contiguous instance range 32 at a time, each lane
// finds its source Gaussian by a binary search over the lanes' start offsets,
// so stores are coalesced whatever the per-Gaussian tile counts are.  Each
// owner lane first tabulates its Gaussian's met columns per tile row (first
// column and running instance count) in shared memory, up to kEmitRows rows;
// taller Gaussians (rare) recompute the rows per instance.  The buffers hold the
// n_inst instances that the projection counted; an order that a lost wait left with
// repeated ids adds up to more or fewer.
constexpr int kEmitRows = 8;

__global__ void __launch_bounds__(256) k_emit(ViewTable vt, BlendParams bp, int N, int total,
                                              const uint32_t *__restrict__ sorted_gv,
                                              const uint64_t *__restrict__ off,
                                              const uint2 *__restrict__ rect,
                                              const float4 *__restrict__ xyzo,
                                              const float4 *__restrict__ conic,
                                              uint32_t *__restrict__ ikey,
                                              uint32_t *__restrict__ ival, uint32_t n_inst) {
    __shared__ uint32_t s_rows[256 / 32][32][kEmitRows];  // first column | (instances before the row << 16)
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int s0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32;
    if (s0 >= total) return;  // warp-uniform
    const int s = s0 + lane;
    const bool in = s < total;
    const uint64_t o = off[in ? s : total];
    const uint64_t o_end = off[min(s0 + 32, total)];
    const uint64_t o_beg = __shfl_sync(full, o, 0);
    uint32_t gv = in ? min(sorted_gv[s], (uint32_t)total - 1u) : 0u;
    uint2 rc = make_uint2(0u, 0u);
    float4 xo = make_float4(0.f, 0.f, 0.f, 1.f), cn = make_float4(1.f, 0.f, 1.f, 0.f);
    const bool mine = in && off[s + 1] > o;
    if (mine) {
        rc = rect[gv];
        xo = xyzo[gv];
        cn = conic[gv];
        const int v = (int)(gv / (uint32_t)N);
        const DevView &cam = vt.v[v];
        const int x0 = rc.x & 0xffff, y0 = rc.x >> 16, x1 = rc.y & 0xffff, y1 = rc.y >> 16;
        if (y1 - y0 < kEmitRows) {
            const Ellipse e = ellipse_of(xo, cn, bp.alpha_min);
            uint32_t before = 0;
            for (int r = y0; r <= y1; ++r) {
                const int2 cc = row_cols(e, r, cam.W, cam.H, x0, x1);
                s_rows[wid][lane][r - y0] = (uint32_t)max(cc.x, 0) | (before << 16);
                if (cc.x <= cc.y) before += (uint32_t)(cc.y - cc.x + 1);
            }
        }
    }
    __syncwarp();
    for (uint64_t b = o_beg; b < o_end; b += 32) {
        const uint64_t i = b + lane;
        int L = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
            uint64_t oc = __shfl_sync(full, o, L + step);
            if (oc <= i) L += step;
        }
        const uint32_t g = __shfl_sync(full, gv, L);
        const uint32_t r0 = __shfl_sync(full, rc.x, L);
        const uint32_t r1 = __shfl_sync(full, rc.y, L);
        const uint64_t oL = __shfl_sync(full, o, L);
        if (i < o_end && i < n_inst) {
            const int v = (int)(g / (uint32_t)N);
            const DevView &cam = vt.v[v];
            const int x0 = r0 & 0xffff, y0 = r0 >> 16, x1 = r1 & 0xffff, y1 = r1 >> 16;
            const int j = (int)(i - oL);
            int tx = x0, ty = y0;
            if (y1 - y0 < kEmitRows) {
                // last tabulated row whose running count is <= j
                int r = 0;
                for (int k = 1; k <= y1 - y0; ++k)
                    if ((int)(s_rows[wid][L][k] >> 16) <= j) r = k;
                const uint32_t e = s_rows[wid][L][r];
                tx = (int)(e & 0xffff) + j - (int)(e >> 16);
                ty = y0 + r;
            } else {
                const Ellipse e = ellipse_of(xyzo[g], conic[g], bp.alpha_min);
                int jj = j;
                for (int r = y0; r <= y1; ++r) {
                    const int2 cc = row_cols(e, r, cam.W, cam.H, x0, x1);
                    const int n = cc.x <= cc.y ? cc.y - cc.x + 1 : 0;
                    if (jj < n) {
                        tx = cc.x + jj;
                        ty = r;
                        break;
                    }
                    jj -= n;
                }
            }
            ikey[i] = (uint32_t)(cam.tile_base + ty * cam.tiles_x + tx);
            ival[i] = g;
        }
    }
    // fewer instances than the buffers were sized for: no tile's
    if (s0 + 32 >= total)
        for (uint64_t i = o_end + lane; i < n_inst; i += 32) {
            ikey[i] = 0xffffffffu;
            ival[i] = 0u;
        }
}

__global__ void k_ranges(const uint32_t *__restrict__ ikey, uint32_t n, uint32_t tiles, uint2 *__restrict__ ranges) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k = ikey[i];
    if (k >= tiles) return;
    if (i == 0 || ikey[i - 1] != k) ranges[k].x = i;
    if (i == n - 1 || ikey[i + 1] != k) ranges[k].y = i + 1;
}

// ---------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------

// The blend backward sets a bit for every Gaussian-view it stages; only those
// have a gradient record that can differ from zero.  At 1M Gaussians and 8 x
// 640x480 it stages 1.7M list entries of 0.18M Gaussian-views, 2 % of the 8M (8 x
// 1280x720: 3.3M entries, 0.13M, 1.6 %), so the projection backward is a zero fill of the gradients, bound by its
// writes (128 B a Gaussian-view at 16 channels), and this kernel over the list
// of set bits (k_list_hits), one Gaussian-view a thread of a grid-stride loop:
// 0.19 ms and 0.01 to clear the records.  A thread per Gaussian-view reading
// every record took 0.47 ms after a 0.14 ms memset of the records; skipping
// those without a flag 0.31 ms (nearly every warp had a lane to evaluate), as
// did CTAs that list the bits of their own words (too few lanes busy); a list
// appended by the blend kernel cost that kernel 0.03 ms of atomic latency.
constexpr int kBwdThreads = 256;

// hits.list = the set bits' Gaussian-views (in order inside a CTA's words);
// *hits.count was zero
__global__ void __launch_bounds__(256) k_list_hits(HitList hits, size_t n_words) {
    __shared__ uint32_t wsum[8];
    __shared__ uint32_t s_at;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t w = (size_t)blockIdx.x * 256 + threadIdx.x;
    uint32_t b = w < n_words ? hits.bits[w] : 0u;
    uint32_t incl = __popc(b);
    const uint32_t c = incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        before += i < wid ? wsum[i] : 0u;
        all += wsum[i];
    }
    if (all == 0) return;
    if (threadIdx.x == 0) s_at = atomicAdd(hits.count, all);
    __syncthreads();
    for (uint32_t at = s_at + before + incl - c; b; b &= b - 1) hits.list[at++] = (uint32_t)(32 * w) + __ffs(b) - 1;
}

__global__ void __launch_bounds__(kBwdThreads) k_project_bwd(
    ViewTable vt, BlendParams bp, int N, int direct, int n_feat, unsigned mask,
    float scale_grad, const float4 *__restrict__ mean_op, const float4 *__restrict__ scale,
    const float4 *__restrict__ quat, const float *__restrict__ g2, HitList hits,
    float4 *__restrict__ d_mean_op, float4 *__restrict__ d_scale, float4 *__restrict__ d_quat,
    float4 *__restrict__ d_color, float *__restrict__ d_feat, float *__restrict__ d_pose) {
    const unsigned full = 0xffffffffu;
    __shared__ float s_pose[UPS_MAX_VIEWS][6];
    for (int i = threadIdx.x; i < 6 * vt.n; i += kBwdThreads) (&s_pose[0][0])[i] = 0.f;
    __syncthreads();
    const int stride = g2_stride(n_feat), lane = threadIdx.x & 31;
    const size_t n_hits = *hits.count;
    for (size_t i0 = (size_t)blockIdx.x * kBwdThreads + threadIdx.x - lane; i0 < n_hits;
         i0 += (size_t)gridDim.x * kBwdThreads) {
        const bool in = i0 + lane < n_hits;
        const size_t gv = in ? hits.list[i0 + lane] : 0u;
        const int v = (int)(gv / (unsigned)N);
        const DevView &cam = vt.v[v];
        // direct: every set is read by one view, so its gradient is written, not
        // accumulated (else the caller zeroed the gradient and views add into it)
        const size_t gs = (size_t)cam.set * N + (gv - (size_t)v * N);
        const float *r = g2 + gv * stride;
        float pose[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        float dmu[3] = {0.f, 0.f, 0.f}, ds[3] = {0.f, 0.f, 0.f}, dq[4] = {0.f, 0.f, 0.f, 0.f};
        float dop = 0.f;
        bool ok = false;
        Geo G;
        if (in) ok = camera_point(cam, bp, mean_op[gs], G.p);
        if (ok) {
            covariance(cam, bp, scale[gs], quat[gs], G);
            float4 ra = *reinterpret_cast<const float4 *>(r);
            float4 rb = *reinterpret_cast<const float4 *>(r + 4);
            float gu = ra.x, gvv = ra.y, gz = ra.z;
            dop = ra.w;
            float ga = rb.x, gb = rb.y, gc = rb.z;
            float A = G.A, B = G.B, Cc = G.C;
            float D = A * Cc - B * B;
            float iD2 = 1.f / (D * D);
            float gA = (-Cc * Cc * ga + B * Cc * gb - B * B * gc) * iD2;
            float gB = (2.f * B * Cc * ga - (A * Cc + B * B) * gb + 2.f * A * B * gc) * iD2;
            float gC = (-B * B * ga + B * A * gb - A * A * gc) * iD2;
            // G2 = [[gA, gB/2], [gB/2, gC]]; Sigma' = T Sigma T^T
            float h = 0.5f * gB;
            const float *T = G.T;
            const float *S = G.Sig;
            // G2 T (2x3)
            float gt0[3], gt1[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                gt0[j] = gA * T[j] + h * T[3 + j];
                gt1[j] = h * T[j] + gC * T[3 + j];
            }
            // dL/dSigma = T^T G2 T (symmetric 3x3, full)
            float GS[9];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) GS[3 * i + j] = T[i] * gt0[j] + T[3 + i] * gt1[j];
            // dL/dT = 2 G2 T Sigma
            float Sf[9] = {S[0], S[1], S[2], S[1], S[3], S[4], S[2], S[4], S[5]};
            float GT[6];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                GT[j] = 2.f * (gt0[0] * Sf[j] + gt0[1] * Sf[3 + j] + gt0[2] * Sf[6 + j]);
                GT[3 + j] = 2.f * (gt1[0] * Sf[j] + gt1[1] * Sf[3 + j] + gt1[2] * Sf[6 + j]);
            }
            // T = J W: dL/dJ = GT W^T, dL/dW(cov) = J^T GT
            const float *W = G.W;
            float GJ[6];
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    GJ[3 * a + j] = GT[3 * a] * W[3 * j] + GT[3 * a + 1] * W[3 * j + 1] +
                                    GT[3 * a + 2] * W[3 * j + 2];
            float iz = 1.f / G.p[2], iz2 = iz * iz, iz3 = iz2 * iz;
            float fx = cam.fx, fy = cam.fy;
            float gp[3];
            gp[0] = GJ[2] * (-fx * iz2) + gu * fx * iz;
            gp[1] = GJ[5] * (-fy * iz2) + gvv * fy * iz;
            gp[2] = GJ[0] * (-fx * iz2) + GJ[2] * (2.f * fx * G.p[0] * iz3) + GJ[4] * (-fy * iz2) +
                    GJ[5] * (2.f * fy * G.p[1] * iz3) - gu * fx * G.p[0] * iz2 -
                    gvv * fy * G.p[1] * iz2 + gz;
#pragma unroll
            for (int i = 0; i < 3; ++i) dmu[i] = W[i] * gp[0] + W[3 + i] * gp[1] + W[6 + i] * gp[2];
            if (mask & UPS_GRAD_POSE) {
                // dW(cov) = J^T GT; J = [[j00 0 j02][0 j11 j12]]
                float j00 = fx * iz, j02 = -fx * G.p[0] * iz2, j11 = fy * iz, j12 = -fy * G.p[1] * iz2;
                float GW[9];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    GW[j] = j00 * GT[j];
                    GW[3 + j] = j11 * GT[3 + j];
                    GW[6 + j] = j02 * GT[j] + j12 * GT[3 + j];
                }
                // A = W GW^T; d phi += vee(A)
                float Am[9];
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        Am[3 * i + j] = W[3 * i] * GW[3 * j] + W[3 * i + 1] * GW[3 * j + 1] +
                                        W[3 * i + 2] * GW[3 * j + 2];
                const float *p = G.p;
                pose[0] = gp[0];
                pose[1] = gp[1];
                pose[2] = gp[2];
                pose[3] = p[1] * gp[2] - p[2] * gp[1] + Am[5] - Am[7];
                pose[4] = p[2] * gp[0] - p[0] * gp[2] + Am[6] - Am[2];
                pose[5] = p[0] * gp[1] - p[1] * gp[0] + Am[1] - Am[3];
            }
            if (mask & UPS_GRAD_GAUSS) {
                // Sigma = (R S)(R S)^T: dL/d(RS) = 2 GS (R S)
                float GR[9];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    float acc = 0.f;
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        float grs = 2.f * (GS[3 * i] * G.Rq[j] * G.s[j] + GS[3 * i + 1] * G.Rq[3 + j] * G.s[j] +
                                           GS[3 * i + 2] * G.Rq[6 + j] * G.s[j]);
                        GR[3 * i + j] = grs * G.s[j];
                        acc += grs * G.Rq[3 * i + j];
                    }
                    ds[j] = acc;
                }
                float w = G.qn[0], x = G.qn[1], y = G.qn[2], z = G.qn[3];
                float dqn[4];
                dqn[0] = 2.f * (-z * GR[1] + y * GR[2] + z * GR[3] - x * GR[5] - y * GR[6] + x * GR[7]);
                dqn[1] = 2.f * (y * GR[1] + z * GR[2] + y * GR[3] - 2.f * x * GR[4] - w * GR[5] +
                                z * GR[6] + w * GR[7] - 2.f * x * GR[8]);
                dqn[2] = 2.f * (-2.f * y * GR[0] + x * GR[1] + w * GR[2] + x * GR[3] + z * GR[5] -
                                w * GR[6] + z * GR[7] - 2.f * y * GR[8]);
                dqn[3] = 2.f * (-2.f * z * GR[0] - w * GR[1] + x * GR[2] + w * GR[3] - 2.f * z * GR[4] +
                                y * GR[5] + x * GR[6] + y * GR[7]);
                float dot = w * dqn[0] + x * dqn[1] + y * dqn[2] + z * dqn[3];
#pragma unroll
                for (int i = 0; i < 4; ++i) dq[i] = (dqn[i] - G.qn[i] * dot) * G.qinv;
            }
        }
        if (in && (mask & UPS_GRAD_GAUSS)) {
            const float4 rc = *reinterpret_cast<const float4 *>(r + 8);  // dr dg db -
            if (direct) {
                // over the zero fill, which holds the mean-scale term of the scales
                d_mean_op[gs] = make_float4(dmu[0], dmu[1], dmu[2], dop);
                d_scale[gs] = make_float4(ds[0] + scale_grad, ds[1] + scale_grad, ds[2] + scale_grad, 0.f);
                d_quat[gs] = make_float4(dq[0], dq[1], dq[2], dq[3]);
                d_color[gs] = make_float4(rc.x, rc.y, rc.z, 0.f);
                // feature gradients as 16-byte moves (n_feat is a multiple of 4; the
                // record's feature part starts 48 bytes into a 16-byte aligned record)
                const float4 *rf = reinterpret_cast<const float4 *>(r + kG2Base);
                float4 *df = reinterpret_cast<float4 *>(d_feat + gs * n_feat);
                for (int c = 0; c < n_feat / 4; ++c) df[c] = rf[c];
            } else if (ok) {
                atomicAdd(d_mean_op + gs, make_float4(dmu[0], dmu[1], dmu[2], dop));
                atomicAdd(d_scale + gs, make_float4(ds[0], ds[1], ds[2], 0.f));
                atomicAdd(d_quat + gs, make_float4(dq[0], dq[1], dq[2], dq[3]));
                atomicAdd(d_color + gs, make_float4(rc.x, rc.y, rc.z, 0.f));
                for (int c = 0; c < n_feat; c += 4)
                    atomicAdd(reinterpret_cast<float4 *>(d_feat + gs * n_feat + c),
                              *reinterpret_cast<const float4 *>(r + kG2Base + c));
            }
        }
        if (!(mask & UPS_GRAD_POSE)) continue;
        // pose: a warp's Gaussian-views are mostly of one view
        const int v0 = __shfl_sync(full, v, 0);
        const bool same = __all_sync(full, !in || v == v0);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            float p = ok ? pose[i] : 0.f;
            if (same) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(full, p, o);
                if (lane == 0) atomicAdd(&s_pose[v0][i], p);
            } else if (ok) {
                atomicAdd(&s_pose[v][i], p);
            }
        }
    }
    if (!(mask & UPS_GRAD_POSE)) return;
    __syncthreads();
    for (int i = threadIdx.x; i < 6 * vt.n; i += kBwdThreads) {
        const float p = (&s_pose[0][0])[i];
        if (p != 0.f) atomicAdd(d_pose + i, p);
    }
}

// Zero gradients of the sets the views read, scale_grad in the scales (the
// mean-scale term).  256 Gaussians a block, a view per grid row.
__global__ void __launch_bounds__(256) k_zero_grads(ViewTable vt, int N, int n_feat, float scale_grad,
                                                    float4 *__restrict__ d_mean_op, float4 *__restrict__ d_scale,
                                                    float4 *__restrict__ d_quat, float4 *__restrict__ d_color,
                                                    float *__restrict__ d_feat) {
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const int g0 = blockIdx.x * 256, g = g0 + threadIdx.x;
    const size_t base = (size_t)vt.v[blockIdx.y].set * N;
    if (g < N) {
        d_mean_op[base + g] = z;
        d_scale[base + g] = make_float4(scale_grad, scale_grad, scale_grad, 0.f);
        d_quat[base + g] = z;
        d_color[base + g] = z;
    }
    float4 *f = reinterpret_cast<float4 *>(d_feat + (base + g0) * n_feat);
    const int n = min(256, N - g0) * (n_feat / 4);
    for (int i = threadIdx.x; i < n; i += 256) f[i] = z;
}

// dL/ds += scale_grad for every scale of n Gaussians (the sets that several
// views read, whose gradients are accumulated)
__global__ void __launch_bounds__(256) k_fill_scales(size_t n, float scale_grad, float4 *__restrict__ d_scale) {
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256)
        d_scale[i] = make_float4(scale_grad, scale_grad, scale_grad, 0.f);
}

// Zeroes the records and bits of the listed Gaussian-views, a few percent of the
// records, instead of a memset of all (0.9 GB at 8M Gaussian-views).
__global__ void __launch_bounds__(256) k_clear_hits(HitList hits, float *__restrict__ g2, int stride) {
    const int q = stride / 4;  // a thread 16 bytes
    const size_t n = (size_t)*hits.count * q;
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
        const size_t h = i / q;
        const int c = (int)(i - h * q);
        const uint32_t gv = hits.list[h];
        if (c == 0) hits.bits[gv >> 5] = 0u;  // every set bit of the word is listed
        reinterpret_cast<float4 *>(g2 + (size_t)gv * stride)[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// CTAs of the grid-stride kernels over a hit list of up to n
int hit_blocks(size_t n, int num_sms) { return (int)std::min<size_t>((n + 255) / 256, (size_t)num_sms * 4); }

}  // namespace

cudaError_t launch_project(const ViewTable &vt, const BlendParams &bp, int N, int total, const ups_gaussians &g,
                           float4 *xyzo, float4 *conic, uint2 *rect, uint32_t *count, uint64_t *dkey, uint32_t *dval,
                           uint4 *span, uint4 *more, unsigned long long *n_inst, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    k_project<<<dim3((N + kProjThreads - 1) / kProjThreads, vt.n), kProjThreads, 0, st>>>(
        vt, bp, N, reinterpret_cast<const float4 *>(g.mean_opacity),
        reinterpret_cast<const float4 *>(g.scale), reinterpret_cast<const float4 *>(g.quat), xyzo,
        conic, rect, count, dkey, dval, nullptr, -1, span, more, n_inst);
    return cudaGetLastError();
}

// Projection writing 32-bit (view, depth) keys (vbits = bits of the view index).
cudaError_t launch_project_k32(const ViewTable &vt, const BlendParams &bp, int N, int total, const ups_gaussians &g,
                               float4 *xyzo, float4 *conic, uint2 *rect, uint32_t *count, uint32_t *dkey32,
                               int vbits, uint4 *span, uint4 *more, unsigned long long *n_inst, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    k_project<<<dim3((N + kProjThreads - 1) / kProjThreads, vt.n), kProjThreads, 0, st>>>(
        vt, bp, N, reinterpret_cast<const float4 *>(g.mean_opacity),
        reinterpret_cast<const float4 *>(g.scale), reinterpret_cast<const float4 *>(g.quat), xyzo,
        conic, rect, count, nullptr, nullptr, dkey32, vbits, span, more, n_inst);
    return cudaGetLastError();
}

cudaError_t launch_gather_counts(const uint32_t *sorted_gv, const uint32_t *count, uint32_t *out,
                                 int total, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    k_gather_counts<<<(total + 255) / 256, 256, 0, st>>>(sorted_gv, count, out, total);
    return cudaGetLastError();
}

cudaError_t launch_emit(const ViewTable &vt, const BlendParams &bp, int N, int total, const uint32_t *sorted_gv,
                        const uint64_t *off, const uint2 *rect, const float4 *xyzo, const float4 *conic,
                        uint32_t *ikey, uint32_t *ival, uint32_t n_inst, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    k_emit<<<(total + 255) / 256, 256, 0, st>>>(vt, bp, N, total, sorted_gv, off, rect, xyzo, conic, ikey, ival, n_inst);
    return cudaGetLastError();
}

cudaError_t launch_ranges(const uint32_t *ikey, uint32_t n, uint32_t tiles, uint2 *ranges, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    k_ranges<<<(n + 255) / 256, 256, 0, st>>>(ikey, n, tiles, ranges);
    return cudaGetLastError();
}

cudaError_t launch_list_hits(const HitList &hits, size_t n_gv, cudaStream_t st) {
    const size_t n_words = (n_gv + 31) / 32;
    if (n_words == 0) return cudaSuccess;
    k_list_hits<<<(unsigned)((n_words + 255) / 256), 256, 0, st>>>(hits, n_words);
    return cudaGetLastError();
}

cudaError_t launch_clear_hits(const HitList &hits, size_t n_gv, float *g2, int n_feat, int num_sms, cudaStream_t st) {
    if (n_gv == 0) return cudaSuccess;
    k_clear_hits<<<hit_blocks(n_gv, num_sms), 256, 0, st>>>(hits, g2, g2_stride(n_feat));
    return cudaGetLastError();
}

cudaError_t launch_project_bwd(const ViewTable &vt, const BlendParams &bp, int N, int n_sets, int direct, int n_feat,
                               unsigned mask, float scale_grad, const ups_gaussians &g, const float *g2,
                               const HitList &hits, const ups_gaussians *grad, float *d_pose, int num_sms,
                               cudaStream_t st) {
    if (N == 0) return cudaSuccess;
    float4 *dm = nullptr, *ds = nullptr, *dq = nullptr, *dc = nullptr;
    float *df = nullptr;
    if (grad && (mask & UPS_GRAD_GAUSS)) {
        dm = reinterpret_cast<float4 *>(grad->mean_opacity);
        ds = reinterpret_cast<float4 *>(grad->scale);
        dq = reinterpret_cast<float4 *>(grad->quat);
        dc = reinterpret_cast<float4 *>(grad->color);
        df = grad->feat;
        if (direct)
            k_zero_grads<<<dim3((N + 255) / 256, vt.n), 256, 0, st>>>(vt, N, n_feat, scale_grad, dm, ds, dq, dc, df);
        else if (scale_grad != 0.f)
            k_fill_scales<<<num_sms * 4, 256, 0, st>>>((size_t)N * n_sets, scale_grad, ds);
    }
    k_project_bwd<<<hit_blocks((size_t)N * vt.n, num_sms), kBwdThreads, 0, st>>>(
        vt, bp, N, direct, n_feat, mask, scale_grad, reinterpret_cast<const float4 *>(g.mean_opacity),
        reinterpret_cast<const float4 *>(g.scale), reinterpret_cast<const float4 *>(g.quat), g2, hits, dm, ds, dq, dc, df,
        d_pose);
    return cudaGetLastError();
}

}  // namespace ups
