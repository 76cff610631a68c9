// Which 16x16 image tiles a projected Gaussian meets (device code shared by
// the projection and the tile-list kernels: all of them must take the same
// decisions).
#pragma once

#include "common.cuh"

namespace ups {

// The alpha >= alpha_min ellipse q(d) = a dx^2 + 2 b dx dy + c dy^2 <= k2,
// k2 = 2 ln(o / alpha_min), of a projected Gaussian at (u, v), conic (a, b, c).
// Tile decisions use a margin so that FP32 rounding never drops a tile the
// blend uses: k2 grown by kMarginQ (relative) and every tile's box of pixel
// centres grown by kMarginPx on each side; the rectangle is the box of that
// grown ellipse, grown by kMarginPx.  A list may thus hold, besides the exact
// tiles, tiles whose box the exact ellipse misses by less than the margin.
constexpr float kMarginQ = 1e-4f;
constexpr float kMarginPx = 1e-3f;

struct Ellipse {
    float u, v, a, b, k2, detc, ry, dyr, ia;
};

__device__ __forceinline__ Ellipse ellipse_of(float4 xo, float4 cn, float alpha_min) {
    Ellipse e;
    e.u = xo.x;
    e.v = xo.y;
    e.a = cn.x;
    e.b = cn.y;
    // a relative margin so FP32 rounding never drops a tile the blend uses
    e.k2 = 2.f * logf(xo.w / alpha_min) * (1.f + kMarginQ);
    e.detc = cn.x * cn.z - cn.y * cn.y;
    e.ry = sqrtf(e.k2 * cn.x / e.detc);               // half-extent in y
    e.dyr = -cn.y * sqrtf(e.k2 / (cn.z * e.detc));    // dy of the point of largest x
    e.ia = 1.f / e.a;
    return e;
}

// Tile columns [c0, c1] of tile row ty (clipped to the rect's columns
// [x0, x1]; c0 > c1: none) whose box of pixel centres the ellipse meets.  The
// ellipse's slice through the row's band of pixel centres is an x interval;
// its ends are the right-most and left-most boundary points, whose dy is the
// unconstrained extreme clamped to the band (the boundary's x is concave /
// convex in dy).
__device__ __forceinline__ int2 row_cols(const Ellipse &e, int ty, int W, int H, int x0, int x1) {
    const float yb0 = (float)(ty * kTile) - kMarginPx,
                yb1 = fminf((float)(ty * kTile + kTile - 1), (float)(H - 1)) + kMarginPx;
    const float lo = fmaxf(yb0 - e.v, -e.ry), hi = fminf(yb1 - e.v, e.ry);
    if (!(lo <= hi)) return make_int2(1, 0);
    const float dr = fminf(fmaxf(e.dyr, lo), hi), dl = fminf(fmaxf(-e.dyr, lo), hi);
    const float xr = (-e.b * dr + sqrtf(fmaxf(e.a * e.k2 - e.detc * dr * dr, 0.f))) * e.ia;
    const float xl = (-e.b * dl - sqrtf(fmaxf(e.a * e.k2 - e.detc * dl * dl, 0.f))) * e.ia;
    const float xlo = fmaxf(e.u + xl - kMarginPx, 0.f), xhi = fminf(e.u + xr + kMarginPx, (float)(W - 1));
    if (!(xlo <= xhi)) return make_int2(1, 0);
    // tile tx holds pixel centres [16 tx, 16 tx + 15]: the first whose box
    // reaches xlo, the last whose box starts at or before xhi
    return make_int2(max((int)ceilf((xlo - (float)(kTile - 1)) * (1.f / kTile)), x0),
                     min((int)floorf(xhi * (1.f / kTile)), x1));
}

// ---------------------------------------------------------------------------
// row spans: the tiles a Gaussian meets, packed
// ---------------------------------------------------------------------------
//
// span (16 bytes a Gaussian-view):
//  x  first column x0 [0, 10) | first row y0 [10, 20) | rows n [20, 25) | columns
//     of its box after x0 [25, 32) (kSpanWide: that many or more)
//  y, z, w  rows 0..5, two a word, 16 bits a row: columns after x0 [0, 8), count [8, 16)
// more (32 bytes): rows 6..21; written and read only for n > 6, so that most
// Gaussian-views cost one 32-byte sector of a gather.
// n = 0: no tile.  A Gaussian of more than 22 rows, or with a row that starts
// or counts more than 255 columns, has n = kSpanTall and its tile rectangle in
// y (x0 | y0 << 16) and z (x1 | y1 << 16): its rows are evaluated again where
// they are needed.
constexpr int kSpanRows1 = 6, kSpanRows = 22;
constexpr int kSpanMore = 2;  // uint4 per Gaussian-view
constexpr uint32_t kSpanTall = 31, kSpanWide = 127;
__device__ __forceinline__ uint32_t span_rows(uint32_t head) { return (head >> 20) & 31u; }

// Columns [c0, c1] of row r of a Gaussian whose spans did not fit the packed
// form.  Not inlined: all kernels of a file run the same instructions.
static __device__ __noinline__ int2 tall_row(float4 xo, float4 cn, float alpha_min, int r, int W, int H, int x0,
                                             int x1) {
    return row_cols(ellipse_of(xo, cn, alpha_min), r, W, H, x0, x1);
}

// f(row, c0, c1) for every tile row that Gaussian-view gv (span s) meets
template <class F>
__device__ __forceinline__ void each_row(uint4 s, uint32_t gv, const uint4 *__restrict__ more,
                                         const float4 *__restrict__ xyzo, const float4 *__restrict__ conic,
                                         float alpha_min, const DevView &cam, F f) {
    const int n = (int)span_rows(s.x), x0 = (int)(s.x & 1023u), y0 = (int)((s.x >> 10) & 1023u);
    if (n == (int)kSpanTall) {
        const int xa = (int)(s.y & 0xffffu), xb = (int)(s.z & 0xffffu), yb = (int)(s.z >> 16);
        const float4 xo = xyzo[gv], cn = conic[gv];
        for (int r = (int)(s.y >> 16); r <= yb; ++r) {
            const int2 cc = tall_row(xo, cn, alpha_min, r, cam.W, cam.H, xa, xb);
            if (cc.x <= cc.y) f(r, cc.x, cc.y);
        }
        return;
    }
    const uint16_t *codes = reinterpret_cast<const uint16_t *>(more + (size_t)kSpanMore * gv);
    uint32_t w = 0u;
    for (int k = 0; k < n; ++k) {
        if (k < kSpanRows1) {
            if ((k & 1) == 0) w = k == 0 ? s.y : k == 2 ? s.z : s.w;
        } else {
            w = __ldg(codes + (k - kSpanRows1));
        }
        const int off = (int)(w & 255u), len = (int)((w >> 8) & 255u);
        w >>= 16;
        if (len) f(y0 + k, x0 + off, x0 + off + len - 1);
    }
}

// Row k of Gaussian-view gv (span head `head`): columns [c0, c1] of row r;
// c0 > c1: none.
struct RowItem {
    int r, c0, c1;
};
__device__ __forceinline__ RowItem row_item(uint32_t gv, uint32_t head, int k, const uint4 *__restrict__ span,
                                            const uint4 *__restrict__ more, const float4 *__restrict__ xyzo,
                                            const float4 *__restrict__ conic, float alpha_min, const DevView &cam) {
    RowItem t;
    t.r = (int)((head >> 10) & 1023u) + k;
    if (span_rows(head) != kSpanTall) {
        const uint16_t *code = k < kSpanRows1 ? reinterpret_cast<const uint16_t *>(span + gv) + 2 + k
                                              : reinterpret_cast<const uint16_t *>(more + (size_t)kSpanMore * gv) +
                                                    (k - kSpanRows1);
        const uint32_t c = __ldg(code);
        t.c0 = (int)(head & 1023u) + (int)(c & 255u);
        t.c1 = t.c0 + (int)(c >> 8) - 1;
    } else {
        const uint4 s = span[gv];
        const int2 cc = tall_row(xyzo[gv], conic[gv], alpha_min, t.r, cam.W, cam.H, (int)(s.y & 0xffffu),
                                 (int)(s.z & 0xffffu));
        t.c0 = cc.x;
        t.c1 = cc.y;
    }
    return t;
}

}  // namespace ups
