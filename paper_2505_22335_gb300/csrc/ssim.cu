// The D-SSIM term of the geometric loss (Eq. 4): scale (1 - SSIM(C~, C)), each
// pixel's (1 - S) weighted by an optional per-pixel weight (the mask of Eq. 14),
// SSIM (Wang et al.) per colour channel of every view with an 11 x 11
// Gaussian window (sigma 1.5, weights summing to 1), C1 = 0.01^2, C2 = 0.03^2
// (data range 1), zero padding, averaged over channels and pixels.
//
// With the window moments mu_x, mu_y, E[x^2], E[y^2], E[xy] of pixel p:
//   A1 = 2 mu_x mu_y + C1, A2 = 2 (E[xy] - mu_x mu_y) + C2,
//   B1 = mu_x^2 + mu_y^2 + C1, B2 = E[x^2] - mu_x^2 + E[y^2] - mu_y^2 + C2,
//   S = A1 A2 / (B1 B2)
// and dS_p/dx_q = w(q - p) (G_mu + 2 x_q G_xx + y_q G_xy)(p) with
//   G_mu = 2 mu_y (A2 - A1) / (B1 B2) - 2 mu_x S (1 / B1 - 1 / B2),
//   G_xx = -S / B2,  G_xy = 2 A1 / (B1 B2),
// (S / A1 and S / A2 written out, so that only B1 and B2 are divided by),
// so the backward correlates the three G maps with the (symmetric) window.
//
// Two launches (forward, backward) over all (view, channel) planes.  A CTA walks
// down a strip of 128 columns, one column a thread: each input row goes through
// shared memory once (double-buffered, the next row's loads in flight), an
// 11-tap horizontal sum per thread, and its contribution to the 11 output rows
// that are open, held in registers (the loop is unrolled by 11 rows, so the
// accumulators rotate by renaming).  Every sum runs over the taps in order, in
// packed pairs of quantities (fma.rn.f32x2 rounds each as a scalar fmaf).
// Bound by instruction issue (two thirds of it FMAs), with the 48 B of traffic
// per channel-pixel behind it.  8 x 640x480 x 3 channels: forward 0.085 and
// backward 0.070 ms, 0.16 ms together, against 0.25 ms for 32 x 16 tiles that
// went through shared memory twice with a load per FMA; seven divisions per
// pixel in place of two and strips of 64 rows (1.3 rounds of CTAs) took 0.23.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace ups {

namespace {

constexpr int kR = 5;                 // window radius
constexpr int kTaps = 2 * kR + 1;
constexpr int kCols = 128;             // columns (threads) of a strip
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

__constant__ float c_win[kTaps];  // 1-D Gaussian window, sums to 1 and is symmetric

// the (view, channel) planes of one call: blockIdx.z selects the plane
constexpr int kMaxPlanes = 3 * UPS_MAX_VIEWS;
struct Planes {
    int n;
    int W[kMaxPlanes], H[kMaxPlanes];
    size_t off[kMaxPlanes];   // offset of the plane's pixel 0 in the colour arrays
    size_t goff[kMaxPlanes];  // offset of its window-term maps in G (3 maps of W * H)
    size_t woff[kMaxPlanes];  // offset of its view's pixel 0 in the weight map
};
struct Plane {
    int W, H;
    size_t off, goff, woff;
};
__device__ __forceinline__ Plane plane_of(const Planes &t) {
    const int z = blockIdx.z;
    return Plane{t.W[z], t.H[z], t.off[z], t.goff[z], t.woff[z]};
}

__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// weight of tap k as a pair (the window is symmetric: six of them)
struct Win {
    f2 w2[kR + 1];
    float w[kR + 1];
    __device__ __forceinline__ Win() {
#pragma unroll
        for (int i = 0; i <= kR; ++i) {
            w[i] = c_win[i];
            w2[i] = f2_make(w[i], w[i]);
        }
    }
    __device__ __forceinline__ static int at(int k) { return k <= kR ? k : 2 * kR - k; }
};

// rows: output rows of a strip
__global__ void __launch_bounds__(kCols) k_ssim_fwd(const Planes pt, int rows, const float *__restrict__ x,
                                                    const float *__restrict__ y, const float *__restrict__ weight,
                                                    float *__restrict__ Gall, float g, float *__restrict__ loss) {
    __shared__ float2 ab[2][kCols + 2 * kR];
    __shared__ float red[kCols / 32];
    const Plane pl = plane_of(pt);
    const int x0 = blockIdx.x * kCols, y0 = blockIdx.y * rows;
    if (x0 >= pl.W || y0 >= pl.H) return;  // grid sized for the largest plane
    const int tid = threadIdx.x, px = x0 + tid;
    const int n_in = min(rows, pl.H - y0) + 2 * kR;  // input rows y0 - kR ..
    float *G = Gall + pl.goff;
    const size_t gstride = (size_t)pl.W * pl.H;
    // this thread's loads of an input row: columns tid and (the first 2 kR threads) kCols + tid
    const int gx0 = x0 - kR + tid, gx1 = gx0 + kCols;
    const bool in0 = gx0 >= 0 && gx0 < pl.W, in1 = tid < 2 * kR && gx1 < pl.W;
    float2 v0, v1;
    auto load = [&](int r) {
        const int gy = y0 - kR + r;
        v0 = v1 = make_float2(0.f, 0.f);
        if (r >= n_in || gy < 0 || gy >= pl.H) return;
        const size_t row = pl.off + (size_t)gy * pl.W;
        if (in0) v0 = make_float2(x[row + gx0], y[row + gx0]);
        if (in1) v1 = make_float2(x[row + gx1], y[row + gx1]);
    };
    auto store = [&](int r) {
        ab[r & 1][tid] = v0;
        if (tid < 2 * kR) ab[r & 1][kCols + tid] = v1;
    };
    const Win win;
    f2 m01[kTaps], m23[kTaps];  // open output rows: (E x, E y), (E x^2, E y^2)
    float m4[kTaps];            // E x y
    float term = 0.f;
    load(0);
    store(0);
    load(1);
    for (int r0 = 0; r0 < n_in; r0 += kTaps) {
#pragma unroll
        for (int j = 0; j < kTaps; ++j) {
            const int r = r0 + j;
            if (r >= n_in) break;  // the same for the CTA
            __syncthreads();
            store(r + 1);
            load(r + 2);
            const float2 *in = ab[r & 1] + tid;
            f2 h01 = 0ull, h23 = 0ull;
            float h4 = 0.f;
#pragma unroll
            for (int k = 0; k < kTaps; ++k) {
                const float2 p = in[k];
                const f2 q = f2_make(p.x, p.y);
                h01 = f2_fma(win.w2[Win::at(k)], q, h01);
                h23 = f2_fma(win.w2[Win::at(k)], f2_mul(q, q), h23);
                h4 = fmaf(win.w[Win::at(k)], p.x * p.y, h4);
            }
            // row r is tap k of output row r - k, which lives in slot (r - k) mod 11
#pragma unroll
            for (int k = 0; k < kTaps; ++k) {
                const int s = (j - k + kTaps) % kTaps;
                m01[s] = f2_fma(win.w2[Win::at(k)], h01, k ? m01[s] : 0ull);
                m23[s] = f2_fma(win.w2[Win::at(k)], h23, k ? m23[s] : 0ull);
                m4[s] = fmaf(win.w[Win::at(k)], h4, k ? m4[s] : 0.f);
            }
            const int o = r - 2 * kR;  // complete
            if (o < 0 || px >= pl.W) continue;
            const int s = (j + 1) % kTaps;
            float mx, my, mxx, myy;
            f2_split(m01[s], mx, my);
            f2_split(m23[s], mxx, myy);
            const float A1 = 2.f * mx * my + kC1, A2 = 2.f * (m4[s] - mx * my) + kC2;
            const float B1 = mx * mx + my * my + kC1, B2 = (mxx - mx * mx) + (myy - my * my) + kC2;
            const float i1 = 1.f / B1, i2 = 1.f / B2, i12 = i1 * i2, S = A1 * A2 * i12;
            const size_t lp = (size_t)(y0 + o) * pl.W + px;  // the G maps are per plane
            const float wp = weight ? weight[pl.woff + lp] : 1.f;
            term += wp * (1.f - S);
            G[lp] = wp * (2.f * (my * ((A2 - A1) * i12) - mx * (S * (i1 - i2))));
            G[gstride + lp] = wp * (-S * i2);
            G[2 * gstride + lp] = wp * (2.f * A1 * i12);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(0xffffffffu, term, o);
    if ((tid & 31) == 0) red[tid >> 5] = term;
    __syncthreads();
    if (tid == 0) {
        float t = 0.f;
        for (int w = 0; w < kCols / 32; ++w) t += red[w];
        atomicAdd(loss, g * t);
    }
}

// dx_q += -g (w * G_mu + 2 x_q w * G_xx + y_q w * G_xy)(q)
__global__ void __launch_bounds__(kCols) k_ssim_bwd(const Planes pt, int rows, const float *__restrict__ x,
                                                    const float *__restrict__ y, const float *__restrict__ Gall,
                                                    float g, float *__restrict__ dx) {
    __shared__ float2 g01[2][kCols + 2 * kR];  // (G_mu, G_xx)
    __shared__ float g2s[2][kCols + 2 * kR];   // G_xy
    const Plane pl = plane_of(pt);
    const int x0 = blockIdx.x * kCols, y0 = blockIdx.y * rows;
    if (x0 >= pl.W || y0 >= pl.H) return;
    const int tid = threadIdx.x, px = x0 + tid;
    const int n_in = min(rows, pl.H - y0) + 2 * kR;
    const size_t gstride = (size_t)pl.W * pl.H;
    const float *G = Gall + pl.goff;
    const int gx0 = x0 - kR + tid, gx1 = gx0 + kCols;
    const bool in0 = gx0 >= 0 && gx0 < pl.W, in1 = tid < 2 * kR && gx1 < pl.W;
    float a0, b0, c0, a1, b1, c1;
    auto load = [&](int r) {
        const int gy = y0 - kR + r;
        a0 = b0 = c0 = a1 = b1 = c1 = 0.f;
        if (r >= n_in || gy < 0 || gy >= pl.H) return;
        const float *row = G + (size_t)gy * pl.W;
        if (in0) {
            a0 = row[gx0];
            b0 = row[gstride + gx0];
            c0 = row[2 * gstride + gx0];
        }
        if (in1) {
            a1 = row[gx1];
            b1 = row[gstride + gx1];
            c1 = row[2 * gstride + gx1];
        }
    };
    auto store = [&](int r) {
        g01[r & 1][tid] = make_float2(a0, b0);
        g2s[r & 1][tid] = c0;
        if (tid < 2 * kR) {
            g01[r & 1][kCols + tid] = make_float2(a1, b1);
            g2s[r & 1][kCols + tid] = c1;
        }
    };
    const Win win;
    f2 m01[kTaps];
    float m2[kTaps];
    load(0);
    store(0);
    load(1);
    for (int r0 = 0; r0 < n_in; r0 += kTaps) {
#pragma unroll
        for (int j = 0; j < kTaps; ++j) {
            const int r = r0 + j;
            if (r >= n_in) break;
            __syncthreads();
            store(r + 1);
            load(r + 2);
            const float2 *p01 = g01[r & 1] + tid;
            const float *p2 = g2s[r & 1] + tid;
            const int o = r - 2 * kR;  // complete after this row
            const bool out = o >= 0 && px < pl.W;
            const size_t p = pl.off + (size_t)(y0 + o) * pl.W + px;
            float xv = 0.f, yv = 0.f, dv = 0.f;
            if (out) {
                xv = x[p];
                yv = y[p];
                dv = dx[p];
            }
            f2 h01 = 0ull;
            float h2 = 0.f;
#pragma unroll
            for (int k = 0; k < kTaps; ++k) {
                const float2 q = p01[k];
                h01 = f2_fma(win.w2[Win::at(k)], f2_make(q.x, q.y), h01);
                h2 = fmaf(win.w[Win::at(k)], p2[k], h2);
            }
#pragma unroll
            for (int k = 0; k < kTaps; ++k) {
                const int s = (j - k + kTaps) % kTaps;
                m01[s] = f2_fma(win.w2[Win::at(k)], h01, k ? m01[s] : 0ull);
                m2[s] = fmaf(win.w[Win::at(k)], h2, k ? m2[s] : 0.f);
            }
            if (!out) continue;
            const int s = (j + 1) % kTaps;
            float t0, t1;
            f2_split(m01[s], t0, t1);
            dx[p] = dv - g * (t0 + 2.f * xv * t1 + yv * m2[s]);
        }
    }
}

// Output rows of a strip.  A strip costs its rows plus the halo of 10, and the
// CTAs run in rounds of `slots`: the rows that make rounds times that cost
// smallest (8 x 640x480: 80 forward, 48 backward, one round each).
int strip_rows(size_t columns, int maxh, int slots) {
    int best = 8;
    size_t cost = (size_t)-1;
    for (int rows = 8; rows <= 256; rows += 8) {
        const size_t n = columns * ((maxh + rows - 1) / rows);
        const size_t c = (n + slots - 1) / slots * (rows + 2 * kR);
        if (c < cost) {
            cost = c;
            best = rows;
        }
    }
    return best;
}

// resident CTAs of kernel k on the device
template <class K>
int resident(K k, int num_sms) {
    int occ = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kCols, 0) != cudaSuccess || occ < 1) occ = 1;
    return occ * num_sms;
}

}  // namespace

cudaError_t ssim_set_window() {
    float w[2 * kR + 1], s = 0.f;
    for (int k = -kR; k <= kR; ++k) s += (w[k + kR] = std::exp(-(float)(k * k) / (2.f * 1.5f * 1.5f)));
    for (float &v : w) v /= s;
    return cudaMemcpyToSymbol(c_win, w, sizeof(w));
}

// Every colour plane of the views in one launch per direction: adds g w (1 - S)
// over all planes to *loss and, if dx, its derivative to dx (w: the per-pixel
// weight of the view's pixels, 1 when null).  G: scratch of 3 x (sum
// of the planes' pixels) floats.
cudaError_t launch_ssim(const ViewTable &vt, const float *x, const float *y, const float *weight, float *G, float g,
                        float *loss, float *dx, int num_sms, cudaStream_t st) {
    Planes pt{};
    int maxw = 0, maxh = 0;
    size_t goff = 0;
    for (int v = 0; v < vt.n; ++v)
        for (int ch = 0; ch < 3; ++ch) {
            const int i = pt.n++;
            pt.W[i] = vt.v[v].W;
            pt.H[i] = vt.v[v].H;
            const size_t HW = (size_t)pt.W[i] * pt.H[i];
            pt.off[i] = 3 * (size_t)vt.v[v].pix_off + ch * HW;
            pt.goff[i] = goff;
            pt.woff[i] = (size_t)vt.v[v].pix_off;
            goff += 3 * HW;
            maxw = std::max(maxw, pt.W[i]);
            maxh = std::max(maxh, pt.H[i]);
        }
    if (pt.n == 0) return cudaSuccess;
    const int strips = (maxw + kCols - 1) / kCols;
    const size_t columns = (size_t)strips * pt.n;
    const int rf = strip_rows(columns, maxh, resident(k_ssim_fwd, num_sms));
    k_ssim_fwd<<<dim3(strips, (maxh + rf - 1) / rf, pt.n), kCols, 0, st>>>(pt, rf, x, y, weight, G, g, loss);
    if (dx) {
        const int rb = strip_rows(columns, maxh, resident(k_ssim_bwd, num_sms));
        k_ssim_bwd<<<dim3(strips, (maxh + rb - 1) / rb, pt.n), kCols, 0, st>>>(pt, rb, x, y, G, g, dx);
    }
    return cudaGetLastError();
}

}  // namespace ups
