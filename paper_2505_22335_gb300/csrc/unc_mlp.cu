// Uncertainty MLP F_u and its loss L_u (Sec. 3.3 "Uncertainty Prediction for
// Mapping", Eq. 5, Eq. 13; App. "MLP Implementation Details"):
//   sigma_p = SoftPlus(w2 . ReLU(W1 F_p + b1) + b2)   (1x1 conv -> ReLU -> 1x1
//   conv -> SoftPlus, hidden 128, one output), F_p the DINO feature of pixel
//   p bilinearly upsampled from the patch grid, and
//   L_u = (1 / P) sum_p [R_p / (2 sigma_p^2) + lambda log sigma_p]   (Eq. 5),
// with the gradient flowing only into F_u's parameters (the mapping and
// uncertainty gradient flows are kept apart, Sec. 3.3).
//
// The first layer is linear, so W1 F_p = sum_c a_c(p) (W1 g_c) over the
// pixel's four patch corners g_c with bilinear weights a_c(p): it runs once
// per patch (Zp = G W1^T, a small GEMM in plain FP32), and every pixel interpolates
// 128 values instead of 384.  Backward, dW1 = sum_p dh_p F_p^T = D^T G with
// D_patch = sum over (pixel, corner) pairs landing on the patch of a_c(p)
// dh_p, so the second small GEMM runs on patches too.  All views' patches go
// through one product each way and all views' cells through one launch.
//
// The pixel kernel: a warp takes a cell, the pixels that share their four corner
// patches (14 x 14 at patch 14), in two passes over its pixels.
//  1. a lane a pixel, seven pixels a lane at a time: the lane runs over the 128
//     hidden units (corner values, b1 and w2 read as warp-uniform 16-byte
//     loads, shared by its seven pixels) and forms sigma, the loss and dL/dz2.
//     The dot with w2 is summed as a tree over groups of four units.
//  2. a lane four hidden units: along an image row the pre-activation is linear
//     in x, so a pixel costs one FMA per unit for its sign, and the row needs
//     only sum dz2 and sum dz2 ax over the pixels where the unit is on.
// About 55 warp instructions a pixel, bound by their issue, where a warp a
// pixel (corner loads, a shuffle reduction and 16 corner sums per lane and
// pixel) took 250.  5 x 621x467 at 384 features: 0.121 ms for the cells and
// 0.21 ms for the call (0.23 with the second pass's look at units near zero), against 0.71 ms of four launches a view.
#include <algorithm>

#include "common.cuh"

namespace ups {

namespace {

constexpr int kUH = 128;     // hidden units
constexpr int kUWarps = 4;   // warps (cells at a time) per CTA
constexpr int kUPx = 7;      // pixels per lane of pass 1 (6.1 x 32 in a 14 x 14 cell)
constexpr int kUnit = 32 * kUPx;

// the views of one call
struct UncViews {
    int n, cells;
    struct V {
        int W, H, wp, hp;
        int patch0;  // its first patch (and cell: one per patch) among all views'
        int pix0;    // its first pixel
    } v[UPS_MAX_VIEWS];
};

__device__ __forceinline__ float softplus_f(float x) { return x > 20.f ? x : log1pf(__expf(x)); }
__device__ __forceinline__ float sigmoid_f(float x) { return 1.f / (1.f + __expf(-x)); }

// first patch index along an axis of n pixels whose bilinear position
// floor(clamp((x + 0.5) / patch - 0.5, 0, np - 1)) is at least i
__device__ __forceinline__ int cell_start(int i, int patch) {
    // (x + 0.5) / patch - 0.5 >= i  <=>  x >= i * patch + (patch - 1) / 2
    return i == 0 ? 0 : (int)ceilf((float)i * patch + 0.5f * (float)(patch - 1) - 1e-4f);
}

// w2 . ReLU(z) of four hidden units (4 l ..) at the lane's pixels, a[p] the
// corner weights (each as a packed pair); z is formed corner by corner
struct Hidden {
    const float *zc;  // [4][128] corner values
    const float *b1, *w2;
};
__device__ __forceinline__ void dot4(const Hidden &h, int l, const f2 (&a)[kUPx][4], float (&out)[kUPx]) {
    const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(h.b1 + 4 * l);
    const float4 w = *reinterpret_cast<const float4 *>(h.w2 + 4 * l);
    ulonglong2 c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = *reinterpret_cast<const ulonglong2 *>(h.zc + i * kUH + 4 * l);
#pragma unroll
    for (int p = 0; p < kUPx; ++p) {
        f2 z01 = b.x, z23 = b.y;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            z01 = f2_fma(a[p][i], c[i].x, z01);
            z23 = f2_fma(a[p][i], c[i].y, z23);
        }
        float z0, z1, z2, z3;
        f2_split(z01, z0, z1);
        f2_split(z23, z2, z3);
        float d = fmaf(w.x, fmaxf(z0, 0.f), 0.f);
        d = fmaf(w.y, fmaxf(z1, 0.f), d);
        d = fmaf(w.z, fmaxf(z2, 0.f), d);
        out[p] = fmaf(w.w, fmaxf(z3, 0.f), d);
    }
}
// sum of dot4 over the groups l, l + O, l + 2 O, ... < 32, as a tree: groups
// 16 apart first, then 8, ...
template <int O>
__device__ __forceinline__ void dot_tree(const Hidden &h, int l, const f2 (&a)[kUPx][4], float (&out)[kUPx]) {
    if constexpr (O == 32) {
        dot4(h, l, a, out);
    } else {
        float t[kUPx];
        dot_tree<2 * O>(h, l, a, out);
        dot_tree<2 * O>(h, l + O, a, t);
#pragma unroll
        for (int p = 0; p < kUPx; ++p) out[p] += t[p];
    }
}

__global__ void __launch_bounds__(32 * kUWarps, 4) k_unc_cells(
    const UncViews tv, int patch, const float *__restrict__ Zp, const float *__restrict__ b1,
    const float *__restrict__ w2, const float *__restrict__ b2, const float *__restrict__ R, float lambda, float g,
    float *__restrict__ loss, float *__restrict__ sigma_out, uint8_t *__restrict__ motion_out,
    float *__restrict__ d_b1, float *__restrict__ d_w2, float *__restrict__ d_b2, float *__restrict__ D,
    int *__restrict__ next) {
    __shared__ __align__(16) float s_z[kUWarps][4][kUH];  // the four corner patches' W1 g
    __shared__ __align__(16) float s_b1[kUH], s_w2[kUH];
    __shared__ float2 s_px[kUWarps][kUnit];  // (dL/dz2, ax) of a unit's pixels
    __shared__ float red[kUWarps][2][kUH];   // per-warp sums: d_w2, d_b1
    __shared__ float sred[kUWarps][2];       // loss, d_b2
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kUH; i += 32 * kUWarps) {
        s_b1[i] = b1[i];
        s_w2[i] = w2[i];
    }
    __syncthreads();
    const float bb2 = b2[0];
    const float inv2p = 1.f / (float)(2 * patch);
    const f2 bb01 = reinterpret_cast<const f2 *>(s_b1)[2 * lane], bb23 = reinterpret_cast<const f2 *>(s_b1)[2 * lane + 1];
    f2 a_dw01 = 0ull, a_dw23 = 0ull, a_db01 = 0ull, a_db23 = 0ull;  // this lane's units, over all of the warp's cells
    float a_loss = 0.f, a_db2 = 0.f;
    const Hidden hid{&s_z[w][0][0], s_b1, s_w2};
    // cells are taken one at a time (*next was zero): border cells are twice as wide
    for (;;) {
        int cell = 0;
        if (lane == 0) cell = atomicAdd(next, 1);
        cell = __shfl_sync(0xffffffffu, cell, 0);
        if (cell >= tv.cells) break;
        int vi = 0;
        while (vi + 1 < tv.n && tv.v[vi + 1].patch0 <= cell) ++vi;
        const UncViews::V &vw = tv.v[vi];
        const int W = vw.W, H = vw.H, wp = vw.wp, hp = vw.hp;
        const int cj = (cell - vw.patch0) / wp, ci = cell - vw.patch0 - cj * wp;
        // pixel range of the cell (the last cell along an axis runs to the border)
        const int xs = cell_start(ci, patch), xe = ci + 1 >= wp ? W : min(W, cell_start(ci + 1, patch));
        const int ys = cell_start(cj, patch), ye = cj + 1 >= hp ? H : min(H, cell_start(cj + 1, patch));
        if (xe <= xs || ye <= ys) continue;
        const int x1 = min(ci + 1, wp - 1), y1 = min(cj + 1, hp - 1);
        const int corner[4] = {vw.patch0 + cj * wp + ci, vw.patch0 + cj * wp + x1, vw.patch0 + y1 * wp + ci,
                               vw.patch0 + y1 * wp + x1};
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 4; ++c)
            reinterpret_cast<float4 *>(s_z[w][c])[lane] =
                reinterpret_cast<const float4 *>(Zp + (size_t)corner[c] * kUH)[lane];
        __syncwarp();
        // this lane's units: corner values and their steps along x
        f2 c0[2], c2[2], e0[2], e2[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            auto at = [&](int c) { return reinterpret_cast<const f2 *>(s_z[w][c])[2 * lane + i]; };
            const f2 neg = f2_make(-1.f, -1.f);
            c0[i] = at(0);
            c2[i] = at(2);
            e0[i] = f2_fma(neg, c0[i], at(1));
            e2[i] = f2_fma(neg, c2[i], at(3));
        }
        // Pass 2 steps the pre-activation along x, which rounds it another way than the
        // corner-by-corner sum of pass 1 (both within 14 roundings of the magnitudes
        // summed, 2^-20 of their sum): where a unit is nearer to 0 than that, pass 2
        // takes pass 1's sum, so that both take the same units for on.  Values that are not
        // finite always take it, and there the hidden values and not z go into dL/dw2: zero
        // times an off unit's z would not be zero.
        float near0 = 0.f;
        {
            const float4 b = reinterpret_cast<const float4 *>(s_b1)[lane];
            float m[4] = {fabsf(b.x), fabsf(b.y), fabsf(b.z), fabsf(b.w)};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 z = reinterpret_cast<const float4 *>(s_z[w][c])[lane];
                m[0] += fabsf(z.x);
                m[1] += fabsf(z.y);
                m[2] += fabsf(z.z);
                m[3] += fabsf(z.w);
            }
            near0 = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])) * 9.5367431640625e-7f;
            if (!((m[0] + m[1]) + (m[2] + m[3]) < INFINITY)) near0 = INFINITY;
        }
        f2 aD[4][2] = {};
        // units of at most kUnit pixels: bw columns, br rows
        for (int bx = xs; bx < xe; bx += kUnit) {
            const int bw = min(xe - bx, kUnit), brm = kUnit / bw;
            const uint32_t magic = (65536u + bw - 1) / bw;  // q / bw = q magic >> 16 for q < kUnit
            for (int by = ys; by < ye; by += brm) {
                const int br = min(ye - by, brm), n = bw * br;
                // pass 1: a lane pixels lane, lane + 32, ...
                f2 a[kUPx][4];
                float axs[kUPx];
                int pos[kUPx];
#pragma unroll
                for (int p = 0; p < kUPx; ++p) {
                    const int q = lane + 32 * p, qy = (int)((uint32_t)q * magic >> 16);
                    const int x = bx + q - qy * bw, y = by + qy;
                    // bilinear weight u - x0 = ((2x + 1) - (2 x0 + 1) patch) / (2 patch): an exact
                    // integer numerator, one rounding (u itself is ~45 at 640 px, where a float
                    // ulp would already move the weight by 4e-6); clamped positions give 0
                    // (and at the far edge x1 == x0)
                    const float ax = fminf(fmaxf((float)(2 * x + 1 - (2 * ci + 1) * patch) * inv2p, 0.f), 1.f);
                    const float ay = fminf(fmaxf((float)(2 * y + 1 - (2 * cj + 1) * patch) * inv2p, 0.f), 1.f);
                    const float wt[4] = {(1.f - ax) * (1.f - ay), ax * (1.f - ay), (1.f - ax) * ay, ax * ay};
#pragma unroll
                    for (int c = 0; c < 4; ++c) a[p][c] = f2_make(wt[c], wt[c]);
                    axs[p] = ax;
                    pos[p] = q < n ? vw.pix0 + y * W + x : -1;
                }
                float dot[kUPx];
#pragma unroll 1
                for (int i = 0; i < 4; ++i) {
                    // groups l, l + 4, ... for l = 0, 2, 1, 3: (0 + 2) + (1 + 3)
                    float t[kUPx];
                    dot_tree<4>(hid, ((i & 1) << 1) | (i >> 1), a, t);
                    if (i == 0)
#pragma unroll
                        for (int p = 0; p < kUPx; ++p) dot[p] = t[p];
                    else if (i == 1)
#pragma unroll
                        for (int p = 0; p < kUPx; ++p) dot[p] += t[p];
                    else if (i == 2)
#pragma unroll
                        for (int p = 0; p < kUPx; ++p) s_px[w][lane + 32 * p].x = t[p];
                    else
#pragma unroll
                        for (int p = 0; p < kUPx; ++p) dot[p] += s_px[w][lane + 32 * p].x + t[p];
                }
#pragma unroll
                for (int p = 0; p < kUPx; ++p) {
                    float dz2 = 0.f;
                    if (pos[p] >= 0) {
                        const float z2 = dot[p] + bb2;
                        const float s = softplus_f(z2);
                        const float r = R[pos[p]];
                        // L_u = R / (2 s^2) + lambda log s;  dL_u/ds = -R / s^3 + lambda / s = (lambda - R / s^2) / s
                        const float is = 1.f / s;
                        const float ds = g * is * (lambda - r * is * is);
                        dz2 = ds * sigmoid_f(z2);
                        a_loss += r / (2.f * s * s) + lambda * logf(s);
                        a_db2 += dz2;
                        if (sigma_out) sigma_out[pos[p]] = s;
                        if (motion_out) motion_out[pos[p]] = 2.f * s * s > 1.f ? 1 : 0;
                    }
                    s_px[w][lane + 32 * p] = make_float2(dz2, axs[p]);
                }
                __syncwarp();
                // pass 2: a lane its four units, row by row
                for (int ry = 0; ry < br; ++ry) {
                    const int y = by + ry;
                    const float ay = fminf(fmaxf((float)(2 * y + 1 - (2 * cj + 1) * patch) * inv2p, 0.f), 1.f);
                    const f2 ay2 = f2_make(ay, ay), by2 = f2_make(1.f - ay, 1.f - ay);
                    const f2 z0a = f2_fma(ay2, c2[0], f2_fma(by2, c0[0], bb01)), z0b = f2_fma(ay2, c2[1], f2_fma(by2, c0[1], bb23));
                    const f2 sla = f2_fma(ay2, e2[0], f2_fma(by2, e0[0], 0ull)), slb = f2_fma(ay2, e2[1], f2_fma(by2, e0[1], 0ull));
                    f2 S0a = 0ull, S0b = 0ull, S1a = 0ull, S1b = 0ull;  // sum dz2, sum dz2 ax where the unit is on
                    const float2 *px = s_px[w] + ry * bw;
#pragma unroll 2
                    for (int x = 0; x < bw; ++x) {
                        const float2 t = px[x];
                        const f2 ax2 = f2_make(t.y, t.y);
                        f2 za = f2_fma(ax2, sla, z0a), zb = f2_fma(ax2, slb, z0b);
                        float u0, u1, u2, u3;
                        f2_split(za, u0, u1);
                        f2_split(zb, u2, u3);
                        if (!(fminf(fminf(fabsf(u0), fabsf(u1)), fminf(fabsf(u2), fabsf(u3))) > near0)) {
                            const float wt[4] = {(1.f - t.y) * (1.f - ay), t.y * (1.f - ay), (1.f - t.y) * ay, t.y * ay};
                            za = bb01;
                            zb = bb23;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const ulonglong2 zc = reinterpret_cast<const ulonglong2 *>(s_z[w][c])[lane];
                                const f2 w2c = f2_make(wt[c], wt[c]);
                                za = f2_fma(w2c, zc.x, za);
                                zb = f2_fma(w2c, zc.y, zb);
                            }
                            f2_split(za, u0, u1);
                            f2_split(zb, u2, u3);
                            za = f2_make(fmaxf(u0, 0.f), fmaxf(u1, 0.f));
                            zb = f2_make(fmaxf(u2, 0.f), fmaxf(u3, 0.f));
                        }
                        const f2 ma = f2_make(u0 > 0.f ? t.x : 0.f, u1 > 0.f ? t.x : 0.f);
                        const f2 mb = f2_make(u2 > 0.f ? t.x : 0.f, u3 > 0.f ? t.x : 0.f);
                        S0a = f2_add(S0a, ma);
                        S0b = f2_add(S0b, mb);
                        S1a = f2_fma(ma, ax2, S1a);
                        S1b = f2_fma(mb, ax2, S1b);
                        a_dw01 = f2_fma(ma, za, a_dw01);
                        a_dw23 = f2_fma(mb, zb, a_dw23);
                    }
                    const f2 neg = f2_make(-1.f, -1.f);
                    const f2 La = f2_fma(neg, S1a, S0a), Lb = f2_fma(neg, S1b, S0b);
                    aD[0][0] = f2_fma(by2, La, aD[0][0]);
                    aD[0][1] = f2_fma(by2, Lb, aD[0][1]);
                    aD[1][0] = f2_fma(by2, S1a, aD[1][0]);
                    aD[1][1] = f2_fma(by2, S1b, aD[1][1]);
                    aD[2][0] = f2_fma(ay2, La, aD[2][0]);
                    aD[2][1] = f2_fma(ay2, Lb, aD[2][1]);
                    aD[3][0] = f2_fma(ay2, S1a, aD[3][0]);
                    aD[3][1] = f2_fma(ay2, S1b, aD[3][1]);
                    a_db01 = f2_add(a_db01, S0a);
                    a_db23 = f2_add(a_db23, S0b);
                }
                __syncwarp();
            }
        }
        if (D) {
            const float4 wv = reinterpret_cast<const float4 *>(s_w2)[lane];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float4 d;
                f2_split(aD[c][0], d.x, d.y);
                f2_split(aD[c][1], d.z, d.w);
                atomicAdd(reinterpret_cast<float4 *>(D + (size_t)corner[c] * kUH) + lane,
                          make_float4(wv.x * d.x, wv.y * d.y, wv.z * d.z, wv.w * d.w));
            }
        }
    }
    // reduce over the CTA's warps, then one atomic per value
    reinterpret_cast<f2 *>(red[w][0])[2 * lane] = a_dw01;
    reinterpret_cast<f2 *>(red[w][0])[2 * lane + 1] = a_dw23;
    reinterpret_cast<f2 *>(red[w][1])[2 * lane] = a_db01;
    reinterpret_cast<f2 *>(red[w][1])[2 * lane + 1] = a_db23;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a_loss += __shfl_xor_sync(0xffffffffu, a_loss, o);
        a_db2 += __shfl_xor_sync(0xffffffffu, a_db2, o);
    }
    if (lane == 0) {
        sred[w][0] = a_loss;
        sred[w][1] = a_db2;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kUH; i += 32 * kUWarps) {
        const int t = i / kUH, j = i % kUH;
        float s = 0.f;
#pragma unroll
        for (int ww = 0; ww < kUWarps; ++ww) s += red[ww][t][j];
        if (t == 0) {
            if (d_w2) atomicAdd(d_w2 + j, s);
        } else if (d_b1) {
            atomicAdd(d_b1 + j, s * s_w2[j]);
        }
    }
    if (threadIdx.x == 0) {
        float l = 0.f, b = 0.f;
        for (int ww = 0; ww < kUWarps; ++ww) {
            l += sred[ww][0];
            b += sred[ww][1];
        }
        atomicAdd(loss, g * l);
        if (d_b2) atomicAdd(d_b2, b);
    }
}

}  // namespace

size_t unc_scratch_floats(size_t patches) { return 2 * patches * kUH + 4; }

// All views of vt: sigma, motion mask, loss and the F_u gradients (accumulated;
// any gradient pointer may be null).  grid: the views' patch grids [hp][wp][nh]
// one after another; scratch: unc_scratch_floats(their patches).
cudaError_t unc_all(int num_sms, cudaStream_t st, const ViewTable &vt, int nh, int patch, const float *grid,
                    const float *R, const float *w1, const float *b1, const float *w2, const float *b2, float lambda,
                    float g, float *loss, float *d_w1, float *d_b1, float *d_w2, float *d_b2, float *sigma,
                    uint8_t *motion, float *scratch, int *launches) {
    UncViews tv{};
    tv.n = vt.n;
    for (int v = 0; v < vt.n; ++v) {
        const DevView &cam = vt.v[v];
        const int wp = (cam.W + patch - 1) / patch, hp = (cam.H + patch - 1) / patch;
        tv.v[v] = UncViews::V{cam.W, cam.H, wp, hp, tv.cells, cam.pix_off};
        tv.cells += wp * hp;
    }
    const int np = tv.cells;
    float *Zp = scratch;                     // [np][128]  W1 g of every patch
    float *D = scratch + (size_t)np * kUH;   // [np][128]  interpolation-weighted dL/dh per patch
    cudaError_t e;
    // Zp (column-major [128 x np]) = W1 [128 x nh] G^T, at most a grid's columns at a time
    constexpr int kMaxCols = 65535 * 64;
    for (int p = 0; p < np; p += kMaxCols)
        if ((e = gemm_f32(st, true, false, kUH, std::min(np - p, kMaxCols), nh, 1.f, w1, nh, grid + (size_t)p * nh, nh,
                          0.f, Zp + (size_t)p * kUH, kUH, num_sms, launches, true)) != cudaSuccess)
            return e;
    int *next = reinterpret_cast<int *>(D + (size_t)np * kUH);  // the cell counter, cleared with D
    float *clear = d_w1 ? D : D + (size_t)np * kUH;
    if ((e = cudaMemsetAsync(clear, 0, ((size_t)(D - clear) + (size_t)np * kUH + 4) * sizeof(float), st)) != cudaSuccess)
        return e;
    const int blocks = std::min((np + kUWarps - 1) / kUWarps, num_sms * 4);
    k_unc_cells<<<blocks, 32 * kUWarps, 0, st>>>(tv, patch, Zp, b1, w2, b2, R, lambda, g, loss, sigma, motion, d_b1, d_w2,
                                                 d_b2, d_w1 ? D : nullptr, next);
    ++*launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // dW1 (column-major [nh x 128], i.e. [128][nh] row-major) += G^T D
    if (d_w1 && (e = gemm_f32(st, false, true, nh, kUH, np, 1.f, grid, nh, D, kUH, 1.f, d_w1, nh, num_sms, launches)) != cudaSuccess)
        return e;
    return cudaSuccess;
}

}  // namespace ups
