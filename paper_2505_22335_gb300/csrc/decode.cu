// Per-anchor MLP decode of K neural Gaussians (Eq. 8-9) and its backward,
// FP32 on the CUDA cores.
//
// Row = (anchor, view).  MLP input x = [f_v, delta_vc, d_vc, sin(pi t),
// cos(pi t)]; four MLPs (opacity, covariance, colour: ReLU hidden; feature
// F_d: SoftPlus hidden) of width `hidden` = 32.  Weights live in shared memory
// and are read as 16-byte broadcasts (every lane of a warp reads the same
// weight); what bounds the loops stands at each kernel.
//
// Backward (FP32 data path): one thread per row recomputes each MLP group's
// hidden layer, forms dL/dY of the group's outputs and propagates it to the
// hidden layer and the MLP input (k_decode_bwd_rows); the hidden activations
// and pre-activation gradients go to a feature-major scratch from which the
// weight gradients are reduced by a separate kernel (decode_bwd_tc.cu).
#include <algorithm>
#include <initializer_list>

#include "decode_bwd.cuh"

namespace ups {

namespace {

constexpr int kH = 32;       // hidden width per MLP
constexpr int kFin = 32;     // anchor feature width
constexpr int kDin = kFin + 6;
constexpr int kDinP = 40;    // padded input width (float4 rows)
constexpr int kDX = kFin + 4;  // MLP inputs with a gradient: f_v, delta_vc, d_vc
constexpr size_t kMaxSmem = 227 * 1024;  // opt-in shared memory per block

__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + __expf(-x)); }
__device__ __forceinline__ float softplus(float x) { return x > 20.f ? x : log1pf(__expf(x)); }
__device__ __forceinline__ float opacity_act(float y, int op_tanh) { return op_tanh ? tanhf(y) : sigm(y); }

struct DecodeArgs {
    int A, K, NF, n_out;
    const float *pos, *afeat, *offs, *ascale;
    const float *w1, *b1, *w2, *b2;
    int op_tanh;  // opacity = tanh(y) (Scaffold-GS form) instead of sigmoid(y)
};

// x (padded to 40) for anchor `an` seen from view `cam`; returns delta and d.
__device__ __forceinline__ void mlp_input(const DecodeArgs &a, const DevView &cam, int an,
                                          float x[kDinP], float delta[3], float &dist) {
    const float4 *f4 = reinterpret_cast<const float4 *>(a.afeat + (size_t)an * kFin);
#pragma unroll
    for (int i = 0; i < kFin / 4; ++i) {
        float4 f = f4[i];
        x[4 * i] = f.x;
        x[4 * i + 1] = f.y;
        x[4 * i + 2] = f.z;
        x[4 * i + 3] = f.w;
    }
    // camera centre o_c = -R^T t
    float oc[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        oc[i] = -(cam.R[i] * cam.t[0] + cam.R[3 + i] * cam.t[1] + cam.R[6 + i] * cam.t[2]);
    float r[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i] = a.pos[3 * an + i] - oc[i];
    dist = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    float id = 1.f / dist;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        delta[i] = r[i] * id;
        x[kFin + i] = delta[i];
    }
    x[kFin + 3] = dist;
    float s, c;
    sincospif(cam.t_norm, &s, &c);
    x[kFin + 4] = s;
    x[kFin + 5] = c;
    x[38] = 0.f;
    x[39] = 0.f;
}

// hidden block g: z = W1_g x + b1_g (32 values, held as 16 packed pairs
// (z_2p, z_2p+1) for fma.rn.f32x2), input-outer so the accumulators stay in
// registers.  W1 is transposed in shared memory ([38][128]: input-major); the
// anchor-feature part of x is read through L1 (rows of the same anchor share
// it), the camera-dependent tail x[32..37] comes in registers.  Each element
// is rounded exactly as a scalar fmaf chain over the inputs in order.
constexpr int kH2 = kH / 2;
__device__ __forceinline__ void hidden_T(const float *sW1T, const float *sb1, int g, const float *afeat_row,
                                         const float xt[6], f2 h[kH2]) {
    const f2 *b2 = reinterpret_cast<const f2 *>(sb1 + g * kH);
#pragma unroll
    for (int p = 0; p < kH2; ++p) h[p] = b2[p];
    const float4 *f4 = reinterpret_cast<const float4 *>(afeat_row);
    // the next four inputs are loaded while the current four are applied (one
    // load in flight per step instead of a stall on each)
    float4 nxt = __ldg(f4);
#pragma unroll 1
    for (int i4 = 0; i4 < kFin / 4; ++i4) {
        const float4 xv = nxt;
        if (i4 + 1 < kFin / 4) nxt = __ldg(f4 + i4 + 1);
        const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW1T + (4 * i4 + u) * 128 + g * kH);
            const f2 xx = f2_make(xs[u], xs[u]);
#pragma unroll
            for (int q = 0; q < kH / 4; ++q) {
                const ulonglong2 ww = w[q];
                h[2 * q] = f2_fma(ww.x, xx, h[2 * q]);
                h[2 * q + 1] = f2_fma(ww.y, xx, h[2 * q + 1]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 6; ++u) {
        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW1T + (kFin + u) * 128 + g * kH);
        const f2 xx = f2_make(xt[u], xt[u]);
#pragma unroll
        for (int q = 0; q < kH / 4; ++q) {
            const ulonglong2 ww = w[q];
            h[2 * q] = f2_fma(ww.x, xx, h[2 * q]);
            h[2 * q + 1] = f2_fma(ww.y, xx, h[2 * q + 1]);
        }
    }
}

// element-wise activation of the packed hidden values: ReLU (act 0) or
// SoftPlus (act 1)
template <int ACT>
__device__ __forceinline__ void activate(f2 h[kH2]) {
#pragma unroll
    for (int p = 0; p < kH2; ++p) {
        float lo, hi;
        f2_split(h[p], lo, hi);
        h[p] = ACT == 0 ? f2_make(fmaxf(lo, 0.f), fmaxf(hi, 0.f)) : f2_make(softplus(lo), softplus(hi));
    }
}

// y_r = W2[r] . h + b2[r] with four partial sums (short dependency chains):
// the pairs (s0, s1) and (s2, s3) of the scalar form, summed (s0+s1)+(s2+s3)
__device__ __forceinline__ float out_row(const float *sW2, const float *sb2, int r, const f2 h[kH2]) {
    const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW2 + r * kH);
    f2 a01 = f2_make(sb2[r], 0.f), a23 = 0ull;
#pragma unroll
    for (int q = 0; q < kH / 4; ++q) {
        const ulonglong2 ww = w[q];
        a01 = f2_fma(ww.x, h[2 * q], a01);
        a23 = f2_fma(ww.y, h[2 * q + 1], a23);
    }
    float s0, s1, s2, s3;
    f2_split(a01, s0, s1);
    f2_split(a23, s2, s3);
    return (s0 + s1) + (s2 + s3);
}

// shared layout of the decode kernels: W1 transposed [38][128], b1 [128],
// W2 [n_out][32], b2 [n_out] (padded to 4)
__device__ __forceinline__ void load_weights_T(const DecodeArgs &a, float *sW1T, float *sb1, float *sW2,
                                               float *sb2) {
    for (int i = threadIdx.x; i < kDin * 4 * kH; i += blockDim.x) {
        const int ii = i / (4 * kH), h = i - ii * (4 * kH);
        sW1T[i] = a.w1[h * kDin + ii];
    }
    for (int i = threadIdx.x; i < 4 * kH; i += blockDim.x) sb1[i] = a.b1[i];
    for (int i = threadIdx.x; i < a.n_out * kH; i += blockDim.x) sW2[i] = a.w2[i];
    for (int i = threadIdx.x; i < a.n_out; i += blockDim.x) sb2[i] = a.b2[i];
}

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------
//
// A warp takes 64 rows on its own, two a lane (rows lane and lane + 32), so that
// every weight, a warp-uniform 16-byte shared load of two wavefronts, feeds both:
// the kernel is bound by shared-memory and store wavefronts, then by the FMA
// pipe.  The rows' inputs lie transposed in the warp's shared memory (one
// wavefront an input and row group); the hidden values stay in registers.
// Gaussians are stored two at a time as 32-byte records (full sectors) where K
// is even and the outputs are 32-byte aligned.  Record of (row, k): row K + k.
// Every element is rounded exactly as a scalar fmaf chain over the inputs in
// order, and an output as four partial sums (s0 + s1) + (s2 + s3).
// 800k rows (100k anchors x 10, 8 views, N_l 16): 0.67 ms; one row a lane 0.90
// ms, a 4 x 4 register tile over lanes in rows and columns 0.81 ms (its 16-byte
// loads take three to four wavefronts).
constexpr int kFwdWarps = 16;  // warps per CTA at most (one CTA per SM)
constexpr int kXT = 64;        // rows of a warp's XT [38][64]

// W1_g x + b1_g of the lane's two rows (XT: at the lane's column), activated
template <int ACT>
__device__ __forceinline__ void hidden2(const float *sW1T, const float *sb1, int g, const float *XT, f2 (&h)[2][kH2]) {
    const ulonglong2 *b = reinterpret_cast<const ulonglong2 *>(sb1 + g * kH);
#pragma unroll
    for (int q = 0; q < kH / 4; ++q) {
        const ulonglong2 v = b[q];
        h[0][2 * q] = h[1][2 * q] = v.x;
        h[0][2 * q + 1] = h[1][2 * q + 1] = v.y;
    }
#pragma unroll 2
    for (int k = 0; k < kDin; ++k) {
        const float x0 = XT[k * kXT], x1 = XT[k * kXT + 32];
        const f2 a = f2_make(x0, x0), c = f2_make(x1, x1);
        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW1T + k * 4 * kH + g * kH);
#pragma unroll
        for (int q = 0; q < kH / 4; ++q) {
            const ulonglong2 v = w[q];
            h[0][2 * q] = f2_fma(v.x, a, h[0][2 * q]);
            h[1][2 * q] = f2_fma(v.x, c, h[1][2 * q]);
            h[0][2 * q + 1] = f2_fma(v.y, a, h[0][2 * q + 1]);
            h[1][2 * q + 1] = f2_fma(v.y, c, h[1][2 * q + 1]);
        }
    }
    activate<ACT>(h[0]);
    activate<ACT>(h[1]);
}

// outputs r .. r + M - 1 of both rows
template <int M>
__device__ __forceinline__ void out2(const float *sW2, const float *sb2, int r, const f2 (&h)[2][kH2], float (&y)[2][M]) {
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW2 + (r + j) * kH);
        f2 a01[2], a23[2];
        a01[0] = a01[1] = f2_make(sb2[r + j], 0.f);
        a23[0] = a23[1] = 0ull;
#pragma unroll
        for (int q = 0; q < kH / 4; ++q) {
            const ulonglong2 v = w[q];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                a01[i] = f2_fma(v.x, h[i][2 * q], a01[i]);
                a23[i] = f2_fma(v.y, h[i][2 * q + 1], a23[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float s0, s1, s2, s3;
            f2_split(a01[i], s0, s1);
            f2_split(a23[i], s2, s3);
            y[i][j] = (s0 + s1) + (s2 + s3);
        }
    }
}

// 32 bytes at a 32-byte aligned address
__device__ __forceinline__ void store8(float *p, float4 a, float4 b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// PAIR: K is even and every output array 32-byte aligned
template <int NF, bool PAIR>
__global__ void __launch_bounds__(32 * kFwdWarps, 1) k_decode_fwd(ViewTable vt, DecodeArgs a, int split,
                                                    float4 *__restrict__ mean_op,
                                                    float4 *__restrict__ scale_out,
                                                    float4 *__restrict__ quat_out,
                                                    float4 *__restrict__ color_out,
                                                    float *__restrict__ feat_out) {
    extern __shared__ float4 smem4[];
    float *sm = reinterpret_cast<float *>(smem4);
    constexpr int P = PAIR ? 2 : 1;  // Gaussians a step
    const int K = a.K, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float *sW1T = sm, *sb1 = sW1T + kDin * 4 * kH, *sW2 = sb1 + 4 * kH, *sb2 = sW2 + a.n_out * kH;
    float *XT = sb2 + ((a.n_out + 3) & ~3) + wid * (kDin * kXT) + lane;
    load_weights_T(a, sW1T, sb1, sW2, sb2);
    __syncthreads();
    const int rows = a.A * vt.n, nw = blockDim.x >> 5;
    const int tiles = (rows + kXT - 1) / kXT;
    // Work items: a tile, or (split) one MLP of a tile, the costliest MLP first:
    // features, covariance, colour, opacity.  They go round the SMs before the
    // warps, so that a last, partial round loads every SM alike.
    constexpr int kMlps = NF > 0 ? 4 : 3;
    const int items = split ? kMlps * tiles : tiles;
    for (int it = blockIdx.x + gridDim.x * wid; it < items; it += gridDim.x * nw) {
        const int tile = it % tiles, first = (split ? it / tiles : 0) + (4 - kMlps), last = split ? first : 3;
        int row[2], an[2];
        bool on[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            row[i] = tile * kXT + 32 * i + lane;
            on[i] = row[i] < rows;
            row[i] = min(row[i], rows - 1);
            const int v = row[i] / a.A;
            an[i] = row[i] - v * a.A;
            float x[kDinP], delta[3], dist;
            mlp_input(a, vt.v[v], an[i], x, delta, dist);
#pragma unroll
            for (int k = 0; k < kDin; ++k) XT[k * kXT + 32 * i] = x[k];  // read back by this lane only
        }
        // the P records from k of row i
        auto put = [&](float4 *base, int i, int k, const float4 (&v)[P]) {
            if (!on[i]) return;
            float4 *p = base + (size_t)row[i] * K + k;
            if constexpr (PAIR)
                store8(reinterpret_cast<float *>(p), v[0], v[P - 1]);
            else
                *p = v[0];
        };
#pragma unroll 1
        for (int order = first; order <= last; ++order) {
            f2 h[2][kH2];
            if (order == 3) {  // opacity, and the mean
                hidden2<0>(sW1T, sb1, 0, XT, h);
#pragma unroll 1
                for (int k = 0; k < K; k += P) {
                    float y[2][P];
                    out2<P>(sW2, sb2, k, h, y);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float *p = a.pos + 3 * an[i], *o3 = a.offs + ((size_t)an[i] * K + k) * 3;
                        float4 m[P];
#pragma unroll
                        for (int j = 0; j < P; ++j)
                            m[j] = make_float4(p[0] + o3[3 * j], p[1] + o3[3 * j + 1], p[2] + o3[3 * j + 2],
                                               opacity_act(y[i][j], a.op_tanh));
                        put(mean_op, i, k, m);
                    }
                }
            } else if (order == 1) {  // covariance: 3 scale + 4 quaternion per Gaussian
                hidden2<0>(sW1T, sb1, 1, XT, h);
#pragma unroll 1
                for (int k = 0; k < K; k += P) {
                    float4 s[2][P];
#pragma unroll
                    for (int j = 0; j < P; ++j) {
                        float y[2][3];
                        out2<3>(sW2, sb2, K + 7 * (k + j), h, y);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const float *l = a.ascale + 3 * an[i];
                            s[i][j] = make_float4(l[0] * sigm(y[i][0]), l[1] * sigm(y[i][1]), l[2] * sigm(y[i][2]), 0.f);
                        }
                    }
                    put(scale_out, 0, k, s[0]);
                    put(scale_out, 1, k, s[1]);
#pragma unroll
                    for (int j = 0; j < P; ++j) {
                        float y[2][4];
                        out2<4>(sW2, sb2, K + 7 * (k + j) + 3, h, y);
#pragma unroll
                        for (int i = 0; i < 2; ++i) s[i][j] = make_float4(y[i][0], y[i][1], y[i][2], y[i][3]);
                    }
                    put(quat_out, 0, k, s[0]);
                    put(quat_out, 1, k, s[1]);
                }
            } else if (order == 2) {  // colour
                hidden2<0>(sW1T, sb1, 2, XT, h);
#pragma unroll 1
                for (int k = 0; k < K; k += P) {
                    float4 c[2][P];
#pragma unroll
                    for (int j = 0; j < P; ++j) {
                        float y[2][3];
                        out2<3>(sW2, sb2, 8 * K + 3 * (k + j), h, y);
#pragma unroll
                        for (int i = 0; i < 2; ++i) c[i][j] = make_float4(sigm(y[i][0]), sigm(y[i][1]), sigm(y[i][2]), 0.f);
                    }
                    put(color_out, 0, k, c[0]);
                    put(color_out, 1, k, c[1]);
                }
            } else if (NF > 0) {
                hidden2<1>(sW1T, sb1, 3, XT, h);
#pragma unroll 1
                for (int f = 0; f < K * NF; f += 8) {
                    float y[2][8];
                    out2<8>(sW2, sb2, 11 * K + f, h, y);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (!on[i]) continue;
                        float *p = feat_out + (size_t)row[i] * K * NF + f;
                        const float4 lo = make_float4(y[i][0], y[i][1], y[i][2], y[i][3]);
                        const float4 hi = make_float4(y[i][4], y[i][5], y[i][6], y[i][7]);
                        if constexpr (PAIR) {
                            store8(p, lo, hi);
                        } else {
                            reinterpret_cast<float4 *>(p)[0] = lo;
                            reinterpret_cast<float4 *>(p)[1] = hi;
                        }
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// backward, per row (FP32)
// ---------------------------------------------------------------------------

// One MLP group of one row: Z = W1_g x + b1 (recomputed), H = act(Z); for each
// output o of the group the pre-activation Y_o (only where the output
// activation has a derivative: opacity, scale, colour), DY_o = dL/dY_o, and
// DH += DY_o W2[o]; DZ = DH * act'(Z); dx += DZ W1_g.  H, DY, DZ go to the
// feature-major scratch for the weight-gradient kernel.
template <int G, int NF>
__device__ __forceinline__ void bwd_group(const dbwd::Args &a, const DecodeArgs &da, const float *sW1T,
                                          const float *sb1, const float *sW2, const float *sb2,
                                          const float xt[6], int an, bool valid, size_t gbase, int lr,
                                          float *sDX, float dls[3]) {
    constexpr int M = G == 0 ? 1 : G == 1 ? 7 : G == 2 ? 3 : NF;
    const int K = a.K;
    const bool want_mlp = a.s.X != nullptr && valid;
    const int ld = a.s.ld;
    f2 h[kH2];
    hidden_T(sW1T, sb1, G, a.afeat + (size_t)an * kFin, xt, h);
    unsigned relu_on = 0;  // ReLU derivative as a bit mask
#pragma unroll
    for (int p = 0; p < kH2; ++p) {
        float lo, hi;
        f2_split(h[p], lo, hi);
        if (G < 3) {
            relu_on |= (lo > 0.f ? 1u : 0u) << (2 * p);
            relu_on |= (hi > 0.f ? 1u : 0u) << (2 * p + 1);
            h[p] = f2_make(fmaxf(lo, 0.f), fmaxf(hi, 0.f));
        } else {
            h[p] = f2_make(softplus(lo), softplus(hi));
        }
    }
    if (want_mlp)
#pragma unroll
        for (int p = 0; p < kH2; ++p) {
            float lo, hi;
            f2_split(h[p], lo, hi);
            a.s.H[(size_t)(G * kH + 2 * p) * ld + lr] = lo;
            a.s.H[(size_t)(G * kH + 2 * p + 1) * ld + lr] = hi;
        }
    f2 dh[kH2];
#pragma unroll
    for (int p = 0; p < kH2; ++p) dh[p] = 0ull;
    const int r0 = dbwd::grp_r0(G, K);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    // dL/dG of Gaussian k for this group, loaded one Gaussian ahead so the
    // loads of k + 1 are in flight while k is processed
    constexpr int NQ = G == 3 ? (NF / 4 > 0 ? NF / 4 : 1) : 2;
    constexpr bool kAhead = UPS_DECB_AHEAD && NQ <= 4;
    auto load = [&](int k, float4 (&q)[NQ]) {
        const size_t gi = gbase + k;
#pragma unroll
        for (int i = 0; i < NQ; ++i) q[i] = z4;
        if (!valid || k >= K) return;
        if (G == 0) q[0] = a.d_mean_op[gi];
        if (G == 1) {
            q[0] = a.d_scale[gi];
            q[1] = a.d_quat[gi];
        }
        if (G == 2) q[0] = a.d_color[gi];
        if (G == 3)
#pragma unroll
            for (int i = 0; i < NF / 4; ++i) q[i] = reinterpret_cast<const float4 *>(a.d_feat + gi * NF)[i];
    };
    float4 nxt[NQ];
    if (kAhead) load(0, nxt);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        float4 cur[NQ];
        if (kAhead) {
#pragma unroll
            for (int i = 0; i < NQ; ++i) cur[i] = nxt[i];
            load(k + 1, nxt);
        } else {
            load(k, cur);
        }
        const float4 g4a = cur[0], g4b = cur[NQ > 1 ? 1 : 0];
#pragma unroll
        for (int c = 0; c < M; ++c) {
            const int o = r0 + M * k + c;
            const bool nl = G == 0 || G == 2 || (G == 1 && c < 3);
            float gin;
            if (G == 0) {
                gin = g4a.w;
            } else if (G == 1) {
                gin = c == 0 ? g4a.x : c == 1 ? g4a.y : c == 2 ? g4a.z : c == 3 ? g4b.x : c == 4 ? g4b.y
                                                                          : c == 5 ? g4b.z : g4b.w;
            } else if (G == 2) {
                gin = c == 0 ? g4a.x : c == 1 ? g4a.y : g4a.z;
            } else {
                const float4 f4 = cur[(c >> 2) < NQ ? (c >> 2) : 0];
                gin = (c & 3) == 0 ? f4.x : (c & 3) == 1 ? f4.y : (c & 3) == 2 ? f4.z : f4.w;
            }
            float dy = gin;
            if (G == 0 && da.op_tanh) {
                const float t = tanhf(out_row(sW2, sb2, o, h));
                dy = gin * (1.f - t * t);
            } else if (nl) {
                const float s = sigm(out_row(sW2, sb2, o, h));
                if (G == 1) {
                    dy = gin * a.ascale[3 * an + c] * s * (1.f - s);
                    dls[c] += gin * s;
                } else {
                    dy = gin * s * (1.f - s);
                }
            }
            if (want_mlp) a.s.DY[(size_t)o * ld + lr] = dy;
            const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW2 + o * kH);
            const f2 dy2 = f2_make(dy, dy);
#pragma unroll
            for (int q = 0; q < kH / 4; ++q) {
                const ulonglong2 ww = w[q];
                dh[2 * q] = f2_fma(dy2, ww.x, dh[2 * q]);
                dh[2 * q + 1] = f2_fma(dy2, ww.y, dh[2 * q + 1]);
            }
        }
    }
    // DZ = DH * act'(Z): ReLU -> mask; SoftPlus -> sigmoid(Z) = 1 - exp(-H)
#pragma unroll
    for (int p = 0; p < kH2; ++p) {
        float d0, d1, h0, h1;
        f2_split(dh[p], d0, d1);
        f2_split(h[p], h0, h1);
        d0 *= G < 3 ? (float)((relu_on >> (2 * p)) & 1u) : -expm1f(-h0);
        d1 *= G < 3 ? (float)((relu_on >> (2 * p + 1)) & 1u) : -expm1f(-h1);
        dh[p] = f2_make(d0, d1);
        if (want_mlp) {
            a.s.DZ[(size_t)(G * kH + 2 * p) * ld + lr] = d0;
            a.s.DZ[(size_t)(G * kH + 2 * p + 1) * ld + lr] = d1;
        }
    }
    // dx += DZ W1_g for the inputs that have a gradient (f_v, delta_vc, d_vc),
    // accumulated in shared memory (column tid of sDX); partial sums as in
    // out_row
#pragma unroll 1
    for (int i = 0; i < kDX; ++i) {
        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(sW1T + i * 128 + G * kH);
        f2 a01 = 0ull, a23 = 0ull;
#pragma unroll
        for (int q = 0; q < kH / 4; ++q) {
            const ulonglong2 ww = w[q];
            a01 = f2_fma(dh[2 * q], ww.x, a01);
            a23 = f2_fma(dh[2 * q + 1], ww.y, a23);
        }
        float s0, s1, s2, s3;
        f2_split(a01, s0, s1);
        f2_split(a23, s2, s3);
        sDX[i * dbwd::kRowsFp32] += (s0 + s1) + (s2 + s3);
    }
}

// One thread per row (anchor-major), kRowsFp32 rows per step of a grid-stride loop;
// weights in shared memory read as broadcasts.
//
// A row's chain through its four MLPs takes about 0.12 ms however few rows there
// are.  Few rows (at most max_split_tiles CTAs' worth, half of what the GPU holds)
// are therefore split by MLP: CTA (x, y) does one MLP of its rows, and as the end of
// a row's backward is linear in dL/dx, every MLP's share goes through it by itself
// (the Gaussians' means with the opacity MLP, the anchor scaling with the
// covariance).  10k rows 0.126 -> 0.086 ms; a tracking request over 500k anchors,
// whose list of rows is short, 2.91 -> 2.82.  More rows than that fill the GPU as
// they are, and the four ends would cost them (SPLIT false: no such choice, and
// fewer registers spilled).
template <int NF, bool SPLIT>
__global__ void __launch_bounds__(dbwd::kRowsFp32, dbwd::kRowsCtasPerSm) k_decode_bwd_rows(ViewTable vt,
                                                                                               dbwd::Args a,
                                                                                               int max_split_tiles) {
    extern __shared__ float4 smem4[];
    __shared__ float aPose[3 * UPS_MAX_VIEWS];
    const int end = a.rows ? (int)*a.n_rows : a.row_end;
    const int step = (int)gridDim.x * dbwd::kRowsFp32;
    const bool split = SPLIT && (end - a.row_begin + dbwd::kRowsFp32 - 1) / dbwd::kRowsFp32 <= max_split_tiles;
    if (!split && blockIdx.y) return;
    // the MLP of this CTA, the costliest first (-1: all)
    constexpr int kFirst = NF > 0 ? 0 : 1;
    const int y = (int)blockIdx.y + kFirst;
    const int only = !split ? -1 : y == 0 ? 3 : y == 1 ? 1 : y == 2 ? 2 : 0;
    auto does = [&](int g) { return !SPLIT || only < 0 || only == g; };
    float *sm = reinterpret_cast<float *>(smem4);
    const int n_out = dbwd::n_out(a.K, NF);
    const DecodeArgs da{a.A, a.K, NF, n_out, a.pos, a.afeat, a.offs, a.ascale, a.w1, a.b1, a.w2, a.b2, a.op_tanh};
    // W1 transposed [38][128] (inputs x hidden), b1, W2 [n_out][32], b2, and
    // the per-row input gradients dx [36][256 rows]
    float *sW1T = sm, *sb1 = sW1T + kDin * 4 * kH, *sW2 = sb1 + 4 * kH, *sb2 = sW2 + n_out * kH;
    float *sDXall = sb2 + ((n_out + 3) & ~3);
    load_weights_T(da, sW1T, sb1, sW2, sb2);
    const int V = vt.n;
    for (int i = threadIdx.x; i < 3 * V; i += blockDim.x) aPose[i] = 0.f;
    __syncthreads();
    const size_t NG = (size_t)a.A * a.K;
    float *sDX = sDXall + threadIdx.x;
    for (int base = a.row_begin + blockIdx.x * dbwd::kRowsFp32; base < end; base += step) {
        const bool valid = base + (int)threadIdx.x < end;
        const int row = a.rows && valid ? (int)a.rows[base + threadIdx.x] : base + (int)threadIdx.x;
        const int an = valid ? row / V : 0, v = valid ? row - an * V : 0;
        const int lr = row - a.row_begin;
        const DevView &cam = vt.v[v];
        const size_t gbase = (size_t)v * NG + (size_t)an * a.K;
        float x[kDinP], delta[3], dist;
        mlp_input(da, cam, an, x, delta, dist);
        if (a.s.X && valid && does(1)) {
            x[38] = 1.f;
#pragma unroll
            for (int i = 0; i < kDinP; ++i) a.s.X[(size_t)i * a.s.ld + lr] = x[i];
        }
        const float xt[6] = {x[kFin], x[kFin + 1], x[kFin + 2], x[kFin + 3], x[kFin + 4], x[kFin + 5]};
#pragma unroll
        for (int i = 0; i < kDX; ++i) sDX[i * dbwd::kRowsFp32] = 0.f;
        float dls[3] = {0.f, 0.f, 0.f};
        if (does(0)) bwd_group<0, NF>(a, da, sW1T, sb1, sW2, sb2, xt, an, valid, gbase, lr, sDX, dls);
        if (does(1)) bwd_group<1, NF>(a, da, sW1T, sb1, sW2, sb2, xt, an, valid, gbase, lr, sDX, dls);
        if (does(2)) bwd_group<2, NF>(a, da, sW1T, sb1, sW2, sb2, xt, an, valid, gbase, lr, sDX, dls);
        if (NF > 0 && does(3)) bwd_group<3, NF>(a, da, sW1T, sb1, sW2, sb2, xt, an, valid, gbase, lr, sDX, dls);
        float dx[kDX];
#pragma unroll
        for (int i = 0; i < kDX; ++i) dx[i] = sDX[i * dbwd::kRowsFp32];
        dbwd::row_epilogue(a, valid ? an : -1, v, gbase, dx, delta, dist, dls, aPose, does(0), does(1));
    }
    __syncthreads();
    dbwd::flush_pose(a, vt, aPose);
}

// Rows whose dL/dG is not all zero, for calls without MLP gradients.  A render
// backward reaches a few percent of a large map's Gaussians (a tracking request
// over 500k anchors: most rows are zero, and a zero row adds nothing), so one
// read of dL/dG (128 B a Gaussian at 16 channels, the bound of this kernel)
// saves the MLP backward of the others.  A warp a row, 32 rows one after another;
// the row's arrays are read until one is not zero.
constexpr int kLiveThreads = 256;
__global__ void __launch_bounds__(kLiveThreads) k_live_rows(dbwd::Args a, int V, int n_rows, uint32_t *__restrict__ rows,
                                                            uint32_t *__restrict__ n_live) {
    __shared__ uint32_t s_bits[kLiveThreads / 32];
    __shared__ uint32_t s_at;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int row0 = blockIdx.x * kLiveThreads + 32 * w;
    const size_t NG = (size_t)a.A * a.K;
    auto nonzero = [](float4 x) { return x.x != 0.f || x.y != 0.f || x.z != 0.f || x.w != 0.f; };  // NaN counts
    uint32_t bits = 0;
    for (int i = 0; i < 32 && row0 + i < n_rows; ++i) {
        const int an = (row0 + i) / V, v = row0 + i - an * V;
        const size_t g = (size_t)v * NG + (size_t)an * a.K;
        bool hit = false;
        if (lane < a.K)
            hit = nonzero(a.d_mean_op[g + lane]) || nonzero(a.d_scale[g + lane]) || nonzero(a.d_quat[g + lane]) ||
                  nonzero(a.d_color[g + lane]);
        const float4 *f = reinterpret_cast<const float4 *>(a.d_feat + g * a.NF);
        for (int k = lane; k < a.K * a.NF / 4 && !hit; k += 32) hit = nonzero(f[k]);
        if (__any_sync(0xffffffffu, hit)) bits |= 1u << i;
    }
    if (lane == 0) s_bits[w] = bits;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < kLiveThreads / 32; ++i) {
        const uint32_t c = __popc(s_bits[i]);
        before += i < w ? c : 0u;
        all += c;
    }
    if (all == 0) return;
    if (threadIdx.x == 0) s_at = atomicAdd(n_live, all);
    __syncthreads();
    if (bits >> lane & 1u) rows[s_at + before + __popc(bits & ((1u << lane) - 1u))] = (uint32_t)(row0 + lane);
}

// shared memory of the backward rows kernel
size_t bwd_rows_smem(int n_out) {
    return sizeof(float) * (kDin * 4 * kH + 4 * kH + n_out * kH + ((n_out + 3) & ~3) + kDX * dbwd::kRowsFp32);
}

size_t fwd_smem(int n_out, int warps) {
    return sizeof(float) * (kDin * 4 * kH + 4 * kH + (size_t)n_out * kH + ((n_out + 3) & ~3) +
                            (size_t)warps * kDin * kXT);
}

}  // namespace

cudaError_t launch_live_rows(const dbwd::Args &a, int V, uint32_t *rows, uint32_t *n_rows, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(n_rows, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    const int n = a.A * V;
    k_live_rows<<<(n + kLiveThreads - 1) / kLiveThreads, kLiveThreads, 0, st>>>(a, V, n, rows, n_rows);
    return cudaGetLastError();
}

cudaError_t launch_decode_bwd_rows_fp32(const ViewTable &vt, const dbwd::Args &a, int num_sms, cudaStream_t st) {
    const size_t smem = bwd_rows_smem(dbwd::n_out(a.K, a.NF));
    if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
    const int rows = a.row_end - a.row_begin;
    const int tiles = (rows + dbwd::kRowsFp32 - 1) / dbwd::kRowsFp32;
    const int blocks = std::max(1, std::min(tiles, num_sms * dbwd::kRowsCtasPerSm));
    // (of a list, whose length only the GPU knows, the kernel decides)
    const int max_split = num_sms * dbwd::kRowsCtasPerSm / 2;
    const bool split = a.rows || tiles <= max_split;
    const dim3 grid(blocks, split ? (a.NF > 0 ? 4 : 3) : 1);
#define UPS_DECB1(NFV, SPLITV)                                                                            \
    do {                                                                                                  \
        const cudaError_t e = allow_smem(k_decode_bwd_rows<NFV, SPLITV>, bwd_rows_smem(dbwd::n_out(16, NFV))); \
        if (e != cudaSuccess) return e;                                                                   \
        k_decode_bwd_rows<NFV, SPLITV><<<grid, dbwd::kRowsFp32, smem, st>>>(vt, a, max_split);            \
    } while (0)
#define UPS_DECB(NFV)              \
    do {                           \
        if (split)                 \
            UPS_DECB1(NFV, true);  \
        else                       \
            UPS_DECB1(NFV, false); \
    } while (0)
    switch (a.NF) {
        case 0: UPS_DECB(0); break;
        case 16: UPS_DECB(16); break;
        case 32: UPS_DECB(32); break;
        default: return cudaErrorInvalidValue;
    }
#undef UPS_DECB
#undef UPS_DECB1
    return cudaGetLastError();
}

cudaError_t launch_decode_fwd(const ViewTable &vt, int A, int K, int NF, const ups_anchors &anc,
                              const ups_mlp &mlp, const ups_gaussians &out, int op_tanh, int num_sms,
                              cudaStream_t st) {
    DecodeArgs a{A, K, NF, K * (11 + NF), anc.pos, anc.feat, anc.offsets, anc.scaling,
                 mlp.w1, mlp.b1, mlp.w2, mlp.b2, op_tanh};
    // as many warps as the weights leave room for (16 at 270 outputs, 15 at 430)
    int warps = kFwdWarps;
    while (warps > 1 && fwd_smem(a.n_out, warps) > kMaxSmem) --warps;
    // one CTA per SM.  Fewer than four rounds of tiles are split by MLP: 10k rows
    // 45 us (77 in tiles), 184k rows 191 (197); with more, sharing a tile's inputs
    // is worth more than even rounds (800k rows 675 against 721).  Eight warps at
    // least, to load the weights.
    const int tiles = (A * vt.n + kXT - 1) / kXT;
    const int split = tiles < 4 * num_sms * warps;
    const int items = split ? tiles * (NF > 0 ? 4 : 3) : tiles;
    warps = std::min(warps, std::max(8, (items + num_sms - 1) / num_sms));
    const size_t smem = fwd_smem(a.n_out, warps);
    if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
    const int blocks = std::max(1, std::min(items, num_sms));
    bool pair = K % 2 == 0;
    for (const void *p : {(const void *)out.mean_opacity, (const void *)out.scale, (const void *)out.quat,
                          (const void *)out.color, (const void *)out.feat})
        pair = pair && reinterpret_cast<uintptr_t>(p) % 32 == 0;
#define UPS_DEC1(NFV, PAIRV)                                                                       \
    do {                                                                                           \
        const cudaError_t e = allow_smem(k_decode_fwd<NFV, PAIRV>, kMaxSmem);                      \
        if (e != cudaSuccess) return e;                                                            \
        k_decode_fwd<NFV, PAIRV><<<blocks, 32 * warps, smem, st>>>(                                \
            vt, a, split, reinterpret_cast<float4 *>(out.mean_opacity),                            \
            reinterpret_cast<float4 *>(out.scale), reinterpret_cast<float4 *>(out.quat),           \
            reinterpret_cast<float4 *>(out.color), out.feat);                                      \
    } while (0)
#define UPS_DEC(NFV)              \
    do {                          \
        if (pair)                 \
            UPS_DEC1(NFV, true);  \
        else                      \
            UPS_DEC1(NFV, false); \
    } while (0)
    switch (NF) {
        case 0: UPS_DEC(0); break;
        case 16: UPS_DEC(16); break;
        case 32: UPS_DEC(32); break;
        default: return cudaErrorInvalidValue;
    }
#undef UPS_DEC
#undef UPS_DEC1
    return cudaGetLastError();
}

}  // namespace ups
