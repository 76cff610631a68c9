// Decode (Eq. 8-9) on the 5th-generation tensor cores (tcgen05), operands rounded
// to BF16, FP32 accumulation.
//
// One 128-thread CTA works on tiles of 128 (anchor, view) rows; thread t owns
// row t, which is also TMEM lane t.  Per tile:
//   Z[128 x 128] = X[128 x 48] . W1^T               (one MMA chain, all four MLPs)
//   H_g = act(Z_g + b1_g), g = 0..3                 (CUDA cores, to shared memory)
//   Y in chunks of up to 64 columns, two TMEM buffers: while a chunk's outputs
//   are activated and stored, the next one's MMAs run
// W2's rows lie in shared memory as the chunks want them: opacity, covariance and
// colour component-major with 16 slots per component (slot = Gaussian index k < K),
// so that each component of all K Gaussians is one aligned 16-column TMEM load;
// features in their own order (k, channel), which is the output's.
// Rows are view-major and a row's records follow the previous row's, so a warp's
// outputs are 32 pieces at a fixed stride: they go through a staging tile of the
// warp (rows of 128 bytes, padded) and out in 16-byte stores of which eight lanes
// fill 128 bytes of a row.
// Bound by the latency of that chain with two CTAs per SM: 800k rows (100k anchors x
// 10, 8 views) at 32 channels 0.574 ms for 1.54 GB of Gaussians (2.7 TB/s); one MMA
// round trip per MLP and chunk and 16-byte stores 160 bytes apart took 1.57 ms.
// 500k rows at 16 channels 0.313 ms (0.481).
#include <algorithm>

#include "common.cuh"
#include "umma.cuh"

namespace ups {

namespace {

using namespace umma;

constexpr int kTCRows = 128;
constexpr int kH = 32;
constexpr int kFin = 32;
constexpr int kDin = kFin + 6;
constexpr int kKin = 48;              // input width padded to the MMA K step
constexpr int kXB = 2 * kKin, kHB = 2 * kH;  // bytes per X and H row
constexpr uint32_t kTmemCols = 256;   // Z: [0, 128), Y buffers of 64: [128, 192), [192, 256)
constexpr uint32_t kYCol = 128;
constexpr int kYN = 64;               // columns of a Y chunk at most
constexpr int kFixed = 16 * 11;       // W2 rows of opacity, covariance and colour
constexpr int kStageF4 = 9;           // float4 per staged row: 8 and one of padding
constexpr int kWaitLimit = 1 << 22;

struct TcArgs {
    int A, K, NF;
    const float *pos, *afeat, *offs, *ascale;
    const float *w1, *b1, *w2, *b2;
    float4 *mean_op, *scale, *quat, *color;
    float4 *feat;
    int *err;
    int op_tanh;  // opacity = tanh(y) instead of sigmoid(y)
};

__device__ __forceinline__ float sig(float x) { return 1.f / (1.f + __expf(-x)); }
__device__ __forceinline__ float softplus(float x) { return x > 20.f ? x : log1pf(__expf(x)); }

// 8 values as BF16, 16 bytes
__device__ __forceinline__ uint4 pack8(const float *v) {
    uint4 r;
    uint32_t *w = &r.x;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t *>(&b);
    }
    return r;
}

struct TcLayout {
    int n_w2rows;  // W2 rows in shared memory
    int oX, oH, oW1, oW2, ob1, ob2, total;
};

__host__ __device__ inline TcLayout tc_layout(int K, int NF) {
    TcLayout L;
    L.n_w2rows = kFixed + K * NF;
    int o = 0;
    auto take = [&](int bytes) { int r = o; o += (bytes + 1023) & ~1023; return r; };
    // X, and (once Z is there) the warps' staging tiles
    const int stage = (kTCRows / 32) * 32 * kStageF4 * 16;
    L.oX = take(kTCRows * kXB > stage ? kTCRows * kXB : stage);
    L.oH = take(4 * kTCRows * kHB);
    L.oW1 = take(4 * kH * kXB);
    L.oW2 = take(L.n_w2rows * kHB);
    L.ob1 = take(4 * kH * 4);
    L.ob2 = take(L.n_w2rows * 4);
    L.total = o;
    return L;
}

template <int NF>
__global__ void __launch_bounds__(kTCRows, 2) k_decode_fwd_tc(ViewTable vt, TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t bar[3];  // Z, the two Y buffers
    __shared__ uint32_t tmem_base;
    const int K = a.K;
    const TcLayout L = tc_layout(K, NF);
    unsigned char *X = smem + L.oX, *Hs = smem + L.oH, *W1 = smem + L.oW1, *W2 = smem + L.oW2;
    float *b1 = reinterpret_cast<float *>(smem + L.ob1), *b2 = reinterpret_cast<float *>(smem + L.ob2);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    float4 *stage = reinterpret_cast<float4 *>(X) + warp * 32 * kStageF4;
    // ---- weights: W1 rows per hidden unit (K-major over inputs), W2 as above
    for (int i = tid; i < 4 * kH * (kKin / 8); i += kTCRows) {
        const int h = i / (kKin / 8), q = i - h * (kKin / 8);
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = 8 * q + c < kDin ? a.w1[h * kDin + 8 * q + c] : 0.f;
        *reinterpret_cast<uint4 *>(W1 + kmajor_offset(h, 8 * q, kXB, 2)) = pack8(v);
    }
    for (int i = tid; i < 4 * kH; i += kTCRows) b1[i] = a.b1[i];
    for (int i = tid; i < L.n_w2rows * (kH / 8); i += kTCRows) {
        const int rr = i / (kH / 8), q = i - rr * (kH / 8);
        int o = -1;  // the output of row rr (-1: an unused slot)
        if (rr >= kFixed) {
            o = 11 * K + rr - kFixed;
        } else {
            const int g = rr < 16 ? 0 : rr < 16 * 8 ? 1 : 2, base = g == 0 ? 0 : g == 1 ? 16 : 16 * 8;
            const int m = g == 0 ? 1 : g == 1 ? 7 : 3, r0 = g == 0 ? 0 : g == 1 ? K : 8 * K;
            const int c = (rr - base) >> 4, k = (rr - base) & 15;
            if (k < K) o = r0 + m * k + c;
        }
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = o >= 0 ? a.w2[(size_t)o * kH + 8 * q + c] : 0.f;
        *reinterpret_cast<uint4 *>(W2 + kmajor_offset(rr, 8 * q, kHB, 2)) = pack8(v);
        if (q == 0) b2[rr] = o >= 0 ? a.b2[o] : 0.f;
    }
    if (tid == 0)
        for (int i = 0; i < 3; ++i) mbar_init(&bar[i], 1);
    if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_base;
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    uint32_t phase[3] = {0u, 0u, 0u};
    const int rows = a.A * vt.n;
    const int ntiles = (rows + kTCRows - 1) / kTCRows;
    const int nchunks = 4 + (K * NF + kYN - 1) / kYN;
    // Y chunk i: opacity, covariance components 0-3 and 4-6, colour, then features
    auto chunk_row = [&](int i) { return i == 0 ? 0 : i == 1 ? 16 : i == 2 ? 80 : i == 3 ? 128 : kFixed + kYN * (i - 4); };
    auto chunk_n = [&](int i) { return i == 0 ? 16 : i == 1 ? 64 : i < 4 ? 48 : min(kYN, K * NF - kYN * (i - 4)); };
    // warp 0: the MMAs of chunk i into buffer i & 1
    auto issue = [&](int i) {
        const int g = i == 0 ? 0 : i < 3 ? 1 : i == 3 ? 2 : 3;
        const uint64_t da = desc(smem_addr(Hs + g * kTCRows * kHB), kHB),
                       db = desc(smem_addr(W2) + (uint32_t)(chunk_row(i) * kHB), kHB);
        const uint32_t id = idesc(kBF16, kTCRows, 0) + ((uint32_t)(chunk_n(i) >> 3) << 17);
#pragma unroll
        for (int ks = 0; ks < kH / 16; ++ks)
            mma_warp<kBF16>(tmem + kYCol + kYN * (i & 1), da + 16u * ks, db + 16u * ks, id, ks > 0 ? 1u : 0u);
        commit_warp(&bar[1 + (i & 1)]);
    };
    bool ok = true;
    int issued = 0, waited = 0;  // commits of this CTA and those waited for
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const int row = tile * kTCRows + tid, row0 = tile * kTCRows + 32 * warp;
        const bool valid = row < rows;
        const int v = valid ? row / a.A : 0, an = valid ? row - v * a.A : 0;
        const DevView &cam = vt.v[v];
        // ---- MLP input of this row
        {
            float x[kKin];
            const float4 *f4 = reinterpret_cast<const float4 *>(a.afeat + (size_t)an * kFin);
#pragma unroll
            for (int i = 0; i < kFin / 4; ++i) {
                float4 f = f4[i];
                x[4 * i] = f.x;
                x[4 * i + 1] = f.y;
                x[4 * i + 2] = f.z;
                x[4 * i + 3] = f.w;
            }
            float oc[3], r[3];
#pragma unroll
            for (int i = 0; i < 3; ++i)
                oc[i] = -(cam.R[i] * cam.t[0] + cam.R[3 + i] * cam.t[1] + cam.R[6 + i] * cam.t[2]);
#pragma unroll
            for (int i = 0; i < 3; ++i) r[i] = a.pos[3 * an + i] - oc[i];
            const float dist = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
            const float id = 1.f / dist;
#pragma unroll
            for (int i = 0; i < 3; ++i) x[kFin + i] = r[i] * id;
            x[kFin + 3] = dist;
            float s, c;
            sincospif(cam.t_norm, &s, &c);
            x[kFin + 4] = s;
            x[kFin + 5] = c;
#pragma unroll
            for (int i = kDin; i < kKin; ++i) x[i] = 0.f;
            if (!valid)
#pragma unroll
                for (int i = 0; i < kDin; ++i) x[i] = 0.f;
            if (tile != blockIdx.x) __syncthreads();  // the staging tiles of the last tile are read
#pragma unroll
            for (int q = 0; q < kKin / 8; ++q)
                *reinterpret_cast<uint4 *>(X + kmajor_offset(tid, 8 * q, kXB, 2)) = pack8(&x[8 * q]);
        }
        fence_async_smem();
        fence_before();
        __syncthreads();
        // Z = X . W1^T -> TMEM columns [0, 128)
        if (warp == 0) {
            fence_after();
            const uint64_t da = desc(smem_addr(X), kXB), db = desc(smem_addr(W1), kXB);
#pragma unroll
            for (int ks = 0; ks < kKin / 16; ++ks)
                mma_warp<kBF16>(tmem, da + 16u * ks, db + 16u * ks, idesc(kBF16, kTCRows, 4 * kH), ks > 0 ? 1u : 0u);
            commit_warp(&bar[0]);
        }
        ++issued;
        bool bad = !mbar_wait(&bar[0], phase[0], kWaitLimit);
        phase[0] ^= 1u;
        if (__syncthreads_or(bad)) {
            ok = false;
            break;
        }
        ++waited;
        fence_after();
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            if (g == 3 && NF == 0) continue;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float h[16];
                tmem_ld16(lane_addr + 32 * g + 16 * p, h);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float zz = h[j] + b1[g * kH + 16 * p + j];
                    h[j] = g < 3 ? fmaxf(zz, 0.f) : softplus(zz);
                }
                unsigned char *Hg = Hs + g * kTCRows * kHB;
                *reinterpret_cast<uint4 *>(Hg + kmajor_offset(tid, 16 * p, kHB, 2)) = pack8(&h[0]);
                *reinterpret_cast<uint4 *>(Hg + kmajor_offset(tid, 16 * p + 8, kHB, 2)) = pack8(&h[8]);
            }
        }
        fence_async_smem();
        fence_before();
        __syncthreads();
        if (warp == 0) {
            fence_after();
            issue(0);
            issue(1);
        }
        issued += 2;
        // the warp's staged float4 (rows of up to 8) to columns [c0, c0 + n) of its rows
        // of dst, `stride` float4 a row
        auto flush = [&](float4 *dst, int stride, int c0, int n) {
            __syncwarp();
            const int c = lane & 7;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = 4 * i + (lane >> 3);
                if (c < n && row0 + r < rows) dst[(size_t)(row0 + r) * stride + c0 + c] = stage[r * kStageF4 + c];
            }
            __syncwarp();
        };
        // K records of the row in two halves of up to 8 Gaussians
        auto put_records = [&](float4 *dst, auto &&rec) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (8 * h >= K) continue;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (8 * h + k < K) stage[lane * kStageF4 + k] = rec(8 * h + k);
                flush(dst, K, 8 * h, min(8, K - 8 * h));
            }
        };
        float qw[16];  // quaternion w, from the chunk before the other components'
        for (int i = 0; i < nchunks; ++i) {
            bad = !mbar_wait(&bar[1 + (i & 1)], i & 1 ? phase[2] : phase[1], kWaitLimit);
            if (i & 1)
                phase[2] ^= 1u;
            else
                phase[1] ^= 1u;
            fence_after();
            const uint32_t yc = lane_addr + kYCol + kYN * (i & 1);
            const int nq = chunk_n(i) >> 4;
            float y[4][16];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nq) tmem_ld16(yc + 16 * q, y[q]);
            fence_before();
            if (__syncthreads_or(bad)) {
                ok = false;
                break;
            }
            ++waited;
            if (i + 2 < nchunks) {  // the buffer is read
                if (warp == 0) {
                    fence_after();
                    issue(i + 2);
                }
                ++issued;
            }
            const float *bb = b2 + chunk_row(i);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nq)
#pragma unroll
                    for (int k = 0; k < 16; ++k) y[q][k] += bb[16 * q + k];
            if (i == 0) {
                // opacity, and the mean
                const float px = a.pos[3 * an], py = a.pos[3 * an + 1], pz = a.pos[3 * an + 2];
                const float *o3 = a.offs + (size_t)an * K * 3;
                put_records(a.mean_op, [&](int k) {
                    return make_float4(px + o3[3 * k], py + o3[3 * k + 1], pz + o3[3 * k + 2],
                                       a.op_tanh ? tanhf(y[0][k]) : sig(y[0][k]));
                });
            } else if (i == 1) {
                // scale x, y, z and quaternion w
                const float lx = a.ascale[3 * an], ly = a.ascale[3 * an + 1], lz = a.ascale[3 * an + 2];
                put_records(a.scale, [&](int k) {
                    return make_float4(lx * sig(y[0][k]), ly * sig(y[1][k]), lz * sig(y[2][k]), 0.f);
                });
#pragma unroll
                for (int k = 0; k < 16; ++k) qw[k] = y[3][k];
            } else if (i == 2) {
                put_records(a.quat, [&](int k) { return make_float4(qw[k], y[0][k], y[1][k], y[2][k]); });
            } else if (i == 3) {
                put_records(a.color, [&](int k) {
                    return make_float4(sig(y[0][k]), sig(y[1][k]), sig(y[2][k]), 0.f);
                });
            } else {
                // up to 64 consecutive floats of the row's features, 32 at a time
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (2 * h >= nq) continue;
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        if (2 * h + q < nq)
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                stage[lane * kStageF4 + 4 * q + c] =
                                    make_float4(y[2 * h + q][4 * c], y[2 * h + q][4 * c + 1], y[2 * h + q][4 * c + 2],
                                                y[2 * h + q][4 * c + 3]);
                    flush(a.feat, K * NF / 4, (kYN / 4) * (i - 4) + 8 * h, min(8, 4 * nq - 8 * h));
                }
            }
        }
    }
    if (!ok) {
        if (tid == 0) atomicExch(a.err, 1);
        // MMAs that a wait gave up on may still run: a bounded wait before their memory goes
        if (issued > waited)
            for (int i = 0; i < 3; ++i) mbar_wait(&bar[i], phase[i] ^ 1u, kWaitLimit);
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace

// (of the most Gaussians an anchor can have)
size_t decode_tc_smem_bytes(int NF) { return (size_t)tc_layout(16, NF).total; }

cudaError_t launch_decode_fwd_tc(const ViewTable &vt, int A, int K, int NF, const ups_anchors &anc,
                                 const ups_mlp &mlp, const ups_gaussians &out, int op_tanh, int *err,
                                 int num_sms, cudaStream_t st) {
    TcArgs a{A, K, NF, anc.pos, anc.feat, anc.offsets, anc.scaling, mlp.w1, mlp.b1, mlp.w2, mlp.b2,
             reinterpret_cast<float4 *>(out.mean_opacity), reinterpret_cast<float4 *>(out.scale),
             reinterpret_cast<float4 *>(out.quat), reinterpret_cast<float4 *>(out.color),
             reinterpret_cast<float4 *>(out.feat), err, op_tanh};
    if (K < 1 || K > 16) return cudaErrorInvalidValue;
    const int rows = A * vt.n;
    const int tiles = (rows + kTCRows - 1) / kTCRows;
    // two CTAs per SM (256 of its 512 TMEM columns each) overlap one's waits with the
    // other's epilogue; more would wait for TMEM
    const size_t smem = (size_t)tc_layout(K, NF).total;
    if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
    const int blocks = std::max(1, std::min(tiles, num_sms * 2));
#define UPS_TC(NFV)                                                                                               \
    do {                                                                                                          \
        const cudaError_t e = allow_smem(k_decode_fwd_tc<NFV>, decode_tc_smem_bytes(NFV));                        \
        if (e != cudaSuccess) return e;                                                                           \
        k_decode_fwd_tc<NFV><<<blocks, kTCRows, smem, st>>>(vt, a);                                               \
    } while (0)
    switch (NF) {
        case 0: UPS_TC(0); break;
        case 16: UPS_TC(16); break;
        case 32: UPS_TC(32); break;
        default: return cudaErrorInvalidValue;
    }
#undef UPS_TC
    return cudaGetLastError();
}

}  // namespace ups
