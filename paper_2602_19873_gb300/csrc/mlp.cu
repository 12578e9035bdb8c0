// Learned smoothing-length start (not in the paper): a small MLP maps
// per-cluster SFC density features to log(h / e64), trained on h values of
// the exact iteration.  8 inputs -> 64 -> 64 -> 64 (SiLU) -> 1, BF16 operands
// on the tensor cores (mma.sync m16n8k16, FP32 accumulate), FP32 master
// weights and Adam.
//
// Features of cluster c (padded SFC order; e(B) = largest side of box B,
// e8 = its cluster box, e64 = its super-cluster box, e512 / e4096 = boxes of
// the 8 / 64 super-clusters around it inside its system, L = largest side
// of the system box, N_s = particles of the system):
//   log(e8/e64), log(e512/e64), log(e4096/e64), log(ex/e8), log(ey/e8),
//   log(ez/e8), log(count/M), log(e64/L) + log(N_s)/3.
// Target: log(mean h of the cluster / e64); the start h of a particle is
// e64 * exp(prediction of its cluster).
#include <cstdint>

#include <cuda_bf16.h>

#include "nl_internal.cuh"
#include "mlp.cuh"

namespace nlg {

__host__ __device__ __forceinline__ int64_t min_i64(int64_t a, int64_t b) { return a < b ? a : b; }

// ---------------------------------------------------------------------------
// Features and targets
// ---------------------------------------------------------------------------
__device__ __forceinline__ float box_extent(const float4 &lo, const float4 &hi)
{
    return fmaxf(fmaxf(hi.x - lo.x, hi.y - lo.y), hi.z - lo.z);
}

__global__ void k_sc_boxes(uint32_t nsc, const float4 *__restrict__ clo, const float4 *__restrict__ chi,
                           float4 *__restrict__ slo, float4 *__restrict__ shi)
{
    uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nsc) return;
    float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    float4 hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
    for (int k = 0; k < kSC; ++k) {
        float4 a = clo[s * kSC + k], b = chi[s * kSC + k];
        lo.x = fminf(lo.x, a.x); lo.y = fminf(lo.y, a.y); lo.z = fminf(lo.z, a.z);
        hi.x = fmaxf(hi.x, b.x); hi.y = fmaxf(hi.y, b.y); hi.z = fmaxf(hi.z, b.z);
    }
    slo[s] = lo;
    shi[s] = hi;
}

__device__ __forceinline__ float region_extent(const float4 *slo, const float4 *shi, int64_t a,
                                               int64_t b)
{
    float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    float4 hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
    for (int64_t s = a; s < b; ++s) {
        float4 p = slo[s], q = shi[s];
        lo.x = fminf(lo.x, p.x); lo.y = fminf(lo.y, p.y); lo.z = fminf(lo.z, p.z);
        hi.x = fmaxf(hi.x, q.x); hi.y = fmaxf(hi.y, q.y); hi.z = fmaxf(hi.z, q.z);
    }
    return box_extent(lo, hi);
}

// one thread per super-cluster: features of its 8 clusters and e64
__global__ void k_features(uint32_t nsc, int M, SysTables t, const float4 *__restrict__ clo,
                           const float4 *__restrict__ chi, const float4 *__restrict__ slo,
                           const float4 *__restrict__ shi, const uint32_t *__restrict__ perm_pad,
                           float *__restrict__ X, float *__restrict__ e64out)
{
    uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nsc) return;
    const uint32_t scp = kSC * M;
    const uint32_t sy = sys_of(t.pad_off, t.nsys, s * scp);
    const int64_t s0 = t.pad_off[sy] / scp, s1 = t.pad_off[sy + 1] / scp;
    const DevBox &b = t.box[sy];
    const float L = fmaxf(fmaxf(b.len[0], b.len[1]), b.len[2]);
    const float ns = (float)(t.off[sy + 1] - t.off[sy]);
    const float fl = 1e-7f * L;  // floor of every length
    const float e64 = fmaxf(box_extent(slo[s], shi[s]), fl);
    const float e512 = fmaxf(region_extent(slo, shi, max(s0, (int64_t)s - 3), min(s1, (int64_t)s + 5)), fl);
    const float e4k = fmaxf(region_extent(slo, shi, max(s0, (int64_t)s - 31), min(s1, (int64_t)s + 33)), fl);
    e64out[s] = e64;
    const float dens = logf(e64 / L) + logf(ns) * (1.f / 3.f);
    for (int k = 0; k < kSC; ++k) {
        const uint32_t c = s * kSC + k;
        uint32_t cnt = 0;
        for (int q = 0; q < M; ++q) cnt += perm_pad[c * M + q] != 0xffffffffu;
        float *x = X + (size_t)c * kMlpF;
        if (cnt == 0) {
            for (int f = 0; f < kMlpF; ++f) x[f] = 0.f;
            continue;
        }
        const float4 lo = clo[c], hi = chi[c];
        const float ex = fmaxf(hi.x - lo.x, fl), ey = fmaxf(hi.y - lo.y, fl), ez = fmaxf(hi.z - lo.z, fl);
        const float e8 = fmaxf(fmaxf(ex, ey), ez);
        x[0] = logf(e8 / e64);
        x[1] = logf(e512 / e64);
        x[2] = logf(e4k / e64);
        x[3] = logf(ex / e8);
        x[4] = logf(ey / e8);
        x[5] = logf(ez / e8);
        x[6] = logf((float)cnt / (float)M);
        x[7] = dens;
    }
}

// target of cluster c: log(mean h of its real particles / e64); w = 0 for
// empty clusters
__global__ void k_targets(uint32_t ncl, int M, const uint32_t *__restrict__ perm_pad,
                          const float *__restrict__ h, const float *__restrict__ e64,
                          float *__restrict__ y, float *__restrict__ w)
{
    uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncl) return;
    float s = 0.f;
    int cnt = 0;
    for (int q = 0; q < M; ++q) {
        uint32_t o = perm_pad[c * M + q];
        if (o != 0xffffffffu) {
            s += h[o];
            ++cnt;
        }
    }
    y[c] = cnt ? logf(s / cnt / e64[c / kSC]) : 0.f;
    w[c] = cnt ? 1.f : 0.f;
}

// start h of every real particle from its cluster's prediction
__global__ void k_apply_h0(uint32_t npad, int M, const uint32_t *__restrict__ perm_pad,
                           const float *__restrict__ pred, const float *__restrict__ e64,
                           float *__restrict__ hq)
{
    uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npad) return;
    const uint32_t c = k / M;
    float h = 0.f;
    if (perm_pad[k] != 0xffffffffu) {
        float p = fminf(fmaxf(pred[c], -20.f), 20.f);
        h = e64[c / kSC] * expf(p);
        if (!(h > 0.f) || !isfinite(h)) h = e64[c / kSC];
    }
    hq[k] = h;
}

cudaError_t mlp_features(uint32_t nsc, int M, const SysTables &t, const float4 *clo,
                         const float4 *chi, const uint32_t *perm_pad, float4 *slo, float4 *shi,
                         float *X, float *e64, cudaStream_t s)
{
    k_sc_boxes<<<(nsc + 255) / 256, 256, 0, s>>>(nsc, clo, chi, slo, shi);
    k_features<<<(nsc + 127) / 128, 128, 0, s>>>(nsc, M, t, clo, chi, slo, shi, perm_pad, X, e64);
    return cudaGetLastError();
}

cudaError_t mlp_targets(uint32_t ncl, int M, const uint32_t *perm_pad, const float *h,
                        const float *e64, float *y, float *w, cudaStream_t s)
{
    k_targets<<<(ncl + 255) / 256, 256, 0, s>>>(ncl, M, perm_pad, h, e64, y, w);
    return cudaGetLastError();
}

cudaError_t mlp_apply_h0(uint32_t npad, int M, const uint32_t *perm_pad, const float *pred,
                         const float *e64, float *hq, cudaStream_t s)
{
    k_apply_h0<<<(npad + 255) / 256, 256, 0, s>>>(npad, M, perm_pad, pred, e64, hq);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Tensor-core building blocks
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// D += A (16x16, row) * B (16x8, col); BF16 operands, FP32 accumulators
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four 8x8 matrices of 16-bit elements from shared memory: lane l gives the
// address of row l % 8 of matrix l / 8; plain: lane (g, t) = (l / 4, l % 4) gets
// elements (g, 2t), (g, 2t + 1) of each matrix; trans: (2t, g), (2t + 1, g).
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}

__device__ __forceinline__ void ldm4t(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + expf(-z)); }

// silu and its derivative from one exponential
__device__ __forceinline__ float silu_d(float z, float &ds)
{
    const float e = 1.f + expf(-z), s = 1.f / e;
    ds = s * (1.f + z * (1.f - s));
    return z / e;
}

// Shared-memory copy of the network: BF16 weights row-major (out x in), FP32
// biases and output row.  Rows are padded by 16 bytes, so that the eight rows of
// an ldmatrix lie in different banks; products with the transposed weights read
// the same copy with ldmatrix.trans.
constexpr int kLd = kMlpH + 8, kLdX = 24;
struct alignas(16) MlpSmem {
    __nv_bfloat16 w1[kMlpH][kLdX];        // inputs padded 8 -> 16 with zeros
    __nv_bfloat16 w2[kMlpH][kLd], w3[kMlpH][kLd];
    float b1[kMlpH], b2[kMlpH], b3[kMlpH], w4[kMlpH];
    float b4;
};

__device__ void load_net(MlpSmem &S, const float *__restrict__ P)
{
    const float *W1 = P, *B1 = W1 + kMlpH * kMlpF, *W2 = B1 + kMlpH, *B2 = W2 + kMlpH * kMlpH;
    const float *W3 = B2 + kMlpH, *B3 = W3 + kMlpH * kMlpH, *W4 = B3 + kMlpH, *B4 = W4 + kMlpH;
    for (int t = threadIdx.x; t < kMlpH * kMlpH; t += blockDim.x) {
        const int o = t / kMlpH, i = t % kMlpH;
        S.w2[o][i] = __float2bfloat16_rn(W2[t]);
        S.w3[o][i] = __float2bfloat16_rn(W3[t]);
    }
    for (int t = threadIdx.x; t < kMlpH * 16; t += blockDim.x) {
        const int o = t / 16, i = t % 16;
        S.w1[o][i] = __float2bfloat16_rn(i < kMlpF ? W1[o * kMlpF + i] : 0.f);
    }
    for (int t = threadIdx.x; t < kMlpH; t += blockDim.x) {
        S.b1[t] = B1[t];
        S.b2[t] = B2[t];
        S.b3[t] = B3[t];
        S.w4[t] = __bfloat162float(__float2bfloat16_rn(W4[t]));
    }
    if (threadIdx.x == 0) S.b4 = B4[0];
}

// C tiles (16 rows x 64) -> A fragments (4 k-blocks of 16) after activation
__device__ __forceinline__ void to_afrag(const float (&h)[8][4], uint32_t (&A)[4][4])
{
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        A[kk][0] = pack_bf16(h[2 * kk][0], h[2 * kk][1]);
        A[kk][1] = pack_bf16(h[2 * kk][2], h[2 * kk][3]);
        A[kk][2] = pack_bf16(h[2 * kk + 1][0], h[2 * kk + 1][1]);
        A[kk][3] = pack_bf16(h[2 * kk + 1][2], h[2 * kk + 1][3]);
    }
}

// z = A(16x64) * W^T + b, W row-major [64][64] in shared memory
__device__ __forceinline__ void dense64(const uint32_t (&A)[4][4], const __nv_bfloat16 (&W)[kMlpH][kLd],
                                       const float *b, float (&z)[8][4])
{
    const unsigned lane = lane_id(), t = lane & 3;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        z[j][0] = b[8 * j + 2 * t];
        z[j][1] = b[8 * j + 2 * t + 1];
        z[j][2] = z[j][0];
        z[j][3] = z[j][1];
#pragma unroll
        for (int kk = 0; kk < 4; kk += 2) {
            uint32_t B[4];
            ldm4(B, &W[8 * j + (lane & 7)][16 * kk + 8 * (lane >> 3)]);
            mma16816(z[j], A[kk], B[0], B[1]);
            mma16816(z[j], A[kk + 1], B[2], B[3]);
        }
    }
}

// z = A0(16x16, inputs) * W1^T + b1
__device__ __forceinline__ void dense_in(const uint32_t (&a0)[4], const MlpSmem &S, float (&z)[8][4])
{
    const unsigned lane = lane_id(), t = lane & 3;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        uint32_t B[4];  // n-tiles j and j + 1
        ldm4(B, &S.w1[8 * j + (lane & 7) + 8 * (lane >> 4)][8 * ((lane >> 3) & 1)]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            z[j + e][0] = S.b1[8 * (j + e) + 2 * t];
            z[j + e][1] = S.b1[8 * (j + e) + 2 * t + 1];
            z[j + e][2] = z[j + e][0];
            z[j + e][3] = z[j + e][1];
            mma16816(z[j + e], a0, B[2 * e], B[2 * e + 1]);
        }
    }
}

// y = b4 + sum_k w4[k] h3[k] of rows g and g + 8; h3 rounded to BF16 like every
// operand (h: this lane's activations, rounded here)
__device__ __forceinline__ void output_row(const MlpSmem &S, float (&h)[8][4], float (&pred)[2])
{
    const unsigned t = lane_id() & 3;
    float p0 = 0.f, p1 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float w0 = S.w4[8 * j + 2 * t], w1 = S.w4[8 * j + 2 * t + 1];
#pragma unroll
        for (int q = 0; q < 4; ++q) h[j][q] = __bfloat162float(__float2bfloat16_rn(h[j][q]));
        p0 += w0 * h[j][0] + w1 * h[j][1];
        p1 += w0 * h[j][2] + w1 * h[j][3];
    }
    p0 += __shfl_xor_sync(0xffffffffu, p0, 1);
    p0 += __shfl_xor_sync(0xffffffffu, p0, 2);
    p1 += __shfl_xor_sync(0xffffffffu, p1, 1);
    p1 += __shfl_xor_sync(0xffffffffu, p1, 2);
    pred[0] = p0 + S.b4;
    pred[1] = p1 + S.b4;
}

// ---------------------------------------------------------------------------
// Inference: one warp per 16 samples, a persistent grid (every block converts
// the network once).  Bound by the FP32 arithmetic of the activations.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 2) k_mlp_predict(int64_t n, const float *__restrict__ X,
                                                     const float *__restrict__ P,
                                                     float *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpSmem &S = *reinterpret_cast<MlpSmem *>(mlp_smem);
    load_net(S, P);
    __syncthreads();
    const unsigned lane = lane_id(), g = lane >> 2, t = lane & 3;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t tile = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); tile * 16 < n;
         tile += warps) {
        const int64_t r0 = tile * 16;
        const int nrows = (int)min_i64(16, n - r0);
        const float *x = X + r0 * kMlpF;
        const bool va = (int)g < nrows, vb = (int)g + 8 < nrows;
        const uint32_t a0[4] = {
            pack_bf16(va ? x[g * kMlpF + 2 * t] : 0.f, va ? x[g * kMlpF + 2 * t + 1] : 0.f),
            pack_bf16(vb ? x[(g + 8) * kMlpF + 2 * t] : 0.f, vb ? x[(g + 8) * kMlpF + 2 * t + 1] : 0.f), 0u, 0u};
        float z[8][4], pred[2];
        uint32_t A[4][4];
        auto act = [&]() {
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) z[j][q] = silu_f(z[j][q]);
        };
        dense_in(a0, S, z);
        act();
        to_afrag(z, A);
        dense64(A, S.w2, S.b2, z);
        act();
        to_afrag(z, A);
        dense64(A, S.w3, S.b3, z);
        act();
        output_row(S, z, pred);
        if (t == 0) {
            if (va) out[r0 + g] = pred[0];
            if (vb) out[r0 + g + 8] = pred[1];
        }
    }
}

// ---------------------------------------------------------------------------
// Training: each CTA (4 warps) takes 64-sample tiles of the minibatch and
// accumulates its gradient in registers (warp w owns output rows 16w..16w+15
// of every weight matrix); the CTA's gradient goes to its own slot of
// `partial`, and k_mlp_reduce_adam sums the slots in a fixed order.
// Activations and deltas lie in shared memory as BF16 rows (padded as the
// weights) and reach the tensor cores by ldmatrix, transposed for the weight
// gradients; the derivatives of the activations stay with the thread that made
// them.  95 KB of shared memory: two CTAs per SM.  With 16-bit loads of the
// fragments, activations evaluated three times over and one 64-sample tile per CTA
// (so that every tile converted the network and wrote a gradient slot), the
// gradient over 262144 samples took 1.25 ms; it takes 0.27 ms now (train kernel 1.08
// -> 0.26 ms, sum of the slots 0.167 -> 0.008 ms, predictions 0.134 -> 0.079 ms).
// ---------------------------------------------------------------------------
struct alignas(16) TrainSmem {
    MlpSmem net;
    __nv_bfloat16 h[2][64][kLd];          // h1, h2 (BF16, as the forward used them)
    __nv_bfloat16 d[2][64][kLd];          // dZ of the current and next layer
    __nv_bfloat16 x[64][kLdX];            // inputs, padded
    float4 ds[2][8][128];                 // derivatives of the first two activations, per thread
    float dy[64];
};

size_t mlp_train_smem() { return sizeof(TrainSmem); }
size_t mlp_predict_smem() { return sizeof(MlpSmem); }

// stripe gradient: G[o in 16w..16w+15][i] += sum_r D[r][o] * Hin[r][i], i over
// NT n-tiles of 8 (K = 64 samples)
template <int NT, int LD>
__device__ __forceinline__ void grad_stripe(const __nv_bfloat16 (*D)[kLd],
                                            const __nv_bfloat16 (*Hin)[LD], float (&G)[NT][4])
{
    const unsigned lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned l8 = lane & 7, m1 = (lane >> 3) & 1, m2 = lane >> 4;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        uint32_t A[4];
        ldm4t(A, &D[16 * kk + 8 * m2 + l8][16 * w + 8 * m1]);
#pragma unroll
        for (int j = 0; j < NT; j += 2) {
            uint32_t B[4];
            ldm4t(B, &Hin[16 * kk + 8 * m1 + l8][8 * j + 8 * m2]);
            mma16816(G[j], A, B[0], B[1]);
            mma16816(G[j + 1], A, B[2], B[3]);
        }
    }
}

// dH (16 rows of this warp) = dZ (rows) * W
__device__ __forceinline__ void back64(const __nv_bfloat16 (*D)[kLd], int row0,
                                      const __nv_bfloat16 (&W)[kMlpH][kLd], float (&dh)[8][4])
{
    const unsigned lane = lane_id();
    const unsigned l8 = lane & 7, m1 = (lane >> 3) & 1, m2 = lane >> 4;
    uint32_t A[4][4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) ldm4(A[kk], &D[row0 + 8 * m1 + l8][16 * kk + 8 * m2]);
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
#pragma unroll
        for (int q = 0; q < 4; ++q) dh[j][q] = dh[j + 1][q] = 0.f;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            uint32_t B[4];
            ldm4t(B, &W[16 * kk + 8 * m1 + l8][8 * j + 8 * m2]);
            mma16816(dh[j], A[kk], B[0], B[1]);
            mma16816(dh[j + 1], A[kk], B[2], B[3]);
        }
    }
}

// A fragments of this warp's 16 rows -> BF16 rows in shared memory
__device__ __forceinline__ void store_rows(__nv_bfloat16 (*H)[kLd], int row0, const uint32_t (&A)[4][4])
{
    const unsigned lane = lane_id(), g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        *reinterpret_cast<uint32_t *>(&H[row0 + g][16 * kk + 2 * t]) = A[kk][0];
        *reinterpret_cast<uint32_t *>(&H[row0 + g + 8][16 * kk + 2 * t]) = A[kk][1];
        *reinterpret_cast<uint32_t *>(&H[row0 + g][16 * kk + 8 + 2 * t]) = A[kk][2];
        *reinterpret_cast<uint32_t *>(&H[row0 + g + 8][16 * kk + 8 + 2 * t]) = A[kk][3];
    }
}

// idx: the samples of the minibatch; NULL: samples 0 .. nb - 1
__global__ void __launch_bounds__(128, 2) k_mlp_train(int64_t nb, const int64_t *__restrict__ idx,
                                                      const float *__restrict__ X,
                                                      const float *__restrict__ Y,
                                                      const float *__restrict__ Wt,
                                                      const float *__restrict__ P, float inv_n,
                                                      float *__restrict__ partial,
                                                      float *__restrict__ loss_out)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(mlp_smem);
    load_net(S.net, P);
    const unsigned lane = lane_id(), g = lane >> 2, t = lane & 3, w = threadIdx.x >> 5;
    const int row0 = 16 * w;
    float gW1[2][4] = {}, gW2[8][4] = {}, gW3[8][4] = {}, gW4[8][2] = {};
    float gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, gb4 = 0.f, lsum = 0.f;
    auto sample = [&](int64_t k) { return idx ? idx[k] : k; };
    // bias gradient of output 16w + lane % 16: lanes l and l + 16 hold halves
    auto bias_sum = [&](const __nv_bfloat16 (*D)[kLd]) {
        const int o = row0 + (lane & 15);
        float sb = 0.f;
        for (int r = (lane >> 4); r < 64; r += 2) sb += __bfloat162float(D[r][o]);
        return sb;
    };
    __syncthreads();
    for (int64_t tile = blockIdx.x; tile * 64 < nb; tile += gridDim.x) {
        const int64_t base = tile * 64;
        const int nrows = (int)min_i64(64, nb - base);
        // inputs to shared memory (padded, BF16)
        for (int q = threadIdx.x; q < 64 * 16; q += blockDim.x) {
            const int r = q / 16, i = q % 16;
            float v = 0.f;
            if (r < nrows && i < kMlpF) v = X[sample(base + r) * kMlpF + i];
            S.x[r][i] = __float2bfloat16_rn(v);
        }
        __syncthreads();
        float z[8][4], ds3[8][4], pred[2];
        uint32_t A[4][4];
        // activation of z; its derivative to shared memory
        auto act = [&](int layer) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float4 ds;
                z[j][0] = silu_d(z[j][0], ds.x);
                z[j][1] = silu_d(z[j][1], ds.y);
                z[j][2] = silu_d(z[j][2], ds.z);
                z[j][3] = silu_d(z[j][3], ds.w);
                S.ds[layer][j][threadIdx.x] = ds;
            }
        };
        const uint32_t a0[4] = {*reinterpret_cast<const uint32_t *>(&S.x[row0 + g][2 * t]),
                                *reinterpret_cast<const uint32_t *>(&S.x[row0 + g + 8][2 * t]), 0u, 0u};
        dense_in(a0, S.net, z);
        act(0);
        to_afrag(z, A);
        store_rows(S.h[0], row0, A);
        dense64(A, S.net.w2, S.net.b2, z);
        act(1);
        to_afrag(z, A);
        store_rows(S.h[1], row0, A);
        dense64(A, S.net.w3, S.net.b3, z);
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) z[j][q] = silu_d(z[j][q], ds3[j][q]);
        output_row(S.net, z, pred);
        if (t == 0) {
            const int ra = row0 + g, rb = row0 + g + 8;
            const int64_t sa = sample(base + min(ra, nrows - 1)), sb = sample(base + min(rb, nrows - 1));
            const float ea = ra < nrows ? (pred[0] - Y[sa]) * Wt[sa] : 0.f;
            const float eb = rb < nrows ? (pred[1] - Y[sb]) * Wt[sb] : 0.f;
            S.dy[ra] = 2.f * ea * inv_n;
            S.dy[rb] = 2.f * eb * inv_n;
            lsum += ea * ea + eb * eb;
        }
        __syncwarp();
        // layer 4 and dZ3 of this warp's rows
        const float dya = S.dy[row0 + g], dyb = S.dy[row0 + g + 8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float w0 = S.net.w4[8 * j + 2 * t], w1 = S.net.w4[8 * j + 2 * t + 1];
            gW4[j][0] += dya * z[j][0];
            gW4[j][1] += dya * z[j][1];
            gW4[j][0] += dyb * z[j][2];
            gW4[j][1] += dyb * z[j][3];
            z[j][0] = dya * w0 * ds3[j][0];
            z[j][1] = dya * w1 * ds3[j][1];
            z[j][2] = dyb * w0 * ds3[j][2];
            z[j][3] = dyb * w1 * ds3[j][3];
        }
        to_afrag(z, A);
        store_rows(S.d[0], row0, A);
        if (lane == 0)
            for (int r = row0; r < row0 + 16; ++r) gb4 += S.dy[r];
        __syncthreads();
        // layer 3: weights (stripe) and dZ2 of this warp's rows
        grad_stripe<8, kLd>(S.d[0], S.h[1], gW3);
        gb3 += bias_sum(S.d[0]);
        auto back = [&](const __nv_bfloat16 (*D)[kLd], const __nv_bfloat16 (&W)[kMlpH][kLd], int layer) {
            back64(D, row0, W, z);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float4 ds = S.ds[layer][j][threadIdx.x];
                z[j][0] *= ds.x;
                z[j][1] *= ds.y;
                z[j][2] *= ds.z;
                z[j][3] *= ds.w;
            }
            to_afrag(z, A);
        };
        back(S.d[0], S.net.w3, 1);
        store_rows(S.d[1], row0, A);
        __syncthreads();
        // layer 2
        grad_stripe<8, kLd>(S.d[1], S.h[0], gW2);
        gb2 += bias_sum(S.d[1]);
        back(S.d[1], S.net.w2, 0);
        // (every warp read d[0] before the last barrier)
        store_rows(S.d[0], row0, A);
        __syncthreads();
        // layer 1 (inputs padded to 16; only i < 8 are real)
        grad_stripe<2, kLdX>(S.d[0], S.x, gW1);
        gb1 += bias_sum(S.d[0]);
        __syncthreads();
    }
    // write this CTA's gradient slot (packing of the parameter vector)
    float *G = partial + (size_t)blockIdx.x * kMlpParams;
    float *gw1 = G, *gbb1 = gw1 + kMlpH * kMlpF, *gw2 = gbb1 + kMlpH, *gbb2 = gw2 + kMlpH * kMlpH;
    float *gw3 = gbb2 + kMlpH, *gbb3 = gw3 + kMlpH * kMlpH, *gw4 = gbb3 + kMlpH, *gbb4 = gw4 + kMlpH;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int i = 8 * j + 2 * t;
        gw2[(row0 + g) * kMlpH + i] = gW2[j][0];
        gw2[(row0 + g) * kMlpH + i + 1] = gW2[j][1];
        gw2[(row0 + g + 8) * kMlpH + i] = gW2[j][2];
        gw2[(row0 + g + 8) * kMlpH + i + 1] = gW2[j][3];
        gw3[(row0 + g) * kMlpH + i] = gW3[j][0];
        gw3[(row0 + g) * kMlpH + i + 1] = gW3[j][1];
        gw3[(row0 + g + 8) * kMlpH + i] = gW3[j][2];
        gw3[(row0 + g + 8) * kMlpH + i + 1] = gW3[j][3];
    }
    if (t < 4) {  // n-tile 0 of layer 1 holds inputs 0..7
        const int i = 2 * t;
        gw1[(row0 + g) * kMlpF + i] = gW1[0][0];
        gw1[(row0 + g) * kMlpF + i + 1] = gW1[0][1];
        gw1[(row0 + g + 8) * kMlpF + i] = gW1[0][2];
        gw1[(row0 + g + 8) * kMlpF + i + 1] = gW1[0][3];
    }
    // biases: lanes l and l+16 hold halves of the same output
    gb1 += __shfl_xor_sync(0xffffffffu, gb1, 16);
    gb2 += __shfl_xor_sync(0xffffffffu, gb2, 16);
    gb3 += __shfl_xor_sync(0xffffffffu, gb3, 16);
    if (lane < 16) {
        gbb1[row0 + lane] = gb1;
        gbb2[row0 + lane] = gb2;
        gbb3[row0 + lane] = gb3;
    }
    // output row: every warp summed its own rows for all 64 inputs
#pragma unroll
    for (int j = 0; j < 8; ++j) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float v = gW4[j][q];
            v += __shfl_xor_sync(0xffffffffu, v, 4);
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            gW4[j][q] = v;
        }
    }
    __shared__ float w4acc[4][kMlpH];
    __shared__ float b4acc[4], lacc[4];
    if (g == 0) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            w4acc[w][8 * j + 2 * t] = gW4[j][0];
            w4acc[w][8 * j + 2 * t + 1] = gW4[j][1];
        }
    }
    lsum += __shfl_xor_sync(0xffffffffu, lsum, 4);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, 8);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, 16);
    if (lane == 0) {
        b4acc[w] = gb4;
        lacc[w] = lsum;
    }
    __syncthreads();
    if (threadIdx.x < kMlpH)
        gw4[threadIdx.x] = w4acc[0][threadIdx.x] + w4acc[1][threadIdx.x] + w4acc[2][threadIdx.x] +
                           w4acc[3][threadIdx.x];
    if (threadIdx.x == 0) {
        gbb4[0] = b4acc[0] + b4acc[1] + b4acc[2] + b4acc[3];
        loss_out[blockIdx.x] = lacc[0] + lacc[1] + lacc[2] + lacc[3];
    }
}

// Sum the CTA slots in a fixed order (32 parameters a block, eight threads each,
// every eighth slot to a thread); optionally apply Adam to the master weights.
__global__ void __launch_bounds__(256) k_mlp_reduce_adam(int nslots, const float *__restrict__ partial,
                                                         float *__restrict__ grad, float *__restrict__ P,
                                                         float *__restrict__ m, float *__restrict__ v,
                                                         int adam, float lr, float b1, float b2, float eps,
                                                         float c1, float c2)
{
    __shared__ float acc[8][32];
    const int part = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + (threadIdx.x & 31);
    float s = 0.f;
    if (k < kMlpParams) {
#pragma unroll 8
        for (int q = part; q < nslots; q += 8) s += partial[(size_t)q * kMlpParams + k];
    }
    acc[part][threadIdx.x & 31] = s;
    __syncthreads();
    if (part != 0 || k >= kMlpParams) return;
    for (int q = 1; q < 8; ++q) s += acc[q][threadIdx.x & 31];
    if (grad) grad[k] = s;
    if (!adam) return;
    const float mk = b1 * m[k] + (1.f - b1) * s;
    const float vk = b2 * v[k] + (1.f - b2) * s * s;
    m[k] = mk;
    v[k] = vk;
    P[k] -= lr * (mk * c1) / (sqrtf(vk * c2) + eps);
}

cudaError_t mlp_predict(int64_t n, const float *X, const float *P, float *out, int num_sms,
                        cudaStream_t s)
{
    cudaError_t e = set_max_dynamic_smem((const void *)k_mlp_predict, mlp_predict_smem());
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + 15) / 16;
    const int grid = (int)min_i64((tiles + 7) / 8, (int64_t)num_sms * 3);
    if (grid > 0) k_mlp_predict<<<grid, 256, mlp_predict_smem(), s>>>(n, X, P, out);
    return cudaGetLastError();
}

cudaError_t mlp_train_step(int64_t nb, const int64_t *idx, const float *X, const float *Y,
                           const float *W, float *P, float *m, float *v, float *partial,
                           int slots, float *grad, float *loss, int adam, float lr, int step,
                           float inv_n, cudaStream_t s)
{
    cudaError_t e = set_max_dynamic_smem((const void *)k_mlp_train, mlp_train_smem());
    if (e != cudaSuccess) return e;
    const int grid = (int)min_i64((nb + 63) / 64, slots);
    if (grid <= 0) return cudaSuccess;
    k_mlp_train<<<grid, 128, mlp_train_smem(), s>>>(nb, idx, X, Y, W, P, inv_n, partial, loss);
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f / (1.f - powf(b1, (float)step)), c2 = 1.f / (1.f - powf(b2, (float)step));
    k_mlp_reduce_adam<<<(kMlpParams + 31) / 32, 256, 0, s>>>(grid, partial, grad, P, m, v, adam, lr,
                                                               b1, b2, 1e-8f, c1, c2);
    return cudaGetLastError();
}

}  // namespace nlg
