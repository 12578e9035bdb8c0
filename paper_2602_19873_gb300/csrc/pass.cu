// Dispatch of the neighborhood passes (kernels in pass_impl.cuh, one
// translation unit per pass kind) and the gather of pass inputs.
#include <algorithm>

#include "nl_internal.cuh"

namespace nlg {

constexpr int kPassBlocksPerSM = 4;
cudaError_t launch_pass_density(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s);
cudaError_t launch_pass_count(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s);
cudaError_t launch_pass_sph(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s);
cudaError_t launch_pass_lj(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s);
cudaError_t launch_pass_ljc(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s);
cudaError_t launch_pass_min(const PassArgs &a, int M, int per, int grid, int threads,
                          cudaStream_t s);

cudaError_t launch_pass(const PassArgs &a0, int kind, int M, int any_periodic, int num_sms,
                        cudaStream_t s, int threads, int blocks_per_sm)
{
    cudaError_t e = cudaMemsetAsync(&a0.st->pass_ticket, 0, 4, s);
    if (e != cudaSuccess) return e;
    const int tpb = threads ? threads : 256;
    const int bps = blocks_per_sm ? blocks_per_sm : kPassBlocksPerSM;
    const int grid = num_sms * bps;
    PassArgs a = a0;
    a.packed = pass_is_packed(kind, M, a.mj, a.support);
    // as many warps of a block share a super-cluster as there are warp slots
    // (two resident blocks per SM) for each
    const uint64_t nwork = a.work ? a.nwork : a.nsc;
    const uint64_t slots = (uint64_t)num_sms * std::min(bps, 2) * (tpb / 32);
    a.split = 1;
    while (a.split * 2 <= tpb / 32 && (a.longs || nwork * a.split * 2 <= slots)) a.split *= 2;
    switch (kind) {
    case PASS_DENSITY: return launch_pass_density(a, M, any_periodic, grid, tpb, s);
    case PASS_COUNT: return launch_pass_count(a, M, any_periodic, grid, tpb, s);
    case PASS_SPH: return launch_pass_sph(a, M, any_periodic, grid, tpb, s);
    case PASS_LJ: return launch_pass_lj(a, M, any_periodic, grid, tpb, s);
    case PASS_LJC: return launch_pass_ljc(a, M, any_periodic, grid, tpb, s);
    case PASS_MIN: return launch_pass_min(a, M, any_periodic, grid, tpb, s);
    default: return cudaErrorInvalidValue;
    }
}

// Gather per-particle pass inputs into SFC order (AuxMode).
template <int MODE>
__global__ void __launch_bounds__(256) k_gather_aux(uint32_t npad, const uint32_t *__restrict__ perm_pad,
                                                    const float4 *__restrict__ pos, float support,
                                                    const float *__restrict__ a, const float *__restrict__ b,
                                                    const float *__restrict__ c, void *__restrict__ aux,
                                                    unsigned int *amax)
{
    constexpr bool MAXIMA = MODE == AUX_MASS || MODE == AUX_SPH4;
    __shared__ unsigned int wm[8], wc[8];
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned int mb = 0, cb = 0;
    if (k < npad) {
        const uint32_t o = perm_pad[k];
        const bool real = o != 0xffffffffu;
        const float x = real ? a[o] : 0.f;
        float y = 0.f, hneg = -INFINITY, hinv = 0.f;
        if (MAXIMA && real) {
            const float h = pos[k].w, r = __fmul_rn(support, h);
            hinv = 1.f / h;
            if (__fmul_rn(r, r) > 0.f) hneg = -0.5f * hinv;
        }
        if ((MODE == AUX_SPH || MODE == AUX_SPH4) && real) {
            const float rho = c[o];
            y = b[o] / (rho * rho);
        }
        if constexpr (MODE == AUX_SPH4) {
            const float c = 0.954929658551372015f * y * hinv * hinv * hinv * hinv;  // 3/pi
            reinterpret_cast<float4 *>(aux)[k] = make_float4(c, x, hneg, y);
            cb = max(__float_as_uint(fabsf(c)), __float_as_uint(fabsf(2.f * c * hinv)));
        } else {
            reinterpret_cast<float2 *>(aux)[k] = make_float2(x, MODE == AUX_MASS ? hneg : y);
        }
        mb = __float_as_uint(fabsf(x));
    }
    if constexpr (MAXIMA) {
        // largest of the block, one atomic per block (non-negative floats
        // order like their bit patterns, NaN above all)
        mb = __reduce_max_sync(0xffffffffu, mb);
        if (MODE == AUX_SPH4) cb = __reduce_max_sync(0xffffffffu, cb);
        if ((threadIdx.x & 31) == 0) {
            wm[threadIdx.x >> 5] = mb;
            wc[threadIdx.x >> 5] = cb;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const bool on = threadIdx.x < (blockDim.x >> 5);
            mb = __reduce_max_sync(0xffffffffu, on ? wm[threadIdx.x] : 0u);
            if (threadIdx.x == 0 && mb) atomicMax(amax, mb);
            if constexpr (MODE == AUX_SPH4) {
                cb = __reduce_max_sync(0xffffffffu, on ? wc[threadIdx.x] : 0u);
                if (threadIdx.x == 0 && cb) atomicMax(amax + 1, cb);
            }
        }
    }
}

// Outputs of a half-list pass: density = (sum in fixed point) * 2^-scale *
// W's normalisation 1/(pi h^3), in the same FP32 form as the full-list pass;
// counts as summed; forces rounded from their FP64 sums.  Real slots only,
// written at perm[k] (or k).
__global__ void __launch_bounds__(256) k_half_finish(PassArgs a, int kind, uint32_t npad)
{
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npad) return;
    const uint32_t pc = a.perm[k];
    if (pc == 0xffffffffu) return;
    const uint32_t o = a.sorted_out ? k : pc;
    if (kind == PASS_COUNT) {
        a.outc[o] = a.hcnt[k];
        return;
    }
    if (kind == PASS_MIN) {  // +inf bits when no neighbor was found
        a.out0[o] = sqrtf(__uint_as_float(a.hcnt[k]));
        return;
    }
    if (kind != PASS_DENSITY) {  // forces: the FP64 sums rounded once to FP32
        a.out0[o] = (float)a.hf[3 * (size_t)k + 0];
        a.out1[o] = (float)a.hf[3 * (size_t)k + 1];
        a.out2[o] = (float)a.hf[3 * (size_t)k + 2];
        return;
    }
    const int ex = half_scale_exp(a.st->m_absmax);
    const double unit = __longlong_as_double((long long)(1023 - ex) << 52);  // 2^-ex
    const float v = (float)((double)(long long)a.hsum[k] * unit);
    const float hinv = 1.f / a.pos[k].w;
    a.out0[o] = v * (0.318309886183790672f * hinv * hinv * hinv);
}

cudaError_t launch_half_finish(const PassArgs &a0, int kind, int M, uint32_t npad, cudaStream_t s)
{
    if (kind < PASS_DENSITY || kind > PASS_MIN) return cudaErrorInvalidValue;
    PassArgs a = a0;
    a.packed = pass_is_packed(kind, M, a.mj, a.support);
    k_half_finish<<<(npad + 255) / 256, 256, 0, s>>>(a, kind, npad);
    return cudaGetLastError();
}

// New positions for a list kept across steps (Verlet buffer): every real
// padded slot takes its particle's caller-order position and keeps its h;
// optionally the largest displacement from the positions the list was built
// on (minimum image on periodic axes), as a float held in an unsigned word
// (non-negative floats order like their bit patterns).
__global__ void __launch_bounds__(256) k_refresh(uint32_t npad, const uint32_t *__restrict__ perm_pad,
                                                 SysTables t, const float *__restrict__ x,
                                                 const float *__restrict__ y,
                                                 const float *__restrict__ z, float4 *__restrict__ pos,
                                                 const float4 *__restrict__ pos_ref,
                                                 unsigned *__restrict__ max_disp)
{
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    float d = 0.f;
    if (k < npad) {
        const uint32_t o = perm_pad[k];
        if (o != 0xffffffffu) {
            const float4 old = pos[k];
            const float4 p = make_float4(x[o], y[o], z[o], old.w);
            pos[k] = p;
            if (max_disp) {
                const PerLen L = per_len(t.box[sys_of(t.pad_off, t.nsys, k)]);
                const float3 dv = pair_dx_acc<true>(pos_ref[k], p, L);
                d = sqrtf(dv.x * dv.x + dv.y * dv.y + dv.z * dv.z);
            }
        }
    }
    if (!max_disp) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d = fmaxf(d, __shfl_xor_sync(0xffffffffu, d, o));
    if ((threadIdx.x & 31) == 0 && d > 0.f) atomicMax(max_disp, __float_as_uint(d));
}

cudaError_t launch_refresh(uint32_t npad, const uint32_t *perm_pad, const SysTables &t,
                           const float *x, const float *y, const float *z, float4 *pos,
                           const float4 *pos_ref, float *max_disp, cudaStream_t s)
{
    if (max_disp) {
        cudaError_t e = cudaMemsetAsync(max_disp, 0, sizeof(float), s);
        if (e != cudaSuccess) return e;
    }
    k_refresh<<<(npad + 255) / 256, 256, 0, s>>>(npad, perm_pad, t, x, y, z, pos, pos_ref,
                                                reinterpret_cast<unsigned *>(max_disp));
    return cudaGetLastError();
}

cudaError_t launch_gather_aux(uint32_t npad, const uint32_t *perm_pad, const float4 *pos, float support,
                              const float *a, const float *b, const float *c, int mode, void *aux,
                              cudaStream_t s, unsigned int *amax)
{
    const unsigned grid = (npad + 255) / 256;
    switch (mode) {
    case AUX_CHARGE: k_gather_aux<AUX_CHARGE><<<grid, 256, 0, s>>>(npad, perm_pad, pos, support, a, b, c, aux, amax); break;
    case AUX_SPH: k_gather_aux<AUX_SPH><<<grid, 256, 0, s>>>(npad, perm_pad, pos, support, a, b, c, aux, amax); break;
    case AUX_MASS: k_gather_aux<AUX_MASS><<<grid, 256, 0, s>>>(npad, perm_pad, pos, support, a, b, c, aux, amax); break;
    case AUX_SPH4: k_gather_aux<AUX_SPH4><<<grid, 256, 0, s>>>(npad, perm_pad, pos, support, a, b, c, aux, amax); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace nlg
