// Record decoding and the number conversions shared by the pass kernels.
#pragma once
#include "nl_internal.cuh"

namespace nlg {

__device__ __forceinline__ uint32_t get_nibble(const uint8_t *body, uint32_t p)
{
    uint32_t b = body[p >> 1];
    return (p & 1u) ? (b >> 4) : (b & 0xfu);
}

// sqrt.approx.f32: the hardware square root approximation (relative error
// about 2^-22); exact 0 for 0, so coincident particles need no guard
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Decode the next 32 entries of a record (one per lane; Sec. II-B): the
// block mask is read at nibble offset pos with a funnel shift, each lane
// finds its info nibble by popcount and its data nibbles by a warp scan of
// data lengths, and a warp scan of the differences rebuilds the j-cluster
// indices from prevJ.  Advances pos and prevJ; uncompressed records hold
// the u32 indices (entry t of lane).
__device__ __forceinline__ uint32_t decode_block(const uint32_t *body, int compress, uint32_t t,
                                                 bool valid, uint32_t &pos, uint32_t &prevJ)
{
    const unsigned lane = lane_id();
    uint32_t J;
    if (compress) {
        const uint8_t *bodyb = reinterpret_cast<const uint8_t *>(body);
        const uint32_t w0 = body[pos >> 3];
        const uint32_t w1 = (pos & 7u) ? body[(pos >> 3) + 1] : 0u;
        const uint32_t bm = __funnelshift_r(w0, w1, (pos & 7u) * 4u);
        const bool bit = (bm >> lane) & 1u;
        const uint32_t nbits = __popc(bm);
        uint32_t info = bit ? get_nibble(bodyb, pos + 8 + __popc(bm & lanemask_lt())) : 0u;
        uint32_t ndat = (bit && info < 8u) ? info + 1u : 0u;
        uint32_t incl = warp_incl_scan(ndat);
        uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        uint32_t pd = pos + 8 + nbits + incl - ndat;
        uint32_t v = 0;
        for (uint32_t q = 0; q < ndat; ++q) v = (v << 4) | get_nibble(bodyb, pd + q);
        uint32_t d = !bit ? 1u : (info >= 8u ? info - 6u : v);
        J = prevJ + warp_incl_scan(d);
        pos += 8 + nbits + tot;
    } else {
        J = valid ? body[t] : 0u;
    }
    prevJ = __shfl_sync(0xffffffffu, J, 31);
    return J;
}

// Nearest integer of x (ties away from zero) as a 64-bit two's complement
// word, with integer operations only; |x| < 2^62.  Subnormal x give 0.
__device__ __forceinline__ unsigned long long fixed_of(float x)
{
    const uint32_t b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xffu) - 150;  // |x| = mant * 2^e
    const unsigned long long m = (unsigned long long)((b & 0x7fffffu) | 0x800000u);
    unsigned long long q;
    if (e >= 0)
        q = m << e;
    else if (e > -25)
        q = (m + (1ull << (-e - 1))) >> (-e);
    else
        q = 0ull;
    if (((b >> 23) & 0xffu) == 0u) q = 0ull;
    return (b >> 31) ? (0ull - q) : q;
}

// The same for 0 <= x < 2^63 in two 32-bit conversions: hi = floor(x / 2^32)
// (exact: x / 2^32 is a float), then the remainder x - hi 2^32, exact in
// FP32 (below 2^32 it is x itself; above, a multiple of ulp(x) >= 2^9 below
// 2^32), rounded to the nearest integer (ties to even; a remainder of x >=
// 2^32 is already an integer)
__device__ __forceinline__ unsigned long long fixed_of_nonneg(float x)
{
    const uint32_t hi = __float2uint_rz(__fmul_rn(x, 0x1p-32f));
    const uint32_t lo = __float2uint_rn(__fmaf_rn(-__uint2float_rn(hi), 0x1p32f, x));
    return ((unsigned long long)hi << 32) | lo;
}

// The same for |x| < 2^63 of either sign, as two's complement.
__device__ __forceinline__ unsigned long long fixed_of_signed(float x)
{
    const unsigned long long q = fixed_of_nonneg(fabsf(x));
    return x < 0.f ? 0ull - q : q;
}

// The FP64 value of x with integer operations only (exact for normal x;
// zero and subnormals, below 1.2e-38, give 0; inf and NaN stay so).
__device__ __forceinline__ double f64_of(float x)
{
    const uint32_t b = __float_as_uint(x);
    const uint32_t e = (b >> 23) & 0xffu;
    if (e == 0u) return 0.0;
    const unsigned long long d = ((unsigned long long)(b >> 31) << 63) |
                                 ((unsigned long long)(e == 255u ? 2047u : e + 896u) << 52) |
                                 ((unsigned long long)(b & 0x7fffffu) << 29);
    return __longlong_as_double((long long)d);
}

}  // namespace nlg
