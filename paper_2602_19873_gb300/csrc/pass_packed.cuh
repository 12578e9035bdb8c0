// Neighborhood passes with packed pair arithmetic: the pass kernel of every
// tile shape with at least 64 pairs (8x8, 16x8, 16x16).
//
// A warp owns a super-cluster, decodes 32 list entries at a time and stages
// the j particles of PK_SE of them in shared memory, two j particles of a
// cluster in each word: (x, x', y, y').  Then it takes the i-clusters two at a
// time: a lane holds one i particle (lane % M) of each, duplicated into packed
// registers once per stage, and walks the staged entries that list them; every
// step of the pair arithmetic is one f32x2 instruction for the lane's two j
// particles.  With the i-clusters outside and the entries inside, the sums of two
// i particles are all the registers a lane needs (the sums of 8 i-clusters held at
// once, with the entries outside, took 126 registers on the force passes), and no
// instruction is spent on i-clusters that an entry does not list.  On half lists
// the shares of the j particles wait in shared memory, one word per lane and
// entry, and are summed and added to memory once a stage.  Neighboring i-clusters
// share two thirds of their entries: such an entry's j words and j shares are read
// and written once for two tiles, and the two tiles' chains overlap.  (One
// i-cluster at a time left the half-list force passes bound by shared memory, 12 of
// 18 wavefronts per tile carrying the j shares: LJ at 4M particles 4.28 -> 3.8 ms,
// LJ + Coulomb 3.73 -> 3.19, pressure force of the 2^21-particle Evrard
// sphere 1.51 -> 1.26; evaluating every entry for both would have cost 18 %
// in pairs that are not listed.)
//
// The pair terms have no branches.  Kernels that vanish with the distance
// (density, pressure force) need no range test at all: with s = 1 - q/2 clamped
// to [0, 1] by the saturating multiply-add and p = q/2, w/2 = min(1/2 - 3 p^2 s,
// s^3) and -w'/3 = min(p, s)(s + u), u = 2s - 1 clamped, are 0 beyond the support.
// The others decide with the canonical FP32 predicate and select their
// coefficient.
//
// Entries with pairs across a periodic face (an eighth of the tiles of LJ at 4M
// particles) take the packed terms with the pair vector wrapped, one i-cluster at
// a time.  A scalar form of the terms is left for tiles that hold self pairs which
// have to be left out, and for all of them when an input is not finite or pressure
// coefficients may overflow (status words of the gather kernel).  (All entries of the own j-clusters and all wrapped
// ones in the scalar form: LJ at 4M 3.8 ms instead of 3.35.)
//
// What bounds it: instruction issue.  The half-list density pass issues 0.69, the
// force passes 0.62 to 0.65 instructions per scheduler and cycle, with the FMA pipe
// 60 % (LJ 31 %) and the shared-memory pipe 46 to 64 % (LJ 29 %) busy; what is left is
// the wait for fixed latencies at 24 to 32 warps per SM, as many as the registers allow.
// Pass stage, scalar kernel -> this one (CUDA events): half-list density on 2^24
// particles 9.10 -> 6.77 ms, pressure force on the 2^21-particle Evrard sphere 2.85
// -> 1.27, LJ at 4M particles 6.92 -> 3.35, LJ + Coulomb 4.83 -> 2.79; full lists:
// density and nearest distance on 2M particles 1.38 -> 1.03, pressure force on 300k
// 0.69 -> 0.29; small systems (split): density of 32k particles 0.48 -> 0.09 ms, of
// 4096 0.32 -> 0.05 ms.
//
// split: W warps of a block share a super-cluster, each working on every W-th
// stage.  Small systems have fewer super-clusters than the chip has warp slots,
// and their passes are bound by the latency of one list.  Lists of more than
// kLongList entries (skip_longer, longs) get a launch of their own in which whole
// blocks, several of them where sums can meet in memory, share one list.
#pragma once
#include <type_traits>

#include "nl_internal.cuh"
#include "pass_decode.cuh"

namespace nlg {

constexpr int PK_THREADS = 256;

__device__ __forceinline__ f32x2 add2_rn(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 dup2(float a) { return pk2(a, a); }

// a * b + 1 clamped to [0, 1]; NaN gives 0
__device__ __forceinline__ float sat_fma1(float a, float b)
{
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, 0f3F800000;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float sqrt_ftz(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_ftz(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// w(q)/2 of the cubic spline: s = sat(1 - q/2), p = q/2.  (Beyond the support s
// = 0; an infinite or NaN p leaves the other operand of the minimum.)  p comes
// from the same rounded 1/h as s and the final 1/h^3: the density hardly depends
// on h, so a rounding of 1/h that all three share cancels.
__device__ __forceinline__ float spline_half_w(float s, float p)
{
    return fminf(fmaf(-3.f, p * p * s, 0.5f), s * s * s);
}

__device__ __forceinline__ f32x2 spline_half_w2(float s0, float s1, f32x2 p)
{
    const f32x2 s = pk2(s0, s1);
    const f32x2 in = fma2_rn(dup2(-3.f), mul2_rn(mul2_rn(p, p), s), dup2(0.5f));
    const f32x2 out = mul2_rn(mul2_rn(s, s), s);
    float i0, i1, o0, o1;
    unpk2(in, i0, i1);
    unpk2(out, o0, o1);
    return pk2(fminf(i0, o0), fminf(i1, o1));
}

// w'(q)/3 of the cubic spline: s = sat(1 - q/2), pn = -q/2.  -max(pn, -s) is
// the smaller of q/2 and 1 - q/2: the factor that goes to 0 with the distance
// keeps its relative accuracy.
__device__ __forceinline__ float spline_third_dw(float s, float pn)
{
    return fmaxf(pn, -s) * (s + __saturatef(fmaf(2.f, s, -1.f)));
}

__device__ __forceinline__ f32x2 spline_third_dw2(float s0, float s1, f32x2 pn)
{
    float p0, p1;
    unpk2(pn, p0, p1);
    const f32x2 u = pk2(__saturatef(fmaf(2.f, s0, -1.f)), __saturatef(fmaf(2.f, s1, -1.f)));
    return mul2_rn(pk2(fmaxf(p0, -s0), fmaxf(p1, -s1)), add2_rn(pk2(s0, s1), u));
}

// Shared memory of one warp.  Own particles: ia = (x, y, z, a) with a = -1/(2h)
// (density, pressure) or the squared range (others), ib the pass inputs.  Staged
// j particles, two (j, j + MJ/2) in a word: ja = (x, x', y, y'), jb = (z, z',
// b, b'), jc = (c, c', d, d'):
//   density    b = m;        jc (half lists) = -1/(2h), 1/(2h)
//   pressure   b = -1/(2h);  jc = C, m
//   LJ + Coulomb b = squared range; jc = q
//   LJ, count, nearest: b = squared range
// js: half lists: the j shares of each lane's pair, per staged entry; full
// lists: the sums of a warp that shares its super-cluster.
template <int M, int MJ, int KIND, bool HL>
struct PkSmem {
    static constexpr bool FORCE = KIND == PASS_SPH || KIND == PASS_LJ || KIND == PASS_LJC;
    static constexpr int G = 32 / M;              // lane groups, each with its own j pairs
    static constexpr int NT = MJ / (2 * G);       // j pairs per lane and entry
    // list entries staged together: half lists, whose j shares take shared
    // memory, 8 of 8 particles (more cost the force passes a resident block, and
    // gave the density pass nothing); full lists 16 (density pass on 2M particles
    // 1.17 -> 1.11 ms against 8), but the pressure force, whose sums cancel, 8:
    // longer partials put it 2 % further from FP64 than the scalar kernel
    static constexpr int SE = HL ? 8 / NT : KIND == PASS_SPH ? 8 : 16;
    static constexpr int NI = kSC * M;
    static constexpr int NP = SE * MJ / 2;        // staged pairs
    static constexpr bool IB = KIND == PASS_SPH || KIND == PASS_LJC || (KIND == PASS_DENSITY && HL);
    static constexpr bool JC = IB;
    static constexpr int NC = FORCE ? 3 : 1;      // components of a sum
    float4 ia[NI];
    float4 ja[NP], jb[NP];
    float4 jc[JC ? NP : 1];
    f32x2 js[HL ? NC * SE * NT * 32 : NC * (kSC / G) * 16];
    float2 ib[IB ? NI : 2];
    uint32_t seen;
    float far;      // x of padding particles (DevBox::far)
    uint32_t pad[2];
};

// Resident blocks of 256 threads the register budget is cut for (half-list
// density at 2^24 particles with 3 / 4: 6.99 / 6.77 ms; half-list LJ at 4M with
// 2 / 3: 3.56 / 3.39 ms, LJ + Coulomb 2.93 / 2.79, pressure force the same).
template <int KIND, bool HL>
constexpr int pk_min_blocks()
{
    return (KIND == PASS_SPH || KIND == PASS_LJ || KIND == PASS_LJC) ? 3 : 4;
}

// One i particle, duplicated into packed registers: position, a as in PkSmem::ia,
// hp = +-a, and its pass inputs u, v.
template <int KIND>
struct IPart {
    f32x2 x, y, z, hp, u, v;
    float a;
};
// Sums of one i particle over a stage: (x, y, z), count or minimum.
struct ISum {
    f32x2 x, y, z;
    uint32_t c;
};

// v += b with the running compensation c (Kahan)
__device__ __forceinline__ void kahan_add(float &v, float &c, float b)
{
    const float y = __fsub_rn(b, c);
    const float t = __fadd_rn(v, y);
    c = __fsub_rn(__fsub_rn(t, v), y);
    v = t;
}

// LONG: the pass over the long lists (a.longs).
template <int M, int MJ, bool PER, int KIND, bool HL, bool LONG>
__global__ void __launch_bounds__(PK_THREADS, (pk_min_blocks<KIND, HL>())) k_pass_packed(PassArgs a)
{
    static_assert(M * MJ >= 64, "a tile fills the lanes with pairs of j particles");
    static_assert(!HL || M == MJ, "half lists have j-clusters of the i-cluster size");
    using Smem = PkSmem<M, MJ, KIND, HL>;
    constexpr uint32_t G = Smem::G, NT = Smem::NT, SE = Smem::SE, HJ = MJ / 2;
    constexpr uint32_t NK = kSC / G;        // i-clusters whose sums a lane keeps
    constexpr uint32_t RJ = M / MJ;
    constexpr bool FORCE = Smem::FORCE;
    constexpr bool INTS = KIND == PASS_COUNT || KIND == PASS_MIN;
    constexpr bool SELF_IN_LOOP = KIND == PASS_DENSITY || KIND == PASS_COUNT;
    constexpr bool NO_SELF = KIND == PASS_LJ || KIND == PASS_LJC || KIND == PASS_MIN;
    constexpr uint32_t NONE = KIND == PASS_MIN ? 0x7f800000u : 0u;  // empty sum (min: +inf)
    extern __shared__ __align__(16) unsigned char pk_smem[];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    Smem *const all = reinterpret_cast<Smem *>(pk_smem);
    Smem &S = all[warp];
    const uint32_t II = lane % M, g = lane / M;
    const uint32_t W = (uint32_t)a.split, wig = warp & (W - 1u), grp = warp / W;
    const uint32_t ngrp = (blockDim.x >> 5) / W;
    // inputs that are not finite: a zero kernel must not multiply them; nor a zero
    // pair vector the pressure terms of coincident particles, at most m 2C/h
    const bool careful =
        KIND == PASS_DENSITY ? __any_sync(0xffffffffu, a.st->m_absmax >= 0x7f800000u)
        : KIND == PASS_SPH
            ? __any_sync(0xffffffffu, !(__uint_as_float(a.st->m_absmax) * __uint_as_float(a.st->c_absmax) < INFINITY))
            : false;
    // fixed-point scale of the half-list density
    const float hscale = (HL && KIND == PASS_DENSITY)
                             ? __int_as_float((half_scale_exp(a.st->m_absmax) + 127) << 23) : 0.f;
    const float sig2 = a.p1 * a.p1, e24 = 24.f * a.p0;
    // running sums take one partial a stage.  Density and pressure (whose sums
    // cancel) compensated: plain adds left the pressure force of the Evrard
    // sphere 10 % further from FP64 than the scalar kernel, 3 % less time.  Lennard-
    // Jones sums are ruled by their nearest pairs: plain adds are as near as the
    // scalar kernel's (median error at 4M particles 3.52e-7, scalar 3.57e-7; with
    // Coulomb terms 4.72e-7, scalar 4.74e-7) and 4 % faster.
    auto sum_add = [](float &v, float &c, float b) {
        if constexpr (KIND == PASS_DENSITY || KIND == PASS_SPH) {
            kahan_add(v, c, b);
            // (a force that overflows stays infinite)
            if (KIND != PASS_DENSITY && !(fabsf(v) < INFINITY)) c = 0.f;
        } else {
            v += b;
        }
    };
    auto merge = [](uint32_t u, uint32_t v) { return KIND == PASS_COUNT ? u + v : min(u, v); };

    constexpr uint32_t JS = SE * NT * 32;  // j shares: between components

    // own particle II of i-cluster k
    auto own_part = [&](uint32_t k) {
        const float4 p = S.ia[k * M + II];
        IPart<KIND> I;
        I.x = dup2(p.x);
        I.y = dup2(p.y);
        I.z = dup2(p.z);
        I.a = p.w;
        if constexpr (KIND == PASS_DENSITY) I.hp = dup2(-p.w);  // 1/(2h)
        if constexpr (KIND == PASS_SPH) I.hp = dup2(p.w);
        if constexpr (Smem::IB) {
            const float2 v = S.ib[k * M + II];
            I.u = dup2(v.x);
            I.v = dup2(v.y);
        }
        return I;
    };
    // the lane's pair tt of staged entry el, with its shares
    struct JPart {
        float4 A, B, C;
        f32x2 x, y, z;
    };
    auto load_j = [&](uint32_t el, uint32_t tt) {
        const uint32_t q = el * HJ + g + tt * G;
        JPart j;
        j.A = S.ja[q];
        j.B = S.jb[q];
        if constexpr (Smem::JC) j.C = S.jc[q];
        if constexpr (HL) {
            const f32x2 *js = S.js + (el * NT + tt) * 32 + lane;
            j.x = js[0];
            if constexpr (FORCE) {
                j.y = js[JS];
                j.z = js[2 * JS];
            }
        }
        return j;
    };
    auto store_j = [&](uint32_t el, uint32_t tt, const JPart &j) {
        if constexpr (HL) {
            f32x2 *js = S.js + (el * NT + tt) * 32 + lane;
            js[0] = j.x;
            if constexpr (FORCE) {
                js[JS] = j.y;
                js[2 * JS] = j.z;
            }
        }
    };
    // Padding particles: counts and nearest distances leave their NaN positions,
    // which are in no range.  Sums of forces need finite differences even of pairs
    // that take no part: there padding lies at (far, 0, 0), where no squared distance
    // is below a squared range (a fixed point would be in range of some box or
    // radius).  To the density, whose padding has no mass, any place will do.
    auto place_padding = [&](float4 &p, float far) {
        if (!INTS && !(p.x == p.x)) {
            p.x = FORCE ? far : 1e18f;
            p.y = p.z = 0.f;
        }
    };

    // the terms of one i particle and the lane's two j particles; wrap: pairs
    // may lie across a periodic face
    auto terms = [&](const IPart<KIND> &I, JPart &j, ISum &T, auto wrap, const PerLen &box) {
        constexpr bool WR = decltype(wrap)::value;
        const float4 &A = j.A, &B = j.B, &C = j.C;
        f32x2 dx = sub2_rn(pk2(A.x, A.y), I.x), dy = sub2_rn(pk2(A.z, A.w), I.y);
        f32x2 dz = sub2_rn(pk2(B.x, B.y), I.z);
        float w0, w1;  // the canonical squared distances of such pairs
        if constexpr (WR) {
            float ix, iy, iz, u;
            unpk2(I.x, ix, u);
            unpk2(I.y, iy, u);
            unpk2(I.z, iz, u);
            if constexpr (KIND != PASS_DENSITY && KIND != PASS_SPH)
                pair_d2_x2<true>(pk2(A.x, A.y), pk2(A.z, A.w), pk2(B.x, B.y), I.x, I.y, I.z, box, w0, w1);
            const float4 pi = make_float4(ix, iy, iz, 0.f);
            const float3 v0 = pair_dx_acc<true>(pi, make_float4(A.x, A.z, B.x, 0.f), box);
            const float3 v1 = pair_dx_acc<true>(pi, make_float4(A.y, A.w, B.y, 0.f), box);
            dx = pk2(v0.x, v1.x);
            dy = pk2(v0.y, v1.y);
            dz = pk2(v0.z, v1.z);
        }
        float d0, d1;
        if constexpr (KIND == PASS_DENSITY) {
            unpk2(fma2_rn(dz, dz, fma2_rn(dy, dy, mul2_rn(dx, dx))), d0, d1);
            const float r0 = sqrt_ftz(d0), r1 = sqrt_ftz(d1);
            const f32x2 r = pk2(r0, r1);
            T.x = fma2_rn(pk2(B.z, B.w), spline_half_w2(sat_fma1(r0, I.a), sat_fma1(r1, I.a), mul2_rn(r, I.hp)), T.x);
            if constexpr (HL)
                j.x = fma2_rn(I.u, spline_half_w2(sat_fma1(r0, C.x), sat_fma1(r1, C.y), mul2_rn(r, pk2(C.z, C.w))), j.x);
        } else if constexpr (KIND == PASS_SPH) {
            // (a self pair: dx = 0, and careful passes aside b is finite; the floor,
            // the smallest normal square, keeps 1/r finite and is so near that w'/r
            // hardly depends on r)
            unpk2(fma2_rn(dz, dz, fma2_rn(dy, dy, mul2_rn(dx, dx))), d0, d1);
            d0 = fmaxf(d0, 1.17549435e-38f);
            d1 = fmaxf(d1, 1.17549435e-38f);
            const f32x2 ir = pk2(rsqrt_ftz(d0), rsqrt_ftz(d1));
            const f32x2 r = mul2_rn(pk2(d0, d1), ir);
            float r0, r1;
            unpk2(r, r0, r1);
            const f32x2 gi = spline_third_dw2(sat_fma1(r0, I.a), sat_fma1(r1, I.a), mul2_rn(r, I.hp));
            const f32x2 gj = spline_third_dw2(sat_fma1(r0, B.z), sat_fma1(r1, B.w), mul2_rn(r, pk2(B.z, B.w)));
            const f32x2 b = mul2_rn(fma2_rn(pk2(C.x, C.y), gj, mul2_rn(I.u, gi)), ir);
            const f32x2 si = mul2_rn(pk2(C.z, C.w), b);
            T.x = fma2_rn(si, dx, T.x);
            T.y = fma2_rn(si, dy, T.y);
            T.z = fma2_rn(si, dz, T.z);
            if constexpr (HL) {
                const f32x2 sj = mul2_rn(I.v, b);
                j.x = fma2_rn(sj, dx, j.x);
                j.y = fma2_rn(sj, dy, j.y);
                j.z = fma2_rn(sj, dz, j.z);
            }
        } else {
            sum_sq_x2(dx, dy, dz, d0, d1);
            if constexpr (!WR) {  // these are the canonical ones
                w0 = d0;
                w1 = d1;
            }
            const bool i0 = w0 < I.a, i1 = w1 < I.a;
            [[maybe_unused]] const bool j0 = HL && w0 < B.z, j1 = HL && w1 < B.w;
            if constexpr (KIND == PASS_COUNT) {
                T.c += (i0 ? 1u : 0u) + (i1 ? 1u : 0u);
                if constexpr (HL) j.x += (j0 ? 1ull : 0ull) + (j1 ? 1ull << 32 : 0ull);
            } else if constexpr (KIND == PASS_MIN) {
                const uint32_t u0 = __float_as_uint(d0), u1 = __float_as_uint(d1);
                if (i0) T.c = min(T.c, u0);
                if (i1) T.c = min(T.c, u1);
                if constexpr (HL) {
                    const uint32_t l = j0 ? min((uint32_t)j.x, u0) : (uint32_t)j.x;
                    const uint32_t h = j1 ? min((uint32_t)(j.x >> 32), u1) : (uint32_t)(j.x >> 32);
                    j.x = ((f32x2)h << 32) | l;
                }
            } else {
                // f: minus the coefficient of dx in the force on j
                float f0, f1;
                if constexpr (KIND == PASS_LJ) {
                    // -1/d2 by the hardware reciprocal and one Newton step.
                    // Denormal d2 (separations below 1.1e-19) count as the
                    // smallest normal one: the coefficient overflows there like
                    // that of 1/d2 unless sigma is below about 1e-18
                    d0 = fmaxf(d0, 1.17549435e-38f);
                    d1 = fmaxf(d1, 1.17549435e-38f);
                    const f32x2 r = pk2(rcp_ftz(-d0), rcp_ftz(-d1));
                    const f32x2 e = fma2_rn(pk2(d0, d1), r, dup2(1.f));
                    const f32x2 ir2 = fma2_rn(r, e, r);
                    const f32x2 s2 = mul2_rn(dup2(sig2), ir2);
                    const f32x2 s6 = mul2_rn(mul2_rn(s2, s2), s2);  // -(sigma/r)^6
                    // (overflows only where the product of all does)
                    unpk2(mul2_rn(mul2_rn(mul2_rn(dup2(e24), ir2), s6), fma2_rn(dup2(2.f), s6, dup2(1.f))), f0, f1);
                } else {
                    const f32x2 ir = pk2(rsqrt_ftz(d0), rsqrt_ftz(d1));
                    const f32x2 ir2 = mul2_rn(ir, ir);
                    const f32x2 s2 = mul2_rn(dup2(-sig2), ir2);
                    const f32x2 s6 = mul2_rn(mul2_rn(s2, s2), s2);
                    const f32x2 lj = mul2_rn(mul2_rn(dup2(e24), s6), fma2_rn(dup2(2.f), s6, dup2(1.f)));
                    const f32x2 qq = mul2_rn(I.u, pk2(C.x, C.y));
                    float t0, t1;
                    unpk2(mul2_rn(ir2, fma2_rn(qq, ir, lj)), t0, t1);
                    f0 = -t0;
                    f1 = -t1;
                }
                // (padding particles are far away: never in range, dx finite)
                const f32x2 fi = pk2(i0 ? f0 : 0.f, i1 ? f1 : 0.f);
                T.x = fma2_rn(fi, dx, T.x);
                T.y = fma2_rn(fi, dy, T.y);
                T.z = fma2_rn(fi, dz, T.z);
                if constexpr (HL) {
                    const f32x2 fj = pk2(j0 ? f0 : 0.f, j1 ? f1 : 0.f);
                    j.x = fma2_rn(fj, dx, j.x);
                    j.y = fma2_rn(fj, dy, j.y);
                    j.z = fma2_rn(fj, dz, j.z);
                }
            }
        }
    };

    // running sums of particle II of the i-clusters cluster_of(q)
    float rx[NK], ry[NK], rz[NK];  // (density: x alone; count, nearest: rc)
    float cx[NK], cy[NK], cz[NK];  // their compensations
    uint32_t rc[NK];
    // lane group g keeps, of the pairs of i-clusters (2p, 2p + 1) with p = g mod
    // G/2, the first (g < G/2) or the second
    auto cluster_of = [&](uint32_t q) { return 2u * (q * (G / 2) + g % (G / 2)) + g / (G / 2); };
    // a stage's sums of i-clusters k, k + 1 over the lanes of the same particle,
    // then to the lanes that keep them
    auto keep = [&](uint32_t k, const ISum &A0, const ISum &A1) {
        const bool up = lane & 16u;  // g >= G/2
        const uint32_t p = k >> 1, mq = p / (G / 2);
        const bool mine = p % (G / 2) == g % (G / 2);
        if constexpr (INTS) {
            uint32_t v = merge(up ? A1.c : A0.c, __shfl_xor_sync(0xffffffffu, up ? A0.c : A1.c, 16));
#pragma unroll
            for (int o = M; o < 16; o <<= 1) v = merge(v, __shfl_xor_sync(0xffffffffu, v, o));
#pragma unroll
            for (uint32_t q = 0; q < NK; ++q)
                if (mine && mq == q) rc[q] = merge(rc[q], v);
        } else {
            auto fold = [&](f32x2 a0, f32x2 a1) {
                float l0, h0, l1, h1;
                unpk2(a0, l0, h0);
                unpk2(a1, l1, h1);
                const float s0 = l0 + h0, s1 = l1 + h1;
                float v = (up ? s1 : s0) + __shfl_xor_sync(0xffffffffu, up ? s0 : s1, 16);
#pragma unroll
                for (int o = M; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                return v;
            };
            const float x = fold(A0.x, A1.x);
            float y = 0.f, z = 0.f;
            if constexpr (FORCE) {
                y = fold(A0.y, A1.y);
                z = fold(A0.z, A1.z);
            }
#pragma unroll
            for (uint32_t q = 0; q < NK; ++q)
                if (mine && mq == q) {
                    sum_add(rx[q], cx[q], x);
                    if constexpr (FORCE) {
                        sum_add(ry[q], cy[q], y);
                        sum_add(rz[q], cz[q], z);
                    }
                }
        }
    };

    const uint32_t nwork = a.work || LONG ? (a.nwork_dev ? min(a.nwork, *a.nwork_dev) : a.nwork) : a.nsc;
    for (uint32_t it = blockIdx.x + gridDim.x * grp;; it += gridDim.x * ngrp) {
        uint32_t s = it, part = 0, seek = kNoSeek;
        if constexpr (LONG) {  // (long list, block of it); first the first blocks of all
            if (it >= nwork * kPassParts) break;
            part = it / nwork;
            const uint2 l = a.longs[it % nwork];
            s = l.x;
            seek = l.y;
            if (a.long_asked && !a.long_asked[s]) continue;
        } else {
            if (W == 1u) {
                if (lane == 0) s = atomicAdd(&a.st->pass_ticket, 1u);
                s = __shfl_sync(0xffffffffu, s, 0);
            }
            if (s >= nwork) break;
            if (a.work) s = a.work[s];
        }
        // a super-cluster whose list was not stored (an overflow inside a graph
        // replay, reported by nl_graph_check) is read as an empty list
        const uint32_t roff = a.rec_off[s];
        const uint32_t *rec = reinterpret_cast<const uint32_t *>(a.list) + (roff == kBadRecord ? 0u : roff);
        const uint32_t cnt = roff == kBadRecord ? 0u : rec[0];
        // blocks that share the list: only where their sums meet in memory
        constexpr bool SHARED = HL || INTS;
        const uint32_t chunks = (cnt + kSeek - 1u) / kSeek;
        uint32_t np = 1;
        if constexpr (LONG) {
            if (SHARED) np = min(kPassParts, (chunks + W - 1u) / W);
            if (part >= np) continue;
        }
        if (!LONG && a.skip_longer && cnt > a.skip_longer) {
            if (a.long_asked && lane == 0) a.long_asked[s] = 1u;
            if constexpr (!HL && INTS) {  // empty results for the blocks to add to
                for (uint32_t t = lane; t < (uint32_t)Smem::NI; t += 32) {
                    const uint32_t i = s * kSC * M + t, pc = a.perm[i];
                    if (pc == 0xffffffffu || wig != 0) continue;
                    const uint32_t o = a.sorted_out ? i : pc;
                    if constexpr (KIND == PASS_COUNT) a.outc[o] = 0u;
                    else a.out0[o] = INFINITY;
                }
            }
            continue;
        }
        const uint32_t VW = W * np, vw = part * W + wig;  // warps that share the list
        const DevBox &sbox = a.sys.box[sys_of(a.sys.pad_off, a.sys.nsys, s * kSC * M)];
        const PerLen box = per_len(sbox);

        // own particles; the box around them (periodic)
        float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
        __syncwarp();
        const float far = FORCE ? sbox.far : 0.f;
        if (FORCE && lane == 0) S.far = far;
#pragma unroll
        for (uint32_t t = lane; t < (uint32_t)Smem::NI; t += 32) {
            const uint32_t i = s * kSC * M + t;
            float4 p = a.pos[i];
            const float r = __fmul_rn(a.support, (KIND == PASS_COUNT && a.hq) ? a.hq[i] : p.w);
            float av = __fmul_rn(r, r);
            if constexpr (KIND == PASS_DENSITY) {
                const float2 x = a.aux[i];
                av = x.y;
                if constexpr (HL) S.ib[t] = make_float2(x.x, 0.f);
            } else if constexpr (KIND == PASS_SPH) {
                const float4 x = a.aux4[i];
                av = x.z;
                S.ib[t] = make_float2(careful ? x.w : x.x, x.y);
            } else if constexpr (KIND == PASS_LJC) {
                av = fminf(av, a.p2);
                S.ib[t] = make_float2(a.p3 * a.aux[i].x, 0.f);
            }
            const bool real = p.x == p.x;
            if constexpr (PER) {
                if (real) {
                    lo[0] = fminf(lo[0], p.x); hi[0] = fmaxf(hi[0], p.x);
                    lo[1] = fminf(lo[1], p.y); hi[1] = fmaxf(hi[1], p.y);
                    lo[2] = fminf(lo[2], p.z); hi[2] = fmaxf(hi[2], p.z);
                }
            }
            place_padding(p, far);
            S.ia[t] = make_float4(p.x, p.y, p.z, av);
        }
        if constexpr (PER) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    lo[x] = fminf(lo[x], __shfl_xor_sync(0xffffffffu, lo[x], o));
                    hi[x] = fmaxf(hi[x], __shfl_xor_sync(0xffffffffu, hi[x], o));
                }
        }
        __syncwarp();

#pragma unroll
        for (uint32_t q = 0; q < NK; ++q) {
            rx[q] = ry[q] = rz[q] = cx[q] = cy[q] = cz[q] = 0.f;
            rc[q] = NONE;
        }
        uint32_t selfseen = 0;  // bit r: the entry of own j-cluster r lists its own i-cluster

        const uint8_t *masks = reinterpret_cast<const uint8_t *>(rec + 1);
        const uint32_t *body = rec + 1 + ((cnt + 3u) >> 2);
        // a long list: every VW-th chunk of kSeek entries, entered at its seek
        // point; else the whole list, of which the warps take stages in turn
        for (uint32_t ch = LONG ? vw : 0u; ch < (LONG ? chunks : 1u); ch += VW) {
        const uint32_t cbeg = LONG ? ch * kSeek : 0u, cend = LONG ? min(cnt, cbeg + kSeek) : cnt;
        const uint2 at = LONG && seek != kNoSeek ? a.seek[seek + ch] : make_uint2(0u, 0xffffffffu);
        uint32_t pos = at.x;
        uint32_t prevJ = at.y;
        for (uint32_t b0 = LONG && seek != kNoSeek ? cbeg : 0u; b0 < cend; b0 += 32) {
            const uint32_t t = b0 + lane;
            const bool valid = t < cnt;
            const uint32_t J = decode_block(body, a.compress, t, valid, pos, prevJ);
            if (LONG && b0 < cbeg) continue;  // (no seek points: decode up to the chunk)
            const uint32_t mk = valid ? masks[t] : 0u;
            const uint32_t rel = J - s * kSC * RJ;  // own j-clusters: below kSC RJ
            const uint32_t own = __ballot_sync(0xffffffffu, valid && rel < kSC * RJ);
            if constexpr (SELF_IN_LOOP) {
                const bool seen = valid && rel < kSC * RJ && ((mk >> (rel / RJ)) & 1u);
                selfseen |= __reduce_or_sync(0xffffffffu, seen ? 1u << rel : 0u);
            }
            // half list: entries beyond the own clusters also feed their j particles
            const uint32_t feeds = HL ? __ballot_sync(0xffffffffu, valid) & ~own : 0u;
            for (uint32_t c = 0; c < min(32u, cnt - b0); c += SE) {
                if (!LONG && W != 1u && (b0 + c) / SE % W != wig) continue;
                const uint32_t ns = min(SE, cnt - b0 - c);
                // stage the j particles of entries c .. c + ns - 1
                uint32_t slow = careful ? 0xffffffffu : 0u;  // bit el: entry c + el takes the scalar terms
                __syncwarp();
#pragma unroll
                for (uint32_t q0 = 0; q0 < (uint32_t)Smem::NP; q0 += 32) {
                    const uint32_t q = q0 + lane;
                    const uint32_t el = q / HJ;
                    const uint32_t src = __shfl_sync(0xffffffffu, J, min(c + el, 31u)) * MJ + q % HJ;
                    bool wr = false;
                    if (el < ns) {
                        float4 p[2];
                        float bv[2] = {0.f, 0.f}, cv[2] = {0.f, 0.f}, dv[2] = {0.f, 0.f};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t j = src + h * HJ;
                            p[h] = a.pos[j];
                            if constexpr (KIND == PASS_DENSITY) {
                                const float2 x = a.aux[j];
                                bv[h] = x.x;
                                cv[h] = x.y;
                                dv[h] = -x.y;
                            } else if constexpr (KIND == PASS_SPH) {
                                const float4 x = a.aux4[j];
                                bv[h] = x.z;
                                cv[h] = careful ? x.w : x.x;
                                dv[h] = x.y;
                            } else {
                                if constexpr (HL) {
                                    const float r = __fmul_rn(a.support, p[h].w);
                                    bv[h] = __fmul_rn(r, r);
                                    if constexpr (KIND == PASS_LJC) bv[h] = fminf(bv[h], a.p2);
                                }
                                if constexpr (KIND == PASS_LJC) cv[h] = a.aux[j].x;
                            }
                            if constexpr (PER) {
                                // (the canonical difference is monotone in both coordinates)
                                const float hx = __fmul_rn(0.5f, box.x), hy = __fmul_rn(0.5f, box.y);
                                const float hz = __fmul_rn(0.5f, box.z);
                                wr = wr || __fsub_rn(p[h].x, lo[0]) > hx || __fsub_rn(p[h].x, hi[0]) < -hx ||
                                     __fsub_rn(p[h].y, lo[1]) > hy || __fsub_rn(p[h].y, hi[1]) < -hy ||
                                     __fsub_rn(p[h].z, lo[2]) > hz || __fsub_rn(p[h].z, hi[2]) < -hz;
                            }
                            place_padding(p[h], FORCE ? S.far : 0.f);
                        }
                        S.ja[q] = make_float4(p[0].x, p[1].x, p[0].y, p[1].y);
                        S.jb[q] = make_float4(p[0].z, p[1].z, bv[0], bv[1]);
                        if constexpr (Smem::JC) S.jc[q] = make_float4(cv[0], cv[1], dv[0], dv[1]);
                    }
                    if constexpr (PER) {
                        const uint32_t wb = __ballot_sync(0xffffffffu, wr);
#pragma unroll
                        for (uint32_t e = 0; e < 32u / HJ; ++e)
                            if ((wb >> (e * HJ)) & ((1u << HJ) - 1u)) slow |= 1u << (q0 / HJ + e);
                    }
                }
                if constexpr (HL) {
                    float4 *z = reinterpret_cast<float4 *>(S.js);
                    const float zv = KIND == PASS_MIN ? INFINITY : 0.f;
#pragma unroll
                    for (uint32_t q = lane; q < sizeof(S.js) / 16; q += 32) z[q] = make_float4(zv, zv, zv, zv);
                }
                __syncwarp();

                // i-clusters k and k + 1 together: entries that list both (about
                // two thirds of those that list one) read their j words, and keep
                // their j shares in registers, once for two tiles
                const uint32_t staged = (1u << SE) - 1u;
                // entries that list i-cluster k and hold its own particles: their
                // self pairs take the scalar terms
                const uint32_t owns = NO_SELF ? (own >> c) & staged : 0u;
                auto diag = [&](uint32_t k) {
                    return owns ? __ballot_sync(0xffffffffu, valid && rel / RJ == k) >> c : 0u;
                };
#pragma unroll 1
                for (uint32_t k = 0; k < kSC; k += 2) {
                    const uint32_t b0w = (__ballot_sync(0xffffffffu, (mk >> k) & 1u) >> c) & staged & ~(slow | diag(k));
                    const uint32_t b1w = (__ballot_sync(0xffffffffu, (mk >> k) & 2u) >> c) & staged & ~(slow | diag(k + 1u));
                    if (!(b0w | b1w)) continue;
                    const IPart<KIND> I0 = own_part(k), I1 = own_part(k + 1);
                    ISum A0{0ull, 0ull, 0ull, NONE}, A1 = A0;
                    for (uint32_t todo = b0w & b1w; todo; todo &= todo - 1u) {
                        const uint32_t el = __ffs(todo) - 1;
#pragma unroll
                        for (uint32_t tt = 0; tt < NT; ++tt) {
                            JPart j = load_j(el, tt);
                            terms(I0, j, A0, std::false_type(), box);
                            terms(I1, j, A1, std::false_type(), box);
                            store_j(el, tt, j);
                        }
                    }
                    for (uint32_t todo = b0w & ~b1w; todo; todo &= todo - 1u) {
                        const uint32_t el = __ffs(todo) - 1;
#pragma unroll
                        for (uint32_t tt = 0; tt < NT; ++tt) {
                            JPart j = load_j(el, tt);
                            terms(I0, j, A0, std::false_type(), box);
                            store_j(el, tt, j);
                        }
                    }
                    for (uint32_t todo = b1w & ~b0w; todo; todo &= todo - 1u) {
                        const uint32_t el = __ffs(todo) - 1;
#pragma unroll
                        for (uint32_t tt = 0; tt < NT; ++tt) {
                            JPart j = load_j(el, tt);
                            terms(I1, j, A1, std::false_type(), box);
                            store_j(el, tt, j);
                        }
                    }
                    keep(k, A0, A1);
                }
                if ((slow | owns) & staged) {
                    // pairs across a periodic face, packed; self pairs and inputs
                    // that are not finite, scalar: canonical predicate, accurate
                    // pair vector
#pragma unroll 1
                    for (uint32_t k = 0; k < kSC; ++k) {
                        const uint32_t lists = (__ballot_sync(0xffffffffu, (mk >> k) & 1u) >> c) & staged;
                        const uint32_t dg = diag(k), bits = careful ? lists : lists & dg;
                        const uint32_t wrapped = PER && !careful ? lists & slow & ~dg : 0u;
                        if (!(bits | wrapped)) continue;
                        ISum T{0ull, 0ull, 0ull, NONE};
                        if constexpr (PER) {
                            if (wrapped) {
                                const IPart<KIND> I = own_part(k);
#pragma unroll 1
                                for (uint32_t todo = wrapped; todo; todo &= todo - 1u) {
                                    const uint32_t el = __ffs(todo) - 1;
#pragma unroll
                                    for (uint32_t tt = 0; tt < NT; ++tt) {
                                        JPart j = load_j(el, tt);
                                        terms(I, j, T, std::true_type(), box);
                                        store_j(el, tt, j);
                                    }
                                }
                            }
                        }
                        const float4 pi = S.ia[k * M + II];
                        const float2 iv = Smem::IB ? S.ib[Smem::IB ? k * M + II : 0] : make_float2(0.f, 0.f);
#pragma unroll 1
                        for (uint32_t todo = bits; todo; todo &= todo - 1u) {
                            const uint32_t el = __ffs(todo) - 1;
                            const uint32_t Je = __shfl_sync(0xffffffffu, J, c + el);
#pragma unroll 1
                            for (uint32_t th = 0; th < 2 * NT; ++th) {
                                const uint32_t tt = th >> 1, h = th & 1u;
                                const uint32_t q = el * HJ + g + tt * G;
                                float *js = reinterpret_cast<float *>(S.js + (el * NT + tt) * 32 + lane) + h;
                                const float *A = reinterpret_cast<const float *>(&S.ja[q]) + h;
                                const float *B = reinterpret_cast<const float *>(&S.jb[q]) + h;
                                const float *C = reinterpret_cast<const float *>(&S.jc[Smem::JC ? q : 0]) + h;
                                const float4 pj = make_float4(A[0], A[2], B[0], B[2]);
                                const float3 dv = pair_dx_acc<PER>(pi, pj, box);
                                const float e2 = d2_of(dv);
                                float fi = 0.f, fj = 0.f;  // coefficients of dv
                                if constexpr (KIND == PASS_DENSITY) {
                                    const float r = sqrt_approx(e2);
                                    const float wi = spline_half_w(sat_fma1(r, pi.w), r * -pi.w);
                                    if (wi > 0.f) T.x = add2_rn(T.x, pk2(pj.w * wi, 0.f));
                                    if constexpr (HL) {
                                        const float wj = spline_half_w(sat_fma1(r, C[0]), r * C[2]);
                                        if (wj > 0.f) *js += iv.x * wj;
                                    }
                                } else if constexpr (KIND == PASS_SPH) {
                                    const float ir = e2 > 0.f ? rsqrtf(e2) : 0.f;  // grad W(0) = 0
                                    const float r = e2 * ir;
                                    // (from P/rho^2: the coefficients may overflow
                                    // where their products with w' do not)
                                    auto grad = [&](float a) {
                                        const float g = spline_third_dw(sat_fma1(r, a), r * a), q = -2.f * a;
                                        return g != 0.f ? g * q * q * q * q : 0.f;
                                    };
                                    const float gi = grad(pi.w), gj = grad(pj.w);
                                    if ((gi != 0.f || gj != 0.f) && e2 > 0.f) {
                                        const float b = ((gi != 0.f ? iv.x * gi : 0.f) + (gj != 0.f ? C[0] * gj : 0.f)) *
                                                        0.954929658551372015f * ir;  // 3/pi
                                        fi = C[2] * b;
                                        fj = iv.y * b;
                                    }
                                } else {
                                    const float d2 = pair_d2<PER>(pi, pj, box);
                                    const bool self = NO_SELF && (s * kSC + k) * M + II == Je * MJ + g + tt * G + h * HJ;
                                    const bool ini = d2 < pi.w && !self;
                                    const bool inj = HL && d2 < pj.w && !self;
                                    if constexpr (KIND == PASS_COUNT) {
                                        T.c += ini ? 1u : 0u;
                                        if (inj) *js = __uint_as_float(__float_as_uint(*js) + 1u);
                                    } else if constexpr (KIND == PASS_MIN) {
                                        if (ini) T.c = min(T.c, __float_as_uint(e2));
                                        if (inj) *js = fminf(*js, e2);
                                    } else if (ini || inj) {
                                        float f;
                                        if constexpr (KIND == PASS_LJ) {
                                            const float ir2 = 1.f / e2;
                                            const float s2 = sig2 * ir2;
                                            const float s6 = s2 * s2 * s2;
                                            f = -(e24 * ir2 * s6 * (2.f * s6 - 1.f));
                                        } else {
                                            const float ir = rsqrtf(e2);
                                            const float ir2 = ir * ir;
                                            const float s2 = sig2 * ir2;
                                            const float s6 = s2 * s2 * s2;
                                            f = -(ir2 * (e24 * s6 * (2.f * s6 - 1.f) + iv.x * C[0] * ir));
                                        }
                                        if (ini) fi = f;
                                        if (inj) fj = f;
                                    }
                                }
                                if constexpr (FORCE) {
                                    if (fi != 0.f) {
                                        T.x = add2_rn(T.x, pk2(fi * dv.x, 0.f));
                                        T.y = add2_rn(T.y, pk2(fi * dv.y, 0.f));
                                        T.z = add2_rn(T.z, pk2(fi * dv.z, 0.f));
                                    }
                                    if constexpr (HL) {
                                        if (fj != 0.f) {
                                            js[0] += fj * dv.x;
                                            js[2 * JS] += fj * dv.y;
                                            js[4 * JS] += fj * dv.z;
                                        }
                                    }
                                }
                            }
                        }
                        const ISum Z{0ull, 0ull, 0ull, NONE};
                        if (k & 1u) keep(k - 1u, Z, T);
                        else keep(k, T, Z);
                    }
                }

                if constexpr (HL) {
                    // the j shares over the M lanes of their i particles (in a fixed
                    // order), then one add per j particle: one task (entry, pair) per
                    // lane; 16-byte reads in an order that spreads over the banks
                    __syncwarp();
                    static_assert(SE * NT * G <= 32, "a task per lane");
                    const uint32_t el = lane / (NT * G), tg = lane % (NT * G);
                    const uint32_t Je = __shfl_sync(0xffffffffu, J, min(c + el, 31u));
                    if (el < ns && ((feeds >> ((c + el) & 31u)) & 1u)) {
                        const uint32_t tt = tg / G, gg = tg % G;
                        const uint32_t j0 = Je * MJ + gg + tt * G;
                        const uint4 *src = reinterpret_cast<const uint4 *>(S.js + (el * NT + tt) * 32 + gg * M);
                        constexpr uint32_t CH = M / 2, JS = SE * NT * 16;
#pragma unroll
                        for (int comp = 0; comp < Smem::NC; ++comp) {
                            f32x2 v = KIND == PASS_MIN ? pk2(INFINITY, INFINITY) : 0ull;
#pragma unroll
                            for (uint32_t ch = 0; ch < CH; ++ch) {
                                const uint4 w = src[comp * JS + (ch ^ ((lane >> 1) & (CH - 1u)))];
                                const f32x2 w0 = ((f32x2)w.y << 32) | w.x, w1 = ((f32x2)w.w << 32) | w.z;
                                if constexpr (INTS) {
                                    const uint32_t l = merge(merge((uint32_t)v, w.x), w.z);
                                    const uint32_t h = merge(merge((uint32_t)(v >> 32), w.y), w.w);
                                    v = ((f32x2)h << 32) | l;
                                } else {
                                    v = add2_rn(v, add2_rn(w0, w1));
                                }
                            }
                            float v0, v1;
                            unpk2(v, v0, v1);
                            if constexpr (KIND == PASS_DENSITY) {  // units of w/2
                                const float x0 = __fmul_rn(v0, hscale) * 2.f, x1 = __fmul_rn(v1, hscale) * 2.f;
                                if (v0 > 0.f) atomicAdd(&a.hsum[j0], fixed_of_nonneg(x0));
                                if (v1 > 0.f) atomicAdd(&a.hsum[j0 + HJ], fixed_of_nonneg(x1));
                                if (fminf(v0, v1) < 0.f) {
                                    if (v0 < 0.f) atomicAdd(&a.hsum[j0], fixed_of_signed(x0));
                                    if (v1 < 0.f) atomicAdd(&a.hsum[j0 + HJ], fixed_of_signed(x1));
                                }
                            } else if constexpr (KIND == PASS_COUNT) {
                                if (__float_as_uint(v0)) atomicAdd(&a.hcnt[j0], __float_as_uint(v0));
                                if (__float_as_uint(v1)) atomicAdd(&a.hcnt[j0 + HJ], __float_as_uint(v1));
                            } else if constexpr (KIND == PASS_MIN) {
                                // (bits of non-negative floats: an integer minimum)
                                if (v0 < INFINITY) atomicMin(&a.hcnt[j0], __float_as_uint(v0));
                                if (v1 < INFINITY) atomicMin(&a.hcnt[j0 + HJ], __float_as_uint(v1));
                            } else {
                                // FP64 adds: their order changes the sum by about
                                // 1e-16 of it, below the FP32 rounding of the output
                                if (v0 != 0.f) atomicAdd(&a.hf[3 * (size_t)j0 + comp], f64_of(-v0));
                                if (v1 != 0.f) atomicAdd(&a.hf[3 * (size_t)(j0 + HJ) + comp], f64_of(-v1));
                            }
                        }
                    }
                }
            }
        }
        }
        if constexpr (INTS) {
#pragma unroll
            for (uint32_t q = 0; q < NK; ++q) rx[q] = __uint_as_float(rc[q]);
        }

        // warps sharing the super-cluster: the first adds the others' sums, in
        // a fixed order (half lists add their sums to memory anyway)
        if (!HL && W != 1u) {
            float *mine = reinterpret_cast<float *>(S.js);
            if (lane == 0) S.seen = selfseen;
            __syncwarp();
#pragma unroll
            for (uint32_t q = 0; q < NK; ++q) {
                mine[q * 32 + lane] = INTS ? rx[q] : __fsub_rn(rx[q], cx[q]);
                if constexpr (FORCE) {
                    mine[(NK + q) * 32 + lane] = __fsub_rn(ry[q], cy[q]);
                    mine[(2 * NK + q) * 32 + lane] = __fsub_rn(rz[q], cz[q]);
                }
            }
            asm volatile("bar.sync %0, %1;" ::"r"(1u + grp), "r"(W * 32u) : "memory");
            if (wig == 0) {
                for (uint32_t w = 1; w < W; ++w) {
                    const float *o = reinterpret_cast<const float *>(all[warp + w].js);
                    selfseen |= all[warp + w].seen;
#pragma unroll
                    for (uint32_t q = 0; q < NK; ++q) {
                        const float v = o[q * 32 + lane];
                        if constexpr (INTS) rx[q] = __uint_as_float(merge(__float_as_uint(rx[q]), __float_as_uint(v)));
                        else sum_add(rx[q], cx[q], v);
                        if constexpr (FORCE) {
                            sum_add(ry[q], cy[q], o[(NK + q) * 32 + lane]);
                            sum_add(rz[q], cz[q], o[(2 * NK + q) * 32 + lane]);
                        }
                    }
                }
            }
            asm volatile("bar.sync %0, %1;" ::"r"(1u + grp), "r"(W * 32u) : "memory");
            if (wig != 0) continue;
        }

        // write in caller order
#pragma unroll
        for (uint32_t q = 0; q < NK; ++q) {
            if constexpr (KIND == PASS_DENSITY || KIND == PASS_SPH) {
                rx[q] = __fsub_rn(rx[q], cx[q]);
                ry[q] = __fsub_rn(ry[q], cy[q]);
                rz[q] = __fsub_rn(rz[q], cz[q]);
            }
            const uint32_t k = cluster_of(q);
            const uint32_t i = (s * kSC + k) * M + II;
            const uint32_t pc = a.perm[i];
            if (pc == 0xffffffffu) continue;  // dummy slot
            const uint32_t o = a.sorted_out ? i : pc;
            // the loop took i = j iff its entry was listed and the range is
            // nonzero (density: -1/(2h) is finite then)
            const float av = S.ia[k * M + II].w;
            const bool seen = (selfseen >> (k * RJ + II / MJ)) & 1u;
            const bool took_self = seen && (KIND == PASS_DENSITY ? isfinite(av) : av > 0.f);
            if constexpr (KIND == PASS_DENSITY) {
                float v = 2.f * rx[q];  // sums are in units of w/2
                // m_i w(0) = m_i  (half lists: the own entries come first, at warp 0)
                if (vw == 0 && !took_self) v += a.aux[i].x;
                if constexpr (HL) {
                    atomicAdd(&a.hsum[i], fixed_of(v * hscale));
                } else {
                    const float hk = 1.f / a.pos[i].w;
                    a.out0[o] = v * (0.318309886183790672f * hk * hk * hk);
                }
            } else if constexpr (KIND == PASS_COUNT) {
                // (of a long list only the warps or block at the own entries saw them)
                const uint32_t v = __float_as_uint(rx[q]) - ((vw == 0 || LONG) && took_self ? 1u : 0u);
                if constexpr (HL) atomicAdd(&a.hcnt[i], v);
                else if (np > 1u) atomicAdd(&a.outc[o], v);
                else a.outc[o] = v;
            } else if constexpr (KIND == PASS_MIN) {
                if constexpr (HL) {
                    if (rx[q] < INFINITY) atomicMin(&a.hcnt[i], __float_as_uint(rx[q]));
                } else if (np > 1u) {
                    atomicMin(reinterpret_cast<unsigned int *>(&a.out0[o]), __float_as_uint(sqrtf(rx[q])));
                } else {
                    a.out0[o] = sqrtf(rx[q]);  // +inf without a neighbor
                }
            } else if constexpr (HL) {
                atomicAdd(&a.hf[3 * (size_t)i + 0], f64_of(rx[q]));
                atomicAdd(&a.hf[3 * (size_t)i + 1], f64_of(ry[q]));
                atomicAdd(&a.hf[3 * (size_t)i + 2], f64_of(rz[q]));
            } else {
                a.out0[o] = rx[q];
                a.out1[o] = ry[q];
                a.out2[o] = rz[q];
            }
        }
    }
}

template <int M, int MJ, int KIND, bool HL>
static cudaError_t launch_packed_mk(const PassArgs &a, int per, int grid, int threads, cudaStream_t s)
{
    // (the periodic arithmetic gives open axes, of infinite length, the open results)
    auto *fn = a.longs ? k_pass_packed<M, MJ, true, KIND, HL, true>
               : per   ? k_pass_packed<M, MJ, true, KIND, HL, false>
                       : k_pass_packed<M, MJ, false, KIND, HL, false>;
    cudaError_t e = set_max_dynamic_smem((const void *)fn, (size_t)(PK_THREADS / 32) * sizeof(PkSmem<M, MJ, KIND, HL>));
    if (e != cudaSuccess) return e;
    fn<<<grid, threads, (size_t)(threads / 32) * sizeof(PkSmem<M, MJ, KIND, HL>), s>>>(a);
    return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_packed(const PassArgs &a, int M, int per, int grid, int threads, cudaStream_t s)
{
    if (threads != 128 && threads != PK_THREADS) return cudaErrorInvalidValue;
    if (a.split != 1 && a.split != 2 && a.split != 4 && (a.split != 8 || threads != 256)) return cudaErrorInvalidValue;
    switch (M * 100 + a.mj) {
    case 808:
        return a.half ? launch_packed_mk<8, 8, KIND, true>(a, per, grid, threads, s)
                      : launch_packed_mk<8, 8, KIND, false>(a, per, grid, threads, s);
    case 1616:
        return a.half ? launch_packed_mk<16, 16, KIND, true>(a, per, grid, threads, s)
                      : launch_packed_mk<16, 16, KIND, false>(a, per, grid, threads, s);
    case 1608:
        return a.half ? cudaErrorInvalidValue : launch_packed_mk<16, 8, KIND, false>(a, per, grid, threads, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace nlg
