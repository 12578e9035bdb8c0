// Cluster-pair search and list encoding (Sec. II-A, II-B, II-C).
//
// One warp per super-cluster (8 i-clusters of M particles), taken from an
// atomic work counter by a persistent grid.  Every step works on 32 items at
// once, one per lane, and hands the survivors to the next:
//   1. the pre-order octree without a stack (skip indices), 32 consecutive
//      nodes at a time against the super-cluster's box inflated by the larger
//      of its radius and the node's (a half search starts at the leaf of its
//      own first particle); where the box is wide against the radii, every
//      particle against the nodes that the box reaches;
//   2. the j-clusters of the leaves reached (MJ particles each, MJ = M or M / 2:
//      the M x MJ tiles of Sec. II-A / III-A), 32 at a time against the boxes of
//      the 8 i-clusters;
//   3. a few single pairs of each candidate tile by the exact FP32 predicate;
//   4. all M x MJ pairs of the tiles still undecided, 32 / M tiles at a time, in
//      fused packed arithmetic whose sign decides them unless it is within its
//      own rounding of zero: then by the exact predicate.
// Periodic systems: only in batches that can hold a wrapped pair (the boxes of
// their j-clusters against the super-cluster's) are the j particles moved to the
// image next to the super-cluster, and the rounding of that is part of the margin
// within which the exact predicate decides.  Differences wrapped pair by pair cost
// twice the open arithmetic, and a second copy of the code for batches without
// wraps waited 2.2 cycles per instruction for the instruction cache.
//
// What bounds it: instruction issue (0.78 per scheduler and cycle on 2^21 particles
// in 64 Plummer spheres), not DRAM; about half of the time goes to step 4, a quarter
// to the walk.  The lane-per-item steps replaced a walk that tested one node, four
// j-clusters and one tile at a time with the whole warp: with fused tile tests 78.7k
// -> 50k warp instructions per super-cluster on those spheres; search stage (half
// lists, CUDA events) 1.18 -> 0.75 ms on the Evrard sphere at 2^21, 15.9 -> 9.2 ms on
// 2^24 particles in 64 Plummer spheres, 3.36 -> 2.22 ms on the 4M-particle fluid.
// Fused tile tests, and images instead of wrapped differences: 0.71, 9.0 and 1.69 ms.
#include <algorithm>
#include <type_traits>

#include "nl_internal.cuh"

namespace nlg {

constexpr int SR_THREADS = 256;
constexpr int SR_WARPS = SR_THREADS / 32;
constexpr int WIN_WORDS = 64;
// A super-cluster is wide, and its particles are tested against the nodes, when
// its box widened by its largest radius exceeds kLoose of its smallest radii, or
// when the boxes alone have reached more than kLooseMin + kLooseRate j-clusters
// per entry found.  Typical lists reach 2.5 to 4 j-clusters per entry; kLoose 3 /
// 5 / 8 gave a search of 9.67 / 9.23 / 9.28 ms on 2^24 particles in 64 Plummer
// spheres and 0.78 / 0.75 / 0.81 ms on a 2^21-particle Evrard sphere; without the
// second condition single super-clusters of the halos ran for 10 ms.
constexpr float kLoose = 5.f;
constexpr uint32_t kLooseMin = 256, kLooseRate = 6;
// Single pairs of every candidate tile that are tested first (search stage on
// the Evrard sphere with 0 / 1 / 2 of them: 0.88 / 0.78 / 0.75 ms).
constexpr int kProbes = 2;

struct SearchCtl {
    const uint32_t *work;   // NULL: super-clusters 0..count-1, else ids
    uint32_t count;
    uint32_t *redo;         // ids that could not be stored this time
    const uint32_t *count_dev;  // optional device count (at most count)
    uint32_t *heavy;            // half search: super-clusters set aside as heavy (NULL: none are)
    unsigned int *n_heavy;
    // the heavy super-clusters in work, nparts j ranges each: phase 1 counts their
    // entries, phase 2 writes them
    int phase;
    uint32_t nparts;
};

__device__ __forceinline__ uint32_t hex_digits(uint32_t v) { return (32u - __clz(v) + 3u) >> 2; }

__device__ __forceinline__ void win_put(uint32_t *win, uint32_t W0, uint32_t p, uint32_t v)
{
    uint32_t l = p - W0;
    atomicOr(&win[l >> 3], v << ((l & 7u) * 4u));
}

// Place of a long record in the list of long records and its seek points
// (kNoSeek: no room), one warp.
__device__ uint32_t long_record(uint32_t cnt, const SearchArgs &a, uint32_t s)
{
    const unsigned lane = lane_id();
    const uint32_t ns = (cnt + kSeek - 1u) / kSeek;
    uint32_t li = 0, seek = 0;
    if (lane == 0) {
        li = atomicAdd(&a.st->n_long, 1u);
        seek = atomicAdd(&a.st->n_seek, ns);
    }
    li = __shfl_sync(0xffffffffu, li, 0);
    seek = __shfl_sync(0xffffffffu, seek, 0);
    const bool room = seek <= a.seek_cap && ns <= a.seek_cap - seek;
    // (the points below the capacity that found no room belong to no record)
    for (uint32_t k = lane; k < ns && seek + k < a.seek_cap; k += 32) a.seek_of[seek + k] = room ? li : kNoSeek;
    if (!room) seek = kNoSeek;
    if (lane == 0) a.long_list[li] = make_uint2(s, seek);
    return seek;
}

// Nibbles of the stream of entries beg .. end (carry: the index before them).
template <class GJ>
__device__ uint32_t stream_nibbles(uint32_t beg, uint32_t end, uint32_t carry, GJ getJ)
{
    const unsigned lane = lane_id();
    uint32_t nib = 0;
    for (uint32_t b0 = beg; b0 < end; b0 += 32) {
        uint32_t t = b0 + lane;
        uint32_t J = t < end ? getJ(t) : 0u;
        uint32_t prev = __shfl_up_sync(0xffffffffu, J, 1);
        if (lane == 0) prev = carry;
        uint32_t d = t < end ? J - prev : 1u;
        uint32_t nb = d == 1u ? 0u : (d <= 9u ? 1u : 1u + hex_digits(d));
        nib += 8u + warp_sum(nb);
        carry = __shfl_sync(0xffffffffu, J, 31);
    }
    return nib;
}

// Mask words of entries beg .. end (beg a multiple of 4).
template <class GM>
__device__ void put_masks(uint32_t *words, uint32_t beg, uint32_t end, GM getM)
{
    for (uint32_t w = beg / 4 + lane_id(); w < (end + 3u) / 4; w += 32) {
        uint32_t v = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t t = 4 * w + q;
            if (t < end) v |= (getM(t) & 0xffu) << (8 * q);
        }
        words[w] = v;
    }
}

// Stream of entries beg .. end from nibble pos on (carry: the index before
// them).  PART: words shared with other stretches (zeroed before) are or-ed in.
// seek: where to note the seek points, or NULL.
template <bool PART, class GJ>
__device__ void put_stream(uint32_t *body, uint32_t *win, uint32_t beg, uint32_t end, uint32_t pos, uint32_t carry,
                           GJ getJ, uint2 *seek)
{
    const unsigned lane = lane_id();
    const unsigned lt = lanemask_lt();
    uint32_t W0 = pos & ~7u;
    bool shared = PART && (pos & 7u);  // the first word of the window
    win[lane] = 0u;
    win[lane + 32] = 0u;
    __syncwarp();
    for (uint32_t b0 = beg; b0 < end; b0 += 32) {
        if (seek && b0 % kSeek == 0 && lane == 0) seek[b0 / kSeek] = make_uint2(pos, carry);
        uint32_t t = b0 + lane;
        bool valid = t < end;
        uint32_t J = valid ? getJ(t) : 0u;
        uint32_t prev = __shfl_up_sync(0xffffffffu, J, 1);
        if (lane == 0) prev = carry;
        uint32_t d = valid ? J - prev : 1u;
        bool bit = d != 1u;
        uint32_t bm = __ballot_sync(0xffffffffu, bit);
        uint32_t ndat = (bit && d > 9u) ? hex_digits(d) : 0u;
        uint32_t info = !bit ? 0u : (d <= 9u ? d + 6u : ndat - 1u);
        uint32_t incl = warp_incl_scan(ndat);
        uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        uint32_t nbits = __popc(bm);
        if (lane < 8) win_put(win, W0, pos + lane, (bm >> (4 * lane)) & 0xfu);
        if (bit) win_put(win, W0, pos + 8 + __popc(bm & lt), info);
        uint32_t pd = pos + 8 + nbits + (incl - ndat);
        for (uint32_t q = 0; q < ndat; ++q) win_put(win, W0, pd + q, (d >> (4 * (ndat - 1 - q))) & 0xfu);
        __syncwarp();
        uint32_t pend = pos + 8 + nbits + tot;
        uint32_t full = (pend - W0) >> 3;
        for (uint32_t w = lane; w < full; w += 32) {
            if (PART && shared && w == 0) atomicOr(&body[W0 >> 3], win[0]);
            else body[(W0 >> 3) + w] = win[w];
        }
        if (full) shared = false;
        __syncwarp();
        uint32_t keep = win[full];
        __syncwarp();
        win[lane] = 0u;
        win[lane + 32] = 0u;
        __syncwarp();
        if (lane == 0) win[0] = keep;
        __syncwarp();
        W0 += full * 8u;
        pos = pend;
        carry = __shfl_sync(0xffffffffu, J, 31);
    }
    if (pos > W0 && lane == 0) {
        if (PART) atomicOr(&body[W0 >> 3], win[0]);
        else body[W0 >> 3] = win[0];
    }
    __syncwarp();
}

// Room for a record of `words` words: its words, or NULL when the list buffer
// is full.  Writes the count and the super-cluster's offset.
__device__ uint32_t *take_record(uint32_t words, uint32_t cnt, const SearchArgs &a, uint32_t s)
{
    const unsigned lane = lane_id();
    unsigned long long off = 0;
    if (lane == 0) off = atomicAdd(&a.st->list_used, (unsigned long long)words * 4ull);
    off = __shfl_sync(0xffffffffu, off, 0);
    if (off + (unsigned long long)words * 4ull > a.list_cap) {
        // reservations only grow, so every record below the lowest failed
        // offset was stored; the host resumes allocation there
        if (lane == 0) atomicMin(&a.st->fail_off, off);
        return nullptr;
    }
    uint32_t *rec = reinterpret_cast<uint32_t *>(a.list + off);
    if (lane == 0) {
        rec[0] = cnt;
        a.rec_off[s] = (uint32_t)(off >> 2);
    }
    return rec;
}

// Encode the list of one super-cluster: entry t is (getJ(t), getM(t)),
// ascending in J.  Returns false when the list buffer is full (nothing
// written for this super-cluster).
// noted: a long record that has its place in the list of long records already.
template <class GJ, class GM>
__device__ bool encode_record(uint32_t cnt, GJ getJ, GM getM, uint32_t *win, const SearchArgs &a,
                              uint32_t s, bool noted = false)
{
    const uint32_t nib = a.compress ? stream_nibbles(0, cnt, 0xffffffffu, getJ) : 0u;  // J_{-1} = -1
    const uint32_t mask_words = (cnt + 3u) >> 2;
    uint32_t *rec = take_record(1u + mask_words + (a.compress ? (nib + 7u) >> 3 : cnt), cnt, a, s);
    if (!rec) return false;
    const uint32_t seek = cnt > kLongList && !noted ? long_record(cnt, a, s) : kNoSeek;
    put_masks(rec + 1, 0, cnt, getM);
    uint32_t *body = rec + 1 + mask_words;
    if (!a.compress) {
        for (uint32_t t = lane_id(); t < cnt; t += 32) body[t] = getJ(t);
        return true;
    }
    put_stream<false>(body, win, 0, cnt, 0, 0xffffffffu, getJ, seek != kNoSeek ? a.seek + seek : nullptr);
    return true;
}

// Half search output of super-cluster s (MJ == M): the staged upper entries
// (J >= 8s, ascending) go to the upper buffer, and every tile (8s+k, J) with
// J beyond the own clusters becomes part of a transposed tuple for
// super-cluster t = J/8: key t * ncl + (8s+k), value = the bits J%8 of all
// such J with the same t (entries of one t are consecutive, at most 8 of
// them, so a group spans at most two 32-entry chunks and is carried over).
// Returns false when a buffer was too small (the reservations still count,
// so the host learns the sizes it needs).
template <class GJ, class GM>
__device__ bool half_tuples(uint32_t cnt, GJ getJ, GM getM, const SearchArgs &a, uint32_t s);

template <class GJ, class GM>
__device__ bool half_output(uint32_t cnt, GJ getJ, GM getM, const SearchArgs &a, uint32_t s)
{
    const unsigned lane = lane_id();
    unsigned long long off = 0;
    if (lane == 0) off = atomicAdd(&a.st->up_used, (unsigned long long)cnt);
    off = __shfl_sync(0xffffffffu, off, 0);
    if (off + cnt > a.up_cap) {
        if (lane == 0) atomicExch(&a.st->half_overflow, 1u);
        return false;
    }
    for (uint32_t t = lane; t < cnt; t += 32) {
        a.uJ[off + t] = getJ(t);
        a.uM[off + t] = (uint8_t)getM(t);
    }
    if (lane == 0) {
        a.up_off[s] = (uint32_t)off;
        a.up_cnt[s] = cnt;
    }
    return half_tuples(cnt, getJ, getM, a, s);
}

// The transposed tuples of entries of super-cluster s (all of one target
// super-cluster together).
template <class GJ, class GM>
__device__ bool half_tuples(uint32_t cnt, GJ getJ, GM getM, const SearchArgs &a, uint32_t s)
{
    const unsigned lane = lane_id();
    constexpr uint32_t NONE = 0xffffffffu;
    const uint32_t own_end = (s + 1) * kSC;  // first cluster after the own ones
    const uint32_t i0 = s * kSC;
    bool ok = true;
    uint32_t carry_t = NONE, carry[kSC];
#pragma unroll
    for (int k = 0; k < kSC; ++k) carry[k] = 0u;
    // reserve and write n tuples of group t from this lane
    auto emit = [&](bool on, uint32_t t, const uint32_t *rows) {
        uint32_t nrow = 0;
#pragma unroll
        for (int k = 0; k < kSC; ++k) nrow += (on && rows[k]) ? 1u : 0u;
        const uint32_t incl = warp_incl_scan(nrow);
        const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        if (tot == 0) return;
        unsigned long long tb = 0;
        if (lane == 0) tb = atomicAdd(&a.st->tu_used, (unsigned long long)tot);
        tb = __shfl_sync(0xffffffffu, tb, 0);
        if (tb + tot > a.tu_cap) {
            ok = false;
            return;
        }
        if (nrow) {
            unsigned long long w = tb + incl - nrow;
#pragma unroll
            for (int k = 0; k < kSC; ++k)
                if (rows[k]) {
                    a.tkey[w] = (uint64_t)t * a.ncl + (i0 + k);
                    a.tval[w] = rows[k];
                    ++w;
                }
            atomicAdd(&a.lower_cnt[t], nrow);
        }
    };
    for (uint32_t b0 = 0; b0 < cnt; b0 += 32) {
        const uint32_t e = b0 + lane;
        const uint32_t J = e < cnt ? getJ(e) : 0u;
        const bool valid = e < cnt && J >= own_end;
        const uint32_t m = valid ? getM(e) : 0u;
        const uint32_t t = valid ? J / kSC : NONE;
        // a carried group that does not continue here is complete
        if (carry_t != NONE && __shfl_sync(0xffffffffu, t, 0) != carry_t) {
            emit(lane == 0, carry_t, carry);
            carry_t = NONE;
        }
        const uint32_t gm = __match_any_sync(0xffffffffu, t);
        uint32_t rows[kSC];
#pragma unroll
        for (int k = 0; k < kSC; ++k) {
            rows[k] = __reduce_or_sync(gm, ((m >> k) & 1u) << (J & 7u));
            if (valid && t == carry_t) rows[k] |= carry[k];
        }
        // the group of the chunk's last entry may continue in the next chunk
        const uint32_t t31 = __shfl_sync(0xffffffffu, t, 31);
        const bool more = b0 + 32 < cnt;
        const bool hold = more && t31 != NONE && t == t31;
#pragma unroll
        for (int k = 0; k < kSC; ++k) carry[k] = __shfl_sync(0xffffffffu, rows[k], 31);
        carry_t = (more && t31 != NONE) ? t31 : NONE;
        emit(valid && lane == (uint32_t)(__ffs(gm) - 1) && !hold, t, rows);
    }
    if (carry_t != NONE) emit(lane == 0, carry_t, carry);
    if (!ok && lane == 0) atomicExch(&a.st->half_overflow, 1u);
    return ok;
}

// j-clusters tested together: one per lane, at most 256 particles staged
template <int MJ>
constexpr uint32_t sr_batch() { return MJ > 8 ? 256 / MJ : 32; }

// Shared memory of one warp: the super-cluster's particles and the boxes of
// its 8 i-clusters, the queue of j-clusters that the walk reached, the staged
// particles of one batch of them, its list of candidate tiles, the masks of
// the tiles found to hold a pair, and the encoder window.  Particles are
// (x, y, z, r^2); squared radii suffice: fl(max(ri, rj)^2) = max(fl(ri^2),
// fl(rj^2)), squaring being monotone.  The boxes are laid out in pairs of
// clusters for packed arithmetic: (lo.x, lo.x', lo.y, lo.y'), (lo.z, lo.z',
// r^2, r'^2), (hi.x, hi.x', hi.y, hi.y'), (hi.z, hi.z', 0, 0).
template <int M, int MJ>
struct SearchSmem {
    float4 ip[kSC * M];                 // i particles
    // j particles of the batch, in pairs (q, q + MJ/2) of a cluster:
    // (x, x', y, y'), (z, z', -r^2, -r'^2)
    float4 ja[sr_batch<MJ>() * MJ / 2], jb[sr_batch<MJ>() * MJ / 2];
    float4 ibox[kSC / 2][4];            // boxes of the i-clusters, in pairs
    uint32_t jq[64];                    // j-clusters to test, ascending (ring)
    uint32_t found[32];                 // per batch slot: tiles holding a pair
    float jrr[32];                      // per batch slot: largest r^2
    uint8_t tl[32 * kSC];               // candidate tiles: slot * 8 + i-cluster
    uint32_t win[WIN_WORDS];
};

// Super-clusters shared by the warps of a block (SPLIT): per batch of
// j-clusters, its first entry in the list and in the staging of the warp that
// tested it.
constexpr uint32_t kSplitBatches = 1024;
struct SplitSmem {
    uint16_t first[kSplitBatches + 1], src[kSplitBatches];
    uint32_t ticket, cnt[SR_WARPS], tiles;
    unsigned long long ttests;
};

// Could some particle of i-cluster box c (pair layout, half e) be a symmetric
// neighbor of one in box B (b squared radius brr)?  The monotone gaps of
// boxes_near.
template <bool PER>
__device__ __forceinline__ void box_pair_near(const float4 *ib, const float4 &blo, const float4 &bhi,
                                              float brr, const PerLen &L, bool &n0, bool &n1)
{
    const float4 A = ib[0], B = ib[1], C = ib[2], D = ib[3];
    float g[3][2];
    if constexpr (PER) {
        g[0][0] = axis_gap_len<true>(A.x, C.x, blo.x, bhi.x, L.x);
        g[0][1] = axis_gap_len<true>(A.y, C.y, blo.x, bhi.x, L.x);
        g[1][0] = axis_gap_len<true>(A.z, C.z, blo.y, bhi.y, L.y);
        g[1][1] = axis_gap_len<true>(A.w, C.w, blo.y, bhi.y, L.y);
        g[2][0] = axis_gap_len<true>(B.x, D.x, blo.z, bhi.z, L.z);
        g[2][1] = axis_gap_len<true>(B.y, D.y, blo.z, bhi.z, L.z);
    } else {
        const f32x2 up[3] = {sub2_rn(pk2(blo.x, blo.x), pk2(C.x, C.y)), sub2_rn(pk2(blo.y, blo.y), pk2(C.z, C.w)),
                             sub2_rn(pk2(blo.z, blo.z), pk2(D.x, D.y))};
        const f32x2 dn[3] = {sub2_rn(pk2(A.x, A.y), pk2(bhi.x, bhi.x)), sub2_rn(pk2(A.z, A.w), pk2(bhi.y, bhi.y)),
                             sub2_rn(pk2(B.x, B.y), pk2(bhi.z, bhi.z))};
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            float u0, u1, d0, d1;
            unpk2(up[ax], u0, u1);
            unpk2(dn[ax], d0, d1);
            g[ax][0] = fmaxf(0.f, fmaxf(u0, d0));
            g[ax][1] = fmaxf(0.f, fmaxf(u1, d1));
        }
    }
    float da, db;
    sum_sq_x2(pk2(g[0][0], g[0][1]), pk2(g[1][0], g[1][1]), pk2(g[2][0], g[2][1]), da, db);
    n0 = da <= fmaxf(B.z, brr);
    n1 = db <= fmaxf(B.w, brr);
}

// Does the canonical difference of some pair of the intervals [a0, a1], [b0, b1]
// wrap around a periodic axis?
__device__ __forceinline__ bool wraps(float a0, float a1, float b0, float b1, float len)
{
    const float half = __fmul_rn(0.5f, len);
    return __fsub_rn(b1, a0) > half || __fsub_rn(b0, a1) < -half;
}

// MODE 0: full list.  MODE 1: half search, upper entries and transposed
// tuples for the record assembly.  MODE 2: half list (each pair stored once,
// Sec. II-D): the half search's upper entries encoded as the record.  MODE 3:
// mode 1 for the parts of heavy super-clusters (ctl.phase).
// SPLIT: the warps of a block share a super-cluster, for systems with fewer of
// them than the chip holds blocks: every warp walks the octree, the batches of
// j-clusters go to the warps in turn, and the first warp encodes the list.
template <int M, int MJ, bool PER, int MODE, bool SPLIT>
__global__ void __launch_bounds__(SR_THREADS, 4) k_search(SearchArgs a, SearchCtl ctl)
{
    static_assert(!SPLIT || MODE != 3, "the parts of heavy super-clusters have a warp each");
    constexpr bool HALF = MODE != 0;  // only j-clusters from the own first one on
    constexpr uint32_t NB = sr_batch<MJ>();
    constexpr uint32_t G = 32 / M;        // tiles tested together, M lanes each
    constexpr uint32_t HJ = MJ / 2;       // pairs of j particles of a cluster
    constexpr int NPI = (kSC * M) / 32;   // i particles per lane
    extern __shared__ __align__(16) unsigned char search_smem[];
    SearchSmem<M, MJ> &S = reinterpret_cast<SearchSmem<M, MJ> *>(search_smem)[threadIdx.x >> 5];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t slot = blockIdx.x * (blockDim.x >> 5) + warp;
    // a warp without staging room stays idle; the work counter hands its
    // super-clusters to the others (warps wait on each other only in a block
    // that shares super-clusters)
    const uint32_t W = blockDim.x >> 5;
    SplitSmem &B = *reinterpret_cast<SplitSmem *>(search_smem + W * sizeof(SearchSmem<M, MJ>));
    if ((SPLIT ? (blockIdx.x + 1u) * W - 1u : slot) >= a.stage_slots) return;
    uint32_t *stJ = a.stageJ + (size_t)slot * a.stage_cap;
    uint8_t *stM = a.stageM + (size_t)slot * a.stage_cap;
    const uint32_t II = lane % M, grp = lane / M;
    // order in which a group of lanes reads the j particles of its tile: the
    // groups read different 16-byte columns of the staged clusters (banks)
    const uint32_t swz = grp & (HJ - 1u);
    const uint32_t gbits = (M == 32 ? 0xffffffffu : ((1u << M) - 1u)) << (grp * M);
    const uint32_t count = ctl.count_dev ? min(ctl.count, *ctl.count_dev) : ctl.count;

    for (;;) {
        uint32_t tk = 0;
        if constexpr (SPLIT) {
            __syncthreads();  // (the last super-cluster is encoded)
            if (threadIdx.x == 0) {
                B.ticket = atomicAdd(&a.st->ticket, 1u);
                B.tiles = 0u;
                B.ttests = 0ull;
            }
            __syncthreads();
            tk = B.ticket;
        } else {
            if (lane == 0) tk = atomicAdd(&a.st->ticket, 1u);
            tk = __shfl_sync(0xffffffffu, tk, 0);
        }
        if (tk >= count) break;
        const uint32_t wi = MODE == 3 ? tk / ctl.nparts : tk;
        const uint32_t s = ctl.work ? ctl.work[wi] : wi;
        const uint32_t base = s * kSC * M;
        // the super-cluster's system: its box and its own octree subtree
        const uint32_t sy = sys_of(a.sys.pad_off, a.sys.nsys, base);
        // particles searched: from the own first one on (half search), or one of
        // nparts ranges of whole super-clusters of them
        uint32_t pbeg = HALF ? base : 0u, pend = 0xffffffffu;
        uint32_t cap = a.stage_cap;
        if constexpr (MODE == 3) {
            const uint32_t n8 = (a.sys.pad_off[sy + 1] - base) / (kSC * M), part = tk % ctl.nparts;
            pbeg = base + (uint32_t)((uint64_t)n8 * part / ctl.nparts) * (kSC * M);
            pend = base + (uint32_t)((uint64_t)n8 * (part + 1) / ctl.nparts) * (kSC * M);
            cap = 0;
            if (ctl.phase == 2) {
                const uint32_t at = a.hpart[tk];
                if (at == kNoPlace) continue;  // (the host starts over)
                stJ = a.uJ + at;
                stM = a.uM + at;
                cap = 0xffffffffu;
            }
            if (pbeg == pend) {
                if (ctl.phase == 1 && lane == 0) a.hpart[tk] = 0u;
                continue;
            }
        }
        const PerLen box = per_len(a.sys.box[sy]);
        // (clamped to the node arrays: after a node overflow in a graph replay
        // the tables may be stale, and the replay is reported as failed)
        const uint32_t vroot = min(a.sys.root[sy], a.nnodes - 1);
        const uint32_t vend = min((uint32_t)__float_as_int(a.nhi[vroot].w), a.nnodes);

        // i-cluster boxes (lane & 7) and the box around all of them
        float4 slo = a.clo[s * kSC + (lane & 7)], shi = a.chi[s * kSC + (lane & 7)];
        __syncwarp();
        if (lane < kSC) {
            float *ib = reinterpret_cast<float *>(&S.ibox[lane >> 1][0]) + (lane & 1);
            ib[0] = slo.x; ib[2] = slo.y; ib[4] = slo.z; ib[6] = __fmul_rn(slo.w, slo.w);
            ib[8] = shi.x; ib[10] = shi.y; ib[12] = shi.z; ib[14] = 0.f;
        }
#pragma unroll
        for (int o = 1; o < kSC; o <<= 1) {
            slo.x = fminf(slo.x, __shfl_xor_sync(0xffffffffu, slo.x, o));
            slo.y = fminf(slo.y, __shfl_xor_sync(0xffffffffu, slo.y, o));
            slo.z = fminf(slo.z, __shfl_xor_sync(0xffffffffu, slo.z, o));
            slo.w = fmaxf(slo.w, __shfl_xor_sync(0xffffffffu, slo.w, o));
            shi.x = fmaxf(shi.x, __shfl_xor_sync(0xffffffffu, shi.x, o));
            shi.y = fmaxf(shi.y, __shfl_xor_sync(0xffffffffu, shi.y, o));
            shi.z = fmaxf(shi.z, __shfl_xor_sync(0xffffffffu, shi.z, o));
            shi.w = fminf(shi.w, __shfl_xor_sync(0xffffffffu, shi.w, o));
        }
#pragma unroll
        for (int t = 0; t < NPI; ++t) {
            const float4 p = a.pos[base + lane + 32 * t];
            const float r = __fmul_rn(a.support, p.w);
            S.ip[lane + 32 * t] = make_float4(p.x, p.y, p.z, __fmul_rn(r, r));
        }
        // a super-cluster whose box is wide against its radii (particles
        // adjacent on the curve can lie far apart in sparse regions) would
        // reach far too many nodes by its box alone: its particles are tested
        // against every node that its box reaches
        const float ext = fmaxf(fmaxf(shi.x - slo.x, shi.y - slo.y), shi.z - slo.z);
        bool loose = !(ext + 2.f * slo.w <= kLoose * shi.w);
        __syncwarp();

        uint32_t cnt = 0, tiles = 0, nvis = 0, lvis = 0, jex = 0, ttests = 0;
        uint32_t qh = 0, qt = 0;  // queue of j-clusters, ring positions
        bool aside = MODE == 1 && !SPLIT && ctl.heavy != nullptr;  // may be set aside
        uint32_t nbatch = 0;                              // SPLIT: batches so far
        // the half search takes only j-clusters from its own first one on
        int lastJ = (int)(pbeg / MJ) - 1;

        // Test a batch of up to NB queued j-clusters.
        auto batch = [&]() {
            const uint32_t nq = min(NB, qt - qh);
            if constexpr (SPLIT) {
                const uint32_t b = nbatch++;
                if (b % W != warp) {  // another warp's
                    qh += nq;
                    return;
                }
                if (lane == 0) B.src[b] = (uint16_t)cnt;
            }
            const uint32_t cnt0 = cnt;
            const uint32_t J = lane < nq ? S.jq[(qh + lane) & 63u] : 0u;
            float4 blo, bhi;
            if (lane < nq) {
                blo = a.jlo[J];
                bhi = a.jhi[J];
            }
            uint32_t mask = 0, cm = 0;
            const float brr = lane < nq ? __fmul_rn(blo.w, blo.w) : 0.f;
            // Periodic: do pairs of the batch wrap?  Not if none of the box corners
            // does (the canonical difference is monotone in both coordinates).  If
            // some may, the j particles are staged in the image next to the
            // super-cluster, where squared distances are within tx of the canonical
            // ones: an image is then the nearest one or beyond every radius if the
            // box and the radii leave room (else all tiles are tested exactly).
            bool wr = false, room = true;
            float tx = 0.f;
            if constexpr (PER) {
                const bool w = lane < nq && (wraps(slo.x, shi.x, blo.x, bhi.x, box.x) ||
                                             wraps(slo.y, shi.y, blo.y, bhi.y, box.y) ||
                                             wraps(slo.z, shi.z, blo.z, bhi.z, box.z));
                wr = __any_sync(0xffffffffu, w);
                if (wr) {
                    // largest radius, and coordinate with its shift
                    float rm = slo.w, am = 0.f;
                    if (lane < nq && blo.x <= bhi.x) {
                        rm = fmaxf(rm, blo.w);
                        am = fmaxf(fmaxf(fmaxf(fabsf(blo.x), fabsf(bhi.x)), fmaxf(fabsf(blo.y), fabsf(bhi.y))),
                                   fmaxf(fabsf(blo.z), fabsf(bhi.z)));
                    }
                    rm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rm)));
                    am = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(am)));
                    auto axis = [&](float lo, float hi, float len) {
                        if (len < INFINITY) {
                            am = fmaxf(am, fmaxf(fabsf(lo), fabsf(hi)) + len);
                            room = room && rm + 0.5f * (hi - lo) < 0.499f * len;
                        }
                    };
                    const float a0 = am;
                    axis(slo.x, shi.x, box.x);
                    axis(slo.y, shi.y, box.y);
                    axis(slo.z, shi.z, box.z);
                    am += a0;
                    // three differences, each at most 2 roundings of am off (margin 2);
                    // where that is not small against the radii (boxes far from the
                    // origin or very large), too many tiles would be left undecided
                    tx = fmaf(am * 1e-6f, rm, am * am * 1e-12f);
                    room = room && tx <= 1e-3f * rm * rm;
                    if (!room) tx = 0.f;
                }
            }
            // 1. box tests, one j-cluster per lane against the 8 i-clusters
            if (lane < nq) {
                S.jrr[lane] = brr;
                if (PER && wr) {
#pragma unroll 1
                    for (int k = 0; k < kSC; k += 2) {
                        bool n0, n1;
                        box_pair_near<PER>(S.ibox[k >> 1], blo, bhi, brr, box, n0, n1);
                        cm |= (n0 ? 1u << k : 0u) | (n1 ? 2u << k : 0u);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < kSC; k += 2) {
                        bool n0, n1;
                        box_pair_near<false>(S.ibox[k >> 1], blo, bhi, brr, box, n0, n1);
                        cm |= (n0 ? 1u << k : 0u) | (n1 ? 2u << k : 0u);
                    }
                }
            }
            if (__any_sync(0xffffffffu, cm != 0u)) {
                // 2. stage the j particles
                for (uint32_t q = lane; q < nq * HJ; q += 32) {
                    const float4 *p = a.pos + S.jq[(qh + q / HJ) & 63u] * MJ + q % HJ;
                    float4 p0 = p[0], p1 = p[HJ];
                    if (PER && wr && room) {
                        auto image = [](float x, float lo, float hi, float len) {
                            const float d = x - 0.5f * (lo + hi);
                            return d > 0.5f * len ? x - len : d < -0.5f * len ? x + len : x;
                        };
                        p0.x = image(p0.x, slo.x, shi.x, box.x);
                        p0.y = image(p0.y, slo.y, shi.y, box.y);
                        p0.z = image(p0.z, slo.z, shi.z, box.z);
                        p1.x = image(p1.x, slo.x, shi.x, box.x);
                        p1.y = image(p1.y, slo.y, shi.y, box.y);
                        p1.z = image(p1.z, slo.z, shi.z, box.z);
                    }
                    const float r0 = __fmul_rn(a.support, p0.w), r1 = __fmul_rn(a.support, p1.w);
                    S.ja[q] = make_float4(p0.x, p1.x, p0.y, p1.y);
                    S.jb[q] = make_float4(p0.z, p1.z, -__fmul_rn(r0, r0), -__fmul_rn(r1, r1));
                }
                __syncwarp();
                // particle jj of batch slot sl
                auto staged = [&](uint32_t sl, uint32_t jj) {
                    const uint32_t q = sl * HJ + (jj & (HJ - 1u)), h = jj / HJ;
                    const float *A = reinterpret_cast<const float *>(&S.ja[q]) + h;
                    const float *B = reinterpret_cast<const float *>(&S.jb[q]) + h;
                    return make_float4(A[0], A[2], B[0], -B[2]);
                };
                // 3. single pairs of every candidate tile, one j-cluster per
                // lane: most tiles that hold a pair are found here (about half
                // of all pairs of such tiles are neighbors)
                if (cm && room) {
                    const float part = wr ? 1.f - 2e-6f : 1.f;  // (1: the canonical predicate)
#pragma unroll
                    for (int q = 0; q < kProbes; ++q) {
                        const float4 pj = staged(lane, (lane + q * HJ) & (MJ - 1));
#pragma unroll
                        for (int k = 0; k < kSC; ++k) {
                            const float4 pi = S.ip[k * M + (q * (M / 2) + M / 4)];
                            const float d2 = pair_d2<false>(pi, pj, box);
                            // (a self pair has d2 = 0)
                            if (d2 < fmaf(fmaxf(pi.w, pj.w), part, -tx) && d2 > 0.f) mask |= 1u << k;
                        }
                    }
                    cm &= ~mask;
                }
                S.found[lane] = mask;
                // list of the other candidate tiles
                const uint32_t pc = __popc(cm);
                const uint32_t incl = warp_incl_scan(pc);
                const uint32_t T = __shfl_sync(0xffffffffu, incl, 31);
                uint32_t at = incl - pc;
                for (uint32_t b = cm; b; b &= b - 1u) S.tl[at++] = (uint8_t)(lane * kSC + __ffs(b) - 1);
                ttests += T;
                __syncwarp();
                // 4. FP32 test of these tiles, G at a time: a lane holds one i
                // particle of its group's tile and takes the MJ j particles in turn
                const uint32_t J0 = S.jq[qh & 63u];
                const bool own = J0 * MJ < base + kSC * M && S.jq[(qh + nq - 1u) & 63u] * MJ >= base;
                for (uint32_t t0 = 0; t0 < T; t0 += G) {
                    const uint32_t e = S.tl[min(t0 + grp, T - 1u)];
                    const uint32_t sl = e >> 3, k = e & 7u;
                    const float4 pi = S.ip[k * M + II];
                    // pair (i, j) is a self pair iff jj == delta
                    const uint32_t Jt = S.jq[(qh + sl) & 63u];
                    const uint32_t delta = base + k * M + II - Jt * MJ;
                    bool hit = false;
                    if (PER && !room) {
#pragma unroll 4
                        for (uint32_t t = 0; t < (uint32_t)MJ; ++t) {
                            const uint32_t jj = t ^ swz;
                            const float4 pj = staged(sl, jj);
                            hit |= pair_d2<PER>(pi, pj, box) < fmaxf(pi.w, pj.w) && jj != delta;
                        }
                    } else {
                        // min of d2 - max(ri^2, rj^2), two j particles at a time in
                        // fused arithmetic.  It and the canonical predicate's sum
                        // are each within 2^-22 of the radius squared (and tx) of the
                        // true value near zero: only a minimum within tol of zero
                        // needs the exact test; so do tiles holding self pairs.
                        const float nri = -pi.w;
                        const f32x2 ix = pk2(pi.x, pi.x), iy = pk2(pi.y, pi.y), iz = pk2(pi.z, pi.z);
                        float mn = INFINITY;
#pragma unroll
                        for (uint32_t t = 0; t < HJ; ++t) {
                            const uint32_t q = sl * HJ + (t ^ swz);
                            const float4 A = S.ja[q], B = S.jb[q];
                            const f32x2 dx = sub2_rn(pk2(A.x, A.y), ix), dy = sub2_rn(pk2(A.z, A.w), iy);
                            const f32x2 dz = sub2_rn(pk2(B.x, B.y), iz);
                            const f32x2 m = pk2(fminf(nri, B.z), fminf(nri, B.w));
                            float d0, d1;
                            unpk2(fma2_rn(dz, dz, fma2_rn(dy, dy, fma2_rn(dx, dx, m))), d0, d1);
                            mn = fminf(mn, fminf(d0, d1));
                        }
                        const float tol = fmaf(fmaxf(pi.w, S.jrr[sl]), 2e-6f, tx + 1e-37f);
                        hit = mn < -tol;
                        const bool exact = (!hit && mn <= tol) || (own && delta < (uint32_t)MJ);
                        if (__any_sync(0xffffffffu, exact)) {  // (particles as they are, not their images)
                            if (exact) hit = false;
#pragma unroll 2
                            for (uint32_t jj = 0; jj < (uint32_t)MJ; ++jj) {
                                const float4 pj = a.pos[(size_t)Jt * MJ + jj];
                                const float r = __fmul_rn(a.support, pj.w);
                                hit |= pair_d2<PER>(pi, pj, box) < fmaxf(pi.w, __fmul_rn(r, r)) && jj != delta;
                            }
                        }
                    }
                    const uint32_t hb = __ballot_sync(0xffffffffu, hit) & gbits;
                    if (II == 0 && hb) atomicOr(&S.found[sl], 1u << k);
                }
                __syncwarp();
                // 5. j-clusters with a tile holding a pair
                mask = S.found[lane];
                const uint32_t has = __ballot_sync(0xffffffffu, mask != 0u);
                const uint32_t o = cnt + __popc(has & lanemask_lt());
                if (mask && o < cap) {
                    stJ[o] = J;
                    stM[o] = (uint8_t)mask;
                }
                cnt += __popc(has);
                tiles += __popc(mask);
                __syncwarp();
            }
            if (SPLIT && lane == 0) B.first[nbatch] = (uint16_t)(cnt - cnt0);
            qh += nq;
        };

        // Stackless pre-order walk of the system's subtree, 32 consecutive
        // nodes at a time: each lane tests one node against the
        // super-cluster's box (the descendants of a node that fails fail too,
        // the gaps being monotone), and the walk continues after the subtree
        // of the last failing node that reaches beyond the chunk.  The
        // j-clusters of the leaves that pass are queued until a batch is full.
        uint32_t v = vroot, leaves = 0;  // leaves: of the current chunk, not queued yet
        if constexpr (HALF) {
            // start at the leaf that holds the first particle: the last node in
            // pre-order whose range begins at or before it (the range starts
            // ascend in pre-order); 32 probes a round
            uint32_t hi = vend;  // nodes [v, hi) may be it; v itself begins early enough
            while (hi - v > 1) {
                const uint32_t step = (hi - v + 31u) >> 5;
                const uint32_t u = v + lane * step;
                const uint32_t m = __ballot_sync(0xffffffffu, u < hi && (uint32_t)a.nrng[min(u, vend - 1)].x <= pbeg);
                const uint32_t last = 31u - __clz(m | 1u);
                v += last * step;
                hi = min(hi, v + step);
            }
        }
        int2 rg = make_int2(0, 0);       // particle range of this lane's node
        int Jlo = 0, Jhi = -1;           // j-clusters of the current leaf, not queued yet
        for (;;) {
            while (qt - qh < NB) {
                if (Jlo <= Jhi) {
                    const uint32_t c = min((uint32_t)(Jhi - Jlo + 1), 32u);
                    if (lane < c) S.jq[(qt + lane) & 63u] = (uint32_t)Jlo + lane;
                    qt += c;
                    Jlo += 32;
                    continue;
                }
                if (leaves) {  // (leaves can share a j-cluster)
                    const int b = __ffs(leaves) - 1;
                    leaves &= leaves - 1u;
                    Jlo = max(__shfl_sync(0xffffffffu, rg.x, b) / MJ, lastJ + 1);
                    Jhi = (__shfl_sync(0xffffffffu, rg.y, b) - 1) / MJ;
                    if (MODE == 3) Jhi = (int)min((uint32_t)Jhi, pend / MJ - 1u);
                    lastJ = max(lastJ, Jhi);
                    ++lvis;
                    jex += (uint32_t)max(Jhi - Jlo + 1, 0);
                    continue;
                }
                if (v >= vend) break;
                const uint32_t u = v + lane;
                float4 nlo = make_float4(0.f, 0.f, 0.f, 0.f), nhi = nlo;
                bool near = false;
                uint32_t skip = 0;
                if (u < vend) {
                    nlo = a.nlo[u];
                    nhi = a.nhi[u];
                    rg = a.nrng[u];
                    skip = (uint32_t)__float_as_int(nhi.w);
                    // (wholly before the first particle: not for a half search)
                    near = (!HALF || (uint32_t)rg.y > pbeg) && (MODE != 3 || (uint32_t)rg.x < pend) &&
                           boxes_near<PER>(slo, shi, nlo, nhi, box);
                }
                uint32_t next = max(v + 32u, __reduce_max_sync(0xffffffffu, near ? 0u : skip));
                if (MODE == 3 && __any_sync(0xffffffffu, u < vend && (uint32_t)rg.x >= pend)) next = vend;
                leaves = __ballot_sync(0xffffffffu, near && skip == u + 1u);
                nvis += min(32u, vend - v);
                // (also when few of the j-clusters reached by boxes hold a pair)
                // (not where warps share it: all must form the same batches)
                loose = loose || (!SPLIT && jex > kLooseMin + kLooseRate * cnt);
                if (loose) {
                    // particles against the leaves and the nodes reaching beyond the chunk
                    const uint32_t big = __ballot_sync(0xffffffffu, near && skip > v + 32u);
                    for (uint32_t todo = leaves | big; todo;) {
                        const int b = __ffs(todo) - 1;
                        todo &= todo - 1u;
                        const float4 lo = make_float4(__shfl_sync(0xffffffffu, nlo.x, b), __shfl_sync(0xffffffffu, nlo.y, b),
                                                      __shfl_sync(0xffffffffu, nlo.z, b), 0.f);
                        const float4 hi = make_float4(__shfl_sync(0xffffffffu, nhi.x, b), __shfl_sync(0xffffffffu, nhi.y, b),
                                                      __shfl_sync(0xffffffffu, nhi.z, b), 0.f);
                        const float nr = __shfl_sync(0xffffffffu, nlo.w, b), nrr = __fmul_rn(nr, nr);
                        bool any = false;
#pragma unroll
                        for (int t = 0; t < NPI; ++t) {
                            const float4 p = S.ip[lane + 32 * t];
                            const float gx = axis_gap_len<PER>(p.x, p.x, lo.x, hi.x, box.x);
                            const float gy = axis_gap_len<PER>(p.y, p.y, lo.y, hi.y, box.y);
                            const float gz = axis_gap_len<PER>(p.z, p.z, lo.z, hi.z, box.z);
                            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)), __fmul_rn(gz, gz));
                            any |= p.x == p.x && d2 <= fmaxf(p.w, nrr);  // (dummies are NaN)
                        }
                        if (__any_sync(0xffffffffu, any)) continue;
                        leaves &= ~(1u << b);
                        if ((big >> b) & 1u) {  // all later nodes of the chunk lie in its subtree
                            leaves &= (1u << b) - 1u;
                            next = max(next, __shfl_sync(0xffffffffu, skip, b));
                            break;
                        }
                    }
                }
                v = next;
            }
            if (qt == qh) break;
            __syncwarp();
            batch();
            if (MODE == 1 && aside && cnt > kLongSearch) {
                // too long for one warp: set aside for the search in parts
                uint32_t h = 0;
                if (lane == 0) {
                    h = atomicAdd(ctl.n_heavy, 1u);
                    if (h < a.hcap) ctl.heavy[h] = s;
                }
                h = __shfl_sync(0xffffffffu, h, 0);
                if (h < a.hcap) break;
                aside = false;
            }
        }
        __syncwarp();
        if (MODE == 1 && aside && cnt > kLongSearch) continue;
        bool staged = cnt <= a.stage_cap;
        if constexpr (SPLIT) {
            // the batches' places in the list; the first warp goes on with it
            tiles = warp_sum(tiles);
            if (lane == 0) {
                B.cnt[warp] = cnt;
                atomicAdd(&B.tiles, tiles);
                atomicAdd(&B.ttests, (unsigned long long)ttests);
            }
            __syncthreads();
            if (warp != 0) continue;
            cnt = 0;
            for (uint32_t w = 0; w < W; ++w) {
                cnt += B.cnt[w];
                staged = staged && B.cnt[w] <= a.stage_cap;
            }
            staged = staged && cnt <= a.stage_cap;
            uint32_t at = 0;
            for (uint32_t b0 = 0; b0 < nbatch; b0 += 32) {
                const uint32_t c = b0 + lane < nbatch ? B.first[b0 + lane + 1] : 0u;
                const uint32_t incl = warp_incl_scan(c);
                if (b0 + lane < nbatch) B.first[b0 + lane + 1] = (uint16_t)(at + incl);
                at += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) B.first[0] = 0;
            __syncwarp();
            tiles = lane == 0 ? B.tiles : 0u;
            ttests = (uint32_t)B.ttests;
        }
        // entry t: in the staging of the warp of its batch
        auto place = [&](uint32_t t) -> size_t {
            if constexpr (!SPLIT) return t;
            uint32_t lo = 0, hi = nbatch;  // first[lo] <= t < first[hi]
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (B.first[mid] <= t) lo = mid;
                else hi = mid;
            }
            return (size_t)(lo % W) * a.stage_cap + B.src[lo] + (t - B.first[lo]);
        };
        auto getJ = [&](uint32_t t) { return stJ[place(t)]; };
        auto getM = [&](uint32_t t) { return (uint32_t)stM[place(t)]; };
        if constexpr (MODE == 3) {
            if (ctl.phase == 1) {
                if (lane == 0) a.hpart[tk] = cnt;
            } else if (!half_tuples(cnt, getJ, getM, a, s) && lane == 0) {
                atomicExch(&a.st->half_overflow, 1u);
            }
            if (lane == 0 && ctl.phase == 2) {
                atomicAdd(&a.st->node_visits, (unsigned long long)nvis);
                atomicAdd(&a.st->leaf_visits, (unsigned long long)lvis);
                atomicAdd(&a.st->j_examined, (unsigned long long)jex);
                atomicAdd(&a.st->tile_tests, (unsigned long long)ttests);
            }
            continue;
        }
        tiles = warp_sum(tiles);
        bool ok = staged;
        if (!staged) {
            if (lane == 0) atomicMax(&a.st->max_count, cnt);
        } else if constexpr (MODE == 1) {
            // a buffer overflow here makes the host re-run every super-cluster
            ok = half_output(cnt, getJ, getM, a, s);
        } else {
            ok = encode_record(cnt, getJ, getM, S.win, a, s);
            if (!ok && lane == 0) atomicExch(&a.st->list_overflow, 1u);
        }
        if (lane == 0) {
            if (!ok) {
                if (MODE != 1 || !staged) {
                    uint32_t r = atomicAdd(&a.st->stage_overflow, 1u);
                    ctl.redo[r] = s;
                }
                a.rec_off[s] = kBadRecord;
            } else if (MODE != 1) {
                atomicAdd(&a.st->n_entries, (unsigned long long)cnt);
                atomicAdd(&a.st->n_tiles, (unsigned long long)tiles);
            }
            atomicAdd(&a.st->node_visits, (unsigned long long)nvis);
            atomicAdd(&a.st->leaf_visits, (unsigned long long)lvis);
            atomicAdd(&a.st->j_examined, (unsigned long long)jex);
            atomicAdd(&a.st->tile_tests, (unsigned long long)ttests);
        }
    }
}

template <int M, int MJ, int MODE, bool SPLIT = false>
static cudaError_t launch_m(const SearchArgs &a, const SearchCtl &c, int per, int grid, int threads,
                            cudaStream_t s)
{
    const size_t extra = SPLIT ? sizeof(SplitSmem) : 0;
    auto *fn = per ? k_search<M, MJ, true, MODE, SPLIT> : k_search<M, MJ, false, MODE, SPLIT>;
    cudaError_t e = set_max_dynamic_smem((const void *)fn, (size_t)SR_WARPS * sizeof(SearchSmem<M, MJ>) + extra);
    if (e != cudaSuccess) return e;
    fn<<<grid, threads, (size_t)(threads / 32) * sizeof(SearchSmem<M, MJ>) + extra, s>>>(a, c);
    return cudaGetLastError();
}

// The warps of a block share a super-cluster when there are at most three of
// them per resident block, unless their lists may hold more batches or entries
// than the block's tables.  Search of an Evrard sphere (half / full lists, ms, a
// warp each -> shared): 512 super-clusters 0.118 / 0.138 -> 0.066 / 0.078, 1216
// 0.134 / 0.145 -> 0.091 / 0.117, 1875 0.141 / 0.153 -> 0.118 / 0.155, 2422 0.149 /
// 0.160 -> 0.148 / 0.197; periodic cubes of 4096 and 32768 particles 0.34 -> 0.14,
// 0.43 -> 0.18.
template <int M, int MJ, int MODE>
static cudaError_t launch_split(const SearchArgs &a, const SearchCtl &c, int per, int grid, int threads,
                                cudaStream_t s)
{
    const uint64_t batches = ((uint64_t)a.nsc * kSC * (M / MJ)) / sr_batch<MJ>() + 2;
    if (a.nsc <= 3u * (uint32_t)grid && batches <= kSplitBatches && a.stage_cap < 65536u / SR_WARPS)
        return launch_m<M, MJ, MODE, true>(a, c, per, (int)std::min<uint32_t>(c.count, (uint32_t)grid), threads, s);
    return launch_m<M, MJ, MODE>(a, c, per, grid, threads, s);
}

cudaError_t launch_search_ctl(const SearchArgs &a, const uint32_t *work, uint32_t count,
                              uint32_t *redo, int M, int any_periodic, int grid, int threads,
                              cudaStream_t s, const uint32_t *count_dev)
{
    SearchCtl c{work, count, redo, count_dev, a.half == 1 ? a.heavy[any_periodic ? 1 : 0] : nullptr,
                &a.st->n_heavy[any_periodic ? 1 : 0], 0, 0};
    if (threads != 128 && threads != SR_THREADS) return cudaErrorInvalidValue;
    if (a.half && a.mj != M) return cudaErrorInvalidValue;  // needs j-clusters = i-clusters
    if (a.half < 0 || a.half > 2) return cudaErrorInvalidValue;
    if (count == 0) return cudaSuccess;
#define NL_SEARCH(M_, MJ_, MODE_) \
    return launch_split<M_, MJ_, MODE_>(a, c, any_periodic, grid, threads, s)
    switch (M * 100 + a.mj) {
    case 404:
        if (a.half == 1) NL_SEARCH(4, 4, 1);
        if (a.half == 2) NL_SEARCH(4, 4, 2);
        NL_SEARCH(4, 4, 0);
    case 808:
        if (a.half == 1) NL_SEARCH(8, 8, 1);
        if (a.half == 2) NL_SEARCH(8, 8, 2);
        NL_SEARCH(8, 8, 0);
    case 804: NL_SEARCH(8, 4, 0);
    case 1616:
        if (a.half == 1) NL_SEARCH(16, 16, 1);
        if (a.half == 2) NL_SEARCH(16, 16, 2);
        NL_SEARCH(16, 16, 0);
    case 1608: NL_SEARCH(16, 8, 0);
    default: return cudaErrorInvalidValue;
    }
#undef NL_SEARCH
}

// Upper entries of a heavy super-cluster from the counts of its parts: one
// reservation, then the place of every part (one warp per super-cluster).  Parts
// with a place are searched to their end also when the tuples have no room left,
// so that the host learns how many there are (stopping at the first that did not
// fit made it start over with a little more room, again and again, until it gave up
// on systems in which most super-clusters are heavy).
__global__ void __launch_bounds__(128) k_heavy_place(SearchArgs a, const uint32_t *heavy, uint32_t count, uint32_t nparts)
{
    const uint32_t h = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (h >= count) return;
    const unsigned lane = lane_id();
    uint32_t *part = a.hpart + (size_t)h * nparts, cnt = 0;
    for (uint32_t p = lane; p < nparts; p += 32) cnt += part[p];
    cnt = warp_sum(cnt);
    unsigned long long off = 0;
    if (lane == 0) off = atomicAdd(&a.st->up_used, (unsigned long long)cnt);
    off = __shfl_sync(0xffffffffu, off, 0);
    if (off + cnt > a.up_cap) {
        for (uint32_t p = lane; p < nparts; p += 32) part[p] = kNoPlace;
        if (lane == 0) atomicExch(&a.st->half_overflow, 1u);
        return;
    }
    if (lane == 0) {
        a.up_off[heavy[h]] = (uint32_t)off;
        a.up_cnt[heavy[h]] = cnt;
    }
    uint32_t at = (uint32_t)off;
    for (uint32_t p0 = 0; p0 < nparts; p0 += 32) {
        const uint32_t c = p0 + lane < nparts ? part[p0 + lane] : 0u;
        const uint32_t incl = warp_incl_scan(c);
        if (p0 + lane < nparts) part[p0 + lane] = at + incl - c;
        at += __shfl_sync(0xffffffffu, incl, 31);
    }
}

cudaError_t launch_search_heavy(const SearchArgs &a, uint32_t count, uint32_t nparts, int M, int per, int grid,
                                int threads, cudaStream_t s)
{
    if (a.half != 1 || !count || !nparts) return cudaErrorInvalidValue;
    const uint32_t *heavy = a.heavy[per ? 1 : 0];
    for (int phase = 1; phase <= 2; ++phase) {
        SearchCtl c{heavy, count * nparts, nullptr, nullptr, nullptr, nullptr, phase, nparts};
        cudaError_t e = cudaMemsetAsync(&a.st->ticket, 0, sizeof(a.st->ticket), s);
        if (e != cudaSuccess) return e;
        switch (M) {
        case 4: e = launch_m<4, 4, 3>(a, c, per, grid, threads, s); break;
        case 8: e = launch_m<8, 8, 3>(a, c, per, grid, threads, s); break;
        case 16: e = launch_m<16, 16, 3>(a, c, per, grid, threads, s); break;
        default: e = cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
        if (phase == 1) k_heavy_place<<<(count + 3) / 4, 128, 0, s>>>(a, heavy, count, nparts);
    }
    return cudaGetLastError();
}

// Record assembly of the half search: one warp per super-cluster t.  Its
// record is the sorted tuples addressed to it (j-clusters below its own
// clusters; keys t * ncl + J, values the mask bits) followed by its upper
// entries, encoded exactly like a record of the full search.
struct AssembleSrc {
    const uint64_t *tkey;
    const uint32_t *tval, *uJ;
    const uint8_t *uM;
    uint64_t kb;
    uint32_t lc, so, uc, uo;
    __device__ AssembleSrc(const SearchArgs &a, uint32_t t)
        : tkey(a.tkey), tval(a.tval), uJ(a.uJ), uM(a.uM), kb((uint64_t)t * a.ncl), lc(a.lower_cnt[t]),
          so(a.seg_off[t]), uc(a.up_cnt[t]), uo(a.up_off[t])
    {
    }
    __device__ uint32_t count() const { return lc + uc; }
    __device__ uint32_t J(uint32_t i) const { return i < lc ? (uint32_t)(tkey[so + i] - kb) : uJ[uo + (i - lc)]; }
    __device__ uint32_t M(uint32_t i) const { return i < lc ? tval[so + i] : (uint32_t)uM[uo + (i - lc)]; }
};

__global__ void __launch_bounds__(SR_THREADS) k_assemble(SearchArgs a)
{
    __shared__ uint32_t wins[SR_WARPS][WIN_WORDS];
    const unsigned lane = lane_id();
    uint32_t *win = wins[threadIdx.x >> 5];
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&a.st->asm_ticket, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= a.nsc) break;
        if (a.st->half_overflow || a.st->stage_overflow) {
            // incomplete tuples or upper entries (a graph replay that outgrew
            // its buffers, reported by nl_graph_check): empty records
            if (lane == 0) a.rec_off[t] = kBadRecord;
            continue;
        }
        const AssembleSrc src(a, t);
        const uint32_t cnt = src.count();
        const bool noted = a.defer_long && cnt > kLongList;
        if (noted && long_record(cnt, a, t) != kNoSeek) continue;
        const bool ok = encode_record(
            cnt, [&](uint32_t i) { return src.J(i); }, [&](uint32_t i) { return src.M(i); }, win, a, t, noted);
        uint32_t tiles = 0;
        for (uint32_t i = lane; i < cnt; i += 32) tiles += __popc(src.M(i));
        tiles = warp_sum(tiles);
        if (lane == 0) {
            if (!ok) {
                atomicExch(&a.st->list_overflow, 1u);
                a.rec_off[t] = kBadRecord;
            } else {
                atomicAdd(&a.st->n_entries, (unsigned long long)cnt);
                atomicAdd(&a.st->n_tiles, (unsigned long long)tiles);
            }
        }
    }
}

// Long records, one warp per stretch of kSeek entries: the nibbles of its stream
// (the seek point holds them and the index before the stretch for now).
__global__ void __launch_bounds__(SR_THREADS) k_long_count(SearchArgs a, uint32_t n_seek)
{
    const uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (q >= n_seek || a.seek_of[q] == kNoSeek) return;
    const uint2 l = a.long_list[a.seek_of[q]];
    const AssembleSrc src(a, l.x);
    const uint32_t beg = (q - l.y) * kSeek, end = min(src.count(), beg + kSeek);
    const uint32_t prev = beg ? src.J(beg - 1u) : 0xffffffffu;
    const uint32_t nib = a.compress ? stream_nibbles(beg, end, prev, [&](uint32_t i) { return src.J(i); }) : 0u;
    if (lane_id() == 0) a.seek[q] = make_uint2(nib, prev);
}

// ... the record's place, the stretches' places in its stream, and zeros in the
// words that stretches share (one warp per record).
__global__ void __launch_bounds__(SR_THREADS) k_long_place(SearchArgs a, uint32_t n_long)
{
    const uint32_t li = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (li >= n_long) return;
    const unsigned lane = lane_id();
    const uint2 l = a.long_list[li];
    if (l.y == kNoSeek) return;  // (encoded by the assembly)
    const uint32_t cnt = AssembleSrc(a, l.x).count(), ns = (cnt + kSeek - 1u) / kSeek;
    uint32_t nib = 0;
    for (uint32_t k0 = 0; k0 < ns; k0 += 32) {
        const uint32_t c = k0 + lane < ns ? a.seek[l.y + k0 + lane].x : 0u;
        const uint32_t incl = warp_incl_scan(c);
        if (k0 + lane < ns) a.seek[l.y + k0 + lane].x = nib + incl - c;
        nib += __shfl_sync(0xffffffffu, incl, 31);
    }
    const uint32_t mask_words = (cnt + 3u) >> 2, body_words = a.compress ? (nib + 7u) >> 3 : cnt;
    uint32_t *rec = take_record(1u + mask_words + body_words, cnt, a, l.x);
    if (!rec) {
        if (lane == 0) {
            atomicExch(&a.st->list_overflow, 1u);
            a.rec_off[l.x] = kBadRecord;
        }
        return;
    }
    if (a.compress) {
        uint32_t *body = rec + 1 + mask_words;
        __syncwarp();
        for (uint32_t k = lane; k < ns; k += 32) body[a.seek[l.y + k].x >> 3] = 0u;
        if (lane == 0) body[body_words - 1u] = 0u;
    }
}

// ... masks and stream of every stretch.
__global__ void __launch_bounds__(SR_THREADS) k_long_put(SearchArgs a, uint32_t n_seek)
{
    __shared__ uint32_t wins[SR_WARPS][WIN_WORDS];
    const uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (q >= n_seek || a.seek_of[q] == kNoSeek) return;
    const unsigned lane = lane_id();
    const uint2 l = a.long_list[a.seek_of[q]];
    const uint32_t roff = a.rec_off[l.x];
    if (roff == kBadRecord) return;  // (no room: the host grows the list and starts over)
    const AssembleSrc src(a, l.x);
    const uint32_t cnt = src.count(), beg = (q - l.y) * kSeek, end = min(cnt, beg + kSeek);
    uint32_t *rec = reinterpret_cast<uint32_t *>(a.list) + roff;
    auto getJ = [&](uint32_t i) { return src.J(i); };
    put_masks(rec + 1, beg, end, [&](uint32_t i) { return src.M(i); });
    uint32_t *body = rec + 1 + ((cnt + 3u) >> 2);
    if (a.compress) {
        const uint2 at = a.seek[q];
        put_stream<true>(body, wins[threadIdx.x >> 5], beg, end, at.x, at.y, getJ, nullptr);
    } else {
        for (uint32_t t = beg + lane; t < end; t += 32) body[t] = getJ(t);
    }
    uint32_t tiles = 0;
    for (uint32_t i = beg + lane; i < end; i += 32) tiles += __popc(src.M(i));
    tiles = warp_sum(tiles);
    if (lane == 0) {
        atomicAdd(&a.st->n_entries, (unsigned long long)(end - beg));
        atomicAdd(&a.st->n_tiles, (unsigned long long)tiles);
    }
}

cudaError_t launch_assemble_long(const SearchArgs &a, uint32_t n_long, uint32_t n_seek, cudaStream_t s)
{
    if (!n_seek) return cudaSuccess;
    k_long_count<<<(n_seek + SR_WARPS - 1) / SR_WARPS, SR_THREADS, 0, s>>>(a, n_seek);
    k_long_place<<<(n_long + SR_WARPS - 1) / SR_WARPS, SR_THREADS, 0, s>>>(a, n_long);
    k_long_put<<<(n_seek + SR_WARPS - 1) / SR_WARPS, SR_THREADS, 0, s>>>(a, n_seek);
    return cudaGetLastError();
}

__global__ void k_classify(const uint32_t *__restrict__ list, uint32_t n, int M, SysTables t,
                           const float4 *__restrict__ clo, const float4 *__restrict__ chi,
                           const float4 *__restrict__ nlo, uint32_t node_cap,
                           uint32_t *__restrict__ out_int, uint32_t *__restrict__ out_bnd,
                           Status *st)
{
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint32_t s = list ? list[k] : k;
    const uint32_t sy = sys_of(t.pad_off, t.nsys, s * kSC * M);
    const DevBox &b = t.box[sy];
    // largest radius of the system: its octree root (clamped as in the search)
    const float R = nlo[min(t.root[sy], node_cap - 1)].w;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int c = 0; c < kSC; ++c) {
        const float4 a = clo[s * kSC + c], z = chi[s * kSC + c];
        lo[0] = fminf(lo[0], a.x); lo[1] = fminf(lo[1], a.y); lo[2] = fminf(lo[2], a.z);
        hi[0] = fmaxf(hi[0], z.x); hi[1] = fmaxf(hi[1], z.y); hi[2] = fmaxf(hi[2], z.z);
    }
    bool interior = true;
    for (int a = 0; a < 3; ++a) {
        if (!b.per[a]) continue;
        // a wrapped pair needs a particle within R of a face; the margin covers
        // the roundings of the gaps here and of the wrapped differences
        const float m = R + R * 1e-5f + b.len[a] * 1e-6f;
        interior = interior && (lo[a] - b.lo[a] > m) && (b.hi[a] - hi[a] > m);
    }
    if (interior)
        out_int[atomicAdd(&st->n_int, 1u)] = s;
    else
        out_bnd[atomicAdd(&st->n_bnd, 1u)] = s;
}

cudaError_t launch_classify(const uint32_t *list, uint32_t n, int M, const SysTables &t,
                            const float4 *clo, const float4 *chi, const float4 *nlo,
                            uint32_t node_cap, uint32_t *out_int, uint32_t *out_bnd, Status *st,
                            cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    k_classify<<<(n + 255) / 256, 256, 0, s>>>(list, n, M, t, clo, chi, nlo, node_cap, out_int,
                                               out_bnd, st);
    return cudaGetLastError();
}

// keys[k] = fill for min(*used, cap) <= k < cap
__global__ void k_fill_keys(uint64_t *keys, uint32_t cap, const unsigned long long *used,
                            uint64_t fill)
{
    const unsigned long long u = *used;
    const uint32_t from = u < cap ? (uint32_t)u : cap;
    for (uint32_t k = from + blockIdx.x * blockDim.x + threadIdx.x; k < cap; k += gridDim.x * blockDim.x)
        keys[k] = fill;
}

cudaError_t launch_fill_keys(uint64_t *keys, uint32_t cap, const unsigned long long *used,
                             uint64_t fill, cudaStream_t s)
{
    k_fill_keys<<<1024, 256, 0, s>>>(keys, cap, used, fill);
    return cudaGetLastError();
}

cudaError_t launch_assemble(const SearchArgs &a, int grid, cudaStream_t s)
{
    k_assemble<<<grid, SR_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace nlg
