// Cost kernels: per-step cardinalities of a schedule (popc over mask AND placement words) and Eq. 1-5.
//
// Four forms. Small schedules, where launches and latency are all there is: score_kernel, one CTA per schedule, groups of
// lanes own whole rows, everything in one launch; score_long_kernel, the same where they have many steps. Large ones, HBM-bound: count_wide_kernel, in which a warp owns 64
// consecutive 16-byte vectors of every row of a step chunk, carries P[s-1] in registers (every word of A and P is read once)
// and adds its per-step counts to global counters; the last CTA of a schedule, or a second launch, turns them into ticks.
// Large batches: count_staged_kernel, the same with rows fetched ahead into shared memory.
#include <string.h>

#include <algorithm>

#include "kvp_common.cuh"

namespace kvp {

namespace {

template <int VEC>
__device__ __forceinline__ uint4 load_vec(const uint32_t* __restrict__ base, size_t row_words, uint32_t row, uint32_t cv)
{
    if (VEC == 4) {
        return __ldg(reinterpret_cast<const uint4*>(base + (size_t)row * row_words) + cv);
    } else {
        return make_uint4(__ldg(base + (size_t)row * row_words + cv), 0u, 0u, 0u);
    }
}

// placement words are read once and never again: stream them through L2 (evict first)
template <int VEC>
__device__ __forceinline__ uint4 load_stream(const uint32_t* __restrict__ base, size_t row_words, uint32_t row, uint32_t cv)
{
    if (VEC == 4) {
        return __ldcs(reinterpret_cast<const uint4*>(base + (size_t)row * row_words) + cv);
    } else {
        return make_uint4(__ldcs(base + (size_t)row * row_words + cv), 0u, 0u, 0u);
    }
}

template <int VEC>
__device__ __forceinline__ uint4 mask_last(uint4 v, uint32_t cv, uint32_t WV, uint32_t pad_mask)
{
    if (cv == WV - 1) {
        if (VEC == 4) v.w &= pad_mask; else v.x &= pad_mask;
    }
    return v;
}

__device__ __forceinline__ uint32_t popc4(uint4 v) { return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w); }
__device__ __forceinline__ uint4 and4(uint4 a, uint4 b) { return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w); }
__device__ __forceinline__ uint4 andn4(uint4 a, uint4 b) { return make_uint4(a.x & ~b.x, a.y & ~b.y, a.z & ~b.z, a.w & ~b.w); }

// counts of one vector: x = hr | mi << 16, y = mo | occ << 16 (each at most 128)
__device__ __forceinline__ uint2 vec_counts(uint4 a, uint4 p, uint4 prev)
{
    const uint32_t hr = popc4(and4(a, p));
    const uint32_t mi = popc4(andn4(p, prev));
    const uint32_t mo = popc4(andn4(prev, p));
    const uint32_t occ = popc4(p);
    return make_uint2(hr | (mi << 16), mo | (occ << 16));
}

// Where the results of a scoring go; every pointer but stepc may be null.
struct ScoreOut {
    const StepC* stepc;
    CostK K;
    uint32_t cap;
    double spt;
    uint64_t* step_ticks; uint64_t* total_ticks;
    double* step_seconds; double* total_seconds;
    int32_t* bad_step;
    uint64_t* hits;
};

// One step's counts c = {hr, mi, mo, occ} (and hb, growing cache) of schedule i into its outputs and the running sums.
struct ScoreSum {
    uint64_t ticks = 0, hits = 0;
    uint32_t bad = 0xFFFFFFFFu;
};
template <bool GROW>
__device__ __forceinline__ void score_step(const ScoreOut& o, uint32_t i, uint32_t S, uint32_t s, uint4 c, uint32_t hb, ScoreSum& sum)
{
    const uint32_t f = GROW ? step_cost_g(c.x, c.y, c.z, hb, __ldg(&o.stepc[s]), o.K) : step_cost(c.x, c.y, c.z, __ldg(&o.stepc[s]), o.K);
    if (o.step_ticks) o.step_ticks[(size_t)i * S + s] = f;
    if (o.step_seconds) o.step_seconds[(size_t)i * S + s] = (double)f * o.spt;
    sum.ticks += f;
    sum.hits += c.x;
    if (c.w > o.cap) sum.bad = min(sum.bad, s);
}
// the CTA's sums into the totals of schedule i; all threads call it
__device__ __forceinline__ void score_total(const ScoreOut& o, uint32_t i, ScoreSum sum)
{
    __shared__ uint64_t s_sum[32], s_hit[32];
    __shared__ uint32_t s_bad[32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        sum.ticks += __shfl_xor_sync(0xFFFFFFFFu, sum.ticks, off);
        sum.hits += __shfl_xor_sync(0xFFFFFFFFu, sum.hits, off);
    }
    sum.bad = __reduce_min_sync(0xFFFFFFFFu, sum.bad);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { s_sum[warp] = sum.ticks; s_hit[warp] = sum.hits; s_bad[warp] = sum.bad; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t w = 1; w < blockDim.x / 32; ++w) { sum.ticks += s_sum[w]; sum.hits += s_hit[w]; sum.bad = min(sum.bad, s_bad[w]); }
        if (o.total_ticks) o.total_ticks[i] = sum.ticks;
        if (o.total_seconds) o.total_seconds[i] = (double)sum.ticks * o.spt;
        if (o.bad_step) o.bad_step[i] = sum.bad == 0xFFFFFFFFu ? -1 : (int32_t)sum.bad;
        if (o.hits) o.hits[i] = sum.hits;
    }
    __syncthreads();
}

// schedule i from its counts in global memory, by a CTA
template <bool GROW>
__device__ __forceinline__ void score_counts(const ScoreOut& o, uint32_t i, uint32_t S, const uint32_t* counts, const uint32_t* hbc)
{
    ScoreSum sum;
    for (uint32_t s = threadIdx.x; s < S; s += blockDim.x)
        score_step<GROW>(o, i, S, s, __ldcg(reinterpret_cast<const uint4*>(counts) + (size_t)i * S + s),
                         GROW ? __ldcg(hbc + (size_t)i * S + s) : 0u, sum);
    score_total(o, i, sum);
}

constexpr int WIDE_WARPS = 8;
constexpr int WIDE_VEC = 2;              // 16-byte vectors per lane and row

// Carry-save adder: three bit-vectors in, (carry, sum) out; each bit position is added independently.
__device__ __forceinline__ void csa(uint32_t& carry, uint32_t& sum, uint32_t a, uint32_t b, uint32_t c)
{
    sum = a ^ b ^ c;
    carry = (a & b) | (c & (a ^ b));
}

// Number of set bits in eight words with four popc instead of eight (Harley-Seal): the words are first added
// bit-position-wise into a 4-bit counter held as four bit-vectors. popc is the scarce instruction of this kernel.
__device__ __forceinline__ uint32_t popc8(const uint32_t (&w)[8])
{
    uint32_t ones, twos, fours, eights, ta, tb, tc, td, fa, fb;
    csa(ta, ones, w[0], w[1], w[2]);
    csa(tb, ones, ones, w[3], w[4]);
    csa(tc, ones, ones, w[5], w[6]);
    td = ones & w[7]; ones ^= w[7];
    csa(fa, twos, ta, tb, tc);
    fb = twos & td; twos ^= td;
    eights = fa & fb; fours = fa ^ fb;
    return __popc(ones) + 2 * __popc(twos) + 4 * __popc(fours) + 8 * __popc(eights);
}

// Wide rows: a warp owns 64 consecutive 16-byte vectors (1 KB) of every row of a step chunk, two per lane.
// Per lane and step only three cardinalities are counted, hits |A&P|, occupancy |P| and stayers |P&Pprev|;
// migrations follow as mi = occ - stay and mo = occ_prev - stay.
// GROW (growing cache): L holds the rows of existing units. Placement bits of units that do not exist yet are
// dropped, and the units born in a step (in L[s], not in L[s-1]) that are placed in HBM are a fourth cardinality
// hb: they were written there, not migrated, so mi = occ - stay - hb.
// NS schedules of a batch share a thread: the access words are loaded once and used for all of them, which halves
// the L2 traffic of a batch (A is the half of the bytes that comes from L2, not DRAM).
// LAST: the last CTA of a group of schedules scores them. (Two kernels: with the scoring behind a test of a parameter the
// loads of the loop are scheduled worse, 419 against 346 us on 96 schedules of 640 x 4096 units x 64 steps.)
template <int VEC, bool GROW, int NS, bool LAST>
__global__ void __launch_bounds__(WIDE_WARPS * 32)
count_wide_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ Ps, uint32_t S, uint32_t W32,
                  uint32_t WV, uint32_t pad_mask, uint32_t SC, uint32_t n, uint32_t* __restrict__ counts,
                  const uint32_t* __restrict__ L, uint32_t* __restrict__ hbc, uint32_t* __restrict__ tickets, const ScoreOut out)
{
    extern __shared__ uint2 acc[];                       // [NS][WIDE_WARPS][SC], then GROW: uint32 [NS][WIDE_WARPS][SC]
    uint32_t* acc_hb = reinterpret_cast<uint32_t*>(acc + NS * WIDE_WARPS * SC);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cv0 = (blockIdx.x * WIDE_WARPS + warp) * (32 * WIDE_VEC) + lane;
    const uint32_t sb = blockIdx.y * SC;
    const uint32_t se = min(S, sb + SC);
    const uint32_t* __restrict__ P[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q)                         // a schedule past the batch re-reads the last one; its counts are dropped
        P[q] = Ps + (size_t)min(blockIdx.z * NS + q, n - 1) * S * W32;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    uint4 prev[NS][WIDE_VEC], lprev[WIDE_VEC];
    uint32_t occ_prev[NS];
#pragma unroll
    for (int j = 0; j < WIDE_VEC; ++j) {
        const uint32_t cv = cv0 + 32 * j;
        if (GROW) lprev[j] = cv < WV ? load_vec<VEC>(L, W32, sb ? sb - 1 : 0, cv) : zero;
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int j = 0; j < WIDE_VEC; ++j) {
            const uint32_t cv = cv0 + 32 * j;
            prev[q][j] = cv < WV ? mask_last<VEC>(load_vec<VEC>(P[q], W32, sb ? sb - 1 : 0, cv), cv, WV, pad_mask) : zero;
            if (GROW) prev[q][j] = and4(prev[q][j], lprev[j]);
            w[4 * j] = prev[q][j].x; w[4 * j + 1] = prev[q][j].y; w[4 * j + 2] = prev[q][j].z; w[4 * j + 3] = prev[q][j].w;
        }
        occ_prev[q] = popc8(w);
    }
#pragma unroll 4
    for (uint32_t s = sb; s < se; ++s) {
        uint4 a[WIDE_VEC], l[WIDE_VEC], p[NS][WIDE_VEC];
#pragma unroll
        for (int j = 0; j < WIDE_VEC; ++j) {
            const uint32_t cv = cv0 + 32 * j;
            const bool valid = cv < WV;
            a[j] = valid ? load_vec<VEC>(A, W32, s, cv) : zero;
            if (GROW) l[j] = valid ? load_vec<VEC>(L, W32, s, cv) : zero;
#pragma unroll
            for (int q = 0; q < NS; ++q)
                p[q][j] = valid ? mask_last<VEC>(load_stream<VEC>(P[q], W32, s, cv), cv, WV, pad_mask) : zero;
        }
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            uint32_t wp[8], wh[8], ws[8], wb[8];
#pragma unroll
            for (int j = 0; j < WIDE_VEC; ++j) {
                uint4 pj = p[q][j];
                if (GROW) {
                    pj = and4(pj, l[j]);
                    const uint4 born = andn4(pj, lprev[j]);          // placed in HBM in the step it is written
                    wb[4 * j] = born.x; wb[4 * j + 1] = born.y; wb[4 * j + 2] = born.z; wb[4 * j + 3] = born.w;
                }
                wp[4 * j] = pj.x; wp[4 * j + 1] = pj.y; wp[4 * j + 2] = pj.z; wp[4 * j + 3] = pj.w;
                wh[4 * j] = a[j].x & pj.x; wh[4 * j + 1] = a[j].y & pj.y;
                wh[4 * j + 2] = a[j].z & pj.z; wh[4 * j + 3] = a[j].w & pj.w;
                ws[4 * j] = pj.x & prev[q][j].x; ws[4 * j + 1] = pj.y & prev[q][j].y;
                ws[4 * j + 2] = pj.z & prev[q][j].z; ws[4 * j + 3] = pj.w & prev[q][j].w;
                prev[q][j] = pj;
            }
            const uint32_t occ = popc8(wp), hr = popc8(wh), stay = popc8(ws);
            uint32_t hb = 0;
            if (GROW) hb = popc8(wb);
            uint2 c = make_uint2(hr | ((occ - stay - hb) << 16), (occ_prev[q] - stay) | (occ << 16));
            occ_prev[q] = occ;
            c.x = __reduce_add_sync(0xFFFFFFFFu, c.x);   // 16-bit fields: 32 lanes * 256 < 65536
            c.y = __reduce_add_sync(0xFFFFFFFFu, c.y);
            if (GROW) hb = __reduce_add_sync(0xFFFFFFFFu, hb);
            if (lane == 0) {
                acc[(q * WIDE_WARPS + warp) * SC + (s - sb)] = c;
                if (GROW) acc_hb[(q * WIDE_WARPS + warp) * SC + (s - sb)] = hb;
            }
        }
        if (GROW) {
#pragma unroll
            for (int j = 0; j < WIDE_VEC; ++j) lprev[j] = l[j];
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        const uint32_t sched = blockIdx.z * NS + q;
        if (sched >= n) break;
        for (uint32_t i = threadIdx.x; i < se - sb; i += blockDim.x) {
            uint32_t hr = 0, mi = 0, mo = 0, occ = 0;
#pragma unroll
            for (int w = 0; w < WIDE_WARPS; ++w) {
                const uint2 c = acc[(q * WIDE_WARPS + w) * SC + i];
                hr += c.x & 0xFFFFu; mi += c.x >> 16; mo += c.y & 0xFFFFu; occ += c.y >> 16;
            }
            uint32_t* dst = counts + ((size_t)sched * S + sb + i) * 4;
            if (hr) atomicAdd(dst + 0, hr);
            if (mi) atomicAdd(dst + 1, mi);
            if (mo) atomicAdd(dst + 2, mo);
            if (occ) atomicAdd(dst + 3, occ);
            if (GROW) {
                uint32_t hb = 0;
#pragma unroll
                for (int w = 0; w < WIDE_WARPS; ++w) hb += acc_hb[(q * WIDE_WARPS + w) * SC + i];
                if (hb) atomicAdd(hbc + (size_t)sched * S + sb + i, hb);
            }
        }
    }
    if (!LAST) return;
    __shared__ uint32_t s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(tickets + blockIdx.z, 1u) + 1u == gridDim.x * gridDim.y ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll 1
    for (uint32_t i = blockIdx.z * NS; i < min(n, (blockIdx.z + 1) * NS); ++i) score_counts<GROW>(out, i, S, counts, hbc);
}

// Large batches of rows of whole 16-byte vectors, no births: count_wide_kernel for pairs of schedules, with the rows of the
// next steps on their way into shared memory by asynchronous copies. Every lane copies its own vectors into slots of its own,
// so there is no barrier, and what is in flight takes no registers: the loads of the other kernel are as far ahead of their
// use as the compiler's schedule happens to put them. Three CTAs per SM (72 KB of rows each, two of three stages in
// flight). Bound by DRAM: 96 schedules of 640 x 4096 units x 64 steps 345 to 376 us before, 329 to 358 now, by box (5.7 to 6.2
// TB/s, 0.88 to 0.96 of a plain copy); the logic pipe is next (68%), hence the cheaper population count, without which this
// form took 372 us on a box where it took 326 with it.
constexpr int kStages = 3;

__device__ __forceinline__ void copy_async(uint4* to, const uint4* from)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}

// Number of set bits in eight words with four popc: seven of the words are added bit-position-wise into ones, twos and
// fours; the eighth is counted as it is, which is cheaper than carrying it through (8 logic instructions, popc8 has 14).
__device__ __forceinline__ uint32_t popc7_1(const uint32_t (&w)[8])
{
    uint32_t ones, other, twos, fours, ta, tb, tc;
    csa(ta, ones, w[0], w[1], w[2]);
    csa(tb, other, w[3], w[4], w[5]);
    csa(tc, ones, ones, other, w[6]);
    csa(fours, twos, ta, tb, tc);
    return __popc(ones) + __popc(w[7]) + 2 * __popc(twos) + 4 * __popc(fours);
}

__global__ void __launch_bounds__(WIDE_WARPS * 32, 3)
count_staged_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ Ps, uint32_t S, uint32_t W32, uint32_t WV,
                    uint32_t pad_mask, uint32_t SC, uint32_t n, uint32_t* __restrict__ counts)
{
    constexpr int NS = 2, kRows = (1 + NS) * WIDE_VEC;
    extern __shared__ uint4 smem4[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint4* const ring = smem4 + (size_t)warp * (kStages * kRows * 32) + lane;    // slot (stage, row, vector) of this lane: stride 32
    uint2* const acc = reinterpret_cast<uint2*>(smem4 + WIDE_WARPS * kStages * kRows * 32);   // [NS][WIDE_WARPS][SC]
    const uint32_t cv0 = (blockIdx.x * WIDE_WARPS + warp) * (32 * WIDE_VEC) + lane;
    const uint32_t sb = blockIdx.y * SC, se = min(S, sb + SC);
    const uint32_t* __restrict__ P[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q)                         // a schedule past the batch re-reads the last one; its counts are dropped
        P[q] = Ps + (size_t)min(blockIdx.z * NS + q, n - 1) * S * W32;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    for (int i = 0; i < kStages * kRows; ++i) ring[i * 32] = zero;               // vectors beyond the row stay zero
    auto fetch = [&](uint32_t s, uint32_t stage) {
        if (s < se) {
#pragma unroll
            for (int j = 0; j < WIDE_VEC; ++j) {
                const uint32_t cv = cv0 + 32 * j;
                if (cv >= WV) continue;
                copy_async(ring + (stage * kRows + j) * 32, reinterpret_cast<const uint4*>(A + (size_t)s * W32) + cv);
#pragma unroll
                for (int q = 0; q < NS; ++q)
                    copy_async(ring + (stage * kRows + (1 + q) * WIDE_VEC + j) * 32, reinterpret_cast<const uint4*>(P[q] + (size_t)s * W32) + cv);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int k = 0; k + 1 < kStages; ++k) fetch(sb + k, k);
    uint4 prev[NS][WIDE_VEC];
    uint32_t occ_prev[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < WIDE_VEC; ++j) {
            const uint32_t cv = cv0 + 32 * j;
            prev[q][j] = cv < WV ? mask_last<4>(load_vec<4>(P[q], W32, sb ? sb - 1 : 0, cv), cv, WV, pad_mask) : zero;
            w[4 * j] = prev[q][j].x; w[4 * j + 1] = prev[q][j].y; w[4 * j + 2] = prev[q][j].z; w[4 * j + 3] = prev[q][j].w;
        }
        occ_prev[q] = popc7_1(w);
    }
    uint32_t stage = 0;
#pragma unroll 1
    for (uint32_t s = sb; s < se; ++s) {
        fetch(s + kStages - 1, stage ? stage - 1 : kStages - 1);   // into the slots read in the step before
        asm volatile("cp.async.wait_group %0;" :: "n"(kStages - 1) : "memory");
        uint4 a[WIDE_VEC];
#pragma unroll
        for (int j = 0; j < WIDE_VEC; ++j) a[j] = ring[(stage * kRows + j) * 32];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            uint32_t wp[8], wh[8], ws[8];
#pragma unroll
            for (int j = 0; j < WIDE_VEC; ++j) {
                const uint4 pj = mask_last<4>(ring[(stage * kRows + (1 + q) * WIDE_VEC + j) * 32], cv0 + 32 * j, WV, pad_mask);
                const uint4 hj = and4(a[j], pj), sj = and4(pj, prev[q][j]);
                wp[4 * j] = pj.x; wp[4 * j + 1] = pj.y; wp[4 * j + 2] = pj.z; wp[4 * j + 3] = pj.w;
                wh[4 * j] = hj.x; wh[4 * j + 1] = hj.y; wh[4 * j + 2] = hj.z; wh[4 * j + 3] = hj.w;
                ws[4 * j] = sj.x; ws[4 * j + 1] = sj.y; ws[4 * j + 2] = sj.z; ws[4 * j + 3] = sj.w;
                prev[q][j] = pj;
            }
            const uint32_t occ = popc7_1(wp), hr = popc7_1(wh), stay = popc7_1(ws);
            uint2 c = make_uint2(hr | ((occ - stay) << 16), (occ_prev[q] - stay) | (occ << 16));
            occ_prev[q] = occ;
            c.x = __reduce_add_sync(0xFFFFFFFFu, c.x);   // 16-bit fields: 32 lanes * 256 < 65536
            c.y = __reduce_add_sync(0xFFFFFFFFu, c.y);
            if (lane == 0) acc[(q * WIDE_WARPS + warp) * SC + (s - sb)] = c;
        }
        stage = stage + 1 < kStages ? stage + 1 : 0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        const uint32_t sched = blockIdx.z * NS + q;
        if (sched >= n) break;
        for (uint32_t i = threadIdx.x; i < se - sb; i += blockDim.x) {
            uint32_t hr = 0, mi = 0, mo = 0, occ = 0;
#pragma unroll
            for (int w = 0; w < WIDE_WARPS; ++w) {
                const uint2 c = acc[(q * WIDE_WARPS + w) * SC + i];
                hr += c.x & 0xFFFFu; mi += c.x >> 16; mo += c.y & 0xFFFFu; occ += c.y >> 16;
            }
            uint32_t* dst = counts + ((size_t)sched * S + sb + i) * 4;
            if (hr) atomicAdd(dst + 0, hr);
            if (mi) atomicAdd(dst + 1, mi);
            if (mo) atomicAdd(dst + 2, mo);
            if (occ) atomicAdd(dst + 3, occ);
        }
    }
}

// Large batches: the counts of schedule i by CTA i, in a launch of its own.
template <bool GROW>
__global__ void __launch_bounds__(256)
score_counts_kernel(const uint32_t* __restrict__ counts, const uint32_t* __restrict__ hbc, uint32_t S, const ScoreOut out)
{
    score_counts<GROW>(out, blockIdx.x, S, counts, hbc);
}

// Small schedules: CTA i scores schedule i. LPR lanes own a row (a power of two; more than 32 vectors: the lanes go round),
// consecutive groups consecutive rows. counts: the four cardinalities, if wanted.
template <int VEC, bool GROW>
__global__ void __launch_bounds__(1024)
score_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ Ps, uint32_t S, uint32_t W32, uint32_t WV, uint32_t LPR,
             uint32_t pad_mask, const uint32_t* __restrict__ L, uint32_t* __restrict__ counts, uint32_t* __restrict__ hbc, const ScoreOut out)
{
    const uint32_t groups = blockDim.x / LPR, g = threadIdx.x / LPR, l = threadIdx.x % LPR, i = blockIdx.x;
    const uint32_t* __restrict__ P = Ps + (size_t)i * S * W32;
    ScoreSum sum;
#pragma unroll 2
    for (uint32_t s0 = 0; s0 < S; s0 += groups) {                 // (all lanes of a warp go through the votes)
        const uint32_t s = s0 + g, sp = s ? s - 1 : 0;
        uint32_t hr = 0, mi = 0, mo = 0, occ = 0, hb = 0;
        if (s < S)
            for (uint32_t cv = l; cv < WV; cv += LPR) {
                const uint4 a = load_vec<VEC>(A, W32, s, cv);
                uint4 p = mask_last<VEC>(load_vec<VEC>(P, W32, s, cv), cv, WV, pad_mask);
                uint4 q = mask_last<VEC>(load_vec<VEC>(P, W32, sp, cv), cv, WV, pad_mask);
                if (GROW) {                                       // see count_wide_kernel
                    const uint4 lq = load_vec<VEC>(L, W32, sp, cv);
                    p = and4(p, load_vec<VEC>(L, W32, s, cv));
                    q = and4(q, lq);
                    const uint32_t born = popc4(andn4(p, lq));
                    hb += born;
                    mi -= born;                                   // written, not migrated in
                }
                const uint2 c = vec_counts(a, p, q);
                hr += c.x & 0xFFFFu; mi += c.x >> 16; mo += c.y & 0xFFFFu; occ += c.y >> 16;
            }
        for (uint32_t off = LPR / 2; off > 0; off >>= 1) {
            hr += __shfl_xor_sync(0xFFFFFFFFu, hr, off);
            mi += __shfl_xor_sync(0xFFFFFFFFu, mi, off);
            mo += __shfl_xor_sync(0xFFFFFFFFu, mo, off);
            occ += __shfl_xor_sync(0xFFFFFFFFu, occ, off);
            if (GROW) hb += __shfl_xor_sync(0xFFFFFFFFu, hb, off);
        }
        if (l == 0 && s < S) {
            const uint4 c = make_uint4(hr, mi, mo, occ);
            if (counts) reinterpret_cast<uint4*>(counts)[(size_t)i * S + s] = c;
            if (GROW && hbc) hbc[(size_t)i * S + s] = hb;
            if (out.stepc) score_step<GROW>(out, i, S, s, c, hb, sum);
        }
    }
    if (out.stepc) score_total(out, i, sum);
}

// The same for schedules of many steps whose rows take 8 lanes or more (and a vector per lane at most). There the lanes that
// hold a row's counts, one in LPR, are too few to score it: the counts go to shared memory, kChunk rows at a time, and every
// thread scores a row. (400 schedules of 2048 units x 2048 steps: 165 -> 89 us, 1024 of 416 x 512: 56 -> 38, 6 of 416 x 2048:
// 35 -> 21; with rows that follow one another in a group, P[s-1] in registers, 155, 38 and 21: too many streams at a time. It
// waits for its loads first; issue slots 65% busy.)
constexpr uint32_t kChunk = 1024;
template <int VEC, bool GROW>
__global__ void __launch_bounds__(1024)
score_long_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ Ps, uint32_t S, uint32_t W32, uint32_t WV, uint32_t LPR,
                  uint32_t pad_mask, const uint32_t* __restrict__ L, uint32_t* __restrict__ counts, uint32_t* __restrict__ hbc, const ScoreOut out)
{
    __shared__ uint4 s_counts[kChunk];
    __shared__ uint32_t s_hb[GROW ? kChunk : 1];
    const uint32_t groups = blockDim.x / LPR, g = threadIdx.x / LPR, l = threadIdx.x % LPR, i = blockIdx.x;
    const uint32_t* __restrict__ P = Ps + (size_t)i * S * W32;
    const bool mine = l < WV;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    auto count = [](uint4 v) {
        if (VEC == 1) return (uint32_t)__popc(v.x);
        uint32_t twos, ones;
        csa(twos, ones, v.x, v.y, v.z);
        return (uint32_t)(__popc(ones) + 2 * __popc(twos) + __popc(v.w));
    };
    auto row = [&](const uint32_t* m, uint32_t s) { return mine ? load_vec<VEC>(m, W32, s, l) : zero; };
    ScoreSum sum;
    for (uint32_t c0 = 0; c0 < S; c0 += kChunk) {
        const uint32_t rows = min(kChunk, S - c0);
#pragma unroll 4
        for (uint32_t r0 = 0; r0 < rows; r0 += groups) {          // (all lanes of a warp go through the sums)
            const uint32_t r = r0 + g, s = min(c0 + r, S - 1), sp = s ? s - 1 : 0;   // rows beyond the chunk: counted and dropped
            const uint4 a = row(A, s);
            uint4 p = mask_last<VEC>(row(P, s), l, WV, pad_mask), q = mask_last<VEC>(row(P, sp), l, WV, pad_mask);
            uint32_t hb = 0;
            if (GROW) {
                const uint4 lq = row(L, sp);
                p = and4(p, row(L, s));
                q = and4(q, lq);
                hb = count(andn4(p, lq));                         // written in HBM, not migrated in
            }
            uint32_t x = count(and4(a, p)) | (count(andn4(p, q)) - hb) << 16, y = count(andn4(q, p)) | count(p) << 16;   // at most 4096 each
            for (uint32_t off = LPR / 2; off > 0; off >>= 1) {
                x += __shfl_xor_sync(0xFFFFFFFFu, x, off);
                y += __shfl_xor_sync(0xFFFFFFFFu, y, off);
                if (GROW) hb += __shfl_xor_sync(0xFFFFFFFFu, hb, off);
            }
            if (l == 0 && r < rows) {
                s_counts[r] = make_uint4(x & 0xFFFFu, x >> 16, y & 0xFFFFu, y >> 16);
                if (GROW) s_hb[r] = hb;
            }
        }
        __syncthreads();
        for (uint32_t r = threadIdx.x; r < rows; r += blockDim.x) {
            const uint4 c = s_counts[r];
            const uint32_t hb = GROW ? s_hb[r] : 0u;
            if (counts) reinterpret_cast<uint4*>(counts)[(size_t)i * S + c0 + r] = c;
            if (GROW && hbc) hbc[(size_t)i * S + c0 + r] = hb;
            if (out.stepc) score_step<GROW>(out, i, S, c0 + r, c, hb, sum);
        }
        __syncthreads();
    }
    if (out.stepc) score_total(out, i, sum);
}

}  // namespace

// lanes of a row in score_kernel
static uint32_t lanes_per_row(uint32_t WV)
{
    uint32_t n = 1;
    while (n < 32 && n < WV) n *= 2;
    return n;
}

// threads of score_kernel and score_long_kernel: one CTA per SM or fewer: as many rows side by side as there are; many CTAs:
// smaller ones. lots: which of the two.
static uint32_t score_threads(const kvp_problem* p, uint32_t n, uint32_t WV, uint32_t LPR, bool* lots)
{
    const uint64_t lanes = (uint64_t)p->S * LPR;
    uint32_t T = (uint32_t)std::min<uint64_t>(n <= 148 ? 1024 : 256, (lanes + 31) / 32 * 32);
    *lots = LPR >= 8 && WV <= LPR && lanes >= 8ull * T;
    if (*lots && n > 148 && n <= 4 * 148) T = 512;
    return T;
}

// Schedules are small when a CTA for each is done with them before the streaming kernel would be. Both estimates in us, from 721
// batches of 1 to 1024 schedules of 32 to 2048 steps x 1 to 2048 words (the choice takes 1.2 times the better kernel's time at
// most, but for two of them; 6 x 6816 units x 512 steps: one CTA each 43.3, streaming 9.9; 148 x 8192 x 128: 12.8, 40.2):
//  - one CTA each: the launch, then by rounds of its threads, longer when the SMs hold more than 1024 threads; at most 2 TB/s;
//  - streaming: the launch and the clearing of the counters, then by steps of a schedule: rows narrower than a CTA's tile (2048
//    words in vectors, 512 in single words) cost as much as a tile.
// Beyond 512 KB a schedule whose rows take a CTA's lanes several times round is no work for one SM (64 x 16,384 x 2048: 239, 173).
static bool is_small(const kvp_problem* p, uint32_t n)
{
    const bool vec4 = p->W32 % 4 == 0;
    const uint32_t WV = vec4 ? p->W32 / 4 : p->W32, LPR = lanes_per_row(WV), per_sm = (n + 147) / 148;
    bool lots;
    const uint32_t T = score_threads(p, n, WV, LPR, &lots);
    const double steps = (double)n * p->S, rounds = (double)(((uint64_t)p->S * LPR + T - 1) / T), more = (WV + LPR - 1) / LPR - 1;
    const double round = lots ? (vec4 ? 0.7 : 0.53) : vec4 ? 1.1 + 0.5 * more : 0.95 + 0.25 * more;
    const double one = 4.0 + std::max(rounds * round * std::max(1.0, per_sm * T / 1024.0), steps * p->W32 * 2e-6);
    const double streaming = 9.5 + steps * (vec4 ? std::max(1.3e-3, 1.4e-6 * p->W32) : 0.47e-3 * ((p->W32 + 511) / 512));
    return one <= streaming && (more == 0 || (size_t)p->S * p->W32 * 4 <= (512u << 10));
}

size_t score_scratch_bytes(const kvp_problem* p, uint32_t n)
{
    return is_small(p, n) ? 0 : (size_t)n * p->S * (p->dL ? 20 : 16) + (size_t)n * 4;
}

// counts [n][S][4] = {hr, mi, mo, occ}, or null if score_scratch_bytes(p, n) is 0; hbc [n][S] for a problem with births,
// likewise; tickets [n] behind counts and hbc, or null. out.stepc null: only the counts are wanted.
static int launch_score_impl(const kvp_problem* p, const uint32_t* schedules, uint32_t n, bool small, uint32_t* counts, uint32_t* hbc,
                             uint32_t* tickets, const ScoreOut& out, cudaStream_t st, uint32_t* launches)
{
    const bool grow = p->dL != nullptr;
    const bool vec4 = (p->W32 % 4 == 0) && ((reinterpret_cast<uintptr_t>(schedules) & 15) == 0);
    const uint32_t WV = vec4 ? p->W32 / 4 : p->W32;
    if (launches) *launches += 1;
    if (small) {
        const uint32_t LPR = lanes_per_row(WV);
        bool lots;
        const uint32_t T = score_threads(p, n, WV, LPR, &lots);
#define KVP_SCORE(VEC, GROW) \
        (lots ? score_long_kernel<VEC, GROW> : score_kernel<VEC, GROW>)<<<n, T, 0, st>>>(p->dA, schedules, p->S, p->W32, WV, LPR, p->pad_mask, p->dL, counts, hbc, out)
        if (grow) { if (vec4) KVP_SCORE(4, true); else KVP_SCORE(1, true); }
        else { if (vec4) KVP_SCORE(4, false); else KVP_SCORE(1, false); }
#undef KVP_SCORE
        KVP_CUDA(cudaGetLastError());
        return KVP_OK;
    }
    // one call clears counts, hbc and tickets where they follow one another
    const size_t cbytes = (size_t)n * p->S * 16, hbytes = grow ? (size_t)n * p->S * 4 : 0, tbytes = tickets ? (size_t)n * 4 : 0;
    KVP_CUDA(cudaMemsetAsync(counts, 0, cbytes + ((char*)hbc == (char*)counts + cbytes || !grow ? hbytes + tbytes : 0), st));
    if (grow && (char*)hbc != (char*)counts + cbytes) KVP_CUDA(cudaMemsetAsync(hbc, 0, hbytes, st));
    const uint32_t col_ctas = (WV + WIDE_WARPS * 32 * WIDE_VEC - 1) / (WIDE_WARPS * 32 * WIDE_VEC);
    // two schedules per thread once a batch is large enough to fill the GPU that way
    const uint32_t NS = n >= 8 ? 2u : 1u;
    const uint32_t nz = (n + NS - 1) / NS;
    // Split the steps until the grid is at least four full waves (148 SMs x 8 resident CTAs), so that the last,
    // partial wave costs little; every chunk re-reads one halo row (1/SC more traffic, mostly from L2).
    uint32_t SC = p->S;
    while (SC > 8 && (uint64_t)col_ctas * ((p->S + SC - 1) / SC) * nz < 148u * 8u * 4u) SC = (SC + 1) / 2;
    // Pairs of schedules with rows of whole vectors can take count_staged_kernel, whose three CTAs per SM leave 3 KB each for
    // the accumulators.
    const bool pairs = NS == 2 && !grow && vec4;
    if (pairs && SC > 24) SC = 24;
    // the per-step accumulators of a chunk live in dynamic shared memory: keep them within the 48 KB a kernel gets
    // without opting in (NS * WIDE_WARPS * SC entries of 8 bytes, 12 with births)
    const uint32_t sc_max = (uint32_t)((47u * 1024u) / (NS * WIDE_WARPS * (sizeof(uint2) + (grow ? 4 : 0))));
    if (SC > sc_max) SC = sc_max;
    dim3 grid(col_ctas, (p->S + SC - 1) / SC, nz);
    const size_t smem = (size_t)NS * WIDE_WARPS * SC * (sizeof(uint2) + (grow ? 4 : 0));
    const int T = WIDE_WARPS * 32;
    // A CTA that takes a ticket waits until its counts have arrived, one or two microseconds. Up to one wave of CTAs that is
    // less than another launch; a large batch pays it in every wave (256 schedules of 65,536 units x 256 steps: 136 us with
    // tickets, 116 with the second launch).
    const bool apart = tickets && (uint64_t)grid.x * grid.y * grid.z > 148u * 8u;
    if (apart) tickets = nullptr;
#define KVP_WIDE(VEC, GROW, NSCH)                                                                                         \
    (tickets ? count_wide_kernel<VEC, GROW, NSCH, true> : count_wide_kernel<VEC, GROW, NSCH, false>)<<<grid, T, smem, st>>>( \
        p->dA, schedules, p->S, p->W32, WV, p->pad_mask, SC, n, counts, GROW ? p->dL : nullptr, GROW ? hbc : nullptr, tickets, out)
    if (pairs && !tickets) {
        const size_t bytes = smem + (size_t)WIDE_WARPS * kStages * (1 + 2) * WIDE_VEC * 32 * sizeof(uint4);
        KVP_CUDA(cudaFuncSetAttribute(count_staged_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 << 10));
        count_staged_kernel<<<grid, T, bytes, st>>>(p->dA, schedules, p->S, p->W32, WV, p->pad_mask, SC, n, counts);
    } else if (NS == 2) {
        if (grow) { if (vec4) KVP_WIDE(4, true, 2); else KVP_WIDE(1, true, 2); }
        else { if (vec4) KVP_WIDE(4, false, 2); else KVP_WIDE(1, false, 2); }
    } else {
        if (grow) { if (vec4) KVP_WIDE(4, true, 1); else KVP_WIDE(1, true, 1); }
        else { if (vec4) KVP_WIDE(4, false, 1); else KVP_WIDE(1, false, 1); }
    }
#undef KVP_WIDE
    KVP_CUDA(cudaGetLastError());
    if (apart) {
        if (grow) score_counts_kernel<true><<<n, 256, 0, st>>>(counts, hbc, p->S, out);
        else score_counts_kernel<false><<<n, 256, 0, st>>>(counts, hbc, p->S, out);
        KVP_CUDA(cudaGetLastError());
        if (launches) *launches += 1;
    }
    return KVP_OK;
}

int launch_score(const kvp_problem* p, const uint32_t* schedules, uint32_t n, void* scratch, uint32_t* counts_out, uint32_t* hbc_out,
                 uint64_t* step_ticks, uint64_t* total_ticks, double* step_seconds, double* total_seconds, int32_t* bad_step,
                 uint64_t* hits, cudaStream_t st, uint32_t* launches)
{
    ScoreOut o;
    o.stepc = p->d_stepc; o.K = p->K; o.cap = p->cap; o.spt = p->spt;
    o.step_ticks = step_ticks; o.total_ticks = total_ticks; o.step_seconds = step_seconds; o.total_seconds = total_seconds;
    o.bad_step = bad_step; o.hits = hits;
    // scratch: counts, hbc (births), tickets
    uint32_t* counts = static_cast<uint32_t*>(scratch);
    uint32_t* hbc = counts && p->dL ? counts + (size_t)n * p->S * 4 : nullptr;
    uint32_t* tickets = counts ? counts + (size_t)n * p->S * (p->dL ? 5 : 4) : nullptr;
    const bool small = is_small(p, n);
    if (small) { counts = counts_out; hbc = hbc_out; }
    int rc = launch_score_impl(p, schedules, n, small, counts, hbc, tickets, o, st, launches);
    if (rc || small) return rc;
    if (counts_out && counts_out != counts) KVP_CUDA(cudaMemcpyAsync(counts_out, counts, (size_t)n * p->S * 16, cudaMemcpyDeviceToDevice, st));
    if (hbc_out && hbc && hbc_out != hbc) KVP_CUDA(cudaMemcpyAsync(hbc_out, hbc, (size_t)n * p->S * 4, cudaMemcpyDeviceToDevice, st));
    return KVP_OK;
}

int launch_counts(const kvp_problem* p, const uint32_t* schedules, uint32_t n, uint32_t* counts, cudaStream_t st)
{
    ScoreOut none;
    memset(&none, 0, sizeof none);
    return launch_score_impl(p, schedules, n, is_small(p, n), counts, nullptr, nullptr, none, st, nullptr);
}

}  // namespace kvp

// The schedule index is a grid dimension limited to 65535: larger batches go in slices.
static const uint32_t kBatchSlice = 32768;

extern "C" int kvp_eval_counts(kvp_problem* p, const uint32_t* schedules, uint32_t n, uint32_t* counts, void* stream)
{
    if (!p || !schedules || !counts || !n) return KVP_ERR_ARG;
    if (p->dL) return KVP_ERR_ARG;                       // four cardinalities do not describe a growing cache
    if ((reinterpret_cast<uintptr_t>(counts) & 15) != 0) return KVP_ERR_ARG;
    KVP_CUDA(cudaSetDevice(p->device));
    p->last_stream = static_cast<cudaStream_t>(stream);
    const size_t sched_words = (size_t)p->S * p->W32;
    for (uint32_t i = 0; i < n; i += kBatchSlice) {
        const uint32_t m = n - i < kBatchSlice ? n - i : kBatchSlice;
        int rc = kvp::launch_counts(p, schedules + i * sched_words, m, counts + (size_t)i * p->S * 4, static_cast<cudaStream_t>(stream));
        if (rc) return rc;
    }
    return KVP_OK;
}

extern "C" int kvp_eval(kvp_problem* p, const uint32_t* schedules, uint32_t n, uint64_t* step_ticks, uint64_t* total_ticks,
                        double* step_seconds, double* total_seconds, int32_t* bad_step, void* stream)
{
    if (!p || !schedules || !total_ticks || !n) return KVP_ERR_ARG;
    KVP_CUDA(cudaSetDevice(p->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t sched_words = (size_t)p->S * p->W32;
    for (uint32_t i = 0; i < n; i += kBatchSlice) {
        const uint32_t m = n - i < kBatchSlice ? n - i : kBatchSlice;
        const size_t so = (size_t)i * p->S, need = kvp::score_scratch_bytes(p, m);
        int rc = need ? kvp::ensure_scratch(p, need, st) : KVP_OK;
        if (rc) return rc;
        p->last_stream = st;
        if ((rc = kvp::launch_score(p, schedules + i * sched_words, m, need ? p->d_scratch : nullptr, nullptr, nullptr,
                                    step_ticks ? step_ticks + so : nullptr, total_ticks + i, step_seconds ? step_seconds + so : nullptr,
                                    total_seconds ? total_seconds + i : nullptr, bad_step ? bad_step + i : nullptr, nullptr, st, nullptr)))
            return rc;
    }
    return KVP_OK;
}

// ---------------------------------------------------------------------------------------------------
// kvp_eval without any allocation: the per-step cardinalities go to a fixed array in the library image.
// Meant for callers that cannot afford or are not allowed a cudaMalloc at this point (a latency-bound
// loop, a process whose memory pool owns the whole device, allocator-free code). See include/kvp.h.
// Behind the counters of n schedules, at most 65,536 of one step, are their tickets.
static __device__ __align__(256) uint32_t g_noalloc_counts[KVP_NOALLOC_SCRATCH_BYTES / 4 + 65536];

namespace {
constexpr int kMaxDevices = 64;
uint32_t* g_noalloc_addr[kMaxDevices];   // device address of g_noalloc_counts, per device; null until looked up
}

// In host code `g_noalloc_counts` names a host-side shadow of the symbol, not device memory: the address a
// kernel may use has to be asked for, once per device and with that device current.
static int noalloc_scratch(int device, uint32_t** out)
{
    if (device < 0 || device >= kMaxDevices) return KVP_ERR_RANGE;
    uint32_t* ptr = __atomic_load_n(&g_noalloc_addr[device], __ATOMIC_ACQUIRE);
    if (!ptr) {
        KVP_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_noalloc_counts));
        if (!ptr) return KVP_ERR_CUDA;
        __atomic_store_n(&g_noalloc_addr[device], ptr, __ATOMIC_RELEASE);   // racing threads store the same value
    }
    *out = ptr;
    return KVP_OK;
}

extern "C" int kvp_eval_noalloc(kvp_problem* p, const uint32_t* schedules, uint32_t n, uint64_t* step_ticks,
                                uint64_t* total_ticks, double* step_seconds, double* total_seconds, int32_t* bad_step,
                                void* stream)
{
    if (!p || !schedules || !total_ticks || !n || p->dL) return KVP_ERR_ARG;
    if ((uint64_t)n * p->S * 16ull > (uint64_t)KVP_NOALLOC_SCRATCH_BYTES) return KVP_ERR_RANGE;   // batch too large
    KVP_CUDA(cudaSetDevice(p->device));
    uint32_t* counts = nullptr;
    int rc = noalloc_scratch(p->device, &counts);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    p->last_stream = st;
    // The array still holds the previous call's numbers: what has to start from zero is cleared on the stream by
    // launch_score. The schedule index is a grid dimension, so a batch of more than kBatchSlice schedules (possible
    // within the limit only for one or two steps) goes in slices.
    const size_t sched_words = (size_t)p->S * p->W32;
    for (uint32_t i = 0; i < n; i += kBatchSlice) {
        const uint32_t m = n - i < kBatchSlice ? n - i : kBatchSlice;
        const size_t so = (size_t)i * p->S;
        if ((rc = kvp::launch_score(p, schedules + i * sched_words, m, counts, nullptr, nullptr, step_ticks ? step_ticks + so : nullptr,
                                    total_ticks + i, step_seconds ? step_seconds + so : nullptr,
                                    total_seconds ? total_seconds + i : nullptr, bad_step ? bad_step + i : nullptr, nullptr, st, nullptr)))
            return rc;
    }
    return KVP_OK;
}
