// Policy kernels: the look-ahead placement policy of Section III-B (window W, migration ratio R) for many (W, R) pairs
// at once, the comparison strategies of Section IV-A, and the paper's own annealer that walks the (W, R) grid.
//
// A policy is sequential in the steps, so what counts is the latency of one step. The warps of a CTA hold the whole
// population in registers, 32 units to a word: the resident bitmap H and the units' keys (accesses in the window, reads of
// the page, time of last use) as bit planes, plane b holding bit b of every unit's key. Then
//   - a window slides by a bit-sliced add of the entering and the leaving access row,
//   - the k-th largest (smallest) key of a set is the one of the step before or close to it: the sets above and at it come
//     from a bit-sliced comparison, their sizes from one reduction; else it is found from the top plane down, a count of
//     the set per plane,
//   - ties go by unit index: a prefix sum over the lanes, then the lowest bits of one word.
// Measured on 4096 units x 512 steps (B200): a CTA of 1024 threads with a frequency byte and a shared-memory histogram
// update per unit and one thread walking the histograms took 9.5 us per step (4.9 ms for one pair, 24.4 ms for the
// 64 x 11 grid); a warp with ~20 dependent reductions per step 1.5 us (0.76 and 1.14 ms); this form 0.67 us (0.34 and
// 0.81), some 300 instructions a warp and step of which a lone warp issues one in four cycles.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "kvp_common.cuh"

namespace kvp {

namespace {

constexpr uint32_t kMaxWindow = 64;
constexpr uint32_t kPolicyMaxUnits = 32768;
constexpr uint32_t TAG_WR = 5;
constexpr int kFreqPlanes = 7;                           // frequencies are at most 64
constexpr int kStampPlanes = 15;                         // times of last use are below 32768
constexpr uint32_t kPolicyMaxWarps = 8;                  // x 32 lanes x 4 words x 32 units = kPolicyMaxUnits

// Sums over the CTA of packed pairs of 16-bit counts (two sets of units are disjoint and hold at most 32768 units
// together, so neither field overflows). One warp: reductions; several: one barrier, the partial sums double-buffered.
template <bool MULTI>
struct CtaSum {
    uint4* buf;                                          // MULTI: [2][kPolicyMaxWarps] shared, zero at first
    uint32_t flip;
    // Three sums at once, so that what a step wants to know costs one round trip. What does not depend on them goes between
    // begin and end: it is worked on while the sums are on their way.
    __device__ __forceinline__ void begin(uint32_t& x, uint32_t& y, uint32_t& z)
    {
        x = __reduce_add_sync(0xFFFFFFFFu, x);
        y = __reduce_add_sync(0xFFFFFFFFu, y);
        z = __reduce_add_sync(0xFFFFFFFFu, z);
    }
    // by, bz: of y and z, what the warps before this one counted
    __device__ __forceinline__ void end(uint32_t& x, uint32_t& y, uint32_t& z, uint32_t& by, uint32_t& bz)
    {
        by = bz = 0u;
        if (!MULTI) return;
        const uint32_t warp = threadIdx.x >> 5;
        uint4* const b = buf + (flip ^= kPolicyMaxWarps);
        if ((threadIdx.x & 31) == 0) b[warp] = make_uint4(x, y, z, 0u);
        __syncthreads();
        x = y = z = 0u;
#pragma unroll
        for (uint32_t h = 0; h < kPolicyMaxWarps; h += 4) {   // the slots of absent warps stay 0
            if (h * 32 >= blockDim.x) break;
#pragma unroll
            for (uint32_t w = h; w < h + 4; ++w) {
                const uint4 v = b[w];
                if (w == warp) { by = y; bz = z; }
                x += v.x; y += v.y; z += v.z;
            }
        }
    }
    __device__ __forceinline__ void end(uint32_t& x, uint32_t& y, uint32_t& z)
    {
        uint32_t by, bz;
        end(x, y, z, by, bz);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t v)
    {
        uint32_t y = 0u, z = 0u;
        begin(v, y, z);
        end(v, y, z);
        return v;
    }
    // the same and what the warps before this one counted
    __device__ __forceinline__ uint32_t operator()(uint32_t v, uint32_t& before)
    {
        uint32_t x = 0u, z = 0u, bz;
        begin(x, v, z);
        end(x, v, z, before, bz);
        return v;
    }
};

template <int WPL>
__device__ __forceinline__ uint32_t popcn(const uint32_t (&m)[WPL])
{
    uint32_t c = 0;
#pragma unroll
    for (int j = 0; j < WPL; ++j) c += __popc(m[j]);
    return c;
}

// Leaves in m, a set of units, its first `take` units in unit order; `before` of them are in the warps before this one.
template <int WPL>
__device__ __forceinline__ void first_units(uint32_t (&m)[WPL], uint32_t take, uint32_t before)
{
    const uint32_t lane = threadIdx.x & 31, mine = popcn(m);
    uint32_t upto = mine;                                // threads own ascending unit indices
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, upto, off);
        if (lane >= (uint32_t)off) upto += o;
    }
    int r = (int)(take - before - (upto - mine));
    uint32_t part = 0, left = 0;                         // the word that is cut, in one lane at most: what stays of it
    int at = -1;
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        const int c = __popc(m[j]);
        if (r > 0 && r < c) { part = m[j]; left = (uint32_t)r; at = j; }
        if (r < c) m[j] = 0u;
        r -= c;
    }
    const uint32_t who = __ballot_sync(0xFFFFFFFFu, at >= 0);
    if (who) {                                           // warp-uniform; its bits are looked at by a lane each
        const int src = __ffs(who) - 1;
        const uint32_t w = __shfl_sync(0xFFFFFFFFu, part, src), n = __shfl_sync(0xFFFFFFFFu, left, src);
        const uint32_t stay = __ballot_sync(0xFFFFFFFFu, ((w >> lane) & 1u) && (uint32_t)__popc(w & ((1u << lane) - 1u)) < n);
#pragma unroll
        for (int j = 0; j < WPL; ++j)
            if (j == at) m[j] = stay;
    }
}

// this thread's words of a row of `words` words; words past the row are 0
template <int WPL>
__device__ __forceinline__ void load_row(const uint32_t* __restrict__ row, uint32_t words, uint32_t w0, uint32_t (&v)[WPL])
{
#pragma unroll
    for (int j = 0; j < WPL; ++j) v[j] = w0 + j < words ? __ldg(row + w0 + j) : 0u;
}

template <int WPL>
__device__ __forceinline__ void store_row(uint32_t* __restrict__ row, uint32_t words, uint32_t w0, const uint32_t (&v)[WPL])
{
    if (WPL == 4 && (words & 3u) == 0) {                 // rows of whole 16-byte vectors (the buffer is 16-byte aligned)
        if (w0 < words) *reinterpret_cast<uint4*>(row + w0) = make_uint4(v[0], v[1], v[2], v[3]);
        return;
    }
#pragma unroll
    for (int j = 0; j < WPL; ++j)
        if (w0 + j < words) row[w0 + j] = v[j];
}

// keys += 1 on the bits of up, -= 1 on the bits of down (disjoint), plane by plane until no carry can be left
template <int WPL, int NP>
__device__ __forceinline__ void slide(uint32_t (&plane)[NP][WPL], int np, const uint32_t (&in)[WPL], const uint32_t (&out)[WPL])
{
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        const uint32_t down = out[j] & ~in[j];
        uint32_t x = in[j] ^ out[j];                     // units whose key changes: carry (up) or borrow (down)
#pragma unroll
        for (int b = 0; b < NP; ++b) {
            const uint32_t old = plane[b][j];
            plane[b][j] = old ^ x;
            x &= old ^ down;                             // a carry goes on where the bit was set, a borrow where it was not
            if (b + 1 >= np) break;
        }
    }
}

// the units whose key is above k, and those whose key is k
template <int WPL, int NP>
__device__ __forceinline__ void split_keys(const uint32_t (&plane)[NP][WPL], uint32_t k, uint32_t (&gt)[WPL], uint32_t (&eq)[WPL])
{
#pragma unroll
    for (int j = 0; j < WPL; ++j) { gt[j] = 0u; eq[j] = 0xFFFFFFFFu; }
#pragma unroll
    for (int b = NP - 1; b >= 0; --b) {
        const uint32_t kb = (uint32_t)((int)(k << (31 - b)) >> 31);
#pragma unroll
        for (int j = 0; j < WPL; ++j) {
            gt[j] |= eq[j] & plane[b][j] & ~kb;
            eq[j] &= ~(plane[b][j] ^ kb);
        }
    }
}

// The look-ahead rule: of the nC candidates (units outside HBM with a key above 0) at most want = nC * permille / 1000 move
// in, the best first; they take the free capacity, then the next ones replace residents of lower key, lowest first.
// kb = want less the free capacity bounds the swaps from one side, the keys from the other: m swaps are possible iff some
// threshold t has insf + m candidates with key >= t and m residents with key < t, so their number is the maximum over t of
// min(C(t) - insf, R(t)), C falling and R rising in t, reached where the two cross.
//   quota: the want-th best candidate and the kb-th lowest resident; right when the first key is above the second.
//   cross: the crossing, the largest t with C(t) >= insf + R(t); right when it gives at most kb swaps, and then its
//          threshold cuts both sets: candidates above it and residents below it move, of those at it as many as are still
//          to move.
// The thresholds of a sliding window seldom move from step to step, so those of the step before are tried first: one
// reduction of the counts above and at them shows whether they hold, and which way to go where they do not. What the
// comparison needs of the keys alone (Keyed) is worked out a step ahead, while the reduction is under way. Where the
// thresholds do not hold, they are moved a few times, then found from the top plane down, a count per plane.
// Measured on 4096 units x 512 steps, the descent in every step against this: one policy 760 -> 342 us, the 64 x 11 grid
// 1143 -> 811; page granularity 463 -> 275. The thresholds hold in 19 of 20 steps at windows of 16 and 32, in 9 of 10 at 64.
struct Cut {
    uint32_t c, r;                                       // thresholds: of the candidates, of the residents (cross: the same)
    bool quota;
};

template <int WPL>
struct Keyed {                                           // units with a key above 0; candidates: above, at; residents: below, level
    uint32_t any[WPL], above[WPL], at[WPL], below[WPL], level[WPL];
};

template <int WPL, int NP>
__device__ __forceinline__ void compare_keys(const uint32_t (&plane)[NP][WPL], const Cut& cut, Keyed<WPL>& k)
{
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        k.any[j] = plane[0][j];
#pragma unroll
        for (int b = 1; b < NP; ++b) k.any[j] |= plane[b][j];
    }
    split_keys(plane, cut.c, k.above, k.at);
    if (cut.r == cut.c) {                                // CTA-uniform
#pragma unroll
        for (int j = 0; j < WPL; ++j) { k.below[j] = ~(k.above[j] | k.at[j]); k.level[j] = k.at[j]; }
    } else {
        split_keys(plane, cut.r, k.below, k.level);
#pragma unroll
        for (int j = 0; j < WPL; ++j) k.below[j] = ~(k.below[j] | k.level[j]);
    }
}

// What a step comes to: the counts, and how many of the ties at the thresholds move.
struct Exchange {
    uint32_t want, insf, kb, swaps, needC, needR;
    bool found, splitC, splitR;                          // the thresholds hold; some of the ties move and some do not
};
// Judges the thresholds by the counts (CTA-uniform) and moves them where they do not hold. False: give up moving.
__device__ __forceinline__ bool judge_cut(Cut& cut, uint32_t top, uint32_t above, uint32_t at, uint32_t below, uint32_t level, Exchange& e)
{
    if (cut.quota) {
        const int dc = above >= e.want ? 1 : above + at < e.want ? -1 : 0;
        const int dr = !e.kb ? 0 : below >= e.kb ? -1 : below + level < e.kb ? 1 : 0;
        e.swaps = e.kb;
        e.needC = e.want - above; e.needR = e.kb ? e.kb - below : 0u;
        e.found = !dc && !dr && (!e.kb || cut.c > cut.r);
        if (!e.found) {
            if (!dc && !dr) { cut.quota = false; cut.c = cut.r; }
            cut.c += dc; cut.r += dr;
        }
    } else {
        const int d = above + at < e.insf + below ? -1 : above >= e.insf + below + level ? 1 : 0;
        e.swaps = max(below, above > e.insf ? above - e.insf : 0u);
        e.needC = e.insf + e.swaps - above; e.needR = e.swaps - below;
        e.found = !d && e.swaps <= e.kb;
        if (!d && !e.found) cut.quota = true;
        cut.c = cut.r = cut.c + d;
    }
    e.splitC = e.needC != 0u && e.needC != at;
    e.splitR = e.needR != 0u && e.needR != level;
    return cut.c <= top && cut.r <= top;                 // (beyond: fewer residents than places, or none)
}

// One step: H is updated, I units came in, `swaps` of them for a resident. k: of this step's keys, for `cut`; ahead():
// works on the next step meanwhile, and again if the thresholds moved; back(): takes the planes back to this step. hits: a count of the caller's, summed.
template <int WPL, int NP, bool MULTI, typename Ahead, typename Back>
__device__ __forceinline__ void exchange_units(uint32_t (&plane)[NP][WPL], int np, const Keyed<WPL>& k, uint32_t permille,
                                               uint32_t free_slots, uint32_t (&H)[WPL], CtaSum<MULTI>& sum, Cut& cut,
                                               uint32_t& I, uint32_t& swaps, uint32_t& hits, Ahead ahead, Back back)
{
    const uint32_t top = (1u << np) - 1u;
    uint32_t mc[WPL], mr[WPL], in[WPL], out[WPL];        // ties at the thresholds, units beyond them
    uint32_t nc = 0, c, r;
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        in[j] = k.above[j] & ~H[j]; mc[j] = k.at[j] & k.any[j] & ~H[j];
        out[j] = k.below[j] & H[j]; mr[j] = k.level[j] & H[j];
        nc += __popc(k.any[j] & ~H[j]);
    }
    nc = nc << 16 | hits;
    c = popcn(in) << 16 | popcn(mc); r = popcn(out) << 16 | popcn(mr);
    uint32_t bc, br;                                      // of the ties, those of the warps before this one
    sum.begin(nc, c, r);
    ahead();
    sum.end(nc, c, r, bc, br);
    hits = nc & 0xFFFFu;
    Exchange e;
    e.want = (nc >> 16) * permille / 1000u;
    I = swaps = 0;
    if (!e.want) return;
    e.insf = min(e.want, free_slots); e.kb = e.want - e.insf;
    const Cut was = cut;
    if (!e.kb) cut.quota = true;                          // nobody has to leave
    bool go = judge_cut(cut, top, c >> 16, c & 0xFFFFu, r >> 16, r & 0xFFFFu, e);
    if (!e.found) {                                       // CTA-uniform
        back();
        uint32_t cand[WPL];
#pragma unroll
        for (int j = 0; j < WPL; ++j) cand[j] = k.any[j] & ~H[j];
#pragma unroll 1
        for (int t = 0; t < 2 && go && !e.found; ++t) {
            Keyed<WPL> n;
            compare_keys(plane, cut, n);
#pragma unroll
            for (int j = 0; j < WPL; ++j) { in[j] = cand[j] & n.above[j]; mc[j] = cand[j] & n.at[j]; out[j] = H[j] & n.below[j]; mr[j] = H[j] & n.level[j]; }
            c = popcn(in) << 16 | popcn(mc); r = popcn(out) << 16 | popcn(mr);
            uint32_t none = 0;
            sum.begin(none, c, r);
            sum.end(none, c, r, bc, br);
            go = judge_cut(cut, top, c >> 16, c & 0xFFFFu, r >> 16, r & 0xFFFFu, e);
        }
        for (bool quota = cut.quota || e.kb == 0; !e.found; quota = !quota) {   // two passes at most
#pragma unroll
            for (int j = 0; j < WPL; ++j) { mc[j] = cand[j]; mr[j] = H[j]; in[j] = 0u; out[j] = 0u; }
            uint32_t above = 0, below = 0;
            cut.quota = quota; cut.c = cut.r = 0;
            e.needC = e.want; e.needR = e.kb;
#pragma unroll
            for (int b = NP - 1; b >= 0; --b) {
                if (b >= np) continue;
                uint32_t n = 0;
#pragma unroll
                for (int j = 0; j < WPL; ++j) n += (__popc(mc[j] & plane[b][j]) << 16) + __popc(mr[j] & ~plane[b][j]);
                n = sum(n);
                const uint32_t cc = n >> 16, cr = n & 0xFFFFu;
                uint32_t tc, tr;                          // all ones: go on among the set bits (C), among the clear ones (R)
                if (quota) {
                    tc = e.needC <= cc ? 0xFFFFFFFFu : 0u;
                    tr = e.needR <= cr ? 0xFFFFFFFFu : 0u;
                    e.needC -= cc & ~tc; e.needR -= cr & ~tr;
                } else {
                    tc = above + cc >= e.insf + below + cr ? 0xFFFFFFFFu : 0u;
                    tr = ~tc;
                    above += cc & ~tc; below += cr & tc;
                }
                cut.c |= tc & (1u << b); cut.r |= ~tr & (1u << b);   // (cross: the same)
#pragma unroll
                for (int j = 0; j < WPL; ++j) {
                    const uint32_t p = plane[b][j];
                    in[j] |= mc[j] & p & ~tc;
                    mc[j] &= ~(p ^ tc);
                    out[j] |= mr[j] & ~p & ~tr;
                    mr[j] &= p ^ tr;
                }
            }
            sum((popcn(mc) << 16) + popcn(mr), bc);
            br = bc; bc >>= 16;
            e.splitC = e.splitR = true;
            if (quota) {
                e.swaps = e.kb;
                e.found = e.kb == 0 || cut.c > cut.r;
            } else {
                e.swaps = max(below, above > e.insf ? above - e.insf : 0u);
                e.needC = e.insf + e.swaps - above; e.needR = e.swaps - below;
                e.found = e.swaps <= e.kb;
            }
        }
    }
    if (cut.c != was.c || cut.r != was.r) ahead();
    swaps = e.swaps;
    I = e.insf + swaps;
    if (!I) return;
    if (e.splitC) first_units(mc, e.needC, bc & 0xFFFFu);  // CTA-uniform
    if (e.splitR) first_units(mr, e.needR, br & 0xFFFFu);
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        const uint32_t gone = e.kb ? out[j] | (e.needR ? mr[j] : 0u) : 0u;
        H[j] = (H[j] & ~gone) | in[j] | (e.needC ? mc[j] : 0u);
    }
}

// the static placement of this thread's words: the row, or the first `cap` of `entities` where there is none
template <int WPL>
__device__ __forceinline__ void initial_row(const uint32_t* __restrict__ row0, uint32_t words, uint32_t w0, uint32_t cap,
                                            uint32_t (&H)[WPL])
{
    if (row0) { load_row(row0, words, w0, H); return; }
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        const uint32_t lo = (w0 + j) * 32;
        H[j] = w0 + j >= words ? 0u : cap >= lo + 32 ? 0xFFFFFFFFu : (cap > lo ? (1u << (cap - lo)) - 1u : 0u);
    }
}

// The look-ahead policy of one (W, R) pair per CTA. Pairs come as arguments (`pairs`), or, for the whole grid
// (n_ratio != 0), from the block index. out: the schedules; totals: T of Eq. 1 of each, summed on the way: the
// cardinalities of Eq. 3-4 are the hits |A & P| and the two counts the policy has anyway.
constexpr uint32_t kPairsPerLaunch = 256;
struct PolicyPairs {
    uint32_t slot[kPairsPerLaunch];                      // which schedule of the call
    uint16_t window[kPairsPerLaunch], permille[kPairsPerLaunch];
};

// DENSE: with four words to a thread, 128 registers, so that an SM holds 16 warps and not the 12 of the 139 it would take. What is
// spilled costs 3 to 6% of a step.
template <int WPL, bool MULTI, bool DENSE = false>
__global__ void __launch_bounds__(MULTI ? 32 * kPolicyMaxWarps : 32, DENSE ? 2 : 0)
lookahead_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ row0, uint32_t S, uint32_t W32, uint32_t cap,
                 uint32_t n_ratio, const __grid_constant__ PolicyPairs pairs, uint32_t* __restrict__ out,
                 const StepC* __restrict__ stepc, CostK K, uint64_t* __restrict__ totals)
{
    __shared__ uint4 s_part[2 * kPolicyMaxWarps];
    if (MULTI) {
        if (threadIdx.x < 2 * kPolicyMaxWarps) s_part[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    CtaSum<MULTI> sum{s_part, 0u};
    const uint32_t i = blockIdx.x;
    const uint32_t W = n_ratio ? i / n_ratio + 1 : pairs.window[i];
    const uint32_t permille = n_ratio ? (1000u * (i % n_ratio)) / (n_ratio - 1) : pairs.permille[i];
    uint32_t* const mine = out ? out + (size_t)pairs.slot[i] * S * W32 : nullptr;
    const uint32_t w0 = threadIdx.x * WPL;
    const int np = 32 - __clz(W);                        // planes of a frequency 0..W
    uint32_t H[WPL], plane[kFreqPlanes][WPL], nR = 0;
    initial_row(row0, W32, w0, cap, H);
    nR = sum(popcn(H));
#pragma unroll
    for (int b = 0; b < kFreqPlanes; ++b)
#pragma unroll
        for (int j = 0; j < WPL; ++j) plane[b][j] = 0u;
    const uint32_t none[WPL] = {};
    if (permille)                                        // the window of step 0, but for its last row
        for (uint32_t t = 0; t + 1 < W && t < S; ++t) {
            uint32_t a[WPL];
            load_row(A + (size_t)t * W32, W32, w0, a);
            slide(plane, np, a, none);
        }
    Cut cut = {1u, 1u, permille < 1000};
    uint64_t total = 0;
    uint32_t mi = 0, mo = 0, hits = 0;                   // of the step before (its hits are reduced with the next step's count)
    uint32_t enter[WPL], now[WPL];                       // rows s + W and s
    Keyed<WPL> k;
    load_row(A + (size_t)min(W - 1, S - 1) * W32, W <= S ? W32 : 0u, w0, enter);
    if (permille) slide(plane, np, enter, none);
    compare_keys(plane, cut, k);
    load_row(A + (size_t)min(W, S - 1) * W32, W < S ? W32 : 0u, w0, enter);
    load_row(A, W32, w0, now);
    for (uint32_t s = 0; s < S; ++s) {
        // the rows of the next step are on their way while this one is worked on
        uint32_t enter2[WPL], now2[WPL], I = 0, swaps = 0;
        load_row(A + (size_t)min(s + 1 + W, S - 1) * W32, s + 1 + W < S ? W32 : 0u, w0, enter2);
        load_row(A + (size_t)min(s + 1, S - 1) * W32, W32, w0, now2);
        if (permille) {
            const Keyed<WPL> of_now = k;
            bool moved = false;                          // the planes are the next step's
            exchange_units(plane, np, of_now, permille, cap - nR, H, sum, cut, I, swaps, hits,
                           [&] {
                               if (!moved) slide(plane, np, enter, now);
                               moved = true;
                               compare_keys(plane, cut, k);
                           },
                           [&] { slide(plane, np, now, enter); moved = false; });
            if (!moved) { slide(plane, np, enter, now); compare_keys(plane, cut, k); }
        } else {
            hits = sum(hits);
        }
        if (totals && s) total += step_cost(hits, mi, mo, __ldg(stepc + s - 1), K);
        nR += I - swaps;
        mi = s ? I : 0u; mo = s ? swaps : 0u;            // the migrations of step 0 are free
        hits = 0;
#pragma unroll
        for (int j = 0; j < WPL; ++j) {
            hits += __popc(now[j] & H[j]);
            now[j] = now2[j]; enter[j] = enter2[j];
        }
        if (mine) store_row(mine + (size_t)s * W32, W32, w0, H);
    }
    if (totals) {
        total += step_cost(sum(hits), mi, mo, __ldg(stepc + S - 1), K);
        if (threadIdx.x == 0) totals[i] = total;
    }
}

// Page Granularity Scheduling: the same rule with W = 1, R = 1 on pages of `page` consecutive units (a power of two <=
// 32); a page's key is how many of its units the step reads. The keys of all steps are laid out as planes first (every
// step at once), then one CTA walks the steps over the page bitmap, then every page bit is spread over its units.
// planes: [S][np][EW32]; a thread per page.
__global__ void __launch_bounds__(256)
page_keys_kernel(const uint32_t* __restrict__ A, uint32_t E, uint32_t page, uint32_t W32, uint32_t EW32, int np,
                 uint32_t* __restrict__ planes)
{
    const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x, s = blockIdx.y;
    uint32_t f = 0;
    if (e < E) {
        const uint32_t first = e * page;                 // the page's units share one row word
        const uint32_t word = __ldg(A + (size_t)s * W32 + (first >> 5)) >> (first & 31);
        f = __popc(page == 32 ? word : word & ((1u << page) - 1u));
    }
    for (int b = 0; b < np; ++b) {
        const uint32_t bits = __ballot_sync(0xFFFFFFFFu, (f >> b) & 1u);
        if ((threadIdx.x & 31) == 0 && (e >> 5) < EW32) planes[((size_t)s * np + b) * EW32 + (e >> 5)] = bits;
    }
}

constexpr int kPagePlanes = 6;                           // at most 32 units of a page are read

template <int WPL, bool MULTI>
__global__ void __launch_bounds__(MULTI ? 32 * kPolicyMaxWarps : 32)
page_kernel(const uint32_t* __restrict__ planes, int np, uint32_t S, uint32_t EW32, uint32_t cap, uint32_t* __restrict__ pages)
{
    __shared__ uint4 s_part[2 * kPolicyMaxWarps];
    if (MULTI) {
        if (threadIdx.x < 2 * kPolicyMaxWarps) s_part[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    CtaSum<MULTI> sum{s_part, 0u};
    const uint32_t w0 = threadIdx.x * WPL;
    uint32_t H[WPL], plane[kPagePlanes][WPL], next[kPagePlanes][WPL], after[kPagePlanes][WPL];   // of this step, the next, the one after
    initial_row<WPL>(nullptr, EW32, w0, cap, H);
    uint32_t nR = sum(popcn(H));
    auto fetch = [&](uint32_t s) {
#pragma unroll
        for (int b = 0; b < kPagePlanes; ++b) load_row(planes + ((size_t)s * np + min(b, np - 1)) * EW32, b < np ? EW32 : 0u, w0, after[b]);
    };
    fetch(0);
#pragma unroll
    for (int b = 0; b < kPagePlanes; ++b)
#pragma unroll
        for (int j = 0; j < WPL; ++j) next[b][j] = after[b][j];
    fetch(min(1u, S - 1));
    Cut cut = {1u, 1u, false};
    Keyed<WPL> k;
    compare_keys(next, cut, k);
    for (uint32_t s = 0; s < S; ++s) {
        const Keyed<WPL> mine = k;
        uint32_t I, swaps, none = 0;
#pragma unroll
        for (int b = 0; b < kPagePlanes; ++b)
#pragma unroll
            for (int j = 0; j < WPL; ++j) { plane[b][j] = next[b][j]; next[b][j] = after[b][j]; }
        fetch(min(s + 2, S - 1));
        exchange_units(plane, np, mine, 1000u, cap - nR, H, sum, cut, I, swaps, none, [&] { compare_keys(next, cut, k); }, [] {});
        nR += I - swaps;
        store_row(pages + (size_t)s * EW32, EW32, w0, H);
    }
}

__global__ void __launch_bounds__(256)
page_expand_kernel(const uint32_t* __restrict__ pages, uint32_t page, uint32_t W32, uint32_t EW32, size_t total,
                   uint32_t* __restrict__ out)
{
    const uint32_t per_word = 32 / page, ones = page == 32 ? 0xFFFFFFFFu : (1u << page) - 1u;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t s = i / W32;
        const uint32_t e0 = (uint32_t)(i % W32) * per_word;
        const uint32_t eb = __ldg(pages + s * EW32 + (e0 >> 5)) >> (e0 & 31);
        uint32_t word = 0;
        for (uint32_t k = 0; k < per_word; ++k)
            if ((eb >> k) & 1u) word |= ones << (k * page);
        out[i] = word;
    }
}

// Reactive Scheduling (Section IV-A): promote on miss, evict the least recently used. One CTA walks the steps; row
// s + 1 follows from row s and the accesses of step s. Keys are the times of last use (step + 1, 0 = never): hits and
// promoted units get the step's, the evicted are the residents with the smallest (key, index). The smallest key among
// the residents never falls, so the class of residents that hold it is kept as a set (`oldest`) and moves on to the next
// key when it is used up: over a whole run no more advances than steps, where a search through the planes cost a
// reduction per plane and step (4096 units x 512 steps: 0.69 ms with it).
template <int WPL, bool MULTI>
__global__ void __launch_bounds__(MULTI ? 32 * kPolicyMaxWarps : 32)
reactive_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ row0, uint32_t S, uint32_t W32, uint32_t cap,
                uint32_t* __restrict__ out)
{
    __shared__ uint4 s_part[2 * kPolicyMaxWarps];
    if (MULTI) {
        if (threadIdx.x < 2 * kPolicyMaxWarps) s_part[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    CtaSum<MULTI> sum{s_part, 0u};
    const uint32_t w0 = threadIdx.x * WPL;
    uint32_t H[WPL], plane[kStampPlanes][WPL], a[WPL], oldest[WPL];
    initial_row(row0, W32, w0, cap, H);
    uint32_t nR = sum(popcn(H)), tau = 0;                // tau: the key of `oldest`
    store_row(out, W32, w0, H);
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        oldest[j] = H[j];
#pragma unroll
        for (int b = 0; b < kStampPlanes; ++b) plane[b][j] = 0u;
    }
    load_row(A, W32, w0, a);
    for (uint32_t s = 0; s + 1 < S; ++s) {
        const int np = 32 - __clz(s + 1);                // planes of a key 0..s+1
        uint32_t a2[WPL], miss[WPL];
        load_row(A + (size_t)(s + 1) * W32, W32, w0, a2);
#pragma unroll
        for (int j = 0; j < WPL; ++j) { miss[j] = a[j] & ~H[j]; oldest[j] &= ~a[j]; }
        uint32_t ahead;                                  // of the two, what the warps before this one have
        const uint32_t both = sum((popcn(miss) << 16) + popcn(oldest), ahead);
        const uint32_t nM = both >> 16;
        uint32_t n_old = both & 0xFFFFu;
        const uint32_t promoted = min(nM, cap), free_slots = cap - nR;
        if (promoted < nM) first_units(miss, promoted, ahead >> 16);   // CTA-uniform
        ahead &= 0xFFFFu;
#pragma unroll
        for (int b = 0; b < kStampPlanes; ++b) {
            if (b >= np) continue;
            const uint32_t v = ((s + 1) >> b) & 1u ? 0xFFFFFFFFu : 0u;
#pragma unroll
            for (int j = 0; j < WPL; ++j) {
                const uint32_t used = (a[j] & H[j]) | miss[j];
                plane[b][j] = (plane[b][j] & ~used) | (v & used);
            }
        }
        uint32_t evict = promoted > free_slots ? promoted - free_slots : 0u;
        nR += promoted - evict;
        while (evict > n_old) {                          // CTA-uniform; at most s + 1 keys exist, and nR >= evict units
            evict -= n_old;
#pragma unroll
            for (int j = 0; j < WPL; ++j) H[j] &= ~oldest[j];
            ++tau;
#pragma unroll
            for (int j = 0; j < WPL; ++j) {
                uint32_t other = 0;
#pragma unroll
                for (int b = 0; b < kStampPlanes; ++b)
                    if (b < np) other |= plane[b][j] ^ ((tau >> b) & 1u ? 0xFFFFFFFFu : 0u);
                oldest[j] = H[j] & ~other;
            }
            n_old = sum(popcn(oldest), ahead);
            if (tau > s + 1) break;                      // never reached: the keys of the residents end at s + 1
        }
        if (evict) {                                     // CTA-uniform
            uint32_t gone[WPL];
#pragma unroll
            for (int j = 0; j < WPL; ++j) gone[j] = oldest[j];
            if (evict < n_old) first_units(gone, evict, ahead);   // CTA-uniform
#pragma unroll
            for (int j = 0; j < WPL; ++j) { H[j] &= ~gone[j]; oldest[j] &= ~gone[j]; }
        }
#pragma unroll
        for (int j = 0; j < WPL; ++j) {
            H[j] |= miss[j]; a[j] = a2[j];
        }
        if (tau == s + 1)                                // the class of this very step: it grows by the promoted
#pragma unroll
            for (int j = 0; j < WPL; ++j) oldest[j] |= miss[j];
        store_row(out + (size_t)(s + 1) * W32, W32, w0, H);
    }
}

struct WRK {
    const uint64_t* table; const uint32_t* acc; const uint32_t* shifts;
    uint32_t w_max, n_ratio, levels, early_permille, w0, r0, seed_lo, seed_hi;
    uint64_t iters, per_level;
};

// The paper's annealer over (W, R): one warp per chain, the objective is a table lookup. The lanes hold the chain's next
// 32 proposals and test all of them against the present point; the first one that is accepted is taken, and the lanes
// after it test again from there. What bounds a walk is the latency of a round, one per accepted move, so all that does not
// depend on the point is worked out when the proposals are drawn: the largest change each lets pass (a search in the level's
// row of thresholds, which fall). A round is then one lookup, a compare, a vote and the shuffles that tell the new point: 64
// walks of 2000 iterations over a 64 x 11 grid 312 -> 193 us (before, each round looked a threshold up behind the cost).
// TSMEM: the table is staged in shared memory. The level's acceptance row always is; the next one is on its way meanwhile.
template <bool TSMEM>
__global__ void __launch_bounds__(32)
wr_anneal_kernel(const WRK k, kvp_wr_result* __restrict__ results)
{
    extern __shared__ uint64_t wr_sm[];                  // the level's row, then the table
    uint32_t* const acc = reinterpret_cast<uint32_t*>(wr_sm);
    uint64_t* const tab_s = wr_sm + KVP_TABLE_Q / 2;
    const uint32_t lane = threadIdx.x, c = blockIdx.x;
    if (TSMEM)
        for (uint32_t i = lane; i < k.w_max * k.n_ratio; i += 32) tab_s[i] = __ldg(k.table + i);
    const uint64_t* const tab = TSMEM ? tab_s : k.table;
    constexpr uint32_t kRow4 = KVP_TABLE_Q / 128;        // uint4 of a row in each lane
    const uint4* const rows = reinterpret_cast<const uint4*>(k.acc) + lane;
    uint4 row[kRow4];
#pragma unroll
    for (uint32_t q = 0; q < kRow4; ++q) row[q] = __ldg(rows + q * 32);
    uint32_t shift = __ldg(k.shifts);
    __syncwarp();
    int w = (int)k.w0 - 1, r = (int)k.r0;                // the point, from 0
    const int w_max = (int)k.w_max, n_ratio = (int)k.n_ratio;
    uint64_t cur = tab[(size_t)w * n_ratio + r];
    kvp_wr_result res;
    res.best_ticks = cur; res.best_w = k.w0; res.best_r = k.r0; res.n_accepted = 0;
    uint64_t bab = res.best_ticks, i = 0;
    for (uint32_t level = 0; level < k.levels && i < k.iters; ++level) {
        if (level) {
            if (k.early_permille && (bab - res.best_ticks) * 1000ull < bab * (uint64_t)k.early_permille) break;
            bab = res.best_ticks;
        }
        __syncwarp();
#pragma unroll
        for (uint32_t q = 0; q < kRow4; ++q) reinterpret_cast<uint4*>(acc)[q * 32 + lane] = row[q];
        __syncwarp();
        const uint32_t bin = shift, next = min(level + 1, k.levels - 1);
#pragma unroll
        for (uint32_t q = 0; q < kRow4; ++q) row[q] = __ldg(rows + (size_t)next * (KVP_TABLE_Q / 4) + q * 32);
        shift = __ldg(k.shifts + next);
        const uint64_t end = level + 1 < k.levels ? min(i + k.per_level, k.iters) : k.iters;
        for (; i < end; i += 32) {
            const uint64_t it = i + lane;
            uint32_t x[4];
            philox4x32_10((uint32_t)it, (uint32_t)(it >> 32), c, TAG_WR, k.seed_lo, k.seed_hi, x);
            const uint32_t sel = x[0] & 255u, d = (x[0] >> 8) & 3u;
            const int dw = sel < 102u || sel >= 204u ? (int)d - (d < 2u ? 2 : 1) : 0;   // window, diagonal: {-2, -1, 1, 2}
            const int dr = sel < 102u ? 0 : ((x[0] >> 10) & 1u) ? 1 : -1;               // ratio, diagonal
            // Metropolis: a change passes if it is 0 or less, or if its bin is among the first `bins`, whose thresholds are
            // above the proposal's uniform
            uint32_t bins = 0;
#pragma unroll
            for (uint32_t step = KVP_TABLE_Q / 2; step > 0; step >>= 1)
                if (x[3] < acc[bins + step - 1]) bins += step;
            if (x[3] < acc[bins]) ++bins;                // (at most KVP_TABLE_Q - 1 before)
            const uint64_t pass = (uint64_t)bins << bin;
            uint32_t open = end - i >= 32 ? 0xFFFFFFFFu : (1u << (uint32_t)(end - i)) - 1u;
            for (;;) {
                const int nw = w + dw, nr = r + dr;
                const bool on = (uint32_t)nw < (uint32_t)w_max && (uint32_t)nr < (uint32_t)n_ratio;   // off the grid: discarded
                const uint64_t cand = tab[on ? (size_t)nw * n_ratio + nr : 0];
                const uint32_t yes = __ballot_sync(0xFFFFFFFFu, on && (cand <= cur || cand - cur < pass)) & open;
                if (!yes) break;
                const int j = __ffs(yes) - 1;
                w = __shfl_sync(0xFFFFFFFFu, nw, j);
                r = __shfl_sync(0xFFFFFFFFu, nr, j);
                cur = __shfl_sync(0xFFFFFFFFu, cand, j);
                ++res.n_accepted;
                if (cur < res.best_ticks) { res.best_ticks = cur; res.best_w = (uint32_t)w + 1u; res.best_r = (uint32_t)r; }
                open &= 0xFFFFFFFEu << j;                // the proposals after the accepted one
            }
        }
        i = end;
    }
    res.iters_done = i; res.final_ticks = cur; res.final_w = (uint32_t)w + 1u; res.final_r = (uint32_t)r;
    if (lane == 0) results[c] = res;
}

}  // namespace

}  // namespace kvp

using namespace kvp;
// Words per thread and threads of a policy CTA. A word to a thread up to 8 warps (8192 units), four above that: what a step
// costs is a warp's instructions, most of them per word. Against a single warp of two or four words to a thread up to 4096
// units and two warps of four up to 8192, on 4096 units x 512 steps: reactive 397 -> 299 us, one policy 530 -> 342, the 704 of
// a grid 955 -> 811 (two warps of two words 791, but on 2470 units x 192 steps 752 against 691 us a search); 6693 x 166: a
// whole search 760 -> 650 us.
#define KVP_POLICY(kernel, words, grid, ...)                                                                    \
    do {                                                                                                        \
        const uint32_t words_ = (words), grid_ = (grid);                                                        \
        if (words_ <= 32) kernel<1, false><<<grid_, 32, 0, st>>>(__VA_ARGS__);                                  \
        else if (words_ <= 32 * kPolicyMaxWarps) kernel<1, true><<<grid_, (words_ + 31) / 32 * 32, 0, st>>>(__VA_ARGS__); \
        else kernel<4, true><<<grid_, (words_ + 127) / 128 * 32, 0, st>>>(__VA_ARGS__);                         \
        KVP_CUDA(cudaGetLastError());                                                                           \
    } while (0)

namespace {

// The look-ahead policies of `grid` CTAs (see lookahead_kernel), in the form that is the faster one for few CTAs (KVP_POLICY) but
// where another takes fewer waves of them.
//  - Up to 8192 units, six to eight warps of a word: two warps of four words, of which an SM holds six CTAs and not three or
//    four. 8192 units x 200 steps, 64 x 11: 631 -> 508 us (two warps in every case, before: 605); 45 x 11 512 -> 429. With five
//    warps of a word it takes longer (5000 x 166, 55 x 11: 338 -> 394).
//  - Above, the dense form of four words: 64 x 11 on 32,768 x 256 2.26 -> 1.73 ms, 32 x 11 1.33 -> 1.11; otherwise the other one
//    (8 x 11: 0.65 against 0.67).
template <typename... Args>
int launch_lookahead(uint32_t words, uint32_t grid, cudaStream_t st, const Args&... args)
{
    if (words > 160 && grid > 1) {
        const bool one = words <= 32 * kPolicyMaxWarps;
        const uint32_t t4 = (words + 127) / 128 * 32;
        const auto usual = one ? &lookahead_kernel<1, true> : &lookahead_kernel<4, true>;
        const auto other = one ? &lookahead_kernel<4, true> : &lookahead_kernel<4, true, true>;
        int dev = 0, sms = 0, n_usual = 0, n_other = 0;
        KVP_CUDA(cudaGetDevice(&dev));
        KVP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        KVP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n_usual, usual, one ? (words + 31) / 32 * 32 : t4, 0));
        KVP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n_other, other, t4, 0));
        auto waves = [&](int held) { return held > 0 ? (grid - 1) / (uint32_t)(held * sms) : 0xFFFFFFFFu; };
        if (waves(n_other) < waves(n_usual)) {
            other<<<grid, t4, 0, st>>>(args...);
            KVP_CUDA(cudaGetLastError());
            return KVP_OK;
        }
    }
    KVP_POLICY(lookahead_kernel, words, grid, args...);
    return KVP_OK;
}

}  // namespace

extern "C" int kvp_policy_reactive(kvp_problem* p, uint32_t init_mode, uint32_t* schedule, void* stream)
{
    if (!p || !schedule || init_mode > KVP_INIT_STATIC_FREQ || p->dL) return KVP_ERR_ARG;   // fixed populations only
    if (p->U > kPolicyMaxUnits) return KVP_ERR_RANGE;
    KVP_CUDA(cudaSetDevice(p->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    p->last_stream = st;
    const uint32_t* row = init_mode == KVP_INIT_STATIC_FREQ ? p->d_row_freq : nullptr;
    KVP_POLICY(reactive_kernel, p->W32, 1, p->dA, row, p->S, p->W32, p->cap, schedule);
    return KVP_OK;
}

extern "C" int kvp_policy_page(kvp_problem* p, uint32_t page_units, uint32_t* schedule, void* stream)
{
    if (p && p->dL) return KVP_ERR_ARG;                      // fixed populations only
    if (!p || !schedule || page_units < 2 || page_units > 32 || (page_units & (page_units - 1)) || p->U % page_units)
        return KVP_ERR_ARG;
    if (p->U > kPolicyMaxUnits) return KVP_ERR_RANGE;
    KVP_CUDA(cudaSetDevice(p->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t E = p->U / page_units, EW32 = (E + 31) / 32;
    int np = 1;
    while ((page_units >> np) != 0) ++np;
    // scratch: the page bitmaps of all steps, then the key planes
    const size_t rows = ((size_t)p->S * EW32 + 63) & ~(size_t)63;
    int rc = ensure_scratch(p, (rows + (size_t)p->S * np * EW32) * 4, st);
    if (rc) return rc;
    uint32_t* pages = static_cast<uint32_t*>(p->d_scratch);
    uint32_t* planes = pages + rows;
    page_keys_kernel<<<dim3((E + 255) / 256, p->S), 256, 0, st>>>(p->dA, E, page_units, p->W32, EW32, np, planes);
    KVP_CUDA(cudaGetLastError());
    KVP_POLICY(page_kernel, EW32, 1, planes, np, p->S, EW32, p->cap / page_units, pages);
    const size_t total = (size_t)p->S * p->W32;
    page_expand_kernel<<<(uint32_t)std::min<size_t>((total + 255) / 256, 148 * 8), 256, 0, st>>>(pages, page_units, p->W32, EW32,
                                                                                                total, schedule);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

extern "C" int kvp_policy_lookahead(kvp_problem* p, uint32_t init_mode, const uint32_t* windows, const uint32_t* ratios_permille,
                                    uint32_t n, uint32_t* schedules, void* stream)
{
    if (!p || !windows || !ratios_permille || !schedules || !n || init_mode > KVP_INIT_STATIC_FREQ) return KVP_ERR_ARG;
    if (p->dL) return KVP_ERR_ARG;                           // fixed populations only
    for (uint32_t i = 0; i < n; ++i)
        if (windows[i] < 1 || windows[i] > kMaxWindow || ratios_permille[i] > 1000) return KVP_ERR_ARG;
    if (p->U > kPolicyMaxUnits) return KVP_ERR_RANGE;
    KVP_CUDA(cudaSetDevice(p->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    p->last_stream = st;
    const uint32_t* row = init_mode == KVP_INIT_STATIC_FREQ ? p->d_row_freq : nullptr;
    PolicyPairs pairs;
    uint32_t used = 0;
    auto flush = [&]() -> int {
        const uint32_t n_pairs = used;
        used = 0;
        return n_pairs ? launch_lookahead(p->W32, n_pairs, st, p->dA, row, p->S, p->W32, p->cap, 0u, pairs, schedules, p->d_stepc, p->K,
                                          (uint64_t*)nullptr)
                       : KVP_OK;
    };
    int rc;
    for (uint32_t i = 0; i < n; ++i) {
        if (ratios_permille[i] == 0) {                       // nothing ever moves: all rows at once
            if (!row) {
                if ((rc = ensure_scratch(p, (size_t)p->W32 * 4, st))) return rc;
                if ((rc = launch_static_first_row(p, static_cast<uint32_t*>(p->d_scratch), st))) return rc;
            }
            if ((rc = launch_broadcast_row(row ? row : static_cast<uint32_t*>(p->d_scratch), p->S, p->W32,
                                           schedules + (size_t)i * p->S * p->W32, st)))
                return rc;
            continue;
        }
        pairs.slot[used] = i; pairs.window[used] = (uint16_t)windows[i]; pairs.permille[used] = (uint16_t)ratios_permille[i];
        if (++used == kPairsPerLaunch && (rc = flush())) return rc;
    }
    if ((rc = flush())) return rc;
    KVP_CUDA(cudaStreamSynchronize(st));
    return KVP_OK;
}

extern "C" int kvp_wr_grid(kvp_problem* p, uint32_t init_mode, uint32_t w_max, uint32_t n_ratio, uint64_t* table, void* stream)
{
    if (!p || !table || w_max < 1 || w_max > kMaxWindow || n_ratio < 2 || n_ratio > 1001 || p->dL) return KVP_ERR_ARG;
    if (init_mode > KVP_INIT_STATIC_FREQ) return KVP_ERR_ARG;
    if (p->U > kPolicyMaxUnits) return KVP_ERR_RANGE;
    KVP_CUDA(cudaSetDevice(p->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    p->last_stream = st;
    // every grid point is simulated and scored by one CTA; no schedule is written
    const PolicyPairs none = {};
    return launch_lookahead(p->W32, w_max * n_ratio, st, p->dA,
                            init_mode == KVP_INIT_STATIC_FREQ ? p->d_row_freq : (const uint32_t*)nullptr, p->S, p->W32, p->cap, n_ratio,
                            none, (uint32_t*)nullptr, p->d_stepc, p->K, table);
}

extern "C" int kvp_wr_anneal(const uint64_t* table, uint32_t w_max, uint32_t n_ratio, const kvp_wr_params* wp,
                             kvp_wr_result* results, kvp_wr_result* best, void* stream)
try {
    if (!table || !wp || w_max < 1 || n_ratio < 2) return KVP_ERR_ARG;
    if (!wp->chains || !wp->levels || wp->levels > 4096 || !wp->iters || wp->reserved) return KVP_ERR_ARG;
    if (wp->w0 < 1 || wp->w0 > w_max || wp->r0 >= n_ratio) return KVP_ERR_ARG;
    if (!(wp->p0 > 0.0 && wp->p0 < 1.0) || !(wp->alpha > 0.0 && wp->alpha <= 1.0)) return KVP_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // temperature ladder from the table itself: the mean uphill step between grid neighbours is accepted with p0
    const size_t cells = (size_t)w_max * n_ratio;
    std::vector<uint64_t> T(cells);
    KVP_CUDA(cudaMemcpyAsync(T.data(), table, cells * 8, cudaMemcpyDeviceToHost, st));
    KVP_CUDA(cudaStreamSynchronize(st));
    uint64_t sum = 0, cnt = 0;
    auto uphill = [&](int dw, int dr) {                      // all grid steps by (dw, dr) that raise T
        const long w_lo = std::max(0, -dw), w_hi = (long)w_max - std::max(0, dw);
        const long r_lo = std::max(0, -dr), r_hi = (long)n_ratio - std::max(0, dr);
        for (long w = w_lo; w < w_hi; ++w) {
            const uint64_t *from = T.data() + w * n_ratio, *to = T.data() + (w + dw) * n_ratio + dr;
            for (long r = r_lo; r < r_hi; ++r)
                if (to[r] > from[r]) { sum += to[r] - from[r]; ++cnt; }
        }
    };
    for (int dw : {-2, -1, 1, 2}) {
        uphill(dw, 0);
        uphill(dw, -1);
        uphill(dw, 1);
    }
    uphill(0, -1);
    uphill(0, 1);
    uint64_t mean = cnt ? sum / cnt : 1;
    if (!mean) mean = 1;
    std::vector<double> temps(wp->levels);
    double C = -(double)mean / log(wp->p0);
    for (uint32_t j = 0; j < wp->levels; ++j) { temps[j] = C; C = C * wp->alpha; }
    std::vector<uint32_t> acc((size_t)wp->levels * KVP_TABLE_Q), shifts(wp->levels);
    int rc = kvp_accept_table(temps.data(), wp->levels, acc.data(), shifts.data());
    if (rc) return rc;
    std::vector<kvp_wr_result> host(wp->chains);
    char* dev = nullptr;
    const size_t acc_bytes = acc.size() * 4, sh_bytes = (shifts.size() * 4 + 255) & ~(size_t)255;
    const size_t res_bytes = (size_t)wp->chains * sizeof(kvp_wr_result);
    KVP_CUDA(cudaMallocAsync(&dev, acc_bytes + sh_bytes + res_bytes, st));
    cudaError_t ce = cudaMemcpyAsync(dev, acc.data(), acc_bytes, cudaMemcpyHostToDevice, st);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(dev + acc_bytes, shifts.data(), shifts.size() * 4, cudaMemcpyHostToDevice, st);
    if (ce != cudaSuccess) {
        cudaFreeAsync(dev, st);
        KVP_CUDA(ce);
    }
    WRK k;
    k.table = table; k.acc = (const uint32_t*)dev; k.shifts = (const uint32_t*)(dev + acc_bytes);
    k.w_max = w_max; k.n_ratio = n_ratio; k.levels = wp->levels;
    k.early_permille = wp->early_stop_permille; k.w0 = wp->w0; k.r0 = wp->r0;
    k.seed_lo = (uint32_t)wp->seed; k.seed_hi = (uint32_t)(wp->seed >> 32);
    k.iters = wp->iters; k.per_level = wp->iters / wp->levels ? wp->iters / wp->levels : 1;
    kvp_wr_result* d_res = (kvp_wr_result*)(dev + acc_bytes + sh_bytes);
    // the table in shared memory beside the acceptance row, within the 48 KB a kernel gets without opting in
    const size_t row_bytes = KVP_TABLE_Q * 4, tab_bytes = cells * 8;
    if (row_bytes + tab_bytes <= 48 * 1024) wr_anneal_kernel<true><<<wp->chains, 32, row_bytes + tab_bytes, st>>>(k, d_res);
    else wr_anneal_kernel<false><<<wp->chains, 32, row_bytes, st>>>(k, d_res);
    cudaError_t le = cudaGetLastError();
    if (le == cudaSuccess) le = cudaMemcpyAsync(host.data(), d_res, res_bytes, cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(dev, st);
    KVP_CUDA(le);
    KVP_CUDA(cudaStreamSynchronize(st));
    if (results) memcpy(results, host.data(), res_bytes);
    if (best) {
        *best = host[0];
        for (uint32_t c = 1; c < wp->chains; ++c)
            if (host[c].best_ticks < best->best_ticks) *best = host[c];
    }
    return KVP_OK;
} catch (const std::bad_alloc&) {
    return KVP_ERR_NOMEM;
}
