// Annealing: the host side, calibration, reduction and the winner's way back. The chains run on one of two kernels, chosen
// per job (see prepare()): the narrow one in kvp_narrow.cuh (one to four warps per chain, 32 proposals prepared at a time
// and evaluated in move order) and the wide one in kvp_chain.cuh (one to four warps per chain, batches of 128 or 256
// proposals, most of them settled by their placement bits or by a lower bound of the cost change).
//
// State of a chain: the schedule in time-packed form (for every unit a bit string over the steps), either
// in shared memory (small problems) or in a private slice of global scratch (a copy-on-write overlay of the initial
// schedule all chains share), and in shared memory per step the two sides {th, te} of Eq. 2 and the occupancy, the
// bitmaps of full steps and of steps where te leads, and the running total T.
//
// A proposal (one Philox4x32-10 block, a pure function of seed, chain and move index) names a run of at most
// 30 consecutive steps and one or two units. Only the run's steps and the step after it change cost. Both kernels leave
// the sequential chain's results: moves are committed in move order with a Metropolis test against the quantised
// exp(-delta/C) table, and what an applied move could have touched is evaluated again. Several warps of a chain take its
// batches in turn (see ChainShared).
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "kvp_common.cuh"

namespace kvp {

namespace {

kvp_test_hooks g_hooks = {0u, 0u, 0u, 0u, 0u};   // kvp_set_test_hooks; read once per call

// What an exchange round of neighbouring rungs needs (by pair of rungs).
struct ExchangeArgs {
    const uint32_t* always; const uint32_t* table; const uint32_t* shifts;
    unsigned long long* counts;  // {tried, accepted}
    uint32_t rungs, seed_lo, seed_hi;
};

// Byte offsets of the parts of a chain's shared memory (see chain_layout).
struct ChainLayout {
    uint32_t occ, full, lead, out, in, hb, have, work;
};

struct ChainParams {
    const uint32_t* Acol;        // [U][S32]
    const StepC* stepc;          // [S]
    const uint4* counters0;      // [S] counters of the initial schedule
    const uint32_t* Pcol0;       // [U][S32] initial schedule
    const uint32_t* table;       // [levels][1024]
    const uint32_t* shifts;      // [levels]
    uint32_t* ws;                // global scratch: [slots][U*S32] (only the global-state variant)
    kvp_chain_result* results;   // indexed by chain - result_base
    uint32_t* dump;              // if set, slot 0 writes its final schedule here (time-packed)
    const uint32_t* full0;       // [S32] full-step bitmap of the initial schedule
    uint32_t* snap;              // if set: [slots][U*S32], each chain's schedule when it reached its best
    uint64_t* undo_log;          // if set: [slots][undo_cap] indices of the moves applied since the best state
    uint32_t* undo_len;          // [slots] how many there were (more than undo_cap: the log overflowed)
    uint32_t undo_cap;
    uint32_t* err;               // set to 1 by a warp that gave up waiting for its turn
    uint32_t drop_first_turn;    // test hook: the owner of batch 0 never passes the turn on, so the next wait runs out
    const uint32_t* birth;       // growing cache: [U] step at which a unit is written (0 = there from the start)
    const uint32_t* hb0;         // growing cache: [S] units written to HBM at birth under the initial schedule
    CostK K;
    uint32_t U, S, S32, cap;
    uint32_t chain_first, chain_count, result_base;
    uint32_t levels, p_swap_256, len_choices;
    uint32_t early_permille, early_from;
    PhiloxKeys keys;             // round keys of the seed
    uint64_t per_level, upto, init_ticks;
    uint32_t* cow_out;           // schedules in global scratch: [slots][cow_slots4 * 4] which buckets of
                                 // units a slot's slice holds when its chain ends (the rest is the initial schedule)
    uint32_t cow_shift;          // a bucket is 2^cow_shift consecutive units
    unsigned long long* work;    // wide kernel: [3] sums over the chains of {n_again, n_listed, n_items}
    // Replica exchange: the call runs rounds round0 .. round1-1; in round t chain c proposes moves
    // t * exch_every .. (t + 1) * exch_every - 1 (up to `upto`) with the table row of the rung it holds,
    // rung_hist[t * hist_stride + (c - hist_base)].
    uint8_t* rung_hist;          // null: the ordinary cooling schedule by temperature levels
    uint64_t exch_every;
    uint32_t round0, round1, hist_stride, hist_base;
    uint4* state;                // if set: [chains][state4] the chain's persistent shared-memory state (and its
                                 // schedule, when that lives in shared memory), indexed like rung_hist
    uint32_t state4;             // uint4 slots per chain in `state`
    uint32_t resume;             // 1: start from `state` instead of the initial schedule
    uint32_t cow_slots4;         // schedules in global scratch: uint4 slots of a chain's bucket bitmap
    // segments seg0 .. seg1 - 1 of seg_len moves (the last one takes what is left up to `upto`), each of
    // seg_bat batches: the temperature levels of the cooling schedule, or rounds of a replica-exchange run
    uint32_t seg0, seg1, seg_bat;
    uint64_t seg_len;
    uint64_t move0;              // narrow kernel: it counts segments from 0, this is the first one's first move
    ChainLayout lay;
    uint32_t warps;              // warps per chain
    uint32_t carry;              // room for accepted proposals: kAccepted (less in tests)
    const float* bounds;         // [levels] C ln 2: see EvalCtx::bound
    uint32_t ladder_ctas;        // replica exchange: a CTA holds whole ladders and exchanges between its rounds itself
    ExchangeArgs ladder;
    uint32_t* n_exchanged;       // replica exchange in the CTA: by chain
};

// A proposal as its lane keeps it in registers: the Philox words and, after evaluation, the verdict.
// Windows of it: Wu, Wv, Nu, Nv = placement of units u, v before (W) and after (N) the move, Au, Av = access bits. Bit k
// belongs to step s0 - 1 + k, so bit 0 is the step before the run (for s0 == 0 it repeats step 0, because P[-1] := P[0]),
// bits 1..run are the run, and the affected steps s0..last are bits 1..nl <= 31. Run lengths stop at 30 so that every
// window fits one 32-bit register.
struct LaneMove {
    uint32_t pk, u, v, w;        // packed (swap | len << 1 | s0 << 8), units, Metropolis uniform
    int delta;
    bool inf, acc, chg;
};

__device__ __forceinline__ void decode_move(const uint32_t r[4], uint32_t p_swap_256, uint32_t len_choices, uint32_t S,
                                            uint32_t U, LaneMove& mv)
{
    const uint32_t swap = (r[0] & 255u) < p_swap_256 ? 1u : 0u;
    const uint32_t k = (((r[0] >> 8) & 255u) * len_choices) >> 8;
    const uint32_t len = min(1u << k, 30u);
    const uint32_t s0 = ((r[0] >> 16) * S) >> 16;
    mv.pk = swap | (len << 1) | (s0 << 8);
    mv.u = __umulhi(r[1], U);
    mv.v = __umulhi(r[2], U);
    mv.w = r[3];
}

// 32 consecutive bits of a time-packed column starting at step s0 - 1 (see LaneMove). Bits that belong to
// steps beyond the horizon are arbitrary; every user masks them.
template <typename Ptr>
__device__ __forceinline__ uint32_t window(Ptr col, uint32_t S32, uint32_t s0)
{
    const uint32_t b0 = s0 ? s0 - 1 : 0u, w = b0 >> 5;
    const uint32_t lo = col[w], hi = col[min(w + 1, S32 - 1)];
    const uint32_t slid = __funnelshift_r(lo, hi, b0 & 31u);
    return s0 ? slid : ((lo << 1) | (lo & 1u));                  // s0 == 0: bit 0 repeats step 0
}

// The same cut for several columns of one proposal: the position is worked out once.
// The word after the first may lie behind the column (its bits are beyond the horizon then, and masked by every user):
// columns are followed by at least four readable bytes everywhere.
struct WinPos {
    uint32_t w, sh;              // first word, shift
    bool first;                  // s0 == 0: bit 0 repeats step 0
};
__device__ __forceinline__ WinPos window_pos(uint32_t s0)
{
    WinPos p;
    const uint32_t b0 = s0 ? s0 - 1 : 0u;
    p.w = b0 >> 5; p.sh = b0 & 31u; p.first = s0 == 0;
    return p;
}
// COLV = 2 or 4: every column is exactly that many words (at most 64 or 128 steps) and comes with one vector load: a
// warp's 32 columns are 32 different lines, and what limits the chains in global memory is the number of such
// scattered loads. (Every column then starts on an 8- or 16-byte boundary; the arrays themselves are 16-byte
// aligned.) COLV = 0: columns of any length, the two words they need. The choice is made at compile time: a test of
// S32 around every load breaks up the straight-line block in which all loads of a batch are issued, and was 1.5x slower.
template <int COLV>
struct Words { using type = uint2; };
template <>
struct Words<4> { using type = uint4; };
template <int COLV, typename Ptr>
__device__ __forceinline__ typename Words<COLV>::type words_at(Ptr col, const WinPos p)
{
    typename Words<COLV>::type x;
    if constexpr (COLV == 0) { x.x = col[p.w]; x.y = col[p.w + 1]; }
    else x = *reinterpret_cast<const typename Words<COLV>::type*>(col);
    return x;
}
template <int COLV>
__device__ __forceinline__ uint32_t cut(const typename Words<COLV>::type q, const WinPos p)
{
    uint32_t lo, hi;
    if constexpr (COLV == 0) { lo = q.x; hi = q.y; }
    else if constexpr (COLV == 2) { lo = p.w ? q.y : q.x; hi = q.y; }
    else {
        lo = p.w == 0 ? q.x : p.w == 1 ? q.y : p.w == 2 ? q.z : q.w;
        hi = p.w == 0 ? q.y : p.w == 1 ? q.z : q.w;
    }
    return p.first ? ((lo << 1) | (lo & 1u)) : __funnelshift_r(lo, hi, p.sh);
}
template <int COLV, typename Ptr>
__device__ __forceinline__ uint32_t window_at(Ptr col, const WinPos p) { return cut<COLV>(words_at<COLV>(col, p), p); }

// born: window bit of the step in which u (low byte) and v (next byte) are written, 0 = not among bits 1..31
struct Windows { uint32_t Wu, Wv, Nu, Nv, Au, Av, s0, born; };

// Growing cache, unit with birth step b seen through the window that starts at step s0 - 1 (-1 for s0 == 0):
// the bits of steps at which it exists, and the bit of the step in which it is written.
__device__ __forceinline__ void alive_born(uint32_t b, uint32_t s0, uint32_t& alive, uint32_t& born)
{
    const int off = (int)b - ((int)s0 - 1);
    alive = (b == 0 || off <= 0) ? 0xFFFFFFFFu : (off >= 32 ? 0u : 0xFFFFFFFFu << off);
    born = (b != 0 && off >= 1 && off < 32) ? 1u << off : 0u;
}

// First half of evaluating a proposal, all in the calling lane and word-parallel over the <= 31 affected
// steps: the windows before and after the move, feasibility (Eq. 5), whether any bit changes, and the set
// of window bits (steps) whose cardinalities, hence cost, change.
// GROW: a move acts only on the steps at which the units it names exist, and a unit that enters HBM in the step
// it is written was written there (it counts in hb), not migrated.
// colu, colv: the time-packed placement columns of unit u and of unit v (of u again for a flip).
template <bool GROW, typename PPtr, typename FPtr>
__device__ __forceinline__ uint32_t lane_windows(PPtr colu, PPtr colv, const uint32_t* __restrict__ Acol, FPtr full,
                                                 const uint32_t* __restrict__ birth, uint32_t S, uint32_t S32,
                                                 LaneMove& mv, Windows& wn)
{
    const bool swap = mv.pk & 1u;
    const uint32_t len = (mv.pk >> 1) & 63u, s0 = mv.pk >> 8;
    const uint32_t run = min(s0 + len, S) - s0;                   // steps whose placement bits change hands
    const uint32_t nl = min(s0 + len, S - 1) - s0 + 1;            // affected steps: the run and the step after it
    const uint32_t M = ((1u << run) - 1u) << 1;
    const uint32_t Sb = ((1u << nl) - 1u) << 1;
    // branch-free: a flip reads unit u twice and ignores the second copy, a swap ignores the full-step window
    const size_t ub = (size_t)mv.u * S32, vb = (size_t)(swap ? mv.v : mv.u) * S32;
    const uint32_t Wu = window(colu, S32, s0), Au = window(Acol + ub, S32, s0);
    const uint32_t wv = window(colv, S32, s0), av = window(Acol + vb, S32, s0);
    const uint32_t Wv = swap ? wv : 0u, Av = swap ? av : 0u;
    const uint32_t Fw = window(full, S32, s0);
    uint32_t Bu = 0u, Bv = 0u, live = 0xFFFFFFFFu;
    if (GROW) {
        uint32_t Lu, Lv;
        alive_born(__ldg(birth + mv.u), s0, Lu, Bu);
        alive_born(__ldg(birth + (swap ? mv.v : mv.u)), s0, Lv, Bv);
        live = Lu & Lv;
        if (!swap) Bv = 0u;
    }
    const uint32_t D = (swap ? (Wu ^ Wv) : 0xFFFFFFFFu) & M & live;      // bits that toggle
    uint32_t Nu = Wu ^ D, Nv = swap ? (Wv ^ D) : 0u;
    if (s0 == 0) {                                                // the virtual step -1 follows step 0
        Nu = (Nu & ~1u) | ((Nu >> 1) & 1u);
        Nv = (Nv & ~1u) | ((Nv >> 1) & 1u);
    }
    wn.Wu = Wu; wn.Wv = Wv; wn.Nu = Nu; wn.Nv = Nv; wn.Au = Au; wn.Av = Av; wn.s0 = s0;
    wn.born = GROW ? ((Bu ? 31u - __clz(Bu) : 0u) | ((Bv ? 31u - __clz(Bv) : 0u) << 8)) : 0u;
    mv.chg = D != 0;
    mv.inf = !swap && (~Wu & D & Fw) != 0;                        // a flip may not raise a full step (Eq. 5)
    const uint32_t hr = (Au ^ Av) & (Wu ^ Nu);                    // a hit is won or lost (v mirrors u in a swap)
    // migrations of a unit at step t are the edges p[t] != p[t-1] (into HBM when p[t] is set, out otherwise):
    // the counts change where an edge appears, disappears or turns around
    // (the edge into the step of birth is no migration; there the placement bit moves a write between H^w and E^w)
    const uint32_t euo = (Wu ^ (Wu << 1)) & ~Bu, eun = (Nu ^ (Nu << 1)) & ~Bu;
    const uint32_t evo = (Wv ^ (Wv << 1)) & ~Bv, evn = (Nv ^ (Nv << 1)) & ~Bv;
    const uint32_t mg = (euo ^ eun) | (euo & eun & (Wu ^ Nu)) | (evo ^ evn) | (evo & evn & (Wv ^ Nv));
    const uint32_t wr = ((Wu ^ Nu) & Bu) | ((Wv ^ Nv) & Bv);
    return mv.inf ? 0u : ((hr | mg | wr) & Sb);
}

// Cost change of the step at window bit k (Eq. 2-4 before and after), from the windows of a proposal.
// hb: the step's count of units written to HBM at birth (GROW only).
template <bool GROW>
__device__ __forceinline__ int item_delta(const Windows& wn, uint32_t k, const uint4 c4, uint32_t hb, const StepC c,
                                          const CostK K)
{
    const uint32_t pu = (wn.Wu >> k) & 1u, qu = (wn.Wu >> (k - 1)) & 1u, npu = (wn.Nu >> k) & 1u, nqu = (wn.Nu >> (k - 1)) & 1u;
    const uint32_t pv = (wn.Wv >> k) & 1u, qv = (wn.Wv >> (k - 1)) & 1u, npv = (wn.Nv >> k) & 1u, nqv = (wn.Nv >> (k - 1)) & 1u;
    const uint32_t au = (wn.Au >> k) & 1u, av = (wn.Av >> k) & 1u;
    const uint32_t hr = c4.x + (au & npu) - (au & pu) + (av & npv) - (av & pv);
    if (GROW) {
        // mu / mv: 1 when the step is an ordinary one for the unit, 0 when it is the step the unit is written in
        const uint32_t mu = (wn.born & 255u) == k ? 0u : 1u, mw = ((wn.born >> 8) & 255u) == k ? 0u : 1u;
        const uint32_t mi = c4.y + mu * ((npu & ~nqu) - (pu & ~qu)) + mw * ((npv & ~nqv) - (pv & ~qv));
        const uint32_t mo = c4.z + (~npu & nqu & 1u) - (~pu & qu & 1u) + (~npv & nqv & 1u) - (~pv & qv & 1u);
        const uint32_t hn = hb + (1u - mu) * (npu - pu) + (1u - mw) * (npv - pv);
        return (int)(step_cost_g(hr, mi, mo, hn, c, K) - step_cost_g(c4.x, c4.y, c4.z, hb, c, K));
    }
    const uint32_t mi = c4.y + (npu & ~nqu) - (pu & ~qu) + (npv & ~nqv) - (pv & ~qv);
    const uint32_t mo = c4.z + (~npu & nqu & 1u) - (~pu & qu & 1u) + (~npv & nqv & 1u) - (~pv & qv & 1u);
    return (int)(step_cost(hr, mi, mo, c, K) - step_cost(c4.x, c4.y, c4.z, c, K));
}

__device__ __forceinline__ bool metropolis(int delta, uint32_t w, const uint32_t* __restrict__ trow, uint32_t shift)
{
    // branch-free: the threshold is loaded whatever delta is (a clamped index), so that the loads of several
    // proposals are in flight together instead of each behind its own branch
    const uint32_t q = (uint32_t)max(delta, 0) >> shift;
    const uint32_t thr = __ldg(trow + min(q, (uint32_t)KVP_TABLE_Q - 1u));
    return delta <= 0 || (q < KVP_TABLE_Q && w < thr);            // quantised exp(-delta/C)
}

// Whole evaluation in one lane (used where there is no warp to share the work with: calibration).
template <bool GROW, typename PPtr, typename CPtr, typename FPtr>
__device__ __forceinline__ void eval_lane(PPtr P, const uint32_t* __restrict__ Acol, CPtr ctr, FPtr full,
                                          const uint32_t* __restrict__ birth, const uint32_t* __restrict__ hb,
                                          const StepC* __restrict__ stepc, const CostK K, uint32_t S, uint32_t S32,
                                          const uint32_t* __restrict__ trow, uint32_t shift, LaneMove& mv)
{
    Windows wn;
    uint32_t todo = lane_windows<GROW>(P + (size_t)mv.u * S32, P + (size_t)((mv.pk & 1u) ? mv.v : mv.u) * S32, Acol, full, birth, S,
                                       S32, mv, wn);
    int delta = 0;
    while (todo) {
        const uint32_t k = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t t = wn.s0 + k - 1;
        delta += item_delta<GROW>(wn, k, ctr[t], GROW ? hb[t] : 0u, __ldg(stepc + t), K);
    }
    mv.delta = delta;
    mv.acc = metropolis(delta, mv.w, trow, shift);
}

// A group of nthr threads (one or more whole warps, this thread being number tid) copies n words. A chain in global
// scratch starts by copying tens of megabytes this way, so eight 16-byte loads per thread are in flight before the
// first store.
__device__ __forceinline__ void copy_words(uint32_t* __restrict__ dst, const uint32_t* __restrict__ src, size_t n,
                                           uint32_t tid, uint32_t nthr = 32)
{
    if ((n & 3) == 0 && ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0) {
        uint4* __restrict__ d4 = reinterpret_cast<uint4*>(dst);
        const uint4* __restrict__ s4 = reinterpret_cast<const uint4*>(src);
        const size_t n4 = n / 4;
        size_t i = tid;
        for (; i + 7 * (size_t)nthr < n4; i += 8 * (size_t)nthr) {
            uint4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = s4[i + (size_t)nthr * j];
#pragma unroll
            for (int j = 0; j < 8; ++j) d4[i + (size_t)nthr * j] = v[j];
        }
        for (; i < n4; i += nthr) d4[i] = s4[i];
    } else {
        for (size_t i = tid; i < n; i += nthr) dst[i] = src[i];
    }
}

// The copies off the hot path (a bucket fetched into a slice, a best state saved) as one function each, so that the
// chain loop stays small enough for the instruction cache.
__device__ __noinline__ void copy_words_cold(uint32_t* dst, const uint32_t* src, size_t n, uint32_t lane)
{
    copy_words(dst, src, n, lane);
}

// Schedules in global scratch are copy-on-write overlays of the one initial schedule that all chains share: the
// units come in buckets of 2^shift consecutive units, a chain's slice holds a bucket only once the chain has
// rewritten a unit of it, and a bitmap in shared memory says which. Chains change few of their units, so nearly
// every placement window is read from the shared initial schedule, which stays in L2, and not from a private slice
// that only DRAM can hold; a chain that rewrites everything ends up copying its whole slice once, bucket by bucket.
// The bitmap takes the shared memory that a full CTA of chains leaves free (kCowBitsMin to kCowBitsMax buckets): a
// chain of a million moves rewrites thousands of units, and every read of a bucket it owns misses L2, so the buckets
// should be small (with 8192 buckets of 512 units a chain of the largest configuration owned two thirds of them at
// its end; with 40,960 of 64 units it owns an eighth).
constexpr uint32_t kCowBitsMin = 8192, kCowBitsMax = 65536;

// A warp copies the buckets of units u and v into the slice where they are not there yet. Both at once, as vectors where
// columns and slices allow it: a bucket of the largest configuration (64 columns of two words) is then one load per lane
// (one word at a time, each iteration waiting for the one before: 8 trips to L2 for a swap, 139 -> 133 ms on that search).
__device__ __forceinline__ void own_buckets(uint32_t* slice, const uint32_t* __restrict__ p0, uint32_t* have, uint32_t shift,
                                            uint32_t U, uint32_t S32, uint32_t u, uint32_t v, uint32_t lane)
{
    const uint32_t bu = u >> shift, bv = v >> shift;
    const bool du = !((have[bu >> 5] >> (bu & 31u)) & 1u), dv = bv != bu && !((have[bv >> 5] >> (bv & 31u)) & 1u);
    if (!du && !dv) return;
    const size_t lu = (size_t)(bu << shift) * S32, lv = (size_t)(bv << shift) * S32;
    const uint32_t nu = du ? (min(U, (bu + 1u) << shift) - (bu << shift)) * S32 : 0u;
    const uint32_t nv = dv ? (min(U, (bv + 1u) << shift) - (bv << shift)) * S32 : 0u, n = max(nu, nv);
    if ((((S32 << shift) | U * S32) & 3u) == 0u) {               // every bucket and every slice begins at a vector
        const uint4 *const su = reinterpret_cast<const uint4*>(p0 + lu), *const sv = reinterpret_cast<const uint4*>(p0 + lv);
        uint4 *const tu = reinterpret_cast<uint4*>(slice + lu), *const tv = reinterpret_cast<uint4*>(slice + lv);
#pragma unroll 1
        for (uint32_t i = lane; 4u * i < n; i += 32) {
            uint4 a, b;
            if (4u * i < nu) a = __ldg(su + i);
            if (4u * i < nv) b = __ldg(sv + i);
            if (4u * i < nu) tu[i] = a;
            if (4u * i < nv) tv[i] = b;
        }
    } else {
#pragma unroll 1
        for (uint32_t i = lane; i < n; i += 32) {
            uint32_t a, b;
            if (i < nu) a = __ldg(p0 + lu + i);
            if (i < nv) b = __ldg(p0 + lv + i);
            if (i < nu) slice[lu + i] = a;
            if (i < nv) slice[lv + i] = b;
        }
    }
    __threadfence_block();
    __syncwarp();
    if (lane == 0) {
        if (du) have[bu >> 5] |= 1u << (bu & 31u);
        if (dv) have[bv >> 5] |= 1u << (bv & 31u);
    }
    __syncwarp();
}

// A whole schedule out of a copy-on-write slice: the buckets the slice holds from it, the rest from the initial one.
__device__ __forceinline__ void copy_merged(uint32_t* __restrict__ dst, const uint32_t* __restrict__ mine,
                                            const uint32_t* __restrict__ p0, const uint32_t* have, uint32_t shift,
                                            uint32_t U, uint32_t S32, uint32_t lane)
{
    const uint32_t nb = (U + (1u << shift) - 1u) >> shift;
    for (uint32_t b = 0; b < nb; ++b) {
        const size_t lo = (size_t)(b << shift) * S32, hi = (size_t)min(U, (b + 1u) << shift) * S32;
        const uint32_t* src = (have[b >> 5] >> (b & 31u)) & 1u ? mine : p0;
        copy_words_cold(dst + lo, src + lo, hi - lo, lane);
    }
}

constexpr uint32_t kLog = 16;    // applied moves a chain's log keeps
// A wait for the turn gives up after this many polls (each at least some tens of nanoseconds apart): the chain then
// reports KVP_ERR_TIMEOUT instead of holding the GPU. A turn lasts microseconds.
constexpr uint32_t kTurnPolls = 1u << 24;

__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); }
__device__ __forceinline__ void st_volatile_u32(uint32_t* p, uint32_t v) { *reinterpret_cast<volatile uint32_t*>(p) = v; }

}  // namespace

}  // namespace kvp

#include "kvp_chain.cuh"
#include "kvp_narrow.cuh"

namespace kvp {

namespace {

// Takes a finished chain's schedule back to its best state: the moves applied after the best were logged, each
// swap or flip is its own inverse, so applying them again in reverse order undoes them. One warp; only the
// schedule words are touched (the counters are not needed any more).
template <bool GROW>
__global__ void __launch_bounds__(32)
undo_kernel(const ChainParams prm, uint32_t slot)
{
    const uint32_t lane = threadIdx.x, S = prm.S, S32 = prm.S32;
    uint32_t* P = prm.ws + (size_t)slot * prm.U * S32;
    const uint64_t* ulog = prm.undo_log + (size_t)slot * prm.undo_cap;
    const uint32_t n = prm.undo_len[slot], chain = prm.chain_first + slot;
    for (uint32_t i = n; i-- > 0;) {
        const uint64_t m = ulog[i];
        uint32_t r[4];
        LaneMove mv;
        philox4x32_10((uint32_t)m, (uint32_t)(m >> 32), chain, TAG_MOVE, prm.keys, r);
        decode_move(r, prm.p_swap_256, prm.len_choices, S, prm.U, mv);
        const bool swap = mv.pk & 1u;
        const uint32_t len = (mv.pk >> 1) & 63u, s0 = mv.pk >> 8, end = min(s0 + len, S);
        if (lane < 2) {
            const uint32_t wj = (s0 >> 5) + lane;
            const uint32_t lo = max(s0, wj * 32u), hi = min(end, wj * 32u + 32u);
            if (hi > lo) {                               // run lengths are at most 30, so never a full word
                uint32_t mask = ((1u << (hi - lo)) - 1u) << (lo - wj * 32u);
                if (GROW) {                              // only the steps at which the units exist were touched
                    const uint32_t b = max(__ldg(prm.birth + mv.u), swap ? __ldg(prm.birth + mv.v) : 0u);
                    if (b >= wj * 32u + 32u) mask = 0u;
                    else if (b > wj * 32u) mask &= 0xFFFFFFFFu << (b - wj * 32u);
                }
                const size_t iu = (size_t)mv.u * S32 + wj, iv = (size_t)mv.v * S32 + wj;
                if (swap) {
                    const uint32_t a = P[iu], b = P[iv], d = (a ^ b) & mask;
                    if (d) { P[iu] = a ^ d; P[iv] = b ^ d; }
                } else {
                    P[iu] ^= mask;
                }
            }
        }
        __syncwarp();
    }
    // the schedule itself is copied out by gather_slice_kernel, on the whole GPU
}

// The schedule a copy-on-write slice of global scratch stands for, copied to dst bucket by bucket, from the slice where it
// holds the bucket and from the initial schedule elsewhere. A warp per bucket.
__global__ void __launch_bounds__(256)
gather_slice_kernel(uint32_t* __restrict__ dst, const uint32_t* __restrict__ mine, const uint32_t* __restrict__ p0,
                    const uint32_t* __restrict__ have, uint32_t shift, uint32_t U, uint32_t S32)
{
    const uint32_t lane = threadIdx.x & 31, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5, nb = (U + (1u << shift) - 1u) >> shift;
    for (uint32_t b = warp; b < nb; b += nwarps) {
        const size_t lo = (size_t)(b << shift) * S32, hi = (size_t)min(U, (b + 1u) << shift) * S32;
        const uint32_t* src = (have[b >> 5] >> (b & 31u)) & 1u ? mine : p0;
        for (size_t i = lo + lane; i < hi; i += 32) dst[i] = src[i];
    }
}

// bit t of full0 is set iff the initial schedule fills the HBM capacity at step t
__global__ void full_mask_kernel(const uint4* __restrict__ counters0, uint32_t S, uint32_t cap, uint32_t* __restrict__ full0)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t bits = __ballot_sync(0xFFFFFFFFu, t < S && counters0[t < S ? t : 0].w == cap);
    if ((threadIdx.x & 31) == 0 && t < ((S + 31) / 32) * 32) full0[t >> 5] = bits;
}

// Calibration of the temperature ladder: proposals (i, 0, 0, TAG_CALIB), i < 1024, are evaluated against the
// initial schedule and never applied; acc = {sum of positive deltas, their number}.
template <bool GROW>
__global__ void __launch_bounds__(256)
calib_kernel(const ChainParams prm, unsigned long long* acc)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= CALIB_N) return;
    uint32_t r[4];
    LaneMove mv;
    philox4x32_10(i, 0u, 0u, TAG_CALIB, prm.keys, r);
    decode_move(r, prm.p_swap_256, prm.len_choices, prm.S, prm.U, mv);
    eval_lane<GROW>(prm.Pcol0, prm.Acol, prm.counters0, prm.full0, prm.birth, prm.hb0, prm.stepc, prm.K, prm.S, prm.S32,
                    prm.table, 0u, mv);
    if (!mv.inf && mv.delta > 0) {
        atomicAdd(acc, (unsigned long long)mv.delta);
        atomicAdd(acc + 1, 1ull);
    }
}

struct ReduceOut {
    uint64_t best_ticks, best_move, moves_total;
    uint32_t best_chain, pad;    // pad: the chains' error word
};

// Cross-chain best-so-far: lexicographic minimum of (best_ticks, chain index), plus the executed-move total.
__global__ void __launch_bounds__(1024)
reduce_kernel(const kvp_chain_result* __restrict__ res, uint32_t chains, const uint32_t* __restrict__ err, ReduceOut* out)
{
    __shared__ uint64_t s_t[32], s_m[32];
    __shared__ uint32_t s_c[32];
    uint64_t bt = ~0ull, moves = 0;
    uint32_t bc = 0xFFFFFFFFu;
    for (uint32_t c = threadIdx.x; c < chains; c += blockDim.x) {
        const uint64_t t = res[c].best_ticks;
        moves += res[c].moves_done;
        if (t < bt || (t == bt && c < bc)) { bt = t; bc = c; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const uint64_t ot = __shfl_xor_sync(0xFFFFFFFFu, bt, off);
        const uint32_t oc = __shfl_xor_sync(0xFFFFFFFFu, bc, off);
        moves += __shfl_xor_sync(0xFFFFFFFFu, moves, off);
        if (ot < bt || (ot == bt && oc < bc)) { bt = ot; bc = oc; }
    }
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { s_t[warp] = bt; s_c[warp] = bc; s_m[warp] = moves; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t w = 1; w < (blockDim.x >> 5); ++w) {
            moves += s_m[w];
            if (s_t[w] < bt || (s_t[w] == bt && s_c[w] < bc)) { bt = s_t[w]; bc = s_c[w]; }
        }
        out->best_ticks = bt; out->best_chain = bc; out->moves_total = moves;
        out->best_move = res[bc].best_move;
        out->pad = *err;                                  // a chain gave up waiting for its turn
    }
}

// One exchange round of a replica-exchange run: in every ladder the pairs of neighbouring rungs (j, j+1) with
// j = t (mod 2) may exchange. The chains keep their states; what changes hands is the rung, i.e. the temperature
// the chain runs at in the next round. A thread per ladder.
//   holder [ladders][rungs] : the chain (index within the call) that holds each rung; updated
//   rung_next [chains]      : the rungs for round t + 1 (the next row of the rung history)
//   counts                  : {exchanges tried, exchanges accepted}
struct ExchangeK {
    const kvp_chain_result* results;   // final_ticks = the chain's present cost
    uint32_t* holder;
    uint8_t* rung_next;
    uint32_t* n_exchanged;
    ExchangeArgs x;
    uint32_t ladders, first_ladder;
    uint64_t t;
};

__global__ void __launch_bounds__(128)
exchange_kernel(const ExchangeK k)
{
    const uint32_t l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= k.ladders) return;
    uint32_t* hold = k.holder + (size_t)l * k.x.rungs;
    uint32_t tried = 0, done = 0;
    for (uint32_t j = (uint32_t)(k.t & 1ull); j + 1 < k.x.rungs; j += 2) {
        const uint32_t hot = hold[j], cold = hold[j + 1];
        const bool accept = exchange_accepts(k.x, k.t, (k.first_ladder + l) * k.x.rungs, j, k.results[hot].final_ticks,
                                             k.results[cold].final_ticks);
        ++tried;
        if (accept) {
            hold[j] = cold; hold[j + 1] = hot;
            ++k.n_exchanged[hot]; ++k.n_exchanged[cold];
            ++done;
        }
    }
    for (uint32_t j = 0; j < k.x.rungs; ++j) k.rung_next[hold[j]] = (uint8_t)j;
    if (tried) {
        atomicAdd(k.x.counts, (unsigned long long)tried);
        atomicAdd(k.x.counts + 1, (unsigned long long)done);
    }
}

__global__ void exchange_init_kernel(uint32_t* holder, uint8_t* rung0, uint32_t* n_exchanged, uint32_t chains, uint32_t rungs)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= chains) return;
    holder[i] = i;                                        // chain i of the call starts on rung i % rungs of ladder i / rungs
    rung0[i] = (uint8_t)(i % rungs);
    n_exchanged[i] = 0u;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Everything a run needs on the device, carved out of the problem's chain workspace.
struct Ctx {
    cudaStream_t st;
    ChainParams prm;
    uint32_t* P0;            // [S][W32] initial schedule, step-major
    uint32_t* Pcol0;         // [U][S32]
    uint32_t* counts0;       // [S][4]
    uint64_t* small;         // [0] total ticks, [1] hits, [2] bad step (int32), [4..5] calibration, [8..] reduce out, [16] err, [24..] work
    char* host;              // host side of the copies: 256 bytes for `small`, then the tables
    size_t host_bytes;
    std::vector<char> host_own;
    // The next call of this thread uses the same block: no way out of a call may leave a copy from or to it in flight.
    struct InFlight {
        cudaStream_t st = nullptr;
        bool any = false;
        ~InFlight() { if (any) cudaStreamSynchronize(st); }
    } copies;
    uint64_t* host_small() const { return reinterpret_cast<uint64_t*>(host); }
    uint32_t* table; uint32_t* shifts;
    kvp_chain_result* results;
    uint32_t* dumpcol;       // [U][S32]
    uint32_t* sched;         // [S][W32]
    uint32_t* slots;         // chain state slices (global variant)
    uint32_t* full0;         // [S32]
    uint32_t* hb0;           // growing cache: [S] written-to-HBM counts of the initial schedule
    bool grow;
    uint32_t* snap;          // best-state snapshots (shared-memory variant), or null
    uint64_t* undo_log;      // undo logs (global variant), or null
    uint32_t* undo_len;
    uint32_t undo_cap;
    uint32_t* cow_out;       // global variant: bucket bitmaps of the slices, or null
    uint32_t cow_shift;
    uint32_t cow_slots4;     // uint4 slots of a chain's bucket bitmap
    bool psmem;
    uint32_t wpb;            // chains per CTA
    uint32_t wpc;            // warps per chain
    uint32_t resident;       // chains per wave
    size_t smem_per_warp;    // shared memory per chain
    size_t smem_shared;      // shared memory of the CTA beside its chains (access bitmap and step constants)
    bool asmem;              // the access bitmap and the step constants are staged in shared memory
    bool wide;               // the wide kernel
    uint32_t S32;            // words per time-packed column
    bool solo;               // narrow kernel, schedules in shared memory: the variant for one warp per chain
    bool ladder_ctas;        // replica exchange: every CTA holds whole ladders (one launch)
    int rows;                // wide kernel: rows of 32 proposals in a batch
    bool ahead;              // wide kernel: placement columns loaded a row ahead
    bool lin;                // kappa_d >= kappa_k: see kvp_chain.cuh
    float* bounds;           // [levels]
    std::vector<double> temps;
    uint64_t init_ticks, calib_mean;
    uint32_t launches;
};

int validate(const kvp_problem* p, const kvp_anneal_params* a)
{
    if (!p || !a) return KVP_ERR_ARG;
    if (!a->chains || !a->moves || !a->levels || a->levels > 4096) return KVP_ERR_ARG;
    if (a->p_swap_256 > 256 || a->max_len_log2 > 5 || a->init_mode > KVP_INIT_USER) return KVP_ERR_ARG;
    if (a->init_mode == KVP_INIT_USER && !a->init_schedule) return KVP_ERR_ARG;
    if (!a->temps && (!(a->p0 > 0.0 && a->p0 < 1.0) || !(a->alpha > 0.0 && a->alpha <= 1.0))) return KVP_ERR_ARG;
    if (a->chains >= (1u << 24) || (uint64_t)a->first_chain + a->chains > (1ull << 31)) return KVP_ERR_RANGE;
    if (a->moves / a->levels + a->levels >= (1ull << 36)) return KVP_ERR_RANGE;   // batches of a level are counted in 32 bits
    return KVP_OK;
}

typedef void (*ChainKernel)(const ChainParams);

template <bool GROW, bool LIN>
ChainKernel narrow_pick(bool psmem, bool asmem, uint32_t S32, bool solo)
{
    if (psmem && solo) return asmem ? narrow_chain_kernel<true, true, true, GROW, LIN, 0> : narrow_chain_kernel<true, true, false, GROW, LIN, 0>;
    if (psmem) return asmem ? narrow_chain_kernel<false, true, true, GROW, LIN, 0> : narrow_chain_kernel<false, true, false, GROW, LIN, 0>;
    return S32 == 2 ? narrow_chain_kernel<false, false, false, GROW, LIN, 2> : S32 == 4 ? narrow_chain_kernel<false, false, false, GROW, LIN, 4>
                                                                                        : narrow_chain_kernel<false, false, false, GROW, LIN, 0>;
}

ChainKernel narrow_kernel_for(bool psmem, bool asmem, bool grow, bool lin, uint32_t S32, bool solo)
{
    if (grow) return lin ? narrow_pick<true, true>(psmem, asmem, S32, solo) : narrow_pick<true, false>(psmem, asmem, S32, solo);
    return lin ? narrow_pick<false, true>(psmem, asmem, S32, solo) : narrow_pick<false, false>(psmem, asmem, S32, solo);
}

template <bool PSMEM, bool ASMEM, bool LIN, int COLV>
ChainKernel wide_pick(bool grow, int rows, bool ahead)
{
    constexpr int kOne = !PSMEM && LIN ? kRowsOne : kRowsMany;
    constexpr bool kAhead = !PSMEM && COLV != 2, kTwo = COLV != 4;     // the forms without births (see load_ahead)
    const bool one = rows == kRowsOne;
    if (grow) return one ? wide_chain_kernel<PSMEM, true, ASMEM, LIN, COLV, kOne, false> : wide_chain_kernel<PSMEM, true, ASMEM, LIN, COLV, kRowsMany, false>;
    if (ahead || !kTwo)
        return one ? wide_chain_kernel<PSMEM, false, ASMEM, LIN, COLV, kOne, kAhead> : wide_chain_kernel<PSMEM, false, ASMEM, LIN, COLV, kRowsMany, kAhead>;
    return one ? wide_chain_kernel<PSMEM, false, ASMEM, LIN, COLV, kOne, !kTwo> : wide_chain_kernel<PSMEM, false, ASMEM, LIN, COLV, kRowsMany, !kTwo>;
}

ChainKernel wide_kernel_for(bool psmem, bool asmem, bool grow, bool lin, uint32_t S32, int rows, bool ahead)
{
    if (!psmem) {
        if (lin && S32 == 2) return wide_pick<false, false, true, 2>(grow, rows, ahead);
        if (lin && S32 == 4) return wide_pick<false, false, true, 4>(grow, rows, ahead);
        return lin ? wide_pick<false, false, true, 0>(grow, rows, ahead) : wide_pick<false, false, false, 0>(grow, rows, ahead);
    }
    if (asmem && lin) return wide_pick<true, true, true, 0>(grow, rows, ahead);
    return lin ? wide_pick<true, false, true, 0>(grow, rows, ahead) : wide_pick<true, false, false, 0>(grow, rows, ahead);
}

ChainKernel kernel_of(const Ctx& c, bool psmem, bool asmem)
{
    return c.wide ? wide_kernel_for(psmem, asmem, c.grow, c.lin, c.S32, c.rows, c.ahead)
                  : narrow_kernel_for(psmem, asmem, c.grow, c.lin, c.S32, c.solo);
}

void report_form(const Ctx& c, kvp_anneal_stats* stats)
{
    stats->wide_kernel = c.wide ? 1u : 0u;
    stats->warps_per_chain = (uint8_t)c.wpc;
    stats->shared_schedules = c.psmem ? 1u : 0u;
    stats->bucket_log2 = (uint8_t)(c.psmem ? 0u : c.cow_shift);
    stats->columns_ahead = c.ahead ? 1u : 0u;
}

int launch_chains(const Ctx& c, ChainParams& prm, uint32_t count)
{
    {
        const bool rounds = prm.rung_hist != nullptr;
        prm.lay = !c.wide ? narrow_layout(prm.S, prm.S32, c.grow, c.psmem, c.lin, c.psmem ? 0u : c.cow_slots4) : chain_layout(prm.S, prm.S32, c.grow, c.psmem, c.lin, c.psmem ? 0u : c.cow_slots4);
        prm.seg_len = rounds ? prm.exch_every : prm.per_level;
        const uint32_t batch = c.wide ? 32u * c.rows : 32u;
        prm.seg_bat = (uint32_t)((prm.seg_len + batch - 1) / batch);
        const uint64_t needed = (prm.upto + prm.seg_len - 1) / prm.seg_len;
        prm.seg0 = rounds ? prm.round0 : 0u;
        prm.seg1 = (uint32_t)std::min<uint64_t>(rounds ? prm.round1 : prm.levels, needed);
        if (rounds && prm.seg1 < needed) prm.upto = prm.seg1 * prm.seg_len;   // the last segment is a whole one
    }
    const uint32_t grid = (count + c.wpb - 1) / c.wpb;
    const size_t smem = (size_t)c.wpb * c.smem_per_warp + c.smem_shared;
    ChainParams k = prm;
    if (!c.wide) {
        k.move0 = k.seg0 * k.seg_len;
        k.seg1 -= k.seg0;
        if (k.rung_hist) k.rung_hist += (size_t)k.seg0 * k.hist_stride;
    }
    kernel_of(c, c.psmem, c.asmem)<<<grid, c.wpb * c.wpc * 32, smem, c.st>>>(k);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int run_chains(Ctx& c, uint32_t first, uint32_t count, uint32_t result_base, kvp_chain_result* results, uint64_t upto,
               uint32_t* dump, uint32_t* snap, bool with_undo = false)
{
    ChainParams prm = c.prm;
    prm.snap = snap;
    prm.undo_log = with_undo ? c.undo_log : nullptr; prm.undo_len = c.undo_len; prm.undo_cap = c.undo_cap;
    prm.cow_out = c.cow_out; prm.cow_shift = c.cow_shift; prm.cow_slots4 = c.cow_slots4;
    prm.chain_first = first; prm.chain_count = count; prm.result_base = result_base;
    prm.results = results; prm.upto = upto; prm.dump = dump;
    ++c.launches;
    return launch_chains(c, prm, count);
}

// bytes of an acceptance table with its shifts and bounds
size_t table_bytes(uint32_t levels) { return (size_t)levels * (KVP_TABLE_Q + 2) * 4; }

// Host side of a call's copies: page-locked, so that a copy neither waits for a staging copy nor holds the host up (the
// tables of 64 levels, 262 KB in three pageable copies: 40 us of a call of 540). Every call ends with a synchronisation, one
// that fails half-way too (Ctx::copies), so one block per thread is enough; it is kept up to 1 MB and freed with the thread.
// Larger calls use ordinary memory.
struct Staging {
    char* p = nullptr;
    size_t bytes = 0;
    ~Staging() { if (p) cudaFreeHost(p); }
};

char* staging(size_t bytes, std::vector<char>& otherwise)
{
    static thread_local Staging mine;
    if (mine.bytes >= bytes) return mine.p;
    if (bytes <= ((size_t)1 << 20)) {
        if (mine.p) cudaFreeHost(mine.p);
        mine = Staging();
        const size_t want = bytes <= ((size_t)512 << 10) ? (size_t)512 << 10 : (size_t)1 << 20;
        if (cudaHostAlloc(reinterpret_cast<void**>(&mine.p), want, cudaHostAllocPortable) == cudaSuccess) {
            mine.bytes = want;
            return mine.p;
        }
        cudaGetLastError();                                       // ordinary memory does as well
        mine.p = nullptr;
    }
    otherwise.resize(bytes);
    return otherwise.data();
}

// Initial schedule, its counters and cost, the temperature ladder and the acceptance table.
// rungs: 0, or the chains of a ladder (replica exchange).
int prepare(kvp_problem* p, const kvp_anneal_params* a, cudaStream_t st, Ctx& c, uint32_t rungs = 0)
{
    int rc = validate(p, a);
    if (rc) return rc;
    KVP_CUDA(cudaSetDevice(p->device));
    c.st = st;
    c.launches = 0;
    // the small block, the table of the levels; replica exchange: the table of the pairs of rungs, the last rungs
    c.host_bytes = 256 + table_bytes(a->levels) + (rungs ? table_bytes(rungs) + a->chains : 0);
    c.host = staging(c.host_bytes, c.host_own);
    const size_t sched_bytes = align256((size_t)p->S * p->W32 * 4);
    const size_t col_bytes = align256((size_t)p->U * p->S32 * 4);

    // shared-memory residency of the schedule, else a slice of global scratch per resident chain
    int dev = p->device, smem_max = 0, sms = 0;
    KVP_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    KVP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t budget = (size_t)smem_max - 1024;
    c.grow = p->dL != nullptr;
    const kvp_test_hooks hooks = g_hooks;
    c.S32 = p->S32;
    const bool exchange = rungs != 0;
    const uint32_t chains_per_sm = (a->chains + sms - 1) / sms;
    const size_t pbytes = (size_t)p->U * p->S32 * 4;
    c.lin = p->K.kd >= p->K.kk;
    c.ladder_ctas = c.solo = false;
    c.rows = kRowsMany;
    c.ahead = false;
    c.cow_slots4 = 0;
    c.cow_shift = 0;
    c.smem_shared = 0;
    c.asmem = false;
    auto fixed_bytes = [&](uint32_t warps, bool shared) {
        if (c.wide) return chain_bytes(p->S, p->S32, c.grow, shared, c.lin, shared ? 0u : c.cow_slots4, warps, c.rows, c.ahead);
        return narrow_bytes(p->S, p->S32, c.grow, shared, c.lin, shared ? 0u : c.cow_slots4, warps);
    };
    // Which kernel, and how many warps per chain (W; an SM holds 16). Measured on 1800 problems of 64 to 524,288 units x 32 to
    // 512 steps, 5 to 20% of the units read per step, 10 to 45% in HBM, even and Zipf importance, 64 to 2368 chains of 10,000 to
    // 100,000 moves, p0 = 1e-6, 0.03 and 0.3; the times below are ratios to the chosen form's, geometric means over such jobs
    // (over all of them the chosen form takes 1.02 to 1.04 times the best one's time, 1.16 to 1.18 with the lines before).
    //  - What decides is how many proposals change the schedule. Many do at a warm start, and at any where the HBM side of Eq. 2
    //    is the larger one in the static placement (busy): such a schedule gets better by moving units out of HBM, and 2 to 14%
    //    of a near-greedy chain's first 20,000 proposals change it, elsewhere 0.02 to 1%. A quiet chain has few proposals to
    //    judge, which the wide kernel's compaction is for; the fewer units are in HBM or read the fewer, and fewer later on.
    //  - Schedules in shared memory: the narrow kernel (wide: 1.2 to 2.35), from p0 = 0.02 on with one warp per chain (two: 1.09
    //    at 0.03, 1.32 at 0.3), below with three up to 5 per SM (two: 1.12, four: 1.02 up to 4), two up to 8 and one beyond; two
    //    at most on fewer than 64 units and on busy short horizons, where moves meet most often. One on fewer than 64 units and
    //    steps (two: 1.07 in the mean of 16 jobs, 0.97 to 1.22; 16 x 32, 64 chains x 10,000: 330 to 365 us by box, there 365 against two
    //    380, three 400), and for 7 and 8 chains per SM where the static placement serves less than half of the reads (two: 1.06
    //    over 66 such jobs, 0.95 to 1.18, on 24 others 1.10, 1.06 to 1.21; 0.99 where it serves more, over 99). The wide one for quiet jobs of more than 8 chains per SM with next to nothing in HBM, if they
    //    are brief or have many units (narrow: 1.1 to 1.2).
    //  - In global memory: the narrow kernel on busy chains, with two warps per chain up to 8 per SM and one beyond (four: 1.77,
    //    wide: 2.1 to 2.2), at warm starts (wide: 1.03 to 1.46) and up to 5 quiet chains per SM, with four warps per chain up to 4,
    //    two up to 8 and one beyond. More quiet chains: the wide one, with two warps per chain up to 8 per SM and one beyond (100,000
    //    moves: narrow 1.05 to 1.8). The limits below are those of jobs of 10,000 moves, whose chains still change much, and of
    //    6 to 8 chains per SM that judge much (where they stop the wide kernel takes 1.0 to 1.25).
    // What counts as chains of an SM (held) is how many it holds at a time when their state takes its shared memory, the waves
    // of the job taken equally large. A ladder given as temperatures is taken for a near-greedy one: what share of the
    // proposals it accepts is not known (256 x 512, 1024 chains x 100,000 moves with the ladder of p0 = 0.8: 23.3 instead of
    // 13.6 ms).
    // kvp_set_test_hooks can force the choice (warps_per_chain 1, 2 or 32 + w: narrow; 3 or 16 + w: wide).
    const double p0 = a->temps ? 0.0 : a->p0;
    const bool busy = (double)p->kh * (double)p->static_hits >= 0.9 * (double)p->ke * (double)(p->total_accessed - p->static_hits);
    c.wide = false;                                               // (for the bytes of a chain)
    c.psmem = fixed_bytes(1, true) + pbytes + 16 <= budget / 2 && p->U < 65536u;
    const uint32_t fit = (uint32_t)((budget - 16) / (c.psmem ? fixed_bytes(1, true) + pbytes : fixed_bytes(1, false) + kCowBitsMin / 8));
    const uint32_t at_a_time = std::min(std::max(fit, 1u), 16u);
    const uint32_t turns = (chains_per_sm + at_a_time - 1) / at_a_time;
    const uint32_t held = turns > 1 ? (chains_per_sm + turns - 1) / turns : chains_per_sm;
    const double in_hbm = (double)p->cap / p->U, read = (double)p->total_accessed / p->S / p->U;
    const bool quiet = !busy && p0 < 0.02, brief = a->moves < 30000;
    if (quiet && c.psmem) c.wide = held > 8 && in_hbm <= 0.15 && (brief || p->U >= 1024u);
    if (quiet && !c.psmem && held > 5)
        c.wide = brief ? in_hbm <= (p->S > 128 ? 0.2 : p->S > 64 ? 0.25 : held > 8 ? 0.4 : 0.3)
                       : held > 8 || p->S <= 64 || read <= 0.1 || in_hbm <= 0.2;
    if (hooks.warps_per_chain) c.wide = hooks.warps_per_chain == 3 || (hooks.warps_per_chain >= 16 && hooks.warps_per_chain < 32);
    // Replica exchange: every round waits for the hottest rungs, which apply the most moves: the narrow kernel, with one warp per
    // chain where schedules live in shared memory. Whole ladders in a CTA (128 of 8 on 256 units x 512 steps, 100,000 moves: 4.5
    // ms, two warps 5.1, wide kernel 7.5; 7 of 4 on 46 x 61, 38,619 moves: 3.5, 5.4, 11.2), or rounds of launches (51 of 20,
    // 50,000 moves: 3.4 ms, wide kernel 5.5; with a slow link 5.2 and 9.8; 128 of 8 on 16,384 x 256, 20,000 moves: 3.8 and 8.0).
    if (exchange && !hooks.warps_per_chain) c.wide = false;
    // Growing caches: the narrow kernel with schedules in shared memory and for warm starts (512 units x 132 steps, 256 chains
    // x 20,000 moves: 0.46 against 0.61 ms, at p0 = 0.8 1.7 against 5.2; 131,072 x 1056, 1024 x 20,000 at p0 = 0.3 1.39
    // against 1.70, at 0.8 4.5 against 6.6); the wide one for near-greedy chains in global memory, most of whose proposals
    // change nothing, which its compaction is for (0.65 against 0.80, at p0 = 0.1 0.90 against 0.93), and, with a slow link,
    // for jobs of many chains (2368 x 10,000 at p0 = 0.8: 16.5 against 20.9; 1024 x 20,000: 10.7 against 7.0).
    if (c.grow && !hooks.warps_per_chain && !exchange) c.wide = !c.psmem && (p0 < 0.2 || (!c.lin && chains_per_sm > 8));
    if (c.wide) c.psmem = fixed_bytes(1, true) + pbytes + 16 <= budget / 2 && p->U < 65536u;
    const uint32_t forced = hooks.warps_per_chain == 3 ? 1u : hooks.warps_per_chain >= 16 ? hooks.warps_per_chain & 15u : hooks.warps_per_chain;
    const uint32_t full = 16;
    auto narrow_warps = [&]() {
        if (c.psmem && (p0 >= 0.02 || (!c.lin && held > 4))) return 1u;
        const uint32_t most = held <= 4 ? 4u : held == 5 ? 3u : held <= 8 ? 2u : 1u;
        if (c.grow && !c.psmem) return c.lin ? std::min(most, 2u) : 1u;
        if (c.psmem && !c.grow && ((p->U < 64u && p->S < 64u) || (held > 6 && 2 * p->static_hits < p->total_accessed))) return 1u;
        if (c.psmem) return std::min(most, p->U < 64u || (busy && p->S < 128u) ? 2u : 3u);
        return busy || p0 >= 0.5 ? std::min(most, 2u) : most;
    };
    uint32_t W = 1;
    if (c.psmem) {
        uint32_t want = held;
        // whole ladders, where a CTA can hold one (256 x 512, 92 ladders of 11, which it cannot: 93 CTAs of 11 chains would
        // leave a third of the SMs idle)
        if (exchange && rungs <= full && rungs * (fixed_bytes(1, true) + pbytes) + 16 <= budget) want = (want + rungs - 1) / rungs * rungs;
        // bytes with the access bitmap staged; columns are followed by readable bytes
        auto with_a = [&](uint32_t chains, uint32_t warps) {
            const size_t a_off = ((size_t)chains * (pbytes / 4) + 3) & ~(size_t)3, c_off = (a_off + pbytes / 4 + 3) & ~(size_t)3;
            return (size_t)chains * fixed_bytes(warps, true) + c_off * 4 + 16;
        };
        if (c.wide) {
            // two warps per chain, four where an SM has three chains or fewer (256 units x 512 steps, 50,000 moves, 148 and
            // 740 chains: one warp 1.62 and 1.79 ms, two 1.12 and 1.34, four 1.05 and 2.40)
            W = chains_per_sm <= 3 ? 4 : 2;
            while (W > 1 && (want * W > full || with_a(want, W) > budget)) W /= 2;
        } else {
            W = exchange ? 1u : narrow_warps();
            while (W > 1 && (fixed_bytes(W, true) + pbytes) * held + 16 > budget) --W;
        }
        if (forced) W = forced;
        if (exchange && !c.wide && (rungs * W > full || rungs * (fixed_bytes(W, true) + pbytes) + 16 > budget)) W = 1;
        c.wpc = W;
        c.smem_per_warp = fixed_bytes(W, true) + pbytes;
        uint32_t wmax = (uint32_t)((budget - 16) / c.smem_per_warp);
        if (wmax > full / W) wmax = full / W;
        if (wmax < 1) return KVP_ERR_RANGE;
        c.wpb = want > wmax ? wmax : want;
        c.solo = !c.wide && W == 1 && c.wpb <= 8u;                // that variant is built for CTAs of up to 256 threads
        if (exchange && rungs <= wmax) {
            c.ladder_ctas = true;
            c.wpb = c.wpb / rungs * rungs;
        }
        c.resident = a->chains;
        c.smem_shared = 16;
        c.asmem = with_a(c.wpb, W) <= budget && (!c.wide || c.lin);
        if (c.asmem) {
            c.smem_shared = with_a(c.wpb, W) - (size_t)c.wpb * c.smem_per_warp;
        }
        KVP_CUDA(cudaFuncSetAttribute(kernel_of(c, true, c.asmem), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget));
    } else {
        // wide: two warps per chain while an SM has at most 8 (more per chain are no faster)
        if (!c.wide) W = narrow_warps();
        else if (!exchange && chains_per_sm <= 8 && !(c.grow && !c.lin)) W = 2;   // (131,072 x 1056 births, slow link: 1.07 against 1.13 ms)
        const bool may_load_ahead = c.wide && load_ahead(c.grow, c.lin, p->S32);
        c.ahead = may_load_ahead;                                 // (the smaller work area)
        while (W > 1 && fixed_bytes(W, false) + kCowBitsMin / 8 > budget) --W;   // very long horizons
        // replica exchange keeps every chain resident: no more warps than leave room for all of them
        while (exchange && W > 1 && std::min<size_t>(full / W, budget / (fixed_bytes(W, false) + kCowBitsMin / 8)) * sms < a->chains) --W;
        if (forced) W = forced;
        if (W == 1 && c.wide && c.lin) c.rows = kRowsOne;
        // Shares the shared memory out and returns how many chains a CTA can hold (0: not one).
        auto share_out = [&](bool ahead) {
            c.ahead = ahead;
            c.cow_shift = c.cow_slots4 = 0;
            uint32_t per_cta = full / W;                          // chains of a full CTA
            if (chains_per_sm < per_cta) per_cta = chains_per_sm ? chains_per_sm : 1u;
            // The bucket bitmap takes what a full CTA of chains leaves of the shared memory: the smaller the buckets, the
            // fewer reads of a long chain go to its private slice.
            const size_t bare = fixed_bytes(W, false);
            if (budget / bare < per_cta) per_cta = (uint32_t)(budget / bare);
            if (per_cta < 1) return 0u;
            const size_t share = budget / per_cta;
            size_t bits = share > bare ? (share - bare) / 16 * 128 : 0;
            if (bits < kCowBitsMin) bits = kCowBitsMin;
            if (bits > kCowBitsMax) bits = kCowBitsMax;
            while (((uint64_t)p->U + (1ull << c.cow_shift) - 1) >> c.cow_shift > bits) ++c.cow_shift;
            if (hooks.overlay == 2 && c.cow_shift < 3) c.cow_shift = 3;   // test hook
            const uint64_t buckets = ((uint64_t)p->U + (1ull << c.cow_shift) - 1) >> c.cow_shift;
            c.cow_slots4 = (uint32_t)((buckets + 127) / 128);
            c.smem_per_warp = fixed_bytes(W, false);
            return (uint32_t)std::min<size_t>(budget / c.smem_per_warp, full / W);
        };
        // Wide kernel: two rows of proposals at a time, or one whose columns were loaded a row ahead (see rows_at_a_time). The
        // first is the faster one by itself (350 jobs: 1.02 to 1.04 in the mean of 16,000 to 50,000 moves, 0.98 to 1.11), but for
        // columns of four words (0.88 to 0.99) and where the last row of a level stands alone in it (0.93 to 0.97 with three
        // rows a level, 0.97 with five in batches of eight, 1.00 in batches of four). The second has the smaller work area: it is
        // taken where a CTA of the first needs more than 196 KB, which leaves 28 KB of an SM's L1 instead of 60 (2368 chains: 1.07 to
        // 1.6 times faster), or more waves (1.27 to 1.7).
        const uint64_t level_rows = (a->moves / a->levels + 31) / 32;
        const bool odd_rows = (level_rows & 1u) && level_rows < (uint64_t)c.rows;
        uint32_t wcap = share_out(may_load_ahead && (exchange || (c.lin && p->S32 == 4) || odd_rows));   // chains per CTA at most
        if (may_load_ahead && !c.ahead) {
            auto waves_of = [&](uint32_t held) { return (a->chains + held * sms - 1) / (held * sms); };
            const uint32_t waves = wcap ? waves_of(wcap) : 0u;
            const uint32_t in_cta = waves ? ((a->chains + waves - 1) / waves + sms - 1) / sms : 0u;
            const bool crowded = !waves || std::min(in_cta, wcap) * c.smem_per_warp + 1024 > ((size_t)196 << 10);
            if (crowded || waves > 1) wcap = share_out(true);
            if (!crowded && waves > 1 && waves_of(wcap) == waves) wcap = share_out(false);
        }
        if (wcap < 1) return KVP_ERR_RANGE;
        c.wpc = W;
        KVP_CUDA(cudaFuncSetAttribute(kernel_of(c, false, false), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget));
        int ctas = 0;
        KVP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, kernel_of(c, false, false), (int)(wcap * W * 32),
                                                               wcap * c.smem_per_warp));
        if (ctas < 1) return KVP_ERR_RANGE;
        uint32_t per_sm = (uint32_t)ctas * wcap;                   // resident chains per SM, at most 32 warps
        if (per_sm * W > 32) per_sm = 32 / W / wcap ? 32 / W / wcap * wcap : wcap;
        size_t cap_r = (size_t)per_sm * sms;
        size_t r = a->chains < cap_r ? a->chains : cap_r;
        // How many slices fit. What the problem holds and what the pool has in reserve is known without asking the driver
        // for the device's free memory, which takes 90 us.
        size_t have = p->chain_ws_bytes;
        {
            cudaMemPool_t pool; uint64_t reserved = 0, used = 0;
            if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess &&
                cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
                cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess && reserved > used)
                have += (size_t)(reserved - used);
        }
        if (p->chain_ws_bytes < r * col_bytes && have / 10 * 9 < r * col_bytes) {
            size_t free_b = 0, total_b = 0;
            KVP_CUDA(cudaMemGetInfo(&free_b, &total_b));
            const size_t fit = (have + free_b) / 10 * 7 / col_bytes;
            if (fit < 1) return KVP_ERR_NOMEM;
            if (r > fit) r = fit;
        }
        // test hook: at most n chains at a time, so that small jobs come in several waves
        if (hooks.resident >= 1 && (size_t)hooks.resident < r) r = hooks.resident;
        const uint32_t waves = (uint32_t)((a->chains + r - 1) / r);
        c.resident = (a->chains + waves - 1) / waves;              // equal waves
        // a wave is spread over all SMs: CTAs of ceil(resident / SMs) chains where one CTA per SM holds them
        const uint32_t even = (c.resident + sms - 1) / sms;
        c.wpb = even < wcap ? even : wcap;
    }
    // a replica-exchange run keeps every chain's slice between its rounds: all chains have to be resident at once
    if (exchange && !c.psmem && a->chains > c.resident) return KVP_ERR_RANGE;

    // workspace layout
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += align256(bytes); return o; };
    const size_t o_P0 = take(sched_bytes), o_col0 = take(col_bytes), o_cnt = take((size_t)p->S * 20 + 4);   // counts, births, ticket
    const size_t o_small = take(256), o_table = take(table_bytes(a->levels));
    const size_t o_res = take((size_t)(a->chains + 1) * sizeof(kvp_chain_result));
    const size_t o_dump = take(col_bytes), o_sched = take(sched_bytes);
    const size_t o_slots = take(c.psmem ? 0 : (size_t)c.resident * col_bytes);
    const size_t o_full = take((size_t)p->S32 * 4);
    // Chains whose schedule lives in shared memory save it to global memory whenever they leave their best state;
    // chains in global scratch do not (a copy would cost as much as thousands of moves): their winner is replayed.
    const size_t snap_bytes = (size_t)a->chains * p->U * p->S32 * 4;
    const bool snapshots = c.psmem && snap_bytes <= ((size_t)2 << 30);
    const size_t o_snap = take(snapshots ? snap_bytes : 0);
    // Chains in global scratch log the moves they apply after their best state (8 bytes each, up to 4096), so that
    // the winner can be walked back instead of replayed from its first move.
    c.undo_cap = c.psmem ? 0u : 4096u;
    const size_t o_ulog = take((size_t)c.resident * c.undo_cap * 8), o_ulen = take(c.psmem ? 0 : (size_t)c.resident * 4);
    // Which buckets of its slice a chain has taken over, for the walk back of the winner.
    const size_t o_cow = take(c.psmem ? 0 : (size_t)c.resident * c.cow_slots4 * 16);
    rc = ensure_chain_ws(p, off, st);
    if (rc) return rc;
    char* base = static_cast<char*>(p->d_chain_ws);
    c.P0 = (uint32_t*)(base + o_P0); c.Pcol0 = (uint32_t*)(base + o_col0); c.counts0 = (uint32_t*)(base + o_cnt);
    c.small = (uint64_t*)(base + o_small); c.table = (uint32_t*)(base + o_table);
    c.shifts = c.table + (size_t)a->levels * KVP_TABLE_Q; c.bounds = (float*)(c.shifts + a->levels);
    c.results = (kvp_chain_result*)(base + o_res); c.dumpcol = (uint32_t*)(base + o_dump);
    c.sched = (uint32_t*)(base + o_sched); c.slots = (uint32_t*)(base + o_slots);
    c.hb0 = c.grow ? c.counts0 + (size_t)p->S * 4 : nullptr;
    c.full0 = (uint32_t*)(base + o_full); c.snap = snapshots ? (uint32_t*)(base + o_snap) : nullptr;
    c.undo_log = c.psmem ? nullptr : (uint64_t*)(base + o_ulog); c.undo_len = c.psmem ? nullptr : (uint32_t*)(base + o_ulen);
    c.cow_out = c.psmem ? nullptr : (uint32_t*)(base + o_cow);

    // initial schedule in both layouts
    KVP_CUDA(cudaMemsetAsync(c.small, 0, 256, st));
    if (a->init_mode == KVP_INIT_USER) {
        if ((rc = launch_clean_copy(a->init_schedule, c.P0, p->S, p->W32, p->pad_mask, st))) return rc;
        // a unit of the initial placement enters HBM when it is written; the chains keep the bits before that clear
        if (c.grow && (rc = launch_and_rows(c.P0, p->dL, (size_t)p->S * p->W32, st))) return rc;
        if ((rc = launch_bit_transpose(c.P0, p->S, p->W32, p->U, c.Pcol0, p->S32, st))) return rc;
        c.launches += c.grow ? 3 : 2;
    } else {
        const uint32_t* row = p->d_row_freq;
        if (a->init_mode == KVP_INIT_STATIC_FIRST) {
            if ((rc = launch_static_first_row(p, c.sched, st))) return rc;
            row = c.sched;
            ++c.launches;
        }
        if ((rc = launch_initial_schedule(p, row, c.P0, c.Pcol0, st))) return rc;
        ++c.launches;
    }
    if ((rc = launch_score(p, c.P0, 1, c.counts0, c.counts0, c.hb0, nullptr, c.small, nullptr, nullptr, (int32_t*)(c.small + 2),
                           c.small + 1, st, &c.launches)))
        return rc;
    full_mask_kernel<<<(p->S32 * 32 + 255) / 256, 256, 0, st>>>((const uint4*)c.counts0, p->S, p->cap, c.full0);
    KVP_CUDA(cudaGetLastError());
    ++c.launches;

    ChainParams& prm = c.prm;
    memset(&prm, 0, sizeof prm);
    prm.Acol = p->dAcol; prm.stepc = p->d_stepc; prm.counters0 = (const uint4*)c.counts0; prm.Pcol0 = c.Pcol0;
    prm.table = c.table; prm.shifts = c.shifts; prm.bounds = c.bounds; prm.warps = c.wpc; prm.ws = c.slots; prm.K = p->K; prm.full0 = c.full0;
    prm.birth = p->d_birth; prm.hb0 = c.hb0;
    prm.err = reinterpret_cast<uint32_t*>(c.small + 16);
    prm.work = nullptr;                                   // set by kvp_anneal for the chains of the search proper
    // test hook (tests of the bounded wait only): one hand-over per chain is withheld, the waiting warp gives up
    // after its poll limit (about a second) and the call returns KVP_ERR_TIMEOUT
    prm.drop_first_turn = hooks.drop_turn ? 1u : 0u;
    // test hook: less room for accepted proposals, so that a batch stops to commit more often
    prm.carry = kAccepted;
    if (hooks.split_queue_plus1 >= 1 && hooks.split_queue_plus1 <= kAccepted) prm.carry = hooks.split_queue_plus1;
    prm.U = p->U; prm.S = p->S; prm.S32 = p->S32; prm.cap = p->cap;
    prm.levels = a->levels; prm.p_swap_256 = a->p_swap_256; prm.len_choices = a->max_len_log2 + 1;
    prm.early_permille = a->early_stop_permille; prm.early_from = a->early_stop_from_level;
    prm.keys = philox_keys((uint32_t)a->seed, (uint32_t)(a->seed >> 32));
    prm.per_level = a->moves / a->levels ? a->moves / a->levels : 1;

    // temperature ladder
    c.temps.resize(a->levels);
    c.calib_mean = 0;
    const bool calibrate = a->temps == nullptr;
    if (calibrate) {
        if (c.grow) calib_kernel<true><<<CALIB_N / 256, 256, 0, st>>>(prm, (unsigned long long*)(c.small + 4));
        else calib_kernel<false><<<CALIB_N / 256, 256, 0, st>>>(prm, (unsigned long long*)(c.small + 4));
        KVP_CUDA(cudaGetLastError());
        ++c.launches;
    }
    uint64_t* const host_small = c.host_small();
    c.copies.st = st;
    c.copies.any = true;
    KVP_CUDA(cudaMemcpyAsync(host_small, c.small, 64, cudaMemcpyDeviceToHost, st));
    KVP_CUDA(cudaStreamSynchronize(st));
    if ((int32_t)(host_small[2] & 0xFFFFFFFFu) >= 0) return KVP_ERR_CAPACITY;   // Eq. 5 on the initial schedule
    c.init_ticks = host_small[0];
    prm.init_ticks = c.init_ticks;
    if (calibrate) {
        uint64_t mean = host_small[5] ? host_small[4] / host_small[5] : 1;
        if (!mean) mean = 1;
        c.calib_mean = mean;
        double C = -(double)mean / log(a->p0);
        for (uint32_t j = 0; j < a->levels; ++j) { c.temps[j] = C; C = C * a->alpha; }
    } else {
        for (uint32_t j = 0; j < a->levels; ++j) c.temps[j] = a->temps[j];
    }
    uint32_t* const table = reinterpret_cast<uint32_t*>(c.host + 256);
    uint32_t* const shifts = table + (size_t)a->levels * KVP_TABLE_Q;
    float* const bounds = reinterpret_cast<float*>(shifts + a->levels);
    if ((rc = kvp_accept_table(c.temps.data(), a->levels, table, shifts))) return rc;
    // the lower bounds of kvp_chain.cuh are sums of at most 31 steps' changes in 32 bits
    const uint64_t step_max = 4ull * std::max({p->K.khF, p->K.kdF, p->K.kkF}) + std::max(p->K.kh, p->K.ke) + 2ull * std::max(p->K.kh, p->K.ke);
    const bool bounded = 31 * step_max < (1ull << 30);
    for (uint32_t j = 0; j < a->levels; ++j) bounds[j] = bounded ? (float)((c.temps[j] >= 1.0 ? c.temps[j] : 1.0) * 0.69314718) : INFINITY;
    KVP_CUDA(cudaMemcpyAsync(c.table, table, table_bytes(a->levels), cudaMemcpyHostToDevice, st));
    return KVP_OK;
}

// Replay `chain` for `upto` proposals and leave its schedule, step-major, in `sched`.
int replay_to_sched(kvp_problem* p, Ctx& c, uint32_t chain, uint64_t upto, kvp_chain_result* result_dev, uint32_t* sched)
{
    int rc;
    if (upto == 0) {
        KVP_CUDA(cudaMemcpyAsync(sched, c.P0, (size_t)p->S * p->W32 * 4, cudaMemcpyDeviceToDevice, c.st));
        return KVP_OK;
    }
    if ((rc = run_chains(c, chain, 1, chain, result_dev, upto, c.dumpcol, nullptr))) return rc;
    if ((rc = launch_bit_transpose(c.dumpcol, p->U, p->S32, p->S, sched, p->W32, c.st))) return rc;
    ++c.launches;
    return KVP_OK;
}

}  // namespace

}  // namespace kvp

using namespace kvp;

extern "C" int kvp_anneal(kvp_problem* p, const kvp_anneal_params* a, uint32_t* best_schedule, uint64_t* best_ticks,
                          double* best_seconds, kvp_anneal_stats* stats, void* stream)
try {
    Ctx c;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = validate(p, a);
    if (rc) return rc;
    KVP_CUDA(cudaSetDevice(p->device));
    struct Events {                                       // destroyed on every way out of the call
        cudaEvent_t e[4];
        int n = 0;
        ~Events() { for (int i = 0; i < n; ++i) cudaEventDestroy(e[i]); }
        cudaEvent_t operator[](int i) const { return e[i]; }
    } ev;
    for (; ev.n < 4; ++ev.n) KVP_CUDA(cudaEventCreate(&ev.e[ev.n]));
    KVP_CUDA(cudaEventRecord(ev[0], st));
    if ((rc = prepare(p, a, st, c))) return rc;
    KVP_CUDA(cudaEventRecord(ev[1], st));

    // the chains, one wave of resident chains after the other
    ReduceOut* red_dev = reinterpret_cast<ReduceOut*>(c.small + 8);
    ReduceOut red;
    memset(&red, 0, sizeof red);
    uint32_t dumped_chain = 0xFFFFFFFFu;                  // call-local index of the chain whose best state is in dumpcol
    uint32_t waves = 0;
    unsigned long long* work_dev = reinterpret_cast<unsigned long long*>(c.small + 24);
    c.prm.work = c.wide ? work_dev : nullptr;
    for (uint32_t first = 0; first < a->chains; first += c.resident, ++waves) {
        const uint32_t count = a->chains - first < c.resident ? a->chains - first : c.resident;
        if ((rc = run_chains(c, a->first_chain + first, count, a->first_chain, c.results, a->moves, nullptr, c.snap,
                             c.undo_log != nullptr)))
            return rc;
        if (c.undo_log) {
            // Best so far over the chains that have finished; if it belongs to this wave, walk that chain back to
            // its best state while its scratch slice still holds its final state.
            reduce_kernel<<<1, 1024, 0, st>>>(c.results, first + count, c.prm.err, red_dev);
            KVP_CUDA(cudaGetLastError());
            ++c.launches;
            KVP_CUDA(cudaMemcpyAsync(&red, red_dev, sizeof red, cudaMemcpyDeviceToHost, st));
            KVP_CUDA(cudaStreamSynchronize(st));
            if (red.pad) return KVP_ERR_TIMEOUT;
            if (red.best_chain >= first && red.best_move != ~0ull) {
                uint32_t len = 0;
                KVP_CUDA(cudaMemcpyAsync(&len, c.undo_len + (red.best_chain - first), 4, cudaMemcpyDeviceToHost, st));
                KVP_CUDA(cudaStreamSynchronize(st));
                if (len <= c.undo_cap) {
                    ChainParams prm = c.prm;
                    prm.chain_first = a->first_chain + first;
                    prm.undo_log = c.undo_log; prm.undo_len = c.undo_len; prm.undo_cap = c.undo_cap;
                    prm.cow_out = c.cow_out; prm.cow_shift = c.cow_shift; prm.cow_slots4 = c.cow_slots4;
                    const uint32_t wslot = red.best_chain - first;
                    if (c.grow) undo_kernel<true><<<1, 32, 0, st>>>(prm, wslot);
                    else undo_kernel<false><<<1, 32, 0, st>>>(prm, wslot);
                    KVP_CUDA(cudaGetLastError());
                    gather_slice_kernel<<<148 * 4, 256, 0, st>>>(c.dumpcol, c.slots + (size_t)wslot * p->U * p->S32, c.Pcol0,
                                                                 c.cow_out + (size_t)wslot * (c.cow_slots4 * 4),
                                                                 c.cow_shift, p->U, p->S32);
                    KVP_CUDA(cudaGetLastError());
                    c.launches += 2;
                    dumped_chain = red.best_chain;
                }
            }
        }
    }
    KVP_CUDA(cudaEventRecord(ev[2], st));
    c.prm.work = nullptr;                                 // a replay of the winner is not part of the count

    // cross-chain reduction, then the winner's schedule (its own snapshot, its walked-back state, or a replay) and a
    // re-score
    uint32_t* const sched = best_schedule ? best_schedule : c.sched;
    uint64_t* const host_small = c.host_small();
    if (!c.undo_log) {
        reduce_kernel<<<1, 1024, 0, st>>>(c.results, a->chains, c.prm.err, red_dev);
        KVP_CUDA(cudaGetLastError());
        ++c.launches;
    }
    if (c.snap) {                                          // the device knows which snapshot: no wait in between
        ChosenInput winner;
        winner.otherwise = c.Pcol0; winner.valid = &red_dev->best_move; winner.index = &red_dev->best_chain;
        if ((rc = launch_bit_transpose(c.snap, p->U, p->S32, p->S, sched, p->W32, st, winner))) return rc;
        ++c.launches;
    } else {
        if (!c.undo_log) {
            KVP_CUDA(cudaMemcpyAsync(&red, red_dev, sizeof red, cudaMemcpyDeviceToHost, st));
            KVP_CUDA(cudaStreamSynchronize(st));
            if (red.pad) return KVP_ERR_TIMEOUT;
        }
        const uint64_t upto = red.best_move == ~0ull ? 0 : red.best_move + 1;
        if (upto && dumped_chain == red.best_chain) {
            if ((rc = launch_bit_transpose(c.dumpcol, p->U, p->S32, p->S, sched, p->W32, st))) return rc;
            ++c.launches;
        } else if ((rc = replay_to_sched(p, c, a->first_chain + red.best_chain, upto, c.results + a->chains, sched))) {
            return rc;
        }
    }
    if ((rc = launch_score(p, sched, 1, c.counts0, nullptr, nullptr, nullptr, c.small, nullptr, nullptr, (int32_t*)(c.small + 2),
                           c.small + 1, st, &c.launches)))
        return rc;
    KVP_CUDA(cudaMemcpyAsync(host_small, c.small, 256, cudaMemcpyDeviceToHost, st));
    if (stats && stats->per_chain)
        KVP_CUDA(cudaMemcpyAsync(stats->per_chain, c.results, (size_t)a->chains * sizeof(kvp_chain_result),
                                 cudaMemcpyDeviceToHost, st));
    KVP_CUDA(cudaEventRecord(ev[3], st));
    KVP_CUDA(cudaStreamSynchronize(st));
    c.copies.any = false;
    memcpy(&red, host_small + 8, sizeof red);
    if (red.pad) return KVP_ERR_TIMEOUT;
    red.best_chain += a->first_chain;                      // the reduction works on call-local indices
    const uint64_t* const work = host_small + 24;
    const bool ok = host_small[0] == red.best_ticks && (int32_t)(host_small[2] & 0xFFFFFFFFu) < 0;
    if (best_ticks) *best_ticks = red.best_ticks;
    if (best_seconds) *best_seconds = (double)red.best_ticks * p->spt;
    if (stats) {
        kvp_chain_result* keep = stats->per_chain;
        memset(stats, 0, sizeof *stats);
        stats->per_chain = keep;
        stats->init_ticks = c.init_ticks; stats->best_ticks = red.best_ticks; stats->best_chain = red.best_chain;
        stats->levels = a->levels; stats->best_move = red.best_move; stats->moves_total = red.moves_total;
        stats->calib_mean_delta = c.calib_mean; stats->temp0 = c.temps[0];
        stats->winner_hits = host_small[1]; stats->winner_accessed = p->total_accessed;
        cudaEventElapsedTime(&stats->ms_init, ev[0], ev[1]);
        cudaEventElapsedTime(&stats->ms_chains, ev[1], ev[2]);
        cudaEventElapsedTime(&stats->ms_finish, ev[2], ev[3]);
        stats->kernel_launches = c.launches;
        stats->chain_launches = waves; stats->resident_chains = c.resident;
        report_form(c, stats);
        stats->work_again = work[0]; stats->work_listed = work[1]; stats->work_items = work[2];
    }
    return ok ? KVP_OK : KVP_ERR_INTERNAL;
} catch (const std::bad_alloc&) {
    return KVP_ERR_NOMEM;
}

extern "C" int kvp_anneal_chain_state(kvp_problem* p, const kvp_anneal_params* a, uint32_t chain, uint64_t upto_moves,
                                      uint32_t* schedule, kvp_chain_result* result, void* stream)
try {
    if (!schedule) return KVP_ERR_ARG;
    Ctx c;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = prepare(p, a, st, c);
    if (rc) return rc;
    if (upto_moves > a->moves) upto_moves = a->moves;
    kvp_chain_result* res_dev = c.results;
    if (upto_moves == 0) {
        kvp_chain_result r0;
        memset(&r0, 0, sizeof r0);
        r0.best_ticks = r0.final_ticks = c.init_ticks; r0.best_move = ~0ull;
        KVP_CUDA(cudaMemcpyAsync(res_dev, &r0, sizeof r0, cudaMemcpyHostToDevice, st));
    }
    if ((rc = replay_to_sched(p, c, chain, upto_moves, res_dev, schedule))) return rc;
    if (result) KVP_CUDA(cudaMemcpyAsync(result, res_dev, sizeof *result, cudaMemcpyDeviceToHost, st));
    uint32_t gave_up = 0;
    KVP_CUDA(cudaMemcpyAsync(&gave_up, c.prm.err, 4, cudaMemcpyDeviceToHost, st));
    KVP_CUDA(cudaStreamSynchronize(st));
    c.copies.any = false;
    return gave_up ? KVP_ERR_TIMEOUT : KVP_OK;
} catch (const std::bad_alloc&) {
    return KVP_ERR_NOMEM;
}

extern "C" void kvp_set_test_hooks(const kvp_test_hooks* hooks)
{
    if (hooks) g_hooks = *hooks;
    else memset(&g_hooks, 0, sizeof g_hooks);
}

extern "C" int kvp_exchange_temps(const double* temps, uint32_t rungs, double* pair_temps, uint32_t* always)
{
    if (!temps || !rungs || (rungs > 1 && (!pair_temps || !always))) return KVP_ERR_ARG;
    for (uint32_t j = 0; j + 1 < rungs; ++j) {
        const double a = temps[j] >= 1.0 ? temps[j] : 1.0, b = temps[j + 1] >= 1.0 ? temps[j + 1] : 1.0;
        if (b > a) return KVP_ERR_ARG;                     // a ladder falls
        const double inv = 1.0 / b - 1.0 / a;
        if (!(inv > 0.0) || 1.0 / inv > 1099511627776.0) { always[j] = 1; pair_temps[j] = 1.0; }
        else { always[j] = 0; pair_temps[j] = 1.0 / inv; }
    }
    return KVP_OK;
}

extern "C" int kvp_anneal_exchange(kvp_problem* p, const kvp_anneal_params* a, const kvp_exchange_params* xp,
                                   uint32_t* best_schedule, uint64_t* best_ticks, double* best_seconds,
                                   kvp_anneal_stats* stats, uint32_t* final_rung, uint32_t* n_exchanged, void* stream)
try {
    Ctx c;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = validate(p, a);
    if (rc) return rc;
    if (!xp || !xp->rungs || xp->rungs > 256 || xp->reserved || !xp->exchange_every) return KVP_ERR_ARG;
    const uint32_t rungs = xp->rungs, chains = a->chains;
    if (a->levels != rungs || chains % rungs || a->first_chain % rungs || a->early_stop_permille) return KVP_ERR_ARG;
    const uint64_t rounds64 = (a->moves + xp->exchange_every - 1) / xp->exchange_every;
    if (rounds64 * chains > (1ull << 30)) return KVP_ERR_RANGE;          // the rung history is kept: one byte per chain and round
    const uint32_t rounds = (uint32_t)rounds64;
    KVP_CUDA(cudaSetDevice(p->device));
    struct Events {
        cudaEvent_t e[4];
        int n = 0;
        ~Events() { for (int i = 0; i < n; ++i) cudaEventDestroy(e[i]); }
        cudaEvent_t operator[](int i) const { return e[i]; }
    } ev;
    for (; ev.n < 4; ++ev.n) KVP_CUDA(cudaEventCreate(&ev.e[ev.n]));
    KVP_CUDA(cudaEventRecord(ev[0], st));
    if ((rc = prepare(p, a, st, c, xp->rungs))) return rc;

    // exchange thresholds of the pairs of neighbouring rungs: the move table's form at the pair temperatures
    const uint32_t pairs = rungs > 1 ? rungs - 1 : 1;
    std::vector<double> pair_temps(pairs, 1.0);
    uint32_t* const xtable = reinterpret_cast<uint32_t*>(c.host + 256 + table_bytes(rungs));
    uint32_t* const xshifts = xtable + (size_t)pairs * KVP_TABLE_Q;
    uint32_t* const always = xshifts + pairs;
    uint8_t* const last_row = reinterpret_cast<uint8_t*>(c.host + 256 + 2 * table_bytes(rungs));
    memset(always, 0, (size_t)pairs * 4);
    if ((rc = kvp_exchange_temps(c.temps.data(), rungs, pair_temps.data(), always))) return rc;
    if ((rc = kvp_accept_table(pair_temps.data(), pairs, xtable, xshifts))) return rc;

    // workspace of the run: rung history, holders, exchange counts, thresholds, the chains' saved states
    const uint32_t cow4 = c.psmem ? 0u : c.cow_slots4;
    const uint32_t persist4 = (c.wide ? chain_layout(p->S, p->S32, c.grow, c.psmem, c.lin, cow4) : narrow_layout(p->S, p->S32, c.grow, c.psmem, c.lin, cow4)).work / 16;
    const size_t pwords = (size_t)p->U * p->S32;
    const uint32_t state4 = persist4 + (c.psmem ? (uint32_t)((pwords + 3) / 4) : 0u);
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += align256(bytes); return o; };
    const size_t o_hist = take((size_t)rounds * chains), o_hold = take((size_t)chains * 4), o_nex = take((size_t)chains * 4);
    const size_t o_xt = take(table_bytes(pairs)), o_state = take(c.ladder_ctas ? 0 : (size_t)chains * state4 * 16);
    char* xw = nullptr;
    KVP_CUDA(cudaMallocAsync(&xw, off, st));
    struct Free {                                          // in stream order, on every way out
        char* ptr; cudaStream_t st;
        ~Free() { cudaFreeAsync(ptr, st); }
    } guard{xw, st};
    uint8_t* hist = (uint8_t*)(xw + o_hist);
    uint32_t* holder = (uint32_t*)(xw + o_hold);
    uint32_t* nex = (uint32_t*)(xw + o_nex);
    unsigned long long* counts = (unsigned long long*)(c.small + 28);   // zero since prepare()
    const uint32_t* const xtable_dev = (const uint32_t*)(xw + o_xt);
    KVP_CUDA(cudaMemcpyAsync(xw + o_xt, xtable, table_bytes(pairs), cudaMemcpyHostToDevice, st));
    exchange_init_kernel<<<(chains + 255) / 256, 256, 0, st>>>(holder, hist, nex, chains, rungs);
    KVP_CUDA(cudaGetLastError());
    ++c.launches;
    KVP_CUDA(cudaEventRecord(ev[1], st));

    ChainParams prm = c.prm;
    prm.snap = c.snap; prm.undo_log = nullptr;
    prm.cow_out = nullptr; prm.cow_shift = c.cow_shift; prm.cow_slots4 = c.cow_slots4;
    prm.chain_first = a->first_chain; prm.chain_count = chains; prm.result_base = a->first_chain;
    prm.results = c.results; prm.upto = a->moves; prm.dump = nullptr;
    prm.rung_hist = hist; prm.exch_every = xp->exchange_every; prm.hist_stride = chains; prm.hist_base = a->first_chain;
    prm.state = (uint4*)(xw + o_state); prm.state4 = state4;
    unsigned long long* work_dev = reinterpret_cast<unsigned long long*>(c.small + 24);
    ExchangeK xk;
    xk.results = c.results; xk.holder = holder; xk.n_exchanged = nex; xk.x.counts = counts;
    xk.x.table = xtable_dev; xk.x.shifts = xtable_dev + (size_t)pairs * KVP_TABLE_Q; xk.x.always = xk.x.shifts + pairs;
    xk.ladders = chains / rungs; xk.x.rungs = rungs; xk.first_ladder = a->first_chain / rungs;
    xk.x.seed_lo = (uint32_t)a->seed; xk.x.seed_hi = (uint32_t)(a->seed >> 32);
    if (c.ladder_ctas) {
        // every CTA holds whole ladders: one launch, the rounds end in a CTA barrier
        prm.round0 = 0; prm.round1 = rounds; prm.state = nullptr;
        prm.ladder_ctas = 1u; prm.ladder = xk.x; prm.n_exchanged = nex; prm.work = c.wide ? work_dev : nullptr;
        if ((rc = launch_chains(c, prm, chains))) return rc;
        ++c.launches;
        prm.ladder_ctas = 0u; prm.n_exchanged = nullptr;
    }
    for (uint32_t t = 0; t < rounds && !c.ladder_ctas; ++t) {
        prm.round0 = t; prm.round1 = t + 1; prm.resume = t > 0 ? 1u : 0u; prm.upto = a->moves;
        prm.work = t + 1 == rounds ? work_dev : nullptr;   // the counts travel with the saved state; the last round reports
        if ((rc = launch_chains(c, prm, chains))) return rc;
        ++c.launches;
        if (t + 1 < rounds) {
            xk.t = t; xk.rung_next = hist + (size_t)(t + 1) * chains;
            exchange_kernel<<<(xk.ladders + 127) / 128, 128, 0, st>>>(xk);
            KVP_CUDA(cudaGetLastError());
            ++c.launches;
        }
    }
    KVP_CUDA(cudaEventRecord(ev[2], st));

    ReduceOut* red_dev = reinterpret_cast<ReduceOut*>(c.small + 8);
    ReduceOut red;
    reduce_kernel<<<1, 1024, 0, st>>>(c.results, chains, c.prm.err, red_dev);
    KVP_CUDA(cudaGetLastError());
    ++c.launches;
    // the winner's schedule: its snapshot, or a replay of that one chain through the rungs it held
    uint32_t* const sched = best_schedule ? best_schedule : c.sched;
    uint64_t* const host_small = c.host_small();
    if (c.snap) {                                          // the device knows which snapshot: no wait in between
        ChosenInput winner;
        winner.otherwise = c.Pcol0; winner.valid = &red_dev->best_move; winner.index = &red_dev->best_chain;
        if ((rc = launch_bit_transpose(c.snap, p->U, p->S32, p->S, sched, p->W32, st, winner))) return rc;
        ++c.launches;
    } else {
        KVP_CUDA(cudaMemcpyAsync(&red, red_dev, sizeof red, cudaMemcpyDeviceToHost, st));
        KVP_CUDA(cudaStreamSynchronize(st));
        if (red.pad) return KVP_ERR_TIMEOUT;
        const uint64_t upto = red.best_move == ~0ull ? 0 : red.best_move + 1;
        if (upto == 0) {
            KVP_CUDA(cudaMemcpyAsync(sched, c.P0, (size_t)p->S * p->W32 * 4, cudaMemcpyDeviceToDevice, st));
        } else {
            ChainParams rp = prm;
            rp.snap = nullptr; rp.state = nullptr; rp.resume = 0u; rp.work = nullptr;
            rp.chain_first = a->first_chain + red.best_chain; rp.chain_count = 1; rp.result_base = rp.chain_first;
            rp.results = c.results + chains; rp.upto = upto; rp.dump = c.dumpcol;
            rp.round0 = 0; rp.round1 = rounds;
            if ((rc = launch_chains(c, rp, 1))) return rc;
            if ((rc = launch_bit_transpose(c.dumpcol, p->U, p->S32, p->S, sched, p->W32, st))) return rc;
            c.launches += 2;
        }
    }
    if ((rc = launch_score(p, sched, 1, c.counts0, nullptr, nullptr, nullptr, c.small, nullptr, nullptr, (int32_t*)(c.small + 2),
                           c.small + 1, st, &c.launches)))
        return rc;
    KVP_CUDA(cudaMemcpyAsync(host_small, c.small, 256, cudaMemcpyDeviceToHost, st));
    if (stats && stats->per_chain)
        KVP_CUDA(cudaMemcpyAsync(stats->per_chain, c.results, (size_t)chains * sizeof(kvp_chain_result), cudaMemcpyDeviceToHost, st));
    if (final_rung) KVP_CUDA(cudaMemcpyAsync(last_row, hist + (size_t)(rounds - 1) * chains, chains, cudaMemcpyDeviceToHost, st));
    if (n_exchanged) KVP_CUDA(cudaMemcpyAsync(n_exchanged, nex, (size_t)chains * 4, cudaMemcpyDeviceToHost, st));
    KVP_CUDA(cudaEventRecord(ev[3], st));
    KVP_CUDA(cudaStreamSynchronize(st));
    c.copies.any = false;
    if (final_rung)
        for (uint32_t i = 0; i < chains; ++i) final_rung[i] = last_row[i];
    memcpy(&red, host_small + 8, sizeof red);
    if (red.pad) return KVP_ERR_TIMEOUT;
    red.best_chain += a->first_chain;
    const uint64_t *const work = host_small + 24, *const xcounts = host_small + 28;
    const bool ok = host_small[0] == red.best_ticks && (int32_t)(host_small[2] & 0xFFFFFFFFu) < 0;
    if (best_ticks) *best_ticks = red.best_ticks;
    if (best_seconds) *best_seconds = (double)red.best_ticks * p->spt;
    if (stats) {
        kvp_chain_result* keep = stats->per_chain;
        memset(stats, 0, sizeof *stats);
        stats->per_chain = keep;
        stats->init_ticks = c.init_ticks; stats->best_ticks = red.best_ticks; stats->best_chain = red.best_chain;
        stats->levels = a->levels; stats->best_move = red.best_move; stats->moves_total = red.moves_total;
        stats->calib_mean_delta = c.calib_mean; stats->temp0 = c.temps[0];
        stats->winner_hits = host_small[1]; stats->winner_accessed = p->total_accessed;
        cudaEventElapsedTime(&stats->ms_init, ev[0], ev[1]);
        cudaEventElapsedTime(&stats->ms_chains, ev[1], ev[2]);
        cudaEventElapsedTime(&stats->ms_finish, ev[2], ev[3]);
        stats->kernel_launches = c.launches;
        stats->chain_launches = rounds; stats->resident_chains = chains;
        report_form(c, stats);
        stats->work_again = work[0]; stats->work_listed = work[1]; stats->work_items = work[2];
        stats->exchange_rounds = rounds; stats->exchanges_tried = xcounts[0]; stats->exchanges_accepted = xcounts[1];
    }
    return ok ? KVP_OK : KVP_ERR_INTERNAL;
} catch (const std::bad_alloc&) {
    return KVP_ERR_NOMEM;
}
