// The wide chain kernel: simulated-annealing chains that walk over placement schedules (included by kvp_anneal.cu only).
//
// State of a chain (shared memory, but for the schedule when it does not fit): the schedule in time-packed form, and per
// step the two sides of Eq. 2, th (Eq. 3) and te (Eq. 4), the occupancy, one bit "HBM is full" and one bit "te >= th".
// When a DRAM channel is no faster than the link (kappa_d >= kappa_k, LIN) the third term of Eq. 4's maximum is always
// the largest, so th and te are linear in the number of hits and of migrations of a step, and the pair is all a
// proposal's cost needs; otherwise (not LIN) the migrations in both directions are kept beside it, and two more step bitmaps
// that say which of the three terms is the largest (the bound of step 3 then takes that term's change where te leads).
//
// A warp takes a batch of 32 * R consecutive moves:
//   1. draw: a Philox block per proposal.
//   2. classify by the placement bits alone: a swap of two units with equal placement over the run changes nothing, a
//      flip into a full step is infeasible (Eq. 5). The rest is listed.
//   3. bound, 32 listed proposals at a time, word-parallel: the masks of the steps at which a hit is won or lost and at
//      which a migration edge appears or vanishes, and from their popcounts over the steps where te leads and where th
//      leads a lower bound of the cost change (the leading side's own change: the new maximum is at least that). With
//      the proposal's uniform w the Metropolis test fails for every cost change above C ln(2^32 / w), so most listed
//      proposals are rejected here, without looking at a single step.
//   4. exact: the survivors' changes of max(th, te), summed over their changed steps.
//   5. commit in move order: usually nothing in the batch changes the schedule and every lane counts its own proposals.
//      Otherwise the warp applies the state-changing moves it meets, marks the proposals whose evaluation an applied one
//      spoiled (see spoiled: a few in a thousand where it was every proposal of overlapping steps), stops at the first of
//      them and evaluates them again.
// Several warps may serve one chain: they take its batches in turn and evaluate ahead of each other's commits (see
// ChainShared). The outcome is that of the sequential chain in every case.
//
// What bounds it (ncu): issue slots and the integer pipe, 13.0 warp instructions per move, 59% of the issue slots busy with 16
// warps per SM in a short launch (65,536 units x 64 steps, 2368 chains x 6,000 moves). Measured on 2.6M units x 64 steps, 8192
// chains x 1M moves: 201 -> 133 ms, on a growing cache of 131,072 units (1024 x 100k) 6.3 -> 2.7 ms against the kernels before, which put
// the changed steps of every listed proposal through a shared-memory queue of (proposal, step) items, each an evaluation of
// Eq. 2-4 from four counters, and had no second warp per chain (work area 6.9 KB a warp, now 3.1).
#pragma once

namespace kvp {

namespace {

// Rows of 32 proposals in a batch. One warp per chain with schedules in global memory (many chains): 8, so that the
// listed proposals of a batch fill the passes that judge them (141 against 144 ms on the largest configuration); else 4.
constexpr int kRowsOne = 8, kRowsMany = 4;
constexpr uint32_t kNone = 256;                           // no proposal (the ids of a batch are below)

// What an applied move changed, as far as evaluations depend on it (see spoiled): its steps; the steps at which a bit of
// the two step bitmaps turned; its units.
struct Applied {
    uint32_t steps;              // s0 | (s0 + len) << 16
    uint32_t bits;               // first | last << 16; first > last: none (narrow kernel: of the bitmap "te >= th")
    uint32_t units;              // low halves of u | v << 16 (u twice for a flip)
    uint32_t fulls;              // narrow kernel: likewise of the bitmap "HBM is full"
};

// The scalars of a chain, its hand-over block when several warps serve it, and the log of its latest applied moves.
// Warp w of W owns batches w, w + W, ... It evaluates a batch against whatever state it finds (another warp may be
// committing an earlier batch meanwhile), waits until `turn` is the index of its batch, evaluates again the proposals
// that a move applied in the meantime spoiled (`napplied` counts them, `applog` keeps the latest), and commits. A read
// of something a commit was just writing is covered: the applied move is in the log before its turn is passed on.
struct ChainShared {
    uint64_t cur, best, best_move, best_at_boundary, n_chg, hash;
    uint64_t n_same, n_inf;      // proposals that change nothing / infeasible ones, added by every warp when it leaves
    uint64_t n_again, n_listed, n_items;   // work of the evaluations (kvp_anneal_stats), likewise
    uint64_t m_end;              // moves done when the stop rule ended the chain
    uint32_t ulen;               // moves applied since the best state
    uint32_t snap_dirty;         // the best state is the current one and not saved yet
    uint32_t turn, napplied, stopped, left;   // left: warps that are done with the chain
    uint32_t rung, n_exchanged;  // replica exchange
    Applied applog[kLog];
};
static_assert(sizeof(ChainShared) % 16 == 0, "uint4 slots");

// Work area of a warp: a ring of listed proposals with their placement windows, the accepted ones that change the schedule
// in move order, by proposal of the batch what spoiled needs and (when it is evaluated again) what became of it, and the
// list of those to evaluate again. A batch with more accepted ones than fit goes on where they end once these are applied.
// Rows of 32 proposals a warp works on side by side: with schedules in global memory two, so that their loads overlap (144
// against 168 ms on the largest configuration, four: 148); in shared memory one, for there the instruction cache counts (four
// rows: 2000 instructions in a batch's path, and a warp waited for the next one a quarter of the time); with births, whose loads
// come first, one (2.7 against 4.6 ms).
// Or, in global memory, one row whose columns were loaded while the row before it was listed and judged (AHEAD), which takes half
// the ring: the choice, and what either measured, is where the shared memory is shared out. Never for columns that are one
// vector of two words, whose loads stay in flight for less than a single row at a time costs (131,072 units x 64 steps, 2368 chains
// x 20,000: 0.74 -> 0.82 ms; the largest configuration 132 -> 138), nor with births (131,072 x 1056: 2.71 -> 2.76); always for
// vectors of four. The second load takes its address from a select: with a branch around it, since a flip has no second column,
// 32,768 x 256, 2368 x 50,000 took 2.30 ms instead of 2.27.
constexpr uint32_t kAccepted = 6;
constexpr bool load_ahead(bool grow, bool lin, uint32_t S32) { return !grow && !(lin && S32 == 2); }   // whether it may be
__host__ __device__ constexpr int rows_at_a_time(bool psmem, bool grow, bool ahead) { return psmem || grow || ahead ? 1 : 2; }
__host__ __device__ constexpr uint32_t ring_size(bool psmem, bool grow, bool ahead) { return rows_at_a_time(psmem, grow, ahead) > 1 ? 128u : 64u; }
__host__ __device__ constexpr uint32_t work4(bool psmem, bool grow, bool ahead, int rows)   // uint4 slots of it
{
    return ring_size(psmem, grow, ahead) * 3 / 2 + 2 * kAccepted + 2 * (uint32_t)rows * 8 + 2 * (uint32_t)rows * 2 + 2;
}
constexpr uint32_t kSame = 1u, kInf = 2u;                 // proposal states: changes nothing (accepted); infeasible

// Byte offsets of the parts of a chain's shared memory. They are kernel parameters, so that a chain's state costs its
// warps two registers of addresses and not two for every part.
inline ChainLayout chain_layout(uint32_t S, uint32_t S32, bool grow, bool psmem, bool lin, uint32_t cow4)
{
    ChainLayout l;
    uint32_t at = sizeof(ChainShared) + 16 * (lin ? (S + 1) / 2 : S);   // {th, te}, or {th, te without migrations, in, out}
    auto take = [&](uint32_t n4) { const uint32_t p = at; at += 16 * n4; return p; };
    l.occ = take(psmem ? (S + 7) / 8 : (S + 3) / 4);
    l.full = take((S32 + 3) / 4);
    l.lead = take((S32 + 3) / 4);
    l.out = take(lin ? 0u : (S32 + 3) / 4);
    l.in = take(lin ? 0u : (S32 + 3) / 4);
    l.hb = take(grow && !lin ? (S + 3) / 4 : 0u);
    l.have = take(cow4);
    l.work = at;                                          // what outlives a batch ends here
    return l;
}
// bytes of a chain of W warps, without a schedule in shared memory
inline size_t chain_bytes(uint32_t S, uint32_t S32, bool grow, bool psmem, bool lin, uint32_t cow4, uint32_t W, int rows, bool ahead)
{
    return chain_layout(S, S32, grow, psmem, lin, cow4).work + (size_t)W * work4(psmem, grow, ahead, rows) * 16;
}

extern __shared__ char chain_smem[];

template <bool PSMEM, bool GROW, bool LIN, int COLV, int R, bool AHEAD>
struct Chain {
    using Occ = typename std::conditional<PSMEM, uint16_t, uint32_t>::type;   // PSMEM: fewer than 2^16 units
    static constexpr uint32_t kRing = ring_size(PSMEM, GROW, AHEAD), kBatch = 32 * R;
    const ChainParams& prm;
    uint32_t cb, wb, pb;         // byte offsets in shared memory: the chain's state, the warp's work area, PSMEM: the schedule
    uint32_t* slice;             // not PSMEM: the chain's slice of global scratch

    template <typename T> __device__ __forceinline__ T* at(uint32_t off) const { return reinterpret_cast<T*>(chain_smem + off); }
    __device__ __forceinline__ ChainShared* sc() const { return at<ChainShared>(cb); }
    __device__ __forceinline__ int2* tt() const { return at<int2>(cb + (uint32_t)sizeof(ChainShared)); }   // LIN: [S] {th, te}
    // not LIN: [S] {th, te without its migration term, units moved in, units moved out}
    __device__ __forceinline__ int4* tm() const { return at<int4>(cb + (uint32_t)sizeof(ChainShared)); }
    __device__ __forceinline__ Occ* occ() const { return at<Occ>(cb + prm.lay.occ); }              // [S]
    __device__ __forceinline__ uint32_t* full() const { return at<uint32_t>(cb + prm.lay.full); }  // [S32] bit t: occ[t] == cap
    __device__ __forceinline__ uint32_t* lead() const { return at<uint32_t>(cb + prm.lay.lead); }  // [S32] bit t: te[t] >= th[t]
    // not LIN: [S32] bit t: the link's outbound (inbound) traffic is the largest term of Eq. 4's maximum (see term_leads)
    __device__ __forceinline__ uint32_t* out() const { return at<uint32_t>(cb + prm.lay.out); }
    __device__ __forceinline__ uint32_t* in() const { return at<uint32_t>(cb + prm.lay.in); }
    __device__ __forceinline__ uint32_t* hb() const { return at<uint32_t>(cb + prm.lay.hb); }      // not LIN, GROW: [S] written to HBM at birth
    __device__ __forceinline__ uint32_t* have() const { return at<uint32_t>(cb + prm.lay.have); }  // not PSMEM: buckets present in the slice
    __device__ __forceinline__ uint4* ring() const { return at<uint4>(wb); }                       // [kRing] {pk | id << 24, u, v, w}
    __device__ __forceinline__ uint2* ring_win() const { return at<uint2>(wb + 16 * kRing); }      // [kRing] {Wu, Wv}
    // [kAccepted][2] {pk | id << 24, u, v, cost change}, {Wu, Wv, Au, Av}
    __device__ __forceinline__ uint4* acc() const { return at<uint4>(wb + 24 * kRing); }
    // [kBatch] {s0 | (s0 + len) << 16, low halves of u | v << 16 (u twice for a flip)}
    __device__ __forceinline__ uint2* reach() const { return at<uint2>(wb + 24 * kRing + 32 * kAccepted); }
    __device__ __forceinline__ uint32_t* close() const { return at<uint32_t>(wb + 24 * kRing + 32 * kAccepted + 8 * kBatch); }   // [R] bit: this proposal's steps were looked at one by one
    // [kBatch] of proposals evaluated again: kSame, kInf or 0
    __device__ __forceinline__ uint8_t* state() const { return at<uint8_t>(wb + 24 * kRing + 32 * kAccepted + 8 * kBatch + 32); }
    __device__ __forceinline__ uint8_t* again() const { return state() + kBatch; }                 // [kBatch] ids to evaluate again, ascending

    // the schedule: shared; or the chain's slice, a copy-on-write overlay of the initial schedule
    __device__ __forceinline__ uint32_t* P() const { return PSMEM ? at<uint32_t>(pb) : slice; }
    __device__ __forceinline__ const uint32_t* col(uint32_t u) const
    {
        if (PSMEM) return at<uint32_t>(pb + 4 * u * prm.S32);
        const uint32_t b = u >> prm.cow_shift;
        // volatile: another warp of the chain may be taking the bucket over (it sets the bit after the copy); a select,
        // not a branch, so that the loads stay in one straight-line block
        const uint32_t w = ld_volatile_u32(have() + (b >> 5));
        return ((w >> (b & 31u)) & 1u ? (const uint32_t*)slice : prm.Pcol0) + (size_t)u * prm.S32;
    }
    // Before unit u is rewritten: its bucket is copied into the slice if it is not there yet (all lanes, u uniform).
    __device__ __forceinline__ void own(uint32_t u, uint32_t lane) const
    {
        const uint32_t b = u >> prm.cow_shift, S32 = prm.S32;
        if ((have()[b >> 5] >> (b & 31u)) & 1u) return;
        const size_t lo = (size_t)(b << prm.cow_shift) * S32, hi = (size_t)min(prm.U, (b + 1u) << prm.cow_shift) * S32;
        for (size_t i = lo + lane; i < hi; i += 32) slice[i] = prm.Pcol0[i];
        __threadfence_block();
        __syncwarp();
        if (lane == 0) have()[b >> 5] |= 1u << (b & 31u);
        __syncwarp();
    }
    // Before units u and v (u again for a flip) are rewritten. Growing caches change few units: one after the other, in less
    // code (131,072 units x 1056 steps, 1024 chains x 100,000, whole call with trace and construction: 3.17 against 3.28 ms).
    __device__ __forceinline__ void own(uint32_t u, uint32_t v, uint32_t lane) const
    {
        if (PSMEM) return;
        if (GROW) {
            own(u, lane);
            if (v != u) own(v, lane);
        } else {
            own_buckets(slice, prm.Pcol0, have(), prm.cow_shift, prm.U, prm.S32, u, v, lane);
        }
    }
};

// what a proposal does to the steps of its window (bit k = step s0 - 1 + k; bits 1..31 count)
struct Effect {
    uint32_t won, lost;          // hits
    uint32_t euo, evo, eun, evn; // migration edges of u and v before and after
    uint32_t Bu, Bv;             // GROW: the steps in which u and v are written, where the move changes their placement
    uint32_t Nu, Nv;             // windows after the move
    uint32_t changed;            // steps whose cost may change
};

// Masks of a proposal from its windows. Wv = 0 and Av = 0 for a flip.
template <bool GROW, bool LIN>
__device__ __forceinline__ Effect effect_of(const uint32_t* __restrict__ birth, uint32_t S, uint32_t pk, uint32_t u, uint32_t v,
                                            uint32_t Wu, uint32_t Wv, uint32_t Au, uint32_t Av)
{
    const bool swap = pk & 1u;
    const uint32_t len = (pk >> 1) & 31u, s0 = (pk >> 8) & 0x7FFFu;
    const uint32_t run = min(len, S - s0), nl = min(len, S - 1 - s0) + 1;   // steps rewritten; affected: and the step after
    const uint32_t M = ((1u << run) - 1u) << 1, Sb = ((1u << nl) - 1u) << 1;
    Effect e;
    uint32_t live = 0xFFFFFFFFu, Bu = 0u, Bv = 0u;
    if (GROW) {
        uint32_t Lu, Lv;
        alive_born(__ldg(birth + u), s0, Lu, Bu);
        alive_born(__ldg(birth + (swap ? v : u)), s0, Lv, Bv);
        live = Lu & Lv;
        if (!swap) Bv = 0u;
    }
    const uint32_t D = (swap ? Wu ^ Wv : 0xFFFFFFFFu) & M & live;          // bits that toggle
    e.Nu = Wu ^ D;
    e.Nv = swap ? Wv ^ D : 0u;
    if (s0 == 0) {                                                // the virtual step -1 follows step 0
        e.Nu = (e.Nu & ~1u) | ((e.Nu >> 1) & 1u);
        e.Nv = (e.Nv & ~1u) | ((e.Nv >> 1) & 1u);
    }
    const uint32_t hit = (Au ^ Av) & D;
    e.won = hit & ~(Au ^ e.Nu);                                   // u in and read, or (swap) v in and read
    e.lost = hit & (Au ^ e.Nu);
    // a unit moves at step t iff p[t] != p[t-1]; the edge into the step in which it is written is no migration
    const uint32_t ku = GROW ? Sb & ~Bu : Sb, kv = GROW ? Sb & ~Bv : Sb;
    e.euo = (Wu ^ (Wu << 1)) & ku; e.eun = (e.Nu ^ (e.Nu << 1)) & ku;
    e.evo = (Wv ^ (Wv << 1)) & kv; e.evn = (e.Nv ^ (e.Nv << 1)) & kv;
    e.Bu = GROW ? Bu & D : 0u;
    e.Bv = GROW ? Bv & D : 0u;
    // LIN: only the number of edges counts; else also an edge that turns around
    uint32_t mg = ((e.euo ^ e.evo) ^ (e.eun ^ e.evn)) | ((e.euo & e.evo) ^ (e.eun & e.evn));
    if (!LIN) mg = (e.euo ^ e.eun) | (e.euo & e.eun & (Wu ^ e.Nu)) | (e.evo ^ e.evn) | (e.evo & e.evn & (Wv ^ e.Nv));
    e.changed = hit | mg | e.Bu | e.Bv;
    return e;
}

// changes at window bit k: hits, edges, writes to HBM at birth
struct BitChange { int hr, mm, hb; };
template <bool GROW>
__device__ __forceinline__ BitChange bit_change(const Effect& e, uint32_t k)
{
    BitChange c;
    c.hr = (int)((e.won >> k) & 1u) - (int)((e.lost >> k) & 1u);
    c.mm = (int)((e.eun >> k) & 1u) + (int)((e.evn >> k) & 1u) - (int)((e.euo >> k) & 1u) - (int)((e.evo >> k) & 1u);
    c.hb = 0;
    if (GROW) {
        const int bu = (e.Bu >> k) & 1u, bv = (e.Bv >> k) & 1u, nu = (e.Nu >> k) & 1u, nv = (e.Nv >> k) & 1u;
        c.hb = bu * (2 * nu - 1) + bv * (2 * nv - 1);             // written to HBM instead of to DRAM, or the reverse
    }
    return c;
}
// not LIN: edges into HBM and out of it separately
__device__ __forceinline__ void edge_change(const Effect& e, uint32_t Wu, uint32_t Wv, uint32_t k, int& mi, int& mo)
{
    mi = (int)(((e.eun & e.Nu) >> k) & 1u) + (int)(((e.evn & e.Nv) >> k) & 1u) - (int)(((e.euo & Wu) >> k) & 1u) -
         (int)(((e.evo & Wv) >> k) & 1u);
    mo = (int)(((e.eun & ~e.Nu) >> k) & 1u) + (int)(((e.evn & ~e.Nv) >> k) & 1u) - (int)(((e.euo & ~Wu) >> k) & 1u) -
         (int)(((e.evo & ~Wv) >> k) & 1u);
}
// Eq. 4's migration and write term
__device__ __forceinline__ int ext_term(int mi, int mo, int hb, const StepC c, const CostK K)
{
    const int e1 = (int)c.y - (int)K.kk * hb + (int)K.kkF * mo, e2 = (int)K.kkF * mi;
    const int e3 = (int)c.z - (int)K.kd * hb + (int)K.kdF * (mi + mo);
    return max(max(e1, e2), e3);
}
// The terms of a step by the step bitmaps, f = {th, te without its migration term, in, out}: bit 0: te leads; bit 1: the
// link's outbound term is the largest of Eq. 4's three; bit 2: the inbound one is.
__device__ __forceinline__ uint32_t term_leads(const int4 f, int hb, const StepC c, const CostK K)
{
    const int e1 = (int)c.y - (int)K.kk * hb + (int)K.kkF * f.w, e2 = (int)K.kkF * f.z;
    const int e3 = (int)c.z - (int)K.kd * hb + (int)K.kdF * (f.z + f.w);
    const bool out = e1 >= e2 && e1 >= e3, in = !out && e2 >= e3;
    return (f.y + max(max(e1, e2), e3) >= f.x ? 1u : 0u) | (out ? 2u : 0u) | (in ? 4u : 0u);
}

// What a warp needs to evaluate, constant over a temperature level or longer.
struct EvalCtx {
    const uint32_t* Acol;        // [U][S32] access bitmap, time-packed (shared or global)
    uint32_t level, shift;       // row of the threshold table, its bin size
    float bound;                 // cost changes above bound * (32 - log2 w) + 2^shift fail the level's Metropolis test
    uint32_t n_again, n_listed, n_items;
};

// Cost change of the step at window bit k, step t.
template <bool PSMEM, bool GROW, bool LIN, int COLV, int R, bool AHEAD>
__device__ __forceinline__ int step_change(const Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>& c, const Effect& e, uint32_t Wu, uint32_t Wv, uint32_t k,
                                           uint32_t t)
{
    const ChainParams& prm = c.prm;
    const int kh = (int)prm.K.kh, ke = (int)prm.K.ke, khF = (int)prm.K.khF, kdF = (int)prm.K.kdF, kd = (int)prm.K.kd;
    const BitChange d = bit_change<GROW>(e, k);
    if (LIN) {
        const int2 f = c.tt()[t];
        return max(f.x + kh * (d.hr + d.hb) + khF * d.mm, f.y - ke * d.hr - kd * d.hb + kdF * d.mm) - max(f.x, f.y);
    }
    const int4 f = c.tm()[t];
    const StepC sc = __ldg(prm.stepc + t);
    const int hb = GROW ? (int)c.hb()[t] : 0;
    int mi, mo;
    edge_change(e, Wu, Wv, k, mi, mo);
    return max(f.x + kh * (d.hr + d.hb) + khF * (mi + mo), f.y - ke * d.hr + ext_term(f.z + mi, f.w + mo, hb + d.hb, sc, prm.K)) -
           max(f.x, f.y + ext_term(f.z, f.w, hb, sc, prm.K));
}

// Steps 3 and 4 for up to 32 listed proposals, from ring position `head` on, one per lane. The accepted ones go to
// c.acc() from `kept` on; where there is no room for all of them, `late` becomes the id of the first that found none.
template <bool PSMEM, bool GROW, bool LIN, int COLV, int R, bool AHEAD>
__device__ __forceinline__ void judge(const Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>& c, EvalCtx& x, uint32_t head, uint32_t count, uint32_t lane,
                                      uint32_t& kept, uint32_t& late)
{
    const ChainParams& prm = c.prm;
    const uint32_t S = prm.S;
    const int kh = (int)prm.K.kh, ke = (int)prm.K.ke, khF = (int)prm.K.khF, kdF = (int)prm.K.kdF, kd = (int)prm.K.kd;
    const bool live = lane < count;
    const uint32_t at = (head + (live ? lane : 0u)) & (c.kRing - 1);
    const uint4 a = c.ring()[at];
    const uint2 b = c.ring_win()[at];
    const uint32_t pk = a.x, s0 = (pk >> 8) & 0x7FFFu;
    const bool swap = pk & 1u;
    const WinPos wp = window_pos(s0);
    const uint32_t Au = window_at<COLV>(x.Acol + (size_t)a.y * prm.S32, wp);
    const uint32_t av = window_at<COLV>(x.Acol + (size_t)(swap ? a.z : a.y) * prm.S32, wp);   // a flip reads unit u twice
    const uint32_t Av = swap ? av : 0u;
    const Effect e = effect_of<GROW, LIN>(prm.birth, S, pk, a.y, a.z, b.x, b.y, Au, Av);
    const uint32_t T = window_at<0>((const uint32_t*)c.lead(), wp);          // steps where te leads
    const int hits_t = __popc(e.won & T) - __popc(e.lost & T), hits = __popc(e.won) - __popc(e.lost);
    int lb;
    if (LIN) {
        const int mm_t = __popc(e.eun & T) + __popc(e.evn & T) - __popc(e.euo & T) - __popc(e.evo & T);
        const int mm = __popc(e.eun) + __popc(e.evn) - __popc(e.euo) - __popc(e.evo);
        lb = kdF * mm_t - ke * hits_t + khF * (mm - mm_t) + kh * (hits - hits_t);
        if (GROW) {
            if (e.Bu) lb += ((e.Nu & e.Bu) != 0 ? 1 : -1) * ((T & e.Bu) != 0 ? -kd : kh);
            if (e.Bv) lb += ((e.Nv & e.Bv) != 0 ? 1 : -1) * ((T & e.Bv) != 0 ? -kd : kh);
        }
    } else {
        // migrations count in the direction of the term that leads (both where th or the DRAM channels do)
        const uint32_t O = T & window_at<0>((const uint32_t*)c.out(), wp), I = T & window_at<0>((const uint32_t*)c.in(), wp);
        const uint32_t iu = e.eun & e.Nu, iv = e.evn & e.Nv, ju = e.euo & b.x, jv = e.evo & b.y;    // into HBM: after, before
        const uint32_t ou = e.eun ^ iu, ov = e.evn ^ iv, pu = e.euo ^ ju, pv = e.evo ^ jv;          // out of it
        auto in = [&](uint32_t m) { return __popc(iu & m) + __popc(iv & m) - __popc(ju & m) - __popc(jv & m); };
        auto out = [&](uint32_t m) { return __popc(ou & m) + __popc(ov & m) - __popc(pu & m) - __popc(pv & m); };
        const uint32_t C = T & ~(O | I);
        const int kk = (int)prm.K.kk, kkF = (int)prm.K.kkF;
        lb = kh * (hits - hits_t) - ke * hits_t + khF * (in(~T) + out(~T)) + kkF * (out(O) + in(I)) + kdF * (in(C) + out(C));
        if (GROW) {
            auto write = [&](uint32_t B) { return (T & B) == 0 ? kh : (O & B) != 0 ? -kk : (I & B) != 0 ? 0 : -kd; };
            if (e.Bu) lb += ((e.Nu & e.Bu) != 0 ? 1 : -1) * write(e.Bu);
            if (e.Bv) lb += ((e.Nv & e.Bv) != 0 ? 1 : -1) * write(e.Bv);
        }
    }
    const bool keep = live && (float)lb <= x.bound * (32.001f - __log2f((float)max(a.w, 1u))) + __uint_as_float((127u + x.shift) << 23);
    const uint32_t kb = __ballot_sync(0xFFFFFFFFu, keep);
    if (!kb) return;
    if (keep) atomicOr(c.close() + (pk >> 29), 1u << ((pk >> 24) & 31u));
    x.n_items += keep ? __popc(e.changed) : 0u;
    // Few survivors: one after the other, a lane per step. Many: every lane walks over its own steps.
    int delta = 0;
    if (__popc(kb) <= 8) {
#pragma unroll 1
        for (uint32_t rest = kb; rest; rest &= rest - 1u) {
            const int src = __ffs(rest) - 1;
            Effect f;
            f.won = __shfl_sync(0xFFFFFFFFu, e.won, src); f.lost = __shfl_sync(0xFFFFFFFFu, e.lost, src);
            f.euo = __shfl_sync(0xFFFFFFFFu, e.euo, src); f.evo = __shfl_sync(0xFFFFFFFFu, e.evo, src);
            f.eun = __shfl_sync(0xFFFFFFFFu, e.eun, src); f.evn = __shfl_sync(0xFFFFFFFFu, e.evn, src);
            f.changed = __shfl_sync(0xFFFFFFFFu, e.changed, src);
            f.Bu = f.Bv = f.Nu = f.Nv = 0u;
            uint32_t Wu = 0u, Wv = 0u;
            if (GROW || !LIN) {
                f.Nu = __shfl_sync(0xFFFFFFFFu, e.Nu, src); f.Nv = __shfl_sync(0xFFFFFFFFu, e.Nv, src);
                f.Bu = __shfl_sync(0xFFFFFFFFu, e.Bu, src); f.Bv = __shfl_sync(0xFFFFFFFFu, e.Bv, src);
            }
            if (!LIN) { Wu = __shfl_sync(0xFFFFFFFFu, b.x, src); Wv = __shfl_sync(0xFFFFFFFFu, b.y, src); }
            const uint32_t first = __shfl_sync(0xFFFFFFFFu, s0, src);
            int d = 0;
            if ((f.changed >> lane) & 1u) d = step_change(c, f, Wu, Wv, lane, first + lane - 1u);
            d = __reduce_add_sync(0xFFFFFFFFu, d);
            if (lane == (uint32_t)src) delta = d;
        }
    } else {
#pragma unroll 1
        for (uint32_t todo = keep ? e.changed : 0u; todo;) {
            const uint32_t j = 31u - __clz(todo);
            todo ^= 1u << j;
            delta += step_change(c, e, b.x, b.y, j, s0 + j - 1u);
        }
    }
    __syncwarp();
    const bool ok = keep && metropolis(delta, a.w, prm.table + (size_t)x.level * KVP_TABLE_Q, x.shift);
    const uint32_t ob = __ballot_sync(0xFFFFFFFFu, ok);
    if (!ob) return;
    const uint32_t to = kept + __popc(ob & ((1u << lane) - 1u));
    if (ok && to < prm.carry) {
        c.acc()[2 * to] = make_uint4(pk, a.y, a.z, (uint32_t)delta);
        c.acc()[2 * to + 1] = make_uint4(b.x, b.y, Au, Av);
    }
    kept += __popc(ob);
    if (kept > prm.carry) {                                       // warp-uniform
        const uint32_t out = __ballot_sync(0xFFFFFFFFu, ok && to == prm.carry);
        late = __shfl_sync(0xFFFFFFFFu, pk >> 24, __ffs(out) - 1);
        kept = prm.carry;
    }
    __syncwarp();
}

// Evaluation of `count` proposals of the batch that starts at move m, against the current state: all of them from the
// first on (fresh), or those listed in c.again(). Draws them, settles what the placement bits settle (into the row masks
// same and inf of a fresh batch, into c.state() otherwise) and judges the rest. The accepted ones that change the schedule
// are left in c.acc() in move order (`kept` of them). Returns the id from which on nothing was evaluated (kNone:
// everything was). One copy of this code for every use keeps the path through a batch short.
template <bool PSMEM, bool GROW, bool LIN, int COLV, int R, bool AHEAD>
__device__ __forceinline__ uint32_t evaluate(const Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>& c, EvalCtx& x, uint64_t m, uint32_t chain, bool fresh,
                                             uint32_t count, uint32_t lane, uint32_t& kept, uint32_t& same, uint32_t& inf)
{
    const ChainParams& prm = c.prm;
    const uint32_t S = prm.S;
    constexpr int UNR = rows_at_a_time(PSMEM, GROW, AHEAD);
    uint32_t head = 0, listed = 0, late = kNone;
    kept = 0;
    auto id_of = [&](uint32_t i) { return fresh ? i : (uint32_t)c.again()[i < count ? i : 0u]; };
    auto draw = [&](uint32_t id, uint32_t& pk, uint32_t& u, uint32_t& v, uint32_t& w) {
        uint32_t r[4];
        const uint64_t mine = m + id;
        philox4x32_10((uint32_t)mine, (uint32_t)(mine >> 32), chain, TAG_MOVE, prm.keys, r);
        LaneMove mv;
        decode_move(r, prm.p_swap_256, prm.len_choices, S, prm.U, mv);
        pk = mv.pk; u = mv.u; v = mv.v; w = mv.w;
    };
    // AHEAD: the row drawn last, its columns under way while the row before it is listed and judged
    uint32_t npk, nu, nv, nw;
    typename Words<COLV>::type qu, qv;
    auto fetch = [&](uint32_t q) {
        draw(id_of(q + lane), npk, nu, nv, nw);
        const WinPos wp = window_pos(npk >> 8);
        qu = words_at<COLV>(c.col(nu), wp);
        // the second window: the other unit's placement for a swap, the full-step bitmap for a flip (one address, no branch)
        qv = words_at<COLV>(npk & 1u ? c.col(nv) : (const uint32_t*)c.full(), wp);
    };
    if constexpr (AHEAD) fetch(0);
#pragma unroll 1
    for (uint32_t q = 0; q < count; q += 32 * UNR) {
        uint32_t id[UNR], pk[UNR], u[UNR], v[UNR], w[UNR], Wu[UNR], W2[UNR], live[UNR];
        if constexpr (AHEAD) {
            static_assert(UNR == 1, "one row at a time");
            id[0] = id_of(q + lane); pk[0] = npk; u[0] = nu; v[0] = nv; w[0] = nw; live[0] = 0xFFFFFFFFu;
            const WinPos wp = window_pos(npk >> 8);
            Wu[0] = cut<COLV>(qu, wp);
            W2[0] = cut<COLV>(qv, wp);
            if (q + 32 < count) fetch(q + 32);
        } else {
#pragma unroll
            for (int j = 0; j < UNR; ++j) {
                id[j] = id_of(q + 32u * j + lane);
                draw(id[j], pk[j], u[j], v[j], w[j]);
            }
#pragma unroll
            for (int j = 0; j < UNR; ++j) {
                const WinPos wp = window_pos(pk[j] >> 8);
                const bool swap = pk[j] & 1u;
                Wu[j] = window_at<COLV>(c.col(u[j]), wp);
                W2[j] = window_at<COLV>(swap ? c.col(v[j]) : (const uint32_t*)c.full(), wp);
                live[j] = 0xFFFFFFFFu;
                if (GROW) {
                    uint32_t La, Lb, Bu, Bv;
                    alive_born(__ldg(prm.birth + u[j]), pk[j] >> 8, La, Bu);
                    alive_born(__ldg(prm.birth + (swap ? v[j] : u[j])), pk[j] >> 8, Lb, Bv);
                    live[j] = La & Lb;
                }
            }
        }
        if (lane == 0) x.n_listed -= listed;                      // (what was left over is counted again below)
#pragma unroll
        for (int j = 0; j < UNR; ++j) {
            if (UNR > 1 && q + 32u * j >= count) break;           // warp-uniform
            const bool named = q + 32u * j + lane < count;
            const uint32_t s0 = pk[j] >> 8, len = (pk[j] >> 1) & 31u;
            const bool swap = pk[j] & 1u;
            const uint32_t M = ((1u << min(len, S - s0)) - 1u) << 1;
            const uint32_t D = (swap ? Wu[j] ^ W2[j] : 0xFFFFFFFFu) & M & live[j];   // a flip toggles every bit of the run
            const bool none = D == 0;                             // nothing changes: always accepted
            const bool bad = !swap && (~Wu[j] & D & W2[j]) != 0;  // a flip may not raise a full step (Eq. 5)
            const bool more = named && !none && !bad;
            if (named) {
                c.reach()[id[j]] = make_uint2(s0 | (s0 + len) << 16, (u[j] & 0xFFFFu) | (swap ? v[j] : u[j]) << 16);
                if (fresh) {                                      // row (q >> 5) + j of this lane
                    const uint32_t bit = 1u << ((q >> 5) + j);
                    if (none) same |= bit;
                    if (bad) inf |= bit;
                } else {
                    atomicAnd(c.close() + (id[j] >> 5), ~(1u << (id[j] & 31u)));
                    c.state()[id[j]] = (uint8_t)(none ? kSame : bad ? kInf : 0u);
                }
            }
            const uint32_t mb = __ballot_sync(0xFFFFFFFFu, more);
            if (more) {
                const uint32_t at = (head + listed + __popc(mb & ((1u << lane) - 1u))) & (c.kRing - 1);
                c.ring()[at] = make_uint4(pk[j] | id[j] << 24, u[j], v[j], w[j]);
                c.ring_win()[at] = make_uint2(Wu[j], swap ? W2[j] : 0u);
            }
            listed += __popc(mb);
        }
        __syncwarp();
        if (lane == 0) x.n_listed += listed;
        const bool last = q + 32 * UNR >= count;
#pragma unroll 1
        while (listed >= 32 || (last && listed)) {                // warp-uniform
            const uint32_t n = min(listed, 32u);
            judge(c, x, head, n, lane, kept, late);
            head += n; listed -= n;
            if (late < kNone) return late;
        }
    }
    return late;
}

// Apply an accepted proposal: all lanes take part, lane j updates the step of window bit j, lanes 0 and 1 rewrite the
// words of the schedule and of the two step bitmaps. Returns the steps at which these turned (Applied::bits).
template <bool PSMEM, bool GROW, bool LIN, int COLV, int R, bool AHEAD>
__device__ __forceinline__ uint32_t apply(const Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>& c, uint32_t lane, const uint4 a, const uint4 win)
{
    const ChainParams& prm = c.prm;
    const uint32_t pk = a.x, u = a.y, v = a.z, s0 = (pk >> 8) & 0x7FFFu, S = prm.S, S32 = prm.S32;
    const bool swap = pk & 1u;
    const uint32_t len = (pk >> 1) & 31u, run = min(len, S - s0), nl = min(len, S - 1 - s0) + 1;
    const Effect e = effect_of<GROW, LIN>(prm.birth, S, pk, u, v, win.x, win.y, win.z, win.w);
    const bool valid = lane >= 1 && lane <= nl;
    const uint32_t j = valid ? lane : 1u, t = s0 + j - 1;
    const BitChange d = bit_change<GROW>(e, j);
    const CostK& K = prm.K;
    bool lead = false, led = false;                               // LIN: te leads, led before
    uint32_t by = 0u, was = 0u;                                   // not LIN: which terms lead, led before
    if (LIN) {
        int2 f = c.tt()[t];
        led = f.y >= f.x;
        f.x += (int)K.kh * (d.hr + d.hb) + (int)K.khF * d.mm;
        f.y += (int)K.kdF * d.mm - (int)K.ke * d.hr - (int)K.kd * d.hb;
        if (valid) c.tt()[t] = f;
        lead = f.y >= f.x;
    } else {
        int4 f = c.tm()[t];
        const StepC sc = __ldg(prm.stepc + t);
        const int hb = GROW ? (int)c.hb()[t] : 0;
        int mi, mo;
        edge_change(e, win.x, win.y, j, mi, mo);
        was = term_leads(f, hb, sc, K);
        f.x += (int)K.kh * (d.hr + d.hb) + (int)K.khF * (mi + mo);
        f.y -= (int)K.ke * d.hr;
        f.z += mi; f.w += mo;
        by = term_leads(f, hb + d.hb, sc, K);
        lead = by & 1u; led = was & 1u;
        if (valid) {
            c.tm()[t] = f;
            if (GROW) c.hb()[t] = (uint32_t)(hb + d.hb);
        }
    }
    uint32_t occ = c.occ()[t];
    const bool was_full = occ == prm.cap;
    occ += ((e.Nu >> j) & 1u) + ((e.Nv >> j) & 1u) - ((win.x >> j) & 1u) - ((win.y >> j) & 1u);
    if (valid) c.occ()[t] = (typename Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>::Occ)occ;
    uint32_t F = __ballot_sync(0xFFFFFFFFu, valid && occ == prm.cap), T = __ballot_sync(0xFFFFFFFFu, valid && lead);
    uint32_t O = 0u, I = 0u;
    if (!LIN) {
        O = __ballot_sync(0xFFFFFFFFu, valid && (by & 2u));
        I = __ballot_sync(0xFFFFFFFFu, valid && (by & 4u));
    }
    const uint32_t turned = __ballot_sync(0xFFFFFFFFu, valid && (lead != led || by != was || (occ == prm.cap) != was_full));
    c.own(u, swap ? v : u, lane);
    if (lane < 2) {
        uint32_t M = ((1u << run) - 1u) << 1, V = ((1u << nl) - 1u) << 1, NU = e.Nu, NV = e.Nv, D = win.x ^ NU, sbit = s0 - 1;
        if (s0 == 0) { F >>= 1; T >>= 1; O >>= 1; I >>= 1; V >>= 1; M >>= 1; NU >>= 1; NV >>= 1; D >>= 1; sbit = 0; }
        const uint32_t wj = (sbit >> 5) + lane, sh = sbit & 31u;
        if (wj < S32 && (lane == 0 || sh != 0)) {
            // lane 0 holds the part of the window that falls into the first word, lane 1 the spill-over
            auto part = [&](uint32_t w) { return lane ? w >> (32 - sh) : w << sh; };
            const uint32_t Vx = part(V), Mx = part(M);
            if (Vx) {
                c.full()[wj] = (c.full()[wj] & ~Vx) | (part(F) & Vx);
                c.lead()[wj] = (c.lead()[wj] & ~Vx) | (part(T) & Vx);
                if (!LIN) {
                    c.out()[wj] = (c.out()[wj] & ~Vx) | (part(O) & Vx);
                    c.in()[wj] = (c.in()[wj] & ~Vx) | (part(I) & Vx);
                }
            }
            if (Mx) {                                             // (many moves in global memory: atomics, which are not waited for)
                uint32_t* const pu = c.P() + (size_t)u * S32 + wj;
                uint32_t* const pv = c.P() + (size_t)v * S32 + wj;
                if (PSMEM || GROW) {
                    *pu = (*pu & ~Mx) | (part(NU) & Mx);
                    if (swap) *pv = (*pv & ~Mx) | (part(NV) & Mx);
                } else if (const uint32_t x = part(D) & Mx) {     // a swap toggles the same bits of both
                    atomicXor(pu, x);
                    if (swap) atomicXor(pv, x);
                }
            }
        }
    }
    __syncwarp();
    return turned ? (s0 + __ffs(turned) - 2u) | (s0 + 30u - __clz(turned)) << 16 : 0xFFFFu;
}

// rows of this lane (row h: proposal 32 h + lane) whose proposal comes before proposal `id`
__device__ __forceinline__ uint32_t rows_before(uint32_t id, uint32_t lane) { return id > lane ? (id - lane + 31u) >> 5 : 0u; }

// the first proposal named by the lanes' row masks, kNone if there is none
__device__ __forceinline__ uint32_t first_of(uint32_t rows, uint32_t lane)
{
    if (!__any_sync(0xFFFFFFFFu, rows != 0u)) return kNone;
    return __reduce_min_sync(0xFFFFFFFFu, rows ? 32u * (__ffs(rows) - 1u) + lane : kNone);
}

// This lane's proposals whose evaluation an applied move spoils. The move rewrote steps s0 .. s0 + len, a proposal reads
// steps s0 - 1 .. s0 + len. Where the two meet, what a proposal came to depends on its units' placement, on the two step
// bitmaps and, if its steps were looked at one by one, on their th and te; on the bitmaps not if it changes nothing.
template <bool PSMEM, bool GROW, bool LIN, int COLV, int R, bool AHEAD>
__device__ __forceinline__ uint32_t spoiled(const Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>& c, const Applied g, uint32_t same, uint32_t lane)
{
    const uint32_t s0b = g.steps & 0xFFFFu, endb = g.steps >> 16, first = g.bits & 0xFFFFu, last = g.bits >> 16;
    const uint32_t bu = g.units & 0xFFFFu, bv = g.units >> 16;
    uint32_t rows = 0;
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const uint2 x = c.reach()[h * 32 + lane];
        const uint32_t r = x.x, lo = x.y & 0xFFFFu, hi = x.y >> 16;
        const bool meets = (r & 0xFFFFu) <= endb + 1u && s0b <= (r >> 16);
        const bool shares = lo == bu || lo == bv || hi == bu || hi == bv;
        const bool turned = first <= (r >> 16) && (r & 0xFFFFu) <= last && !((same >> h) & 1u);
        const bool close = (c.close()[h] >> lane) & 1u;
        if (meets && (shares || close || turned)) rows |= 1u << h;
    }
    return rows;
}

// Whether the rungs j (hotter, at cost Eh) and j + 1 of the ladder that starts at rung index first_rung exchange in
// round t (see kvp_anneal_exchange).
__device__ __forceinline__ bool exchange_accepts(const ExchangeArgs& k, uint64_t t, uint32_t first_rung, uint32_t j, uint64_t Eh,
                                                 uint64_t Ec)
{
    if (Eh <= Ec || k.always[j]) return true;                     // the colder rung holds the worse schedule (or an equal one)
    uint32_t x[4];
    philox4x32_10((uint32_t)t, (uint32_t)(t >> 32), first_rung + j, TAG_EXCHANGE, k.seed_lo, k.seed_hi, x);
    const uint64_t q = (Eh - Ec) >> k.shifts[j];
    return q < KVP_TABLE_Q && x[3] < k.table[(size_t)j * KVP_TABLE_Q + q];
}

// One exchange round of the ladders a CTA holds, after round `t`: a thread per pair of neighbouring rungs. holder: ladder
// by ladder the chain (index within the CTA) on each rung. stride: bytes from chain to chain.
template <typename C>
__device__ __forceinline__ void exchange_round(const C& c, uint8_t* holder, uint32_t stride, uint32_t cpb, uint32_t t)
{
    const ChainParams& prm = c.prm;
    const ExchangeArgs& k = prm.ladder;
    const uint32_t par = t & 1u, npairs = (k.rungs - par) / 2;
    const uint32_t ladders = min(cpb, prm.chain_count - blockIdx.x * cpb) / k.rungs;
    if (threadIdx.x >= ladders * npairs) return;
    const uint32_t l = threadIdx.x / npairs, j = 2 * (threadIdx.x % npairs) + par;
    uint8_t* const hold = holder + l * k.rungs;
    ChainShared* const hot = c.template at<ChainShared>(hold[j] * stride);
    ChainShared* const cold = c.template at<ChainShared>(hold[j + 1] * stride);
    const bool yes = exchange_accepts(k, t, prm.chain_first + blockIdx.x * cpb + l * k.rungs, j, hot->cur, cold->cur);
    if (yes) {
        const uint8_t h = hold[j]; hold[j] = hold[j + 1]; hold[j + 1] = h;
        hot->rung = j + 1; cold->rung = j;
        ++hot->n_exchanged; ++cold->n_exchanged;
    }
    atomicAdd(k.counts, 1ull);
    if (yes) atomicAdd(k.counts + 1, 1ull);
}

// A warp of a chain waits until it is batch b's turn. 0: go on; 1: the chain has ended; 2: the wait ran out.
__device__ __forceinline__ uint32_t wait_turn(ChainShared* sc, uint32_t b)
{
    uint32_t polls = 0, now;
    for (;;) {
        now = __shfl_sync(0xFFFFFFFFu, ld_volatile_u32(&sc->turn), 0);
        if (now == b || ++polls > kTurnPolls) break;
        __nanosleep(40);
    }
    __threadfence_block();
    if (now != b) return 2u;
    return __shfl_sync(0xFFFFFFFFu, ld_volatile_u32(&sc->stopped), 0) ? 1u : 0u;
}

// The chain's scalars after move m was applied (one lane).
__device__ __forceinline__ void record(const ChainParams& prm, ChainShared* sc, uint64_t m, uint64_t after, bool leaving,
                                       const Applied& g, uint32_t slot)
{
    if (leaving) sc->snap_dirty = 0u;
    sc->cur = after;
    ++sc->n_chg;
    sc->hash = (sc->hash ^ m) * 0x9E3779B97F4A7C15ull + after;
    if (after < sc->best) { sc->best = after; sc->best_move = m; sc->snap_dirty = 1u; sc->ulen = 0u; }
    else if (prm.undo_log) {                                      // every move is its own inverse: remember it
        const uint32_t ulen = sc->ulen;
        if (ulen < prm.undo_cap) prm.undo_log[(size_t)slot * prm.undo_cap + ulen] = m;
        if (ulen <= prm.undo_cap) sc->ulen = ulen + 1u;
    }
    if (prm.warps > 1) {                                          // tell the warps that are evaluating later batches
        const uint32_t napp = sc->napplied;
        sc->applog[napp % kLog] = g;
        __threadfence_block();
        st_volatile_u32(&sc->napplied, napp + 1u);
    }
}

// PSMEM: the schedules live in shared memory; otherwise a chain's slice of global scratch is a copy-on-write overlay of
// the initial schedule (see kCowBitsMin).
// ASMEM (only with PSMEM): the access bitmap, which every chain of the CTA reads, is staged in shared memory.
// COLV (only without PSMEM): 2 or 4 when every column has exactly that many words, else 0 (see window_at).
// A CTA has blockDim / 32 / W chains of W warps each (W = prm.warps, a power of two).
template <bool PSMEM, bool GROW, bool ASMEM, bool LIN, int COLV, int R, bool AHEAD>
__global__ void __launch_bounds__(512, 1)
wide_chain_kernel(const __grid_constant__ ChainParams prm)
{
    static_assert(PSMEM || !ASMEM, "shared access bitmap only beside shared schedules");
    static_assert(!PSMEM || COLV == 0, "vector columns only for schedules in global scratch");
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = prm.warps;
    const uint32_t cpb = (blockDim.x >> 5) / W, cic = warp / W, sub = warp % W;   // chains per CTA; chain; warp of the chain
    const uint32_t slot = blockIdx.x * cpb + cic;
    const bool active = slot < prm.chain_count;
    const uint32_t chain = prm.chain_first + slot;
    const uint32_t S = prm.S, S32 = prm.S32, U = prm.U;
    const size_t pwords = (size_t)U * S32;
    const uint32_t cow_words = PSMEM ? 0u : prm.cow_slots4 * 4;
    const uint32_t stride = prm.lay.work + W * work4(PSMEM, GROW, AHEAD, R) * 16;       // bytes of a chain
    Chain<PSMEM, GROW, LIN, COLV, R, AHEAD> c{prm, cic * stride, cic * stride + prm.lay.work + sub * work4(PSMEM, GROW, AHEAD, R) * 16,
                                       cpb * stride + cic * U * S32 * 4, PSMEM ? nullptr : prm.ws + (size_t)slot * pwords};
    ChainShared* const sc = c.sc();
    EvalCtx x;
    x.Acol = prm.Acol;
    x.n_again = x.n_listed = x.n_items = 0u;
    if (ASMEM) {
        uint32_t* const a_s = c.template at<uint32_t>((cpb * stride + cpb * U * S32 * 4 + 15u) & ~15u);
        copy_words(a_s, prm.Acol, pwords, threadIdx.x, blockDim.x);
        x.Acol = a_s;
    }
    const uint32_t tid = sub * 32 + lane, nthr = W * 32;          // thread of the chain
    uint4* const saved = prm.state ? prm.state + (size_t)(chain - prm.hist_base) * prm.state4 : nullptr;
    const uint32_t persist4 = prm.lay.work / 16;                  // of what outlives a batch
    if (active && !(saved && prm.resume)) {
        for (uint32_t w = sub; w < S32; w += W) {                 // 32 steps at a time, for the two bitmaps
            const uint32_t t = w * 32 + lane, i = min(t, S - 1);
            const uint4 n = __ldg(prm.counters0 + i);             // {hr, mi, mo, occ}
            const StepC k = __ldg(prm.stepc + i);
            const uint32_t hb = GROW ? __ldg(prm.hb0 + i) : 0u;
            const int th = (int)(k.x + prm.K.kh * (n.x + hb) + prm.K.khF * (n.y + n.z));
            const int ext = ext_term((int)n.y, (int)n.z, (int)hb, k, prm.K), base = (int)(k.w - prm.K.ke * n.x);
            if (t < S) {
                if (LIN) c.tt()[t] = make_int2(th, base + ext);
                else c.tm()[t] = make_int4(th, base, (int)n.y, (int)n.z);
                if (GROW && !LIN) c.hb()[t] = hb;
                c.occ()[t] = (typename Chain<PSMEM, GROW, LIN, COLV, R, AHEAD>::Occ)n.w;
            }
            const uint32_t F = __ballot_sync(0xFFFFFFFFu, t < S && n.w == prm.cap);
            const uint32_t T = __ballot_sync(0xFFFFFFFFu, t < S && base + ext >= th);
            if (lane == 0) { c.full()[w] = F; c.lead()[w] = T; }
            if (!LIN) {
                const uint32_t by = term_leads(make_int4(th, base, (int)n.y, (int)n.z), (int)hb, k, prm.K);
                const uint32_t O = __ballot_sync(0xFFFFFFFFu, t < S && (by & 2u)), I = __ballot_sync(0xFFFFFFFFu, t < S && (by & 4u));
                if (lane == 0) { c.out()[w] = O; c.in()[w] = I; }
            }
        }
        if (tid == 0) {
            ChainShared z = {};
            z.cur = z.best = z.best_at_boundary = prm.init_ticks;
            z.best_move = ~0ull;
            *sc = z;
        }
        if (!PSMEM)
            for (uint32_t i = tid; i < cow_words; i += nthr) c.have()[i] = 0u;   // the slice holds nothing yet
        else
            copy_words(c.P(), prm.Pcol0, pwords, tid, nthr);
    } else if (active) {
        uint4* const mine4 = c.template at<uint4>(c.cb);
        for (uint32_t i = tid; i < persist4; i += nthr) mine4[i] = saved[i];
        if (PSMEM) copy_words(c.P(), reinterpret_cast<const uint32_t*>(saved + persist4), pwords, tid, nthr);
    }
    __syncthreads();
    const bool fused = prm.ladder_ctas != 0u;                     // whole ladders in this CTA: exchange between segments
    if (!active && !fused) return;
    __shared__ uint8_t s_holder[16];                              // fused: the chain (within the CTA) on each rung
    if (fused) {
        if (threadIdx.x < 16) s_holder[threadIdx.x] = (uint8_t)threadIdx.x;
        if (active && tid == 0) sc->rung = cic % prm.ladder.rungs;
        __syncthreads();
    }

    uint32_t n_same = 0, n_inf = 0;                               // per lane: of the proposals this lane owned
    // A segment of moves at one temperature: a level of the cooling schedule, or a round of a replica-exchange run. All
    // but the last have the same length, so the batches of the run are numbered without a counter.
    const bool exchange = prm.rung_hist != nullptr;
    bool over = !active;                                          // this warp is done with its chain
    bool silent = false;                                          // ... because a wait ran out
    uint32_t win = 32 * R;                                        // proposals evaluated at a time
    for (uint32_t seg = prm.seg0; seg < prm.seg1; ++seg) {
        const uint64_t len = min(seg + 1 == prm.seg1 ? ~(uint64_t)0 : prm.seg_len, prm.upto - seg * prm.seg_len);
        const uint32_t nbat = (uint32_t)((len + 32 * R - 1) / (32 * R)), last_nb = (uint32_t)(len - (uint64_t)(nbat - 1) * (32 * R));
        const uint32_t base = (seg - prm.seg0) * prm.seg_bat;     // index of the segment's first batch (mod 2^32)
        if (!over) {
            x.level = !exchange ? seg : fused ? sc->rung : prm.rung_hist[(size_t)seg * prm.hist_stride + (chain - prm.hist_base)];
            x.shift = __ldg(prm.shifts + x.level);
            x.bound = __ldg(prm.bounds + x.level);
        }
#pragma unroll 1
        for (uint32_t bi = (sub - base) & (W - 1); bi < nbat && !over; bi += W) {
            const uint32_t nb = bi + 1 < nbat ? 32u * R : last_nb;
            const uint32_t mine = (1u << rows_before(nb, lane)) - 1u;   // row mask (row h: proposal 32 h + lane): this lane's proposals
            uint32_t n0 = 0;
            if (W > 1) {
                // moves applied from now on may be half visible to the reads below: they are checked for at the turn
                n0 = __shfl_sync(0xFFFFFFFFu, ld_volatile_u32(&sc->napplied), 0);
                __threadfence_block();
            }
            uint32_t settled = 0u, todo = mine;                   // committed so far; row mask: not evaluated, or no longer right
            if (lane < (uint32_t)R) c.close()[lane] = 0u;
            __syncwarp();
            uint32_t same = 0u, inf = 0u;                         // row masks of what is evaluated: changes nothing, infeasible
            uint32_t kept = 0u, count = min(nb, win), upto = count;   // upto: the ids below it are in the list
            bool at_turn = false;
#pragma unroll 1
            for (;;) {
                const uint64_t m = seg * prm.seg_len + (uint64_t)bi * (32 * R);
                upto = min(upto, evaluate(c, x, m, chain, !at_turn, count, lane, kept, same, inf));
                const uint32_t good = todo & ((1u << rows_before(upto, lane)) - 1u);
                if (at_turn) {                                    // what became of this lane's rows among them
                    same &= ~good; inf &= ~good;
#pragma unroll 1
                    for (uint32_t rest = good; rest; rest &= rest - 1u) {
                        const uint32_t h = __ffs(rest) - 1u, state = c.state()[h * 32 + lane];
                        if (state == kSame) same |= 1u << h;
                        if (state == kInf) inf |= 1u << h;
                    }
                }
                todo &= ~good;
                if (!at_turn) {
                    at_turn = true;
                    if (W > 1) {
                        const uint32_t b = base + bi;
                        const uint32_t left = wait_turn(sc, b);
                        if (left) {                               // gave up: flag it; or the chain has ended: pass on, leave
                            if (lane == 0) {
                                if (left > 1u) {
                                    atomicExch(prm.err, 1u);
                                    st_volatile_u32(&sc->stopped, 1u);
                                    __threadfence_block();
                                }
                                st_volatile_u32(&sc->turn, b + 1u);
                            }
                            over = true;
                            silent = left > 1u;
                            break;
                        }
                        const uint32_t napp = sc->napplied;
                        if (napp - n0 > kLog) todo = mine;
                        else
#pragma unroll 1
                            for (uint32_t k = n0; k != napp; ++k) todo |= spoiled(c, sc->applog[k % kLog], same, lane) & mine;
                    }
                    if (!exchange && bi == 0 && seg > 0) {        // the level's first batch: stop rule, new reference
                        const uint64_t best = sc->best, before = sc->best_at_boundary;
                        if (prm.early_permille && seg >= prm.early_from &&
                            (before - best) * 1000ull < before * (uint64_t)prm.early_permille) {
                            if (lane == 0) {
                                sc->m_end = m;
                                st_volatile_u32(&sc->stopped, 1u);
                                __threadfence_block();
                                st_volatile_u32(&sc->turn, base + bi + 1u);
                            }
                            over = true;
                            break;
                        }
                        __syncwarp();
                        if (lane == 0) sc->best_at_boundary = best;
                        __syncwarp();
                    }
                }
                // Commit in move order up to the first proposal that is not evaluated or no longer right. Nearly always
                // that is all of them, and none changes the schedule.
                uint32_t limit = first_of(todo, lane), e = 0;
#pragma unroll 1
                for (; e < kept; ++e) {
                    const uint4 a = c.acc()[2 * e], w = c.acc()[2 * e + 1];
                    const uint32_t id = a.x >> 24, s0b = (a.x >> 8) & 0x7FFFu;
                    if (id >= limit) break;
                    const uint64_t after = (uint64_t)((int64_t)sc->cur + (int)a.w);
                    const bool leaving = prm.snap && sc->snap_dirty && after >= sc->best;
                    if (leaving) copy_words_cold(prm.snap + (size_t)slot * pwords, c.P(), pwords, lane);   // save the best state first
                    __syncwarp();
                    Applied g;
                    g.steps = s0b | (s0b + ((a.x >> 1) & 31u)) << 16;
                    g.units = (a.y & 0xFFFFu) | ((a.x & 1u) ? a.z : a.y) << 16;
                    g.fulls = 0u;
                    g.bits = apply(c, lane, a, w);
                    if (lane == 0) record(prm, sc, m + id, after, leaving, g, slot);
                    __syncwarp();
                    // what comes after it and depends on what it changed is no longer right
                    todo |= spoiled(c, g, same, lane) & mine & ~((1u << rows_before(id + 1, lane)) - 1u);
                    limit = first_of(todo, lane);
                }
                const uint32_t from = settled;
                settled = min(limit, nb);
                const uint32_t rows = (1u << rows_before(settled, lane)) - (1u << rows_before(from, lane));
                n_inf += __popc(inf & rows);
                n_same += __popc(same & rows);
                // as many proposals at a time as are likely to be committed together
                if (settled >= min(upto, nb)) win = min(32u * R, 2 * win);
                else if (4 * (settled - from) < win) win = max(32u, win / 2);
                if (limit >= kNone) break;
                // next: what is to be evaluated, and with it the accepted ones behind `limit`
#pragma unroll 1
                for (; e < kept; ++e) {
                    const uint32_t id = c.acc()[2 * e].x >> 24;
                    if ((id & 31u) == lane) todo |= 1u << (id >> 5);
                }
                count = 0;
                upto = kNone;
#pragma unroll 1
                for (uint32_t h = limit >> 5; h < (uint32_t)R; ++h) {
                    const uint32_t rb = __ballot_sync(0xFFFFFFFFu, (todo >> h) & 1u);
                    if ((todo >> h) & 1u) c.again()[count + __popc(rb & ((1u << lane) - 1u))] = (uint8_t)(h * 32 + lane);
                    count += __popc(rb);
                    if (count >= win) { upto = h * 32 + 32; break; }
                }
                __syncwarp();
                if (count > win) { upto = c.again()[win]; count = win; }
                if (lane == 0) x.n_again += count;
            }
            if (over) break;
            if (W > 1) {                                          // hand the chain to the owner of the next batch
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    if (!(prm.drop_first_turn && base + bi == 0)) st_volatile_u32(&sc->turn, base + bi + 1u);
                }
            }
        }
        if (over && !fused) break;
        if (__any_sync(0xFFFFFFFFu, (n_same | n_inf) >> 30)) {    // the lanes' counters are emptied before they run over
            atomicAdd(reinterpret_cast<unsigned long long*>(&sc->n_same), (unsigned long long)n_same);
            atomicAdd(reinterpret_cast<unsigned long long*>(&sc->n_inf), (unsigned long long)n_inf);
            n_same = n_inf = 0u;
        }
        if (fused && seg + 1 < prm.seg1) {
            __syncthreads();                                      // every chain of the CTA has done its round
            exchange_round(c, s_holder, stride, cpb, seg);
            __syncthreads();
            if (active && tid == 0) prm.rung_hist[(size_t)(seg + 1) * prm.hist_stride + (chain - prm.hist_base)] = (uint8_t)sc->rung;
        }
    }
    if (!active || silent) return;
    // every warp adds what it counted; the last one to leave reports for the chain
    auto add = [](uint64_t* p, uint64_t v) { atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v); };
    add(&sc->n_same, n_same); add(&sc->n_inf, n_inf); add(&sc->n_items, x.n_items);
    uint32_t last = 0u;
    if (lane == 0) { add(&sc->n_again, x.n_again); add(&sc->n_listed, x.n_listed); }
    __threadfence_block();
    __syncwarp();
    if (lane == 0) last = atomicAdd(&sc->left, 1u) == W - 1u ? 1u : 0u;
    last = __shfl_sync(0xFFFFFFFFu, last, 0);
    if (!last) return;
    __threadfence_block();
    if (lane == 0) {
        kvp_chain_result res;
        res.best_ticks = sc->best; res.best_move = sc->best_move; res.final_ticks = sc->cur;
        res.moves_done = sc->m_end ? sc->m_end : min(prm.upto, exchange ? prm.seg1 * prm.seg_len : ~(uint64_t)0);
        res.n_accepted = sc->n_same + sc->n_chg; res.n_changed = sc->n_chg; res.n_infeasible = sc->n_inf; res.traj_hash = sc->hash;
        prm.results[chain - prm.result_base] = res;
        if (prm.n_exchanged) prm.n_exchanged[chain - prm.hist_base] = sc->n_exchanged;
        if (prm.work) {
            atomicAdd(prm.work, (unsigned long long)sc->n_again);
            atomicAdd(prm.work + 1, (unsigned long long)sc->n_listed);
            atomicAdd(prm.work + 2, (unsigned long long)sc->n_items);
        }
        sc->turn = 0u; sc->napplied = 0u; sc->left = 0u;          // the hand-over of a chain taken up again starts anew
    }
    __syncwarp();
    if (saved) {                                                  // the next round goes on from here
        const uint4* const mine4 = c.template at<uint4>(c.cb);
        for (uint32_t i = lane; i < persist4; i += 32) saved[i] = mine4[i];
        if (PSMEM) copy_words_cold(reinterpret_cast<uint32_t*>(saved + persist4), c.P(), pwords, lane);
    }
    if (prm.snap && sc->snap_dirty) copy_words_cold(prm.snap + (size_t)slot * pwords, c.P(), pwords, lane);
    if (prm.undo_log && lane == 0) prm.undo_len[slot] = sc->ulen;
    if (!PSMEM && prm.cow_out)                                    // which buckets the slice holds (for the walk back)
        for (uint32_t i = lane; i < cow_words; i += 32) prm.cow_out[(size_t)slot * cow_words + i] = c.have()[i];
    if (prm.dump && slot == 0) {
        if (PSMEM) copy_words_cold(prm.dump, c.P(), pwords, lane);
        else copy_merged(prm.dump, c.P(), prm.Pcol0, c.have(), prm.cow_shift, U, S32, lane);
    }
}

}  // namespace

}  // namespace kvp
