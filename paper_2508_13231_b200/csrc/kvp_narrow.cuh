// The narrow chain kernel (included by kvp_anneal.cu only): for jobs of few chains per SM and for chains that apply many of
// their moves, such as hot starts, where a fifth to a quarter of the proposals change the schedule, and the hot rungs of
// replica exchange (whole ladders in a CTA, or a launch per round).
//
// There, evaluations of cost changes ahead of the commits do not last. What lasts is what depends on a proposal's own units:
// a warp takes 32 consecutive proposals, one per lane, and prepares them word-parallel: the windows, what the placement bits
// settle, the masks of hits won and lost and of migration edges, the largest cost change its uniform lets pass, and the
// lower bound of kvp_chain.cuh, which rejects most of the rest. An applied move spoils a later preparation only if both name
// a unit and have steps in common; a flip is checked again if one of its steps became full or free, a bounded rejection if
// the leading side of one of its steps changed. The proposals that are left are evaluated in move order, against the state
// as it is, a lane per step of the window (two side by side where the registers allow it: their steps seldom meet); what
// bounds a chain is the latency of these dependent steps (votes, sums over the warp, shared-memory loads).
// W warps may serve a chain: they take its batches in turn and prepare ahead of each other's commits (see ChainShared).
//
// The kernel before evaluated its 32 proposals in full, ahead of the commits, through a work queue of (proposal, step)
// items, one move applied per pass. Measured (B200), before and now: 256 units x 512 steps at p0 = 0.8, 1024
// chains x 100,000 moves: 25.5 -> 13.6 ms; 16 x 32, 64 x 10,000: 0.43 -> 0.33 to 0.37 by box; 16,384 x 256, 1024 x 200,000: 15.7 -> 10.8.
// A link slower than the DRAM channels (not LIN), which for a while only the wide kernel served, without a bound: 256 x 512,
// 1024 x 20,000 at p0 = 0.8: 8.5 -> 3.2 ms (the kernel before 4.4); 16,384 x 256, 1024 x 100,000: 12.3 -> 7.0 (7.3).
// Growing caches, likewise: 512 units x 132 steps, 256 x 20,000 0.61 -> 0.45 ms (0.69), at p0 = 0.8 5.2 -> 1.7 (3.4);
// 131,072 x 1056, 1024 x 20,000 at p0 = 0.8 6.6 -> 4.5 (5.8).
#pragma once

namespace kvp {

namespace {

// uint4 slots of a warp's prepared proposals
__host__ __device__ constexpr uint32_t prepared4(bool lin) { return lin ? 4 * 32 : 5 * 32; }

inline ChainLayout narrow_layout(uint32_t S, uint32_t S32, bool grow, bool psmem, bool lin, uint32_t cow4)
{
    ChainLayout l;
    uint32_t at = sizeof(ChainShared) + 16 * (lin ? (S + 1) / 2 : S);   // {th, te}, or {th, te without migrations, in, out}
    auto take = [&](uint32_t n4) { const uint32_t p = at; at += 16 * n4; return p; };
    l.occ = take(psmem ? (S + 7) / 8 : (S + 3) / 4);
    l.full = take((S32 + 4) / 4);                         // (a bitmap is followed by a readable word)
    l.lead = take((S32 + 4) / 4);
    l.out = take(lin ? 0u : (S32 + 4) / 4);
    l.in = take(lin ? 0u : (S32 + 4) / 4);
    l.hb = take(grow && !lin ? (S + 3) / 4 : 0u);
    l.have = take(cow4);
    l.work = at;
    return l;
}
// bytes of a chain of W warps, without a schedule in shared memory
inline size_t narrow_bytes(uint32_t S, uint32_t S32, bool grow, bool psmem, bool lin, uint32_t cow4, uint32_t W)
{
    return narrow_layout(S, S32, grow, psmem, lin, cow4).work + (size_t)W * prepared4(lin) * 16;
}

// where a chain and a warp of it keep their state in shared memory
template <bool PSMEM>
struct Narrow {
    using Occ = typename std::conditional<PSMEM, uint16_t, uint32_t>::type;   // PSMEM: fewer than 2^16 units
    const ChainParams& prm;
    uint32_t cb, wb;             // byte offsets: the chain's state, the warp's prepared proposals
    template <typename T> __device__ __forceinline__ T* at(uint32_t off) const { return reinterpret_cast<T*>(chain_smem + off); }
    __device__ __forceinline__ ChainShared* sc() const { return at<ChainShared>(cb); }
    // [S] {th, te}, or {th, te without its migration term, units moved in, units moved out}
    template <typename Sides> __device__ __forceinline__ Sides* sides() const { return at<Sides>(cb + (uint32_t)sizeof(ChainShared)); }
    __device__ __forceinline__ Occ* occ() const { return at<Occ>(cb + prm.lay.occ); }              // [S]
    __device__ __forceinline__ uint32_t* full() const { return at<uint32_t>(cb + prm.lay.full); }  // [S32] bit t: occ[t] == cap
    __device__ __forceinline__ uint32_t* lead() const { return at<uint32_t>(cb + prm.lay.lead); }  // [S32] bit t: te[t] >= th[t]
    // not LIN: [S32] bit t: the link's outbound (inbound) traffic is the largest term of Eq. 4's maximum (see term_leads)
    __device__ __forceinline__ uint32_t* out() const { return at<uint32_t>(cb + prm.lay.out); }
    __device__ __forceinline__ uint32_t* in() const { return at<uint32_t>(cb + prm.lay.in); }
    __device__ __forceinline__ uint32_t* hb() const { return at<uint32_t>(cb + prm.lay.hb); }      // GROW, not LIN: [S] written to HBM at birth
    __device__ __forceinline__ uint32_t* have() const { return at<uint32_t>(cb + prm.lay.have); }  // not PSMEM: buckets the slice holds
    // [4][32] prepared proposals: {s0 | end << 16, hit, lost, one}, {two, neg, largest accepted change, changed},
    // {u, v, D's two words}, {D, placement after, Metropolis uniform, GROW: the step at which a unit is written to HBM (bit 0
    // set) or to DRAM instead of the other}; not LIN: one, two and neg are of the units moved in,
    // and a fifth row has those of the units moved out
    __device__ __forceinline__ uint4* rec() const { return at<uint4>(wb); }
};

// By how much a count rises at each step, given the up to two events that add to it after (na, nb) and before (oa, ob) a
// move, one bit a step: one and two are the bits of the absolute value, neg its sign.
struct Rise { uint32_t one, two, neg; };
__device__ __forceinline__ Rise rise_of(uint32_t na, uint32_t nb, uint32_t oa, uint32_t ob)
{
    const uint32_t n1 = na ^ nb, n2 = na & nb, o1 = oa ^ ob, o2 = oa & ob;
    Rise r;
    r.two = (n2 & ~(o1 | o2)) | (o2 & ~(n1 | n2));
    r.one = n1 ^ o1;
    r.neg = (o2 & ~n2) | (o1 & ~(n1 | n2));
    return r;
}
// its sum over the steps of a mask
__device__ __forceinline__ int rise_over(const Rise& r, uint32_t m)
{
    return __popc(r.one & m) + 2 * (__popc(r.two & m) - __popc(r.one & r.neg & m)) - 4 * __popc(r.two & r.neg & m);
}
// its value at a step
__device__ __forceinline__ int rise_at(uint32_t one, uint32_t two, uint32_t neg, uint32_t bit)
{
    const int n = (int)((one >> bit) & 1u) + 2 * (int)((two >> bit) & 1u);
    return (neg >> bit) & 1u ? -n : n;
}

// PSMEM: schedules in shared memory; otherwise a chain's slice of global scratch is a copy-on-write overlay of the initial
// schedule. ASMEM: the access bitmap staged there, too. SOLO: one warp per chain (W == 1).
// LIN: kappa_d >= kappa_k, th and te are linear in hits and migrations (see kvp_chain.cuh). Otherwise te is the largest of
// three linear terms, migrations in and out count separately, and the lower bound follows the term that leads at each step:
// th, or Eq. 4 with the term that is the largest of its three (the new maximum is at least that one's new value).
// GROW: units have steps of birth. A move acts where both its units exist; of the steps in which they are written at most one
// is among these (the later one: if both are written in the same step, a swap leaves that step's writes as they are).
template <bool SOLO, bool PSMEM, bool ASMEM, bool GROW, bool LIN, int COLV>
__global__ void __launch_bounds__(SOLO ? 256 : 512, 1)
narrow_chain_kernel(const __grid_constant__ ChainParams prm)
{
    static_assert(PSMEM ? COLV == 0 : !ASMEM && !SOLO, "vector columns only for schedules in global scratch");
    constexpr int kSide = SOLO ? 2 : 1;                           // (registers: 157; two in the other variants spill)
    constexpr uint32_t kPrepared4 = prepared4(LIN);
    using Sides = typename std::conditional<LIN, int2, int4>::type;
    using Occ = typename Narrow<PSMEM>::Occ;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = SOLO ? 1u : prm.warps;
    const uint32_t cpb = (blockDim.x >> 5) / W, cic = warp / W, sub = warp % W;   // chains per CTA; chain; warp of the chain
    const uint32_t slot = blockIdx.x * cpb + cic, chain = prm.chain_first + slot;
    const bool active = slot < prm.chain_count;
    const uint32_t S = prm.S, S32 = prm.S32, U = prm.U;
    const size_t pwords = (size_t)U * S32;
    const uint32_t o4 = PSMEM ? 0u : prm.cow_slots4, stride = prm.lay.work + W * kPrepared4 * 16;   // bytes of a chain
    const uint32_t cb = cic * stride, wb = cb + prm.lay.work + sub * kPrepared4 * 16;
    const Narrow<PSMEM> c{prm, cb, wb};
    uint32_t* const pool = reinterpret_cast<uint32_t*>(chain_smem + cpb * stride);
    uint32_t* const P = PSMEM ? pool + cic * (uint32_t)pwords : prm.ws + (size_t)slot * pwords;
    const uint32_t* A = prm.Acol;
    if (ASMEM) {
        uint32_t* const a_s = pool + ((cpb * (uint32_t)pwords + 3u) & ~3u);
        copy_words(a_s, prm.Acol, pwords, threadIdx.x, blockDim.x);
        A = a_s;
    }
    // rounds of launches: what the chain left behind in the round before (see ChainParams::state)
    const bool resumed = prm.resume != 0u;
    if (active && resumed) {
        if (sub == 0) {
            const uint32_t* const saved = reinterpret_cast<const uint32_t*>(prm.state + (size_t)(chain - prm.hist_base) * prm.state4);
            copy_words_cold(c.template at<uint32_t>(cb), saved, prm.lay.work / 4, lane);
            if (PSMEM) copy_words_cold(P, saved + prm.lay.work / 4, pwords, lane);
        }
    } else if (active) {
        for (uint32_t w = sub; w < S32; w += W) {                 // 32 steps at a time, for the two bitmaps
            const uint32_t t = w * 32 + lane, i = min(t, S - 1);
            const uint4 n = __ldg(prm.counters0 + i);             // {hr, mi, mo, occ}
            const StepC k = __ldg(prm.stepc + i);
            const int hb = GROW ? (int)__ldg(prm.hb0 + i) : 0;
            const int4 f = make_int4((int)(k.x + prm.K.kh * (n.x + hb) + prm.K.khF * (n.y + n.z)), (int)(k.w - prm.K.ke * n.x), (int)n.y, (int)n.z);
            const int te = f.y + ext_term(f.z, f.w, hb, k, prm.K);
            if (t < S) {
                if constexpr (LIN) c.template sides<int2>()[t] = make_int2(f.x, te);
                else c.template sides<int4>()[t] = f;
                if constexpr (GROW && !LIN) c.hb()[t] = (uint32_t)hb;
                c.occ()[t] = (Occ)n.w;
            }
            const uint32_t F = __ballot_sync(0xFFFFFFFFu, t < S && n.w == prm.cap), T = __ballot_sync(0xFFFFFFFFu, t < S && te >= f.x);
            if (lane == 0) { c.full()[w] = F; c.lead()[w] = T; }
            if constexpr (!LIN) {
                const uint32_t by = term_leads(f, hb, k, prm.K);
                const uint32_t O = __ballot_sync(0xFFFFFFFFu, t < S && (by & 2u)), I = __ballot_sync(0xFFFFFFFFu, t < S && (by & 4u));
                if (lane == 0) { c.out()[w] = O; c.in()[w] = I; }
            }
        }
        if (sub == 0 && lane == 0) {
            ChainShared z = {};
            z.cur = z.best = z.best_at_boundary = prm.init_ticks;
            z.best_move = ~0ull;
            *c.sc() = z;
        }
        if (!PSMEM)
            for (uint32_t i = sub * 32 + lane; i < o4 * 4; i += W * 32) c.have()[i] = 0u;   // the slice holds nothing yet
        else
            copy_words(P, prm.Pcol0, pwords, sub * 32 + lane, W * 32);
    }
    __syncthreads();
    const bool fused = PSMEM && prm.ladder_ctas != 0u;            // whole ladders in this CTA: exchange between segments
    if (!active && !fused) return;
    __shared__ uint8_t s_holder[PSMEM ? 16 : 1];                  // fused: the chain (within the CTA) on each rung
    if (fused) {
        if (threadIdx.x < 16) s_holder[threadIdx.x] = (uint8_t)threadIdx.x;
        if (active && sub == 0 && lane == 0) c.sc()->rung = cic % prm.ladder.rungs;
        __syncthreads();
    }
    auto column = [&](uint32_t u) -> const uint32_t* {
        if (PSMEM) return P + u * S32;
        const uint32_t b = u >> prm.cow_shift, w = ld_volatile_u32(c.have() + (b >> 5));   // (another warp may be taking it over)
        return ((w >> (b & 31u)) & 1u ? (const uint32_t*)P : prm.Pcol0) + (size_t)u * S32;
    };
    // not PSMEM, before unit u is rewritten: its bucket is copied into the slice if it is not there yet
    auto own = [&](uint32_t u) {
        const uint32_t b = u >> prm.cow_shift;
        if ((c.have()[b >> 5] >> (b & 31u)) & 1u) return;
        const size_t lo = (size_t)(b << prm.cow_shift) * S32, hi = (size_t)min(U, (b + 1u) << prm.cow_shift) * S32;
#pragma unroll 1
        for (size_t i = lo + lane; i < hi; i += 32) P[i] = prm.Pcol0[i];
        __threadfence_block();
        __syncwarp();
        if (lane == 0) c.have()[b >> 5] |= 1u << (b & 31u);
        __syncwarp();
    };

    // The chain's scalars: SOLO in registers, otherwise in `sc`.
    uint64_t cur = prm.init_ticks, best = cur, best_move = ~0ull, hash = 0, n_chg = 0;
    bool unsaved = false;                                         // the best state is the current one and not saved yet
    if (SOLO && resumed) {
        const ChainShared* const was = c.sc();
        cur = was->cur; best = was->best; best_move = was->best_move; hash = was->hash; n_chg = was->n_chg;
        unsaved = was->snap_dirty != 0u;
    }

    uint32_t n_same = 0, n_inf = 0;                               // per lane
    const int kh = (int)prm.K.kh, ke = (int)prm.K.ke, khF = (int)prm.K.khF, kdF = (int)prm.K.kdF, kkF = (int)prm.K.kkF;
    const int kd = (int)prm.K.kd, kk = (int)prm.K.kk;
    const bool exchange = prm.rung_hist != nullptr;               // a level is a round of a replica-exchange run
    bool over = !active, silent = false;                          // this warp is done with its chain; because a wait ran out
    for (uint32_t level = 0; level < prm.seg1; ++level) {
        if (over && !fused) break;
        const uint64_t lvl_start = prm.move0 + level * prm.seg_len, lvl_len = min(level + 1 == prm.seg1 ? ~(uint64_t)0 : prm.seg_len, prm.upto - lvl_start);
        const uint32_t nbat = (uint32_t)((lvl_len + 31) / 32), last_nb = (uint32_t)(lvl_len - (uint64_t)(nbat - 1) * 32);
        const uint32_t base = level * prm.seg_bat;                // index of the level's first batch (mod 2^32)
        // row of the acceptance table
        const uint32_t rank = over ? 0u : !exchange ? level : fused ? c.sc()->rung : prm.rung_hist[(size_t)level * prm.hist_stride + (chain - prm.hist_base)];
        const uint32_t shift = __ldg(prm.shifts + rank);
        const uint32_t* const row = prm.table + (size_t)rank * KVP_TABLE_Q;
        const float scale = __ldg(prm.bounds + rank) * __uint_as_float((127u - shift) << 23);   // C ln 2 in bins
        const uint32_t bin = shift < 31 ? 1u << shift : 0x7FFFFFFFu;
        const bool bounded = scale < 1e30f;                       // the lower bounds fit 32 bits
#pragma unroll 1
        for (uint32_t bi = (sub + W - base % W) % W; bi < nbat && !over; bi += W) {
            const uint64_t m = lvl_start + (uint64_t)bi * 32;
            const uint32_t nb = bi + 1 < nbat ? 32u : last_nb;
            uint32_t n0 = 0;
            if (W > 1) {
                // moves applied from now on may be half visible to the reads below: they are checked for at the turn
                n0 = __shfl_sync(0xFFFFFFFFu, ld_volatile_u32(&c.sc()->napplied), 0);
                __threadfence_block();
            }
            LaneMove mv;
            {
                uint32_t r[4];
                const uint64_t mine = m + lane;
                philox4x32_10((uint32_t)mine, (uint32_t)(mine >> 32), chain, TAG_MOVE, prm.keys, r);
                decode_move(r, prm.p_swap_256, prm.len_choices, S, U, mv);
            }
            const uint32_t s0 = mv.pk >> 8, len = (mv.pk >> 1) & 31u, send = s0 + len;
            const bool swap = mv.pk & 1u;
            const uint32_t run = min(len, S - s0), nl = min(len, S - 1 - s0) + 1;   // steps rewritten; affected
            const uint32_t Sb = ((1u << nl) - 1u) << 1;
            uint32_t M = ((1u << run) - 1u) << 1;
            const WinPos wp = window_pos(s0);
            const uint32_t u = mv.u, v = swap ? mv.v : mv.u, units = (u & 0xFFFFu) | v << 16;
            uint32_t Bu = 0u, Bv = 0u;                            // GROW: the steps in which u and v are written
            if constexpr (GROW) {
                uint32_t Lu, Lv;
                alive_born(__ldg(prm.birth + u), s0, Lu, Bu);
                alive_born(__ldg(prm.birth + v), s0, Lv, Bv);
                M &= Lu & Lv;
            }
            const uint32_t Au = window_at<COLV>(A + (size_t)u * S32, wp), av = window_at<COLV>(A + (size_t)v * S32, wp);
            const uint32_t Av = swap ? av : 0u;
            // A cost change passes the Metropolis test if its bin q has q + 1/2 < X = C ln(2^32 / w) in bins, up to the
            // rounding of the thresholds and of the logarithm here, far less than a tenth of a bin from w = 4096 on: bins up
            // to X - 0.6 pass, of the next one the table decides should a change fall into it, those above do not.
            // (Two or three dependent table loads per batch before: 2.85 -> 2.69 ms on 256 units x 512 steps, 1024 chains x
            // 100,000 moves; the hot rungs of replica exchange 4.47 -> 4.10.)
            int dmax;                                             // the largest change that passes for certain
            if (bounded && mv.w >= 4096u) {
                const int q = min((int)floorf(scale * (32.0f - __log2f((float)mv.w)) - 0.6f), (int)KVP_TABLE_Q - 1);
                dmax = q >= 0 ? (int)min(((uint64_t)(q + 1) << shift) - 1u, (uint64_t)0x7FFFFFFF) : 0;
            } else {
                int q = -1;
#pragma unroll 1
                for (int step = KVP_TABLE_Q / 2; step > 0; step >>= 1)
                    if (mv.w < __ldg(row + q + step)) q += step;
                if (q + 1 < (int)KVP_TABLE_Q && mv.w < __ldg(row + q + 1)) ++q;
                dmax = q >= 0 ? (int)min(((uint64_t)(q + 1) << shift) - 1u, (uint64_t)0x7FFFFFFF) : 0;
            }
            uint32_t pend = nb >= 32 ? 0xFFFFFFFFu : (1u << nb) - 1u;   // not committed
            uint32_t prep = pend, check = 0u;                     // to be prepared (again); flips to be checked again
            uint32_t Wu = 0u;
            bool none = false, bad = false, rejected = false, at_turn = false;
            // what an applied move makes of the preparations of this batch
            auto mark = [&](const Applied& g) {
                const uint32_t bu = g.units & 0xFFFFu, bv = g.units >> 16, lo = units & 0xFFFFu, hi = units >> 16;
                const bool meets = s0 <= (g.steps >> 16) + 1u && (g.steps & 0xFFFFu) <= send;
                const bool anew = meets && (lo == bu || lo == bv || hi == bu || hi == bv);
                const bool open = rejected && (g.bits & 0xFFFFu) <= send && s0 <= (g.bits >> 16);
                const bool flip = !swap && (g.fulls & 0xFFFFu) <= send && s0 <= (g.fulls >> 16);
                if (__ballot_sync(0xFFFFFFFFu, anew || open || flip) & pend) {
                    if (open) rejected = false;                   // looked at after all
                    prep |= __ballot_sync(0xFFFFFFFFu, anew) & pend;
                    check |= __ballot_sync(0xFFFFFFFFu, flip) & pend;
                    return true;
                }
                return false;
            };
#pragma unroll 1
            for (;;) {
                if (prep) {                                       // warp-uniform
                    const uint32_t T = window_at<0>(c.lead(), wp);    // steps where te leads
                    uint32_t wu, W2;
                    if constexpr (PSMEM) {
                        wu = window_at<0>(column(u), wp);
                        W2 = window_at<0>(swap ? column(v) : c.full(), wp);
                    } else if constexpr (COLV == 4) {             // (eight registers less: 1.32 against 1.35 ms on 131,072 x 100, 500 x 20,000)
                        wu = window_at<COLV>(column(u), wp);
                        W2 = swap ? window_at<COLV>(column(v), wp) : window_at<0>(c.full(), wp);
                    } else {
                        // No branch in between, so that all loads are under way before the first is waited for; a flip's second
                        // one is of the same words (16,384 units x 256 steps, 1024 x 200,000: 11.5 -> 10.8 ms).
                        const typename Words<COLV>::type qu = words_at<COLV>(column(u), wp), qv = words_at<COLV>(column(v), wp);
                        const uint32_t F = window_at<0>(c.full(), wp);
                        wu = cut<COLV>(qu, wp);
                        W2 = swap ? cut<COLV>(qv, wp) : F;
                    }
                    const uint32_t D = (swap ? wu ^ W2 : 0xFFFFFFFFu) & M;   // a flip toggles every bit of the run
                    const uint32_t Wv = swap ? W2 : 0u;
                    uint32_t Nu = wu ^ D, Nv = swap ? Wv ^ D : 0u;
                    if (s0 == 0) {                                // the virtual step -1 follows step 0
                        Nu = (Nu & ~1u) | ((Nu >> 1) & 1u);
                        Nv = (Nv & ~1u) | ((Nv >> 1) & 1u);
                    }
                    const uint32_t hit = (Au ^ Av) & D, lost = hit & (Au ^ Nu);
                    uint32_t eun = Nu ^ (Nu << 1), euo = wu ^ (wu << 1), evn = Nv ^ (Nv << 1), evo = Wv ^ (Wv << 1);
                    uint32_t born = 0u;                           // GROW: a step whose write goes elsewhere, bit 0: to HBM
                    if constexpr (GROW) {                         // the edge into the step in which a unit is written is no migration
                        eun &= ~Bu; euo &= ~Bu; evn &= ~Bv; evo &= ~Bv;
                        born = (Bu ^ (swap ? Bv : 0u)) & D;
                        if (born) born |= ((Bu & D) ? Nu & born : Nv & born) ? 1u : 0u;
                    }
                    const int ht = __popc(hit & T) - 2 * __popc(lost & T), hs = __popc(hit) - 2 * __popc(lost) - ht;
                    int lb = kh * hs - ke * ht;                   // the change of the side that leads
                    Rise go, leave;                               // migrations gained at a step; not LIN: into HBM, out of it
                    if constexpr (LIN) {
                        go = rise_of(eun & Sb, evn & Sb, euo & Sb, evo & Sb);
                        const int mt = rise_over(go, T), ms = rise_over(go, 0xFFFFFFFFu) - mt;
                        lb += kdF * mt + khF * ms;
                        if (GROW && born) lb += (born & 1u ? 1 : -1) * ((T & born & ~1u) ? -kd : kh);
                    } else {
                        go = rise_of(eun & Nu & Sb, evn & Nv & Sb, euo & wu & Sb, evo & Wv & Sb);
                        leave = rise_of(eun & ~Nu & Sb, evn & ~Nv & Sb, euo & ~wu & Sb, evo & ~Wv & Sb);
                        const uint32_t O = window_at<0>(c.out(), wp), I = window_at<0>(c.in(), wp), C = T & ~(O | I);
                        lb += khF * (rise_over(go, ~T) + rise_over(leave, ~T)) + kkF * (rise_over(leave, T & O) + rise_over(go, T & I)) +
                              kdF * (rise_over(go, C) + rise_over(leave, C));
                        if (GROW && born) {
                            const uint32_t B = born & ~1u;
                            lb += (born & 1u ? 1 : -1) * (!(T & B) ? kh : O & B ? -kk : I & B ? 0 : -kd);
                        }
                    }
                    uint32_t turns = hit | go.one | go.two | (born & ~1u);
                    if constexpr (!LIN) turns |= leave.one | leave.two;
                    __syncwarp();
                    if ((prep >> lane) & 1u) {
                        Wu = wu;
                        none = D == 0u;                           // nothing changes: always accepted
                        bad = !swap && (~wu & D & W2) != 0u;      // a flip may not raise a full step (Eq. 5)
                        rejected = bounded && lb > dmax && (uint32_t)(lb - dmax) > bin;
                        const uint32_t d = s0 ? D : D >> 1;       // aligned to step s0 - 1 (0)
                        c.rec()[lane] = make_uint4(s0 | (s0 + 31u - __clz(D)) << 16, hit, lost, go.one);
                        c.rec()[32 + lane] = make_uint4(go.two, go.neg, (uint32_t)dmax, turns | (swap ? 1u : 0u));   // (bit 0 is no step)
                        if constexpr (!LIN) c.rec()[128 + lane] = make_uint4(leave.one, leave.two, leave.neg, 0u);
                        c.rec()[64 + lane] = make_uint4(u, v, d << wp.sh, wp.sh ? d >> (32u - wp.sh) : 0u);
                        c.rec()[96 + lane] = make_uint4(D, Nu, mv.w, born);
                    } else if ((check >> lane) & 1u) {
                        bad = (~wu & D & W2) != 0u;
                    }
                    prep = check = 0u;
                    __syncwarp();
                } else if (check) {
                    const uint32_t F = window_at<0>(c.full(), wp);
                    if ((check >> lane) & 1u) bad = (~Wu & M & F) != 0u;
                    check = 0u;
                }
                if (!at_turn) {
                    at_turn = true;
                    if (W > 1) {
                        const uint32_t b = base + bi, left = wait_turn(c.sc(), b);
                        if (left) {                               // gave up: flag it; or the chain has ended: pass on, leave
                            if (lane == 0) {
                                if (left > 1u) {
                                    atomicExch(prm.err, 1u);
                                    st_volatile_u32(&c.sc()->stopped, 1u);
                                    __threadfence_block();
                                }
                                st_volatile_u32(&c.sc()->turn, b + 1u);
                            }
                            over = true;
                            silent = left > 1u;
                            break;
                        }
                    }
                    if (!exchange && bi == 0 && level > 0) {                   // the level's first batch: stop rule, new reference
                        if (!SOLO) best = c.sc()->best;
                        const uint64_t before = c.sc()->best_at_boundary;
                        if (prm.early_permille && level >= prm.early_from &&
                            (before - best) * 1000ull < before * (uint64_t)prm.early_permille) {
                            if (lane == 0) {
                                c.sc()->m_end = m;
                                st_volatile_u32(&c.sc()->stopped, 1u);
                                __threadfence_block();
                                st_volatile_u32(&c.sc()->turn, base + bi + 1u);
                            }
                            over = true;
                            break;
                        }
                        __syncwarp();
                        if (lane == 0) c.sc()->best_at_boundary = best;
                        __syncwarp();
                    }
                    if (W > 1) {
                        const uint32_t napp = c.sc()->napplied;
                        if (napp - n0 > kLog) prep = pend;
                        else
#pragma unroll 1
                            for (uint32_t k = n0; k != napp; ++k) mark(c.sc()->applog[k % kLog]);
                        if (prep | check) continue;
                    }
                }
                uint32_t survivors = __ballot_sync(0xFFFFFFFFu, !none && !bad && !rejected) & pend;
                if (!survivors) break;
#pragma unroll 1
                while (survivors) {
                    // up to kSide of the survivors: cost changes against the present state
                    Sides g[kSide], f[kSide];
                    uint32_t id[kSide], t[kSide], chg[kSide], steps[kSide];
                    int delta[kSide], most[kSide];
                    uint32_t rest = survivors;
#pragma unroll
                    for (int j = 0; j < kSide; ++j) {
                        id[j] = rest ? __ffs(rest) - 1u : 32u;
                        rest &= rest - 1u;
                        const uint32_t k = id[j] & 31u;
                        const uint4 a = c.rec()[k], b = c.rec()[32 + k];
                        chg[j] = b.w; steps[j] = a.x; most[j] = (int)b.z;
                        t[j] = min((a.x & 0xFFFFu) + max(lane, 1u) - 1u, S - 1u);   // lane l: window bit l, step s0 - 1 + l
                        f[j] = c.template sides<Sides>()[t[j]];
                        const int h = (a.y >> lane) & 1u, hr = (a.z >> lane) & 1u ? -h : h, mi = rise_at(a.w, b.x, b.y, lane);
                        int hb = 0;                               // GROW: writes to HBM gained
                        if constexpr (GROW) {
                            const uint32_t born = c.rec()[96 + k].w;
                            if (lane != 0u && ((born >> lane) & 1u)) hb = born & 1u ? 1 : -1;
                        }
                        if constexpr (LIN) {
                            g[j] = make_int2(f[j].x + kh * (hr + hb) + khF * mi, f[j].y - ke * hr + kdF * mi - kd * hb);
                            delta[j] = max(g[j].x, g[j].y) - max(f[j].x, f[j].y);   // 0 where nothing changes
                        } else {
                            const uint4 o = c.rec()[128 + k];
                            const int mo = rise_at(o.x, o.y, o.z, lane);
                            const StepC sc = __ldg(prm.stepc + t[j]);
                            const int was = GROW ? (int)c.hb()[t[j]] : 0;
                            g[j] = make_int4(f[j].x + kh * (hr + hb) + khF * (mi + mo), f[j].y - ke * hr, f[j].z + mi, f[j].w + mo);
                            delta[j] = max(g[j].x, g[j].y + ext_term(g[j].z, g[j].w, was + hb, sc, prm.K)) -
                                       max(f[j].x, f[j].y + ext_term(f[j].z, f[j].w, was, sc, prm.K));
                        }
                    }
#pragma unroll
                    for (int j = 0; j < kSide; ++j) delta[j] = __reduce_add_sync(0xFFFFFFFFu, delta[j]);
                    uint32_t first = 0xFFFFu, last = 0u;          // steps rewritten by the moves applied in this group
                    bool marked = false;
#pragma unroll
                    for (int j = 0; j < kSide; ++j) {
                        if (id[j] >= 32u) break;                  // (all of this is warp-uniform)
                        const uint32_t b0 = steps[j] & 0xFFFFu, bend = steps[j] >> 16;   // bend: the step after the last rewritten
                        if (j > 0 && b0 <= last && first <= bend) break;   // its steps changed meanwhile
                        survivors &= ~(1u << id[j]);
                        pend &= 0xFFFFFFFEu << id[j];
                        if (delta[j] > most[j]) {                 // rejected by the Metropolis test, unless the table says else
                            if ((uint32_t)(delta[j] - most[j]) > bin) continue;
                            const uint32_t q = (uint32_t)delta[j] >> shift;
                            if (q >= KVP_TABLE_Q || c.rec()[96 + id[j]].z >= __ldg(row + q)) continue;
                        }
                        const uint64_t after = (uint64_t)((int64_t)(SOLO ? cur : c.sc()->cur) + delta[j]);
                        const bool leaving = prm.snap && (SOLO ? unsaved && after >= best : c.sc()->snap_dirty && after >= c.sc()->best);
                        if (leaving) copy_words_cold(prm.snap + (size_t)slot * pwords, P, pwords, lane);   // save the best state first
                        const uint4 r = c.rec()[64 + id[j]];
                        const bool sw = chg[j] & 1u, mine = lane != 0u && (chg[j] >> lane) & 1u;
                        const uint32_t bit0 = b0 ? b0 - 1u : 0u;
                        __syncwarp();
                        if (mine) c.template sides<Sides>()[t[j]] = g[j];
                        uint32_t lturn, oturn = 0u, iturn = 0u, fturn = 0u;   // steps at which the bitmaps turn
                        if constexpr (LIN) {
                            lturn = __ballot_sync(0xFFFFFFFFu, mine && (g[j].y >= g[j].x) != (f[j].y >= f[j].x));
                        } else {
                            const StepC sc = __ldg(prm.stepc + t[j]);
                            int was = 0, hb = 0;
                            if constexpr (GROW) {
                                const uint32_t born = c.rec()[96 + id[j]].w;
                                was = (int)c.hb()[t[j]];
                                hb = was + (lane != 0u && ((born >> lane) & 1u) ? (born & 1u ? 1 : -1) : 0);
                                __syncwarp();
                                if (mine) c.hb()[t[j]] = (uint32_t)hb;
                            }
                            const uint32_t turn = mine ? term_leads(g[j], hb, sc, prm.K) ^ term_leads(f[j], was, sc, prm.K) : 0u;
                            lturn = __ballot_sync(0xFFFFFFFFu, turn & 1u);
                            oturn = __ballot_sync(0xFFFFFFFFu, turn & 2u);
                            iturn = __ballot_sync(0xFFFFFFFFu, turn & 4u);
                        }
                        if (!sw) {                                // a flip: occupancy and the full-step bitmap
                            const uint2 e = *reinterpret_cast<const uint2*>(c.rec() + 96 + id[j]);
                            const bool in = (e.x >> lane) & 1u;
                            uint32_t o = c.occ()[t[j]];
                            const bool was = o == prm.cap;
                            o += (e.y >> lane) & 1u ? 1u : 0xFFFFFFFFu;
                            if (in) c.occ()[t[j]] = (Occ)o;
                            fturn = __ballot_sync(0xFFFFFFFFu, in && was != (o == prm.cap));
                        }
                        if (PSMEM) {
                            if (lane < (sw ? 4u : 2u)) {          // two words of u, two of v
                                const uint32_t part = lane & 1u ? r.w : r.z;
                                if (part) P[(lane & 2u ? r.y : r.x) * S32 + (bit0 >> 5) + (lane & 1u)] ^= part;
                            }
                        } else if (prm.cow_shift == 0 && S32 <= 16) {
                            // a bucket is a column: half a warp takes it over and rewrites it in one go
                            const uint32_t unit = lane & 16u ? r.y : r.x, k = lane & 15u, off = k - (bit0 >> 5);
                            const uint32_t part = off == 0u ? r.z : off == 1u ? r.w : 0u;
                            const bool owned = (c.have()[unit >> 5] >> (unit & 31u)) & 1u;
                            uint32_t* const p = P + (size_t)unit * S32 + k;
                            if (k < S32 && (lane < 16u || sw)) {
                                if (!owned) *p = __ldg(prm.Pcol0 + (size_t)unit * S32 + k) ^ part;
                                else if (part) atomicXor(p, part);   // not waited for
                            }
                            __threadfence_block();
                            __syncwarp();
                            if (!owned && (lane == 0 || (lane == 16 && sw))) atomicOr(c.have() + (unit >> 5), 1u << (unit & 31u));
                        } else {
                            own(r.x);
                            if (sw) own(r.y);
                            if (lane < (sw ? 4u : 2u)) {
                                const uint32_t part = lane & 1u ? r.w : r.z;
                                if (part) atomicXor(P + (size_t)(lane & 2u ? r.y : r.x) * S32 + (bit0 >> 5) + (lane & 1u), part);
                            }
                        }
                        Applied a;
                        a.steps = b0 | bend << 16;
                        a.units = (r.x & 0xFFFFu) | r.y << 16;
                        a.bits = a.fulls = 0xFFFFu;
                        if (lturn | fturn | oturn | iturn) {
                            const uint32_t sh = bit0 & 31u, x0 = lane < 2 ? lturn : lane < 4 || LIN ? fturn : lane < 6 ? oturn : iturn, x = b0 ? x0 : x0 >> 1;
                            const uint32_t part = lane & 1u ? (sh ? x >> (32u - sh) : 0u) : x << sh;
                            if (lane < (LIN ? 4u : 8u) && part)
                                (lane < 2 ? c.lead() : lane < 4 || LIN ? c.full() : lane < 6 ? c.out() : c.in())[(bit0 >> 5) + (lane & 1u)] ^= part;
                            lturn |= oturn | iturn;
                            if (lturn) a.bits = (b0 + __ffs(lturn) - 2u) | (b0 + 30u - __clz(lturn)) << 16;
                            if (fturn) a.fulls = (b0 + __ffs(fturn) - 2u) | (b0 + 30u - __clz(fturn)) << 16;
                        }
                        __syncwarp();
                        const uint64_t mb = m + id[j];
                        if (SOLO) {
                            cur = after;
                            ++n_chg;
                            if (leaving) unsaved = false;
                            hash = (hash ^ mb) * 0x9E3779B97F4A7C15ull + after;
                            if (after < best) { best = after; best_move = mb; unsaved = true; }
                        } else {
                            if (lane == 0) record(prm, c.sc(), mb, after, leaving, a, slot);
                            __syncwarp();
                        }
                        first = min(first, b0); last = max(last, bend);
                        if (mark(a)) { marked = true; break; }
                    }
                    if (marked) break;
                }
                if (!(prep | check) && !(__ballot_sync(0xFFFFFFFFu, !none && !bad && !rejected) & pend)) break;
            }
            if (over) break;
            n_same += lane < nb && none ? 1u : 0u;
            n_inf += lane < nb && bad ? 1u : 0u;
            if (W > 1) {                                          // hand the chain to the owner of the next batch
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    if (!(prm.drop_first_turn && base + bi == 0)) st_volatile_u32(&c.sc()->turn, base + bi + 1u);
                }
            }
        }
        if (__any_sync(0xFFFFFFFFu, (n_same | n_inf) >> 31)) {    // the lanes' counters are emptied before they run over
            atomicAdd(reinterpret_cast<unsigned long long*>(&c.sc()->n_same), (unsigned long long)n_same);
            atomicAdd(reinterpret_cast<unsigned long long*>(&c.sc()->n_inf), (unsigned long long)n_inf);
            n_same = n_inf = 0u;
        }
        if (fused && level + 1 < prm.seg1) {
            if (SOLO && active && lane == 0) c.sc()->cur = cur;
            __syncthreads();                                      // every chain of the CTA has done its round
            exchange_round(c, s_holder, stride, cpb, level);
            __syncthreads();
            if (active && sub == 0 && lane == 0)
                prm.rung_hist[(size_t)(level + 1) * prm.hist_stride + (chain - prm.hist_base)] = (uint8_t)c.sc()->rung;
        }
    }
    if (!active || silent) return;
    // every warp adds what it counted; the last one to leave reports for the chain
    atomicAdd(reinterpret_cast<unsigned long long*>(&c.sc()->n_same), (unsigned long long)n_same);
    atomicAdd(reinterpret_cast<unsigned long long*>(&c.sc()->n_inf), (unsigned long long)n_inf);
    if (SOLO && lane == 0) {
        c.sc()->cur = cur; c.sc()->best = best; c.sc()->best_move = best_move; c.sc()->hash = hash; c.sc()->n_chg = n_chg; c.sc()->snap_dirty = unsaved ? 1u : 0u;
    }
    uint32_t done = 0u;
    __threadfence_block();
    __syncwarp();
    if (lane == 0) done = atomicAdd(&c.sc()->left, 1u) == W - 1u ? 1u : 0u;
    if (!__shfl_sync(0xFFFFFFFFu, done, 0)) return;
    __threadfence_block();
    if (lane == 0) {
        kvp_chain_result res;
        res.best_ticks = c.sc()->best; res.best_move = c.sc()->best_move; res.final_ticks = c.sc()->cur;
        res.moves_done = c.sc()->m_end ? c.sc()->m_end : min(prm.upto, exchange ? prm.move0 + prm.seg1 * prm.seg_len : ~(uint64_t)0);
        res.n_accepted = c.sc()->n_same + c.sc()->n_chg; res.n_changed = c.sc()->n_chg; res.n_infeasible = c.sc()->n_inf; res.traj_hash = c.sc()->hash;
        prm.results[chain - prm.result_base] = res;
        if (prm.n_exchanged) prm.n_exchanged[chain - prm.hist_base] = c.sc()->n_exchanged;
        c.sc()->turn = 0u; c.sc()->napplied = 0u; c.sc()->left = 0u;   // the hand-over of a chain taken up again starts anew
    }
    __syncwarp();
    if (prm.state) {                                              // the next round goes on from here
        uint32_t* const saved = reinterpret_cast<uint32_t*>(prm.state + (size_t)(chain - prm.hist_base) * prm.state4);
        copy_words_cold(saved, c.template at<uint32_t>(cb), prm.lay.work / 4, lane);
        if (PSMEM) copy_words_cold(saved + prm.lay.work / 4, P, pwords, lane);
    }
    if (prm.snap && c.sc()->snap_dirty) copy_words_cold(prm.snap + (size_t)slot * pwords, P, pwords, lane);
    if (prm.undo_log && lane == 0) prm.undo_len[slot] = c.sc()->ulen;
    if (!PSMEM && prm.cow_out)                                       // which buckets the slice holds (for the walk back)
        for (uint32_t i = lane; i < o4 * 4; i += 32) prm.cow_out[(size_t)slot * (o4 * 4) + i] = c.have()[i];
    if (prm.dump && slot == 0) {
        if (!PSMEM) copy_merged(prm.dump, P, prm.Pcol0, c.have(), prm.cow_shift, U, S32, lane);
        else copy_words_cold(prm.dump, P, pwords, lane);
    }
}

}  // namespace

}  // namespace kvp
