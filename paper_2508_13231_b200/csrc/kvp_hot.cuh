// The chain kernel for chains that apply many of their moves (included by kvp_anneal.cu only): hot starts, where a fifth to
// a quarter of the proposals change the schedule. One warp per chain.
//
// An evaluation of cost changes ahead of the commits does not last there: the batched kernels evaluated every proposal two
// to three times. What lasts is what depends on a proposal's own units: 32 proposals, one per lane, are drawn and prepared
// word-parallel (windows, what the placement bits settle, the masks of hits won and lost and of migration edges), and an
// applied move spoils a later proposal's preparation only if both name a unit and a step in common, or if a step that a
// flip enters became full or free. The proposals that need it are then evaluated in move order, against the state as it is,
// a lane per step of the window; kSide of them side by side, since their steps seldom meet those of one another, and
// what bounds the chain is the latency of these dependent steps (votes, sums over the warp, shared-memory loads).
#pragma once

namespace kvp {

namespace {

#ifndef KVP_SIDE
#define KVP_SIDE 2
#endif
constexpr int kSide = KVP_SIDE;

// bytes of a chain besides its schedule: {th, te} and occupancy of every step, the full-step bitmap, the level's
// thresholds, 32 prepared proposals
__host__ __device__ inline uint32_t hot_stride(uint32_t S, uint32_t S32)
{
    return 16 * ((S + 1) / 2 + (S + 7) / 8 + (S32 + 4) / 4) + 4 * KVP_TABLE_Q + 3 * 32 * 16;
}

// LIN only (kappa_d >= kappa_k: th and te are linear in hits and migrations, see kvp_chain.cuh), no births.
template <bool ASMEM>
__global__ void __launch_bounds__(256, 1)
hot_chain_kernel(const __grid_constant__ ChainParams prm)
{
    const uint32_t lane = threadIdx.x & 31, cic = threadIdx.x >> 5, cpb = blockDim.x >> 5;
    const uint32_t slot = blockIdx.x * cpb + cic, chain = prm.chain_first + slot;
    const bool active = slot < prm.chain_count;
    const uint32_t S = prm.S, S32 = prm.S32, U = prm.U;
    const size_t pwords = (size_t)U * S32;
    char* at = chain_smem + cic * hot_stride(S, S32);
    auto take = [&](uint32_t n4) { char* p = at; at += 16 * n4; return p; };
    int2* const tt = reinterpret_cast<int2*>(take((S + 1) / 2));
    uint16_t* const occ = reinterpret_cast<uint16_t*>(take((S + 7) / 8));
    uint32_t* const full = reinterpret_cast<uint32_t*>(take((S32 + 4) / 4));   // (a column is followed by a readable word)
    uint32_t* const row = reinterpret_cast<uint32_t*>(take(KVP_TABLE_Q / 4));
    uint4* const rec = reinterpret_cast<uint4*>(at);              // [3][32] prepared proposals
    uint32_t* const pool = reinterpret_cast<uint32_t*>(chain_smem + cpb * hot_stride(S, S32));
    uint32_t* const P = pool + cic * (uint32_t)pwords;
    const uint32_t* A = prm.Acol;
    if (ASMEM) {
        uint32_t* const a_s = pool + ((cpb * (uint32_t)pwords + 3u) & ~3u);
        copy_words(a_s, prm.Acol, pwords, threadIdx.x, blockDim.x);
        A = a_s;
    }
    if (active) {
        for (uint32_t w = 0; w < S32; ++w) {
            const uint32_t t = w * 32 + lane, i = min(t, S - 1);
            const uint4 n = __ldg(prm.counters0 + i);             // {hr, mi, mo, occ}
            const StepC k = __ldg(prm.stepc + i);
            if (t < S) {
                tt[t] = make_int2((int)(k.x + prm.K.kh * n.x + prm.K.khF * (n.y + n.z)),
                                  (int)(k.w - prm.K.ke * n.x) + ext_term((int)n.y, (int)n.z, 0, k, prm.K));
                occ[t] = (uint16_t)n.w;
            }
            const uint32_t F = __ballot_sync(0xFFFFFFFFu, t < S && n.w == prm.cap);
            if (lane == 0) full[w] = F;
        }
        copy_words(P, prm.Pcol0, pwords, lane);
    }
    __syncthreads();
    if (!active) return;

    uint64_t cur = prm.init_ticks, best = cur, best_move = ~0ull, reference = cur, n_chg = 0, hash = 0;
    uint64_t n_same = 0, n_inf = 0;                               // per lane
    bool unsaved = false;                                         // the best state is the current one and not saved yet
    const int kh = (int)prm.K.kh, ke = (int)prm.K.ke, khF = (int)prm.K.khF, kdF = (int)prm.K.kdF;
    uint64_t m = 0;
    for (uint32_t level = 0; level < prm.seg1; ++level) {
        if (level > 0) {
            if (prm.early_permille && level >= prm.early_from && (reference - best) * 1000ull < reference * (uint64_t)prm.early_permille) break;
            reference = best;
        }
        const uint64_t end = level + 1 < prm.seg1 ? (level + 1) * prm.seg_len : prm.upto;
        const uint32_t shift = __ldg(prm.shifts + level);
        __syncwarp();
        copy_words(row, prm.table + (size_t)level * KVP_TABLE_Q, KVP_TABLE_Q, lane);
#pragma unroll 1
        for (; m < end; m += 32) {
            LaneMove mv;
            {
                uint32_t r[4];
                const uint64_t mine = m + lane;
                philox4x32_10((uint32_t)mine, (uint32_t)(mine >> 32), chain, TAG_MOVE, prm.keys, r);
                decode_move(r, prm.p_swap_256, prm.len_choices, S, U, mv);
            }
            const uint32_t s0 = mv.pk >> 8, len = (mv.pk >> 1) & 31u;
            const bool swap = mv.pk & 1u;
            const uint32_t run = min(len, S - s0), nl = min(len, S - 1 - s0) + 1;   // steps rewritten; affected
            const uint32_t M = ((1u << run) - 1u) << 1, Sb = ((1u << nl) - 1u) << 1;
            const WinPos wp = window_pos(s0);
            const uint32_t v = swap ? mv.v : mv.u;
            const uint32_t Au = window_at<0>(A + mv.u * S32, wp), Av = swap ? window_at<0>(A + v * S32, wp) : 0u;
            uint32_t pend = end - m >= 32 ? 0xFFFFFFFFu : (1u << (uint32_t)(end - m)) - 1u;   // not committed
            uint32_t prep = pend;                                 // to be prepared (again)
            bool none = false, bad = false;
            uint32_t survivors = 0;
#pragma unroll 1
            do {
                if (prep) {
                    const uint32_t Wu = window_at<0>(P + mv.u * S32, wp), W2 = window_at<0>(swap ? P + v * S32 : full, wp);
                    const uint32_t D = (swap ? Wu ^ W2 : 0xFFFFFFFFu) & M;   // a flip toggles every bit of the run
                    const bool mine = (prep >> lane) & 1u;
                    if (mine) {
                        none = D == 0u;                           // nothing changes: always accepted
                        bad = !swap && (~Wu & D & W2) != 0u;      // a flip may not raise a full step (Eq. 5)
                    }
                    const uint32_t Wv = swap ? W2 : 0u;
                    uint32_t Nu = Wu ^ D, Nv = swap ? Wv ^ D : 0u;
                    if (s0 == 0) {                                // the virtual step -1 follows step 0
                        Nu = (Nu & ~1u) | ((Nu >> 1) & 1u);
                        Nv = (Nv & ~1u) | ((Nv >> 1) & 1u);
                    }
                    const uint32_t hit = (Au ^ Av) & D, lost = hit & (Au ^ Nu);
                    const uint32_t eun = Nu ^ (Nu << 1), euo = Wu ^ (Wu << 1), evn = Nv ^ (Nv << 1), evo = Wv ^ (Wv << 1);
                    // migrations gained at a step: (eun + evn) - (euo + evo), as sign and two bits of the absolute value
                    const uint32_t n1 = (eun ^ evn) & Sb, n2 = eun & evn & Sb, o1 = (euo ^ evo) & Sb, o2 = euo & evo & Sb;
                    const uint32_t two = (n2 & ~(o1 | o2)) | (o2 & ~(n1 | n2)), one = n1 ^ o1;
                    const uint32_t neg = (o2 & ~n2) | (o1 & ~(n1 | n2));
                    __syncwarp();
                    if (mine) {
                        rec[lane] = make_uint4(s0, hit, lost, one);
                        rec[32 + lane] = make_uint4(two, neg, mv.w, hit | one | two);
                        rec[64 + lane] = make_uint4(mv.u * S32, v * S32, D | (swap ? 1u : 0u), Nu);   // bit 0 of D is never set
                    }
                    survivors = __ballot_sync(0xFFFFFFFFu, !none && !bad) & pend;
                    prep = 0;
                    __syncwarp();
                }
                // up to kSide of the survivors: cost changes against the present state
                int2 g[kSide];
                uint32_t id[kSide], t[kSide], chg[kSide];
                int delta[kSide];
                uint32_t rest = survivors;
#pragma unroll
                for (int j = 0; j < kSide; ++j) {
                    id[j] = rest ? __ffs(rest) - 1u : 32u;
                    rest &= rest - 1u;
                    const uint32_t k = id[j] & 31u;
                    const uint4 a = rec[k], b = rec[32 + k];
                    chg[j] = b.w;
                    t[j] = min(a.x + max(lane, 1u) - 1u, S - 1u); // lane l: window bit l, step s0 - 1 + l
                    const int2 f = tt[t[j]];
                    const int h = (a.y >> lane) & 1u, mg = (int)((a.w >> lane) & 1u) + 2 * (int)((b.x >> lane) & 1u);
                    const int hr = (a.z >> lane) & 1u ? -h : h, mm = (b.y >> lane) & 1u ? -mg : mg;
                    g[j] = make_int2(f.x + kh * hr + khF * mm, f.y - ke * hr + kdF * mm);
                    delta[j] = max(g[j].x, g[j].y) - max(f.x, f.y);   // 0 where nothing changes
                }
#pragma unroll
                for (int j = 0; j < kSide; ++j) delta[j] = __reduce_add_sync(0xFFFFFFFFu, delta[j]);
                bool ok[kSide];
#pragma unroll
                for (int j = 0; j < kSide; ++j) {
                    const uint32_t q = (uint32_t)max(delta[j], 0) >> shift;
                    ok[j] = delta[j] <= 0 || (q < KVP_TABLE_Q && rec[32 + (id[j] & 31u)].z < row[min(q, KVP_TABLE_Q - 1u)]);   // quantised exp(-delta/C)
                }
                uint32_t first = 0xFFFFu, last = 0u;              // steps rewritten by the moves applied in this group
#pragma unroll
                for (int j = 0; j < kSide; ++j) {
                    if (id[j] >= 32u) break;                      // (all of this is warp-uniform)
                    const uint4 c = rec[64 + id[j]];
                    const uint32_t b0 = rec[id[j]].x;
                    if (j > 0 && first <= last) {
                        const uint32_t e0 = min(b0 + 31u - __clz(chg[j]), S);
                        if (b0 <= last && first <= e0) break;     // its steps changed meanwhile
                    }
                    survivors &= ~(1u << id[j]);
                    pend &= 0xFFFFFFFEu << id[j];
                    if (!ok[j]) continue;
                    const uint64_t after = (uint64_t)((int64_t)cur + delta[j]);
                    if (unsaved && after >= best && prm.snap) {   // leaving the best state: save it first
                        copy_words_cold(prm.snap + (size_t)slot * pwords, P, pwords, lane);
                        unsaved = false;
                    }
                    __syncwarp();
                    if ((chg[j] >> lane) & 1u) tt[t[j]] = g[j];
                    const uint32_t Db = c.z & ~1u, bit0 = b0 ? b0 - 1u : 0u, d = b0 ? Db : Db >> 1, sh = bit0 & 31u, wd = bit0 >> 5;
                    uint32_t turned = 0u;
                    if (!(c.z & 1u)) {                            // a flip: occupancy and the full-step bitmap
                        const bool mine = (Db >> lane) & 1u;
                        uint32_t o = occ[t[j]];
                        const bool was = o == prm.cap;
                        o += (c.w >> lane) & 1u ? 1u : 0xFFFFFFFFu;
                        if (mine) occ[t[j]] = (uint16_t)o;
                        turned = __ballot_sync(0xFFFFFFFFu, mine && was != (o == prm.cap));
                    }
                    if (lane < 6) {                               // two words each of u, v and the full-step bitmap
                        const uint32_t x = lane < 4 ? d : b0 ? turned : turned >> 1;
                        const uint32_t part = lane & 1u ? (sh ? x >> (32u - sh) : 0u) : x << sh;
                        uint32_t* const p = (lane < 2 ? P + c.x : lane < 4 ? P + c.y : full) + wd + (lane & 1u);
                        if (part && (lane < 2 || lane >= 4 || (c.z & 1u))) *p ^= part;
                    }
                    __syncwarp();
                    cur = after;
                    ++n_chg;
                    const uint64_t mb = m + id[j];
                    hash = (hash ^ mb) * 0x9E3779B97F4A7C15ull + after;
                    if (after < best) { best = after; best_move = mb; unsaved = true; }
                    const uint32_t bend = b0 + 31u - __clz(Db);   // steps b0 .. bend changed bits or costs
                    first = min(first, b0); last = max(last, bend);
                    // preparations that no longer hold: a common unit and step, or a flip's step that became full or free
                    const uint32_t end_s = s0 + len;
                    const bool meets = s0 <= bend + 1u && b0 <= end_s;
                    const bool shares = mv.u * S32 == c.x || mv.u * S32 == c.y || v * S32 == c.x || v * S32 == c.y;
                    const bool flips = !swap && turned != 0u;
                    prep |= __ballot_sync(0xFFFFFFFFu, meets && (shares || flips)) & pend;
                    if (prep) break;
                }
            } while (survivors | prep);
            const bool valid = m + lane < end;
            n_same += valid && none ? 1 : 0;
            n_inf += valid && bad ? 1 : 0;
        }
        m = end;
    }
    if (prm.snap && unsaved) copy_words_cold(prm.snap + (size_t)slot * pwords, P, pwords, lane);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        n_same += __shfl_xor_sync(0xFFFFFFFFu, n_same, off);
        n_inf += __shfl_xor_sync(0xFFFFFFFFu, n_inf, off);
    }
    if (lane == 0) {
        kvp_chain_result res;
        res.best_ticks = best; res.best_move = best_move; res.final_ticks = cur; res.moves_done = m;
        res.n_accepted = n_same + n_chg; res.n_changed = n_chg; res.n_infeasible = n_inf; res.traj_hash = hash;
        prm.results[chain - prm.result_base] = res;
    }
    if (prm.dump && slot == 0) copy_words_cold(prm.dump, P, pwords, lane);
}

}  // namespace

}  // namespace kvp
