// Policy kernels: the look-ahead placement policy of Section III-B (window W, migration ratio R) for many (W, R) pairs
// at once, the comparison strategies of Section IV-A, and the paper's own annealer that walks the (W, R) grid.
//
// A policy is sequential in the steps, so what counts is the latency of one step. A warp (up to 4096 units; several
// warps of one CTA above that) holds the whole population in registers, 32 units to a word: the resident bitmap H and
// the units' keys (accesses in the window, reads of the page, time of last use) as bit planes, plane b holding bit b of
// every unit's key. Then
//   - a window slides by a bit-sliced add of the entering and the leaving access row,
//   - the k-th largest (smallest) key of a set is found from the top plane down, one popc count of the set per plane and
//     one warp reduction, which also leaves the set of units beyond the threshold and the set of ties at it,
//   - ties go by unit index: a prefix sum over the lanes, then the lowest bits of one word.
// Measured on 4096 units x 512 steps (B200): a CTA of 1024 threads with a frequency byte and a shared-memory histogram
// update per unit and one thread walking the histograms took 9.5 us per step (4.9 ms for one pair, 24.4 ms for the
// 64 x 11 grid, which is 4.8 CTAs per SM); this form is bound by the latency of its ~20 dependent reductions per step.
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

// Sums over the CTA of a packed pair of 16-bit counts (two sets of units are disjoint and hold at most 32768 units
// together, so neither field overflows). One warp: a reduction; several: one barrier, the partial sums double-buffered.
template <bool MULTI>
struct CtaSum {
    uint32_t* buf;                                       // MULTI: [2][kPolicyMaxWarps] shared
    uint32_t flip;
    __device__ __forceinline__ uint32_t operator()(uint32_t v)
    {
        v = __reduce_add_sync(0xFFFFFFFFu, v);
        if (!MULTI) return v;
        uint32_t* b = buf + (flip ^= kPolicyMaxWarps);
        if ((threadIdx.x & 31) == 0) b[threadIdx.x >> 5] = v;
        __syncthreads();
        const uint4 x = *reinterpret_cast<const uint4*>(b), y = *reinterpret_cast<const uint4*>(b + 4);
        return x.x + x.y + x.z + x.w + y.x + y.y + y.z + y.w;   // the slots of absent warps stay 0
    }
    // sum over the threads before this one (threads own ascending unit indices)
    __device__ __forceinline__ uint32_t before(uint32_t v)
    {
        const uint32_t lane = threadIdx.x & 31;
        uint32_t incl = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (lane >= (uint32_t)off) incl += o;
        }
        uint32_t base = 0;
        if (MULTI) {
            uint32_t* b = buf + (flip ^= kPolicyMaxWarps);
            if (lane == 31) b[threadIdx.x >> 5] = incl;
            __syncthreads();
            for (uint32_t w = 0; w < (threadIdx.x >> 5); ++w) base += b[w];
        }
        return base + incl - v;
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

// the r lowest set bits of w (0 < r < popc(w))
__device__ __forceinline__ uint32_t lowest_bits(uint32_t w, uint32_t r)
{
    uint32_t pos = 0;                                    // the largest cut with at most r bits below it
#pragma unroll
    for (uint32_t step = 16; step > 0; step >>= 1)
        if (__popc(w & ((1u << (pos + step)) - 1u)) <= r) pos += step;
    return w & ((1u << pos) - 1u);
}

// Leaves in m its first `take` bits in unit order, given how many bits of the set lie in the threads before this one.
template <int WPL>
__device__ __forceinline__ void first_bits(uint32_t (&m)[WPL], uint32_t before, uint32_t take)
{
    int r = (int)take - (int)before;
#pragma unroll
    for (int j = 0; j < WPL; ++j) {
        const int c = __popc(m[j]);
        if (r <= 0) m[j] = 0u;
        else if (r < c) m[j] = lowest_bits(m[j], (uint32_t)r);
        r -= c;
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

// One step of the look-ahead rule: at most `want` of the candidates move in, the best first; they take the free
// capacity, then the next ones replace residents of lower key, lowest first. H is updated; I units came in, `swaps` of
// them for a resident. kb = want less the free capacity bounds the swaps from one side, the keys from the other: m swaps
// are possible iff some threshold t has insf + m candidates with key >= t and m residents with key < t, so their number
// is the maximum over t of min(C(t) - insf, R(t)), C falling and R rising in t, reached where the two cross.
//   quota: the want-th best candidate and the kb-th lowest resident, both descents side by side; right when the first
//          key is above the second.
//   cross: the crossing, one descent over both sets; right when it gives at most kb swaps, and then its threshold cuts
//          both sets: candidates above it and residents below it move, of those at it as many as are still to move.
// Either is one count per plane. `limited` remembers which was right at the step before and goes first.
template <int WPL, int NP, bool MULTI>
__device__ __forceinline__ void exchange_units(const uint32_t (&plane)[NP][WPL], int np, const uint32_t (&cand)[WPL],
                                               uint32_t want, uint32_t free_slots, uint32_t (&H)[WPL],
                                               CtaSum<MULTI>& sum, bool& limited, uint32_t& I, uint32_t& swaps)
{
    const uint32_t insf = min(want, free_slots), kb = want - insf;
    uint32_t mc[WPL], mr[WPL], in[WPL], out[WPL], needC, needR;   // ties at the thresholds, units beyond them
    for (bool quota = limited || kb == 0;; quota = !quota) {      // two passes at most
#pragma unroll
        for (int j = 0; j < WPL; ++j) { mc[j] = cand[j]; mr[j] = H[j]; in[j] = 0u; out[j] = 0u; }
        uint32_t above = 0, below = 0, keyC = 0, keyR = 0;
        needC = want; needR = kb;
#pragma unroll
        for (int b = NP - 1; b >= 0; --b) {
            if (b >= np) continue;
            uint32_t c = 0;
#pragma unroll
            for (int j = 0; j < WPL; ++j) c += (__popc(mc[j] & plane[b][j]) << 16) + __popc(mr[j] & ~plane[b][j]);
            c = sum(c);
            const uint32_t cc = c >> 16, cr = c & 0xFFFFu;
            uint32_t tc, tr;                              // all ones: go on among the set bits (C), among the clear ones (R)
            if (quota) {
                tc = needC <= cc ? 0xFFFFFFFFu : 0u;
                tr = needR <= cr ? 0xFFFFFFFFu : 0u;
                needC -= cc & ~tc; needR -= cr & ~tr;
                keyC |= tc & (1u << b); keyR |= ~tr & (1u << b);
            } else {
                tc = above + cc >= insf + below + cr ? 0xFFFFFFFFu : 0u;
                tr = ~tc;
                above += cc & ~tc; below += cr & tc;
            }
#pragma unroll
            for (int j = 0; j < WPL; ++j) {
                const uint32_t p = plane[b][j];
                in[j] |= mc[j] & p & ~tc;
                mc[j] &= ~(p ^ tc);
                out[j] |= mr[j] & ~p & ~tr;
                mr[j] &= p ^ tr;
            }
        }
        if (quota) {
            swaps = kb;
            if (kb == 0 || keyC > keyR) break;
            limited = false;
        } else {
            swaps = max(below, above > insf ? above - insf : 0u);
            needC = insf + swaps - above; needR = swaps - below;
            if (swaps <= kb) break;
            limited = true;
        }
    }
    I = insf + swaps;
    if (!I) return;
    const uint32_t bf = sum.before((popcn(mc) << 16) + popcn(mr));
    first_bits(mc, bf >> 16, needC);
    first_bits(mr, bf & 0xFFFFu, needR);
#pragma unroll
    for (int j = 0; j < WPL; ++j) H[j] = (H[j] & ~(out[j] | mr[j])) | in[j] | mc[j];
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

template <int WPL, bool MULTI>
__global__ void __launch_bounds__(MULTI ? 32 * kPolicyMaxWarps : 32)
lookahead_kernel(const uint32_t* __restrict__ A, const uint32_t* __restrict__ row0, uint32_t S, uint32_t W32, uint32_t cap,
                 uint32_t n_ratio, const __grid_constant__ PolicyPairs pairs, uint32_t* __restrict__ out,
                 const StepC* __restrict__ stepc, CostK K, uint64_t* __restrict__ totals)
{
    __shared__ __align__(16) uint32_t s_part[2 * kPolicyMaxWarps];
    if (MULTI) {
        if (threadIdx.x < 2 * kPolicyMaxWarps) s_part[threadIdx.x] = 0u;
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
    bool limited = permille < 1000;
    uint64_t total = 0;
    uint32_t mi = 0, mo = 0, hits = 0;                   // of the step before (its hits are reduced with the next step's count)
    uint32_t enter[WPL], leave[WPL] = {}, now[WPL];      // rows s + W - 1, s - 1 and s
    load_row(A + (size_t)min(W - 1, S - 1) * W32, W <= S ? W32 : 0u, w0, enter);
    load_row(A, W32, w0, now);
    for (uint32_t s = 0; s < S; ++s) {
        // the rows of the next step are on their way while this one is worked on
        uint32_t enter2[WPL], now2[WPL];
        load_row(A + (size_t)min(s + W, S - 1) * W32, s + W < S ? W32 : 0u, w0, enter2);
        load_row(A + (size_t)min(s + 1, S - 1) * W32, W32, w0, now2);
        uint32_t cand[WPL], I = 0, swaps = 0;
        if (permille) {
            slide(plane, np, enter, leave);
#pragma unroll
            for (int j = 0; j < WPL; ++j) {
                uint32_t any = plane[0][j];
#pragma unroll
                for (int b = 1; b < kFreqPlanes; ++b) any |= plane[b][j];
                cand[j] = any & ~H[j];
            }
        } else {
#pragma unroll
            for (int j = 0; j < WPL; ++j) cand[j] = 0u;
        }
        const uint32_t both = sum((popcn(cand) << 16) + hits);
        const uint32_t nC = both >> 16;
        if (totals && s) total += step_cost(both & 0xFFFFu, mi, mo, __ldg(stepc + s - 1), K);
        const uint32_t want = nC * permille / 1000u;
        if (want) {
            exchange_units(plane, np, cand, want, cap - nR, H, sum, limited, I, swaps);
            nR += I - swaps;
        }
        mi = s ? I : 0u; mo = s ? swaps : 0u;            // the migrations of step 0 are free
        hits = 0;
#pragma unroll
        for (int j = 0; j < WPL; ++j) {
            hits += __popc(now[j] & H[j]);
            leave[j] = now[j]; now[j] = now2[j]; enter[j] = enter2[j];
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
    __shared__ __align__(16) uint32_t s_part[2 * kPolicyMaxWarps];
    if (MULTI) {
        if (threadIdx.x < 2 * kPolicyMaxWarps) s_part[threadIdx.x] = 0u;
        __syncthreads();
    }
    CtaSum<MULTI> sum{s_part, 0u};
    const uint32_t w0 = threadIdx.x * WPL;
    uint32_t H[WPL], plane[kPagePlanes][WPL], next[kPagePlanes][WPL];
    initial_row<WPL>(nullptr, EW32, w0, cap, H);
    uint32_t nR = sum(popcn(H));
    auto fetch = [&](uint32_t s) {
#pragma unroll
        for (int b = 0; b < kPagePlanes; ++b) load_row(planes + ((size_t)s * np + min(b, np - 1)) * EW32, b < np ? EW32 : 0u, w0, next[b]);
    };
    fetch(0);
    bool limited = false;
    for (uint32_t s = 0; s < S; ++s) {
        uint32_t cand[WPL], I = 0, swaps = 0;
#pragma unroll
        for (int j = 0; j < WPL; ++j) {
            uint32_t any = 0;
#pragma unroll
            for (int b = 0; b < kPagePlanes; ++b) { plane[b][j] = next[b][j]; any |= next[b][j]; }
            cand[j] = any & ~H[j];
        }
        fetch(min(s + 1, S - 1));
        const uint32_t nC = sum(popcn(cand));
        if (nC) {
            exchange_units(plane, np, cand, nC, cap - nR, H, sum, limited, I, swaps);
            nR += I - swaps;
        }
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
    __shared__ __align__(16) uint32_t s_part[2 * kPolicyMaxWarps];
    if (MULTI) {
        if (threadIdx.x < 2 * kPolicyMaxWarps) s_part[threadIdx.x] = 0u;
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
        const uint32_t both = sum((popcn(miss) << 16) + popcn(oldest));
        const uint32_t nM = both >> 16;
        uint32_t n_old = both & 0xFFFFu;
        const uint32_t promoted = min(nM, cap), free_slots = cap - nR;
        if (promoted < nM) first_bits(miss, sum.before(popcn(miss)), promoted);   // CTA-uniform
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
            n_old = sum(popcn(oldest));
            if (tau > s + 1) break;                      // never reached: the keys of the residents end at s + 1
        }
        if (evict) {                                     // CTA-uniform
            uint32_t gone[WPL];
#pragma unroll
            for (int j = 0; j < WPL; ++j) gone[j] = oldest[j];
            first_bits(gone, sum.before(popcn(gone)), evict);
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
// after it test again from there. A walk of n iterations so costs n / 32 draws plus one short round per accepted move (a
// few tests in flight at once, 0.1 us) instead of n times the latency of a draw and two lookups (0.25 us).
// TSMEM: the table is staged in shared memory. The level's acceptance row always is.
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
    __syncwarp();
    uint32_t w = k.w0, r = k.r0;
    uint64_t cur = tab[(size_t)(w - 1) * k.n_ratio + r];
    kvp_wr_result res;
    res.best_ticks = cur; res.best_w = w; res.best_r = r; res.n_accepted = 0;
    uint64_t bab = cur, i = 0;
    for (uint32_t level = 0; level < k.levels && i < k.iters; ++level) {
        if (level) {
            if (k.early_permille && (bab - res.best_ticks) * 1000ull < bab * (uint64_t)k.early_permille) break;
            bab = res.best_ticks;
        }
        __syncwarp();
        const uint4* src = reinterpret_cast<const uint4*>(k.acc + (size_t)level * KVP_TABLE_Q);
#pragma unroll
        for (uint32_t q = 0; q < KVP_TABLE_Q / 128; ++q) reinterpret_cast<uint4*>(acc)[q * 32 + lane] = __ldg(src + q * 32 + lane);
        __syncwarp();
        const uint32_t shift = __ldg(k.shifts + level);
        const uint64_t end = level + 1 < k.levels ? min(i + k.per_level, k.iters) : k.iters;
        for (; i < end; i += 32) {
            const uint64_t it = i + lane;
            uint32_t x[4];
            philox4x32_10((uint32_t)it, (uint32_t)(it >> 32), c, TAG_WR, k.seed_lo, k.seed_hi, x);
            const uint32_t sel = x[0] & 255u, d = (x[0] >> 8) & 3u;
            const int dw = sel < 102u || sel >= 204u ? (int)d - (d < 2u ? 2 : 1) : 0;   // window, diagonal: {-2, -1, 1, 2}
            const int dr = sel < 102u ? 0 : ((x[0] >> 10) & 1u) ? 1 : -1;               // ratio, diagonal
            uint32_t open = end - i >= 32 ? 0xFFFFFFFFu : (1u << (uint32_t)(end - i)) - 1u;
            for (;;) {
                const int nw = (int)w + dw, nr = (int)r + dr;
                const bool on = nw >= 1 && nw <= (int)k.w_max && nr >= 0 && nr < (int)k.n_ratio;   // off the grid: discarded
                const uint64_t cand = tab[on ? (size_t)(nw - 1) * k.n_ratio + nr : 0];
                const uint64_t q = cand <= cur ? 0 : (cand - cur) >> shift;
                const uint32_t thr = acc[min(q, (uint64_t)KVP_TABLE_Q - 1)];
                const bool accept = on && (cand <= cur || (q < KVP_TABLE_Q && x[3] < thr));        // Metropolis
                const uint32_t yes = __ballot_sync(0xFFFFFFFFu, accept) & open;
                if (!yes) break;
                const int j = __ffs(yes) - 1;
                w = __shfl_sync(0xFFFFFFFFu, (uint32_t)nw, j);
                r = __shfl_sync(0xFFFFFFFFu, (uint32_t)nr, j);
                cur = __shfl_sync(0xFFFFFFFFu, cand, j);
                ++res.n_accepted;
                if (cur < res.best_ticks) { res.best_ticks = cur; res.best_w = w; res.best_r = r; }
                open &= 0xFFFFFFFEu << j;                // the proposals after the accepted one
            }
        }
        i = end;
    }
    res.iters_done = i; res.final_ticks = cur; res.final_w = w; res.final_r = r;
    if (lane == 0) results[c] = res;
}

}  // namespace

}  // namespace kvp

using namespace kvp;

// Words per thread and threads of a policy CTA: one warp holds up to 128 words (4096 units); more warps above that.
#define KVP_POLICY(kernel, words, grid, ...)                                                                    \
    do {                                                                                                        \
        const uint32_t words_ = (words);                                                                        \
        if (words_ <= 32) kernel<1, false><<<grid, 32, 0, st>>>(__VA_ARGS__);                                   \
        else if (words_ <= 64) kernel<2, false><<<grid, 32, 0, st>>>(__VA_ARGS__);                              \
        else if (words_ <= 128) kernel<4, false><<<grid, 32, 0, st>>>(__VA_ARGS__);                             \
        else kernel<4, true><<<grid, (words_ + 127) / 128 * 32, 0, st>>>(__VA_ARGS__);                          \
        KVP_CUDA(cudaGetLastError());                                                                           \
    } while (0)

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
        if (used)
            KVP_POLICY(lookahead_kernel, p->W32, used, p->dA, row, p->S, p->W32, p->cap, 0u, pairs, schedules, p->d_stepc, p->K,
                       (uint64_t*)nullptr);
        used = 0;
        return KVP_OK;
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
    KVP_POLICY(lookahead_kernel, p->W32, w_max * n_ratio, p->dA,
               init_mode == KVP_INIT_STATIC_FREQ ? p->d_row_freq : (const uint32_t*)nullptr, p->S, p->W32, p->cap, n_ratio, none,
               (uint32_t*)nullptr, p->d_stepc, p->K, table);
    return KVP_OK;
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
