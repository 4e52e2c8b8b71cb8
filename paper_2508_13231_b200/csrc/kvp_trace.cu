// Trace kernels: synthetic importance per unit and step, top-k per (layer, kv-head) group, packed into uint32
// bitmaps. Two passes by default: the first writes a score matrix (large traces: a thread per unit walks the steps;
// small ones: the draws in parallel over units and steps, the AR(1) recurrence, sequential in time, by one lane per
// unit); then one CTA per (group, step) finds the k-th largest score: the first eight bits of its range by a
// shared-memory histogram, the rest by ranking the keys of that bin, ties going to the lower unit index. A fused single-pass form
// (one CTA per group walking the steps, state in registers) serves layered or growing traces and those whose score
// matrix would exceed the scratch budget.
#include "kvp_common.cuh"

namespace kvp {

namespace {

struct TraceK {
    uint32_t groups, n, steps, topk, W32;
    PhiloxKeys keys;         // round keys of the seed
    int32_t rho_q, c_q, sigma_q, burst_jump;
    uint32_t burst_thr;
    const int32_t* base;
    uint32_t* out;
    int aligned;             // n % 32 == 0: whole output words belong to one group
    uint32_t layers;         // >= 1; step t belongs to token t / layers and layer t % layers
    uint32_t per_layer;      // groups per layer
    const uint32_t* birth;   // or null: unit u can be read from step birth[u] on
};

// Irwin-Hall(8) noise with unit variance in Q16.16: the sum of the eight 16-bit halves of one Philox block, centred
// and scaled by floor(sum * 80265 / 2^16). |result| <= 321,057. The operands are shifted up by 12 and 4 bits so that the
// floor is the high word of a 32-bit product: a 64-bit product and a shift take twice the multiplier's time, which is
// what the score kernels wait for.
__device__ __forceinline__ int32_t noise_q16(const PhiloxKeys& keys, uint32_t u, uint32_t t)
{
    uint32_t r[4];
    philox4x32_10(u, t, 0u, TAG_NOISE, keys, r);
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) sum = __dp2a_lo(r[i], 0x0101u, sum);      // + low half + high half
    return __mulhi(((int32_t)sum - 262140) * 4096, 80265 * 16);
}

// Sum of a per-thread value over the CTA; every thread gets the result. slot: one of 32 shared counters.
__device__ __forceinline__ uint32_t block_sum(uint32_t v, uint32_t* slot)
{
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(slot, v);
    __syncthreads();
    return *slot;
}

constexpr int kDigitBits = 8;                        // the search fixes this many bits of the threshold per pass
constexpr int kBins = 1 << kDigitBits;
constexpr uint32_t kListCap = 256;                   // a threshold bin of up to this many keys is finished by ranking
constexpr int32_t kNoKey = INT32_MIN;                // a slot without a unit; no score has this value

struct SelectSmem {
    alignas(16) uint32_t hist[kBins];            // how many keys with the threshold's higher bits have each digit
    uint32_t cnt[4];                 // block-wide counts beside the search ([1]: keys in `list`)
    int32_t list[kListCap];          // the keys of the threshold's bin after the first pass
    uint32_t warp[32];
    uint32_t run;
    int32_t hi, lo;                  // largest key of the step, and a lower bound of the k-th largest
    int32_t K;                       // lower edge of the threshold's bin, at last the threshold
    uint32_t need, equal;            // how many keys are still to find in that bin, and how many it holds
};

// State of one selection; a barrier must follow before select_step.
__device__ __forceinline__ void select_reset(SelectSmem& sm)
{
    for (uint32_t i = threadIdx.x; i < kBins; i += blockDim.x) sm.hist[i] = 0;
    if (threadIdx.x < 4) sm.cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) { sm.hi = INT32_MIN; sm.lo = INT32_MAX; }
}

// Top-k of one (group, step): the CTA holds the n keys (UPT per thread, unit i = j*T + tid, kNoKey past n) and sets the
// bits of the k largest, ties to the lower unit index. select_reset and a barrier come first.
// topk: how many to pick (at most the number of keys other than kNoKey).
//
// What bounds it: instructions per key, then the latency of the barriers. So keys that cannot be picked are dropped first.
// Every warp looks at the largest key of each lane and finds, by six ballots, a value that `want` = ceil(k / warps) of them
// reach; the smallest such value over the warps is reached by at least k keys of the step, so the k-th largest is not
// below it. (Where that would take more than 24 of the 32 lanes, `want` is 0 and the bound is the smallest key; so it is with
// fewer than eight keys per thread, where the search costs more than it saves: 411 groups of 268 units 171 against 161 us.) Keys from
// the bound up, about 9% of them at k = 5%, are counted per digit of (key - bound) in a shared-memory histogram, one
// warp walks it from the top until the counts reach what is needed, and the keys of the bin found there, a few, are
// ranked against each other. A bin with many keys (ties) takes more histogram passes, eight bits each.
// 640 groups of 4096 units x 64 steps, 205 picked: 323 us with every key in the histogram and eight keys per thread, 240 now.
// Groups that do not begin at a word set their bits by two atomics per 32 units (123 groups of 2326 units x 106 steps, the whole
// call: 166 us, 273 when they took the way of the ties, 186 with an atomic per bit).
// FULL: the CTA's UPT * T slots are exactly the n units, so no slot needs a bounds test.
template <int UPT, bool FULL = false>
__device__ __forceinline__ void select_step(const int32_t (&key)[UPT], const TraceK& k, uint32_t want, uint32_t topk, uint32_t gbase,
                                            uint32_t t, SelectSmem& sm)
{
    const uint32_t T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        int32_t mine = key[0];
#pragma unroll
        for (int j = 1; j < UPT; ++j) mine = max(mine, key[j]);
        const int32_t mx = __reduce_max_sync(0xFFFFFFFFu, mine);
        int32_t bound;
        if (UPT >= 8 && want) {
            const int32_t mn = __reduce_min_sync(0xFFFFFFFFu, mine);
            const uint32_t d = (uint32_t)mine - (uint32_t)mn;
            const int shift = max(26 - __clz((uint32_t)mx - (uint32_t)mn), 0);
            uint32_t x = 0;
#pragma unroll
            for (int i = 5; i >= 0; --i) {
                const uint32_t trial = x + (1u << (i + shift));
                if (__popc(__ballot_sync(0xFFFFFFFFu, d >= trial)) >= want) x = trial;
            }
            bound = (int32_t)((uint32_t)mn + x);
        } else {
            bound = INT32_MAX;
#pragma unroll
            for (int j = 0; j < UPT; ++j)
                if (FULL || j * T + tid < k.n) bound = min(bound, key[j]);
            bound = __reduce_min_sync(0xFFFFFFFFu, bound);
        }
        if (lane == 0) { atomicMax(&sm.hi, mx); atomicMin(&sm.lo, bound); }
    }
    __syncthreads();
    int32_t K = sm.lo;
    int rem = 32 - __clz((uint32_t)sm.hi - (uint32_t)K);     // bits still open; 0 when all these keys are equal
    uint32_t need = topk, equal = ~0u;                        // one value only: ties, if there is any key
    for (int pass = 0; rem > 0; ++pass) {
        const int sh = rem < kDigitBits ? 0 : rem - kDigitBits;
        if (pass) {
            for (uint32_t i = tid; i < kBins; i += T) sm.hist[i] = 0;
            __syncthreads();
        }
        // one predicated instruction per key, no branch: d >> sh stays inside the histogram for the keys that count
        const uint32_t hist = (uint32_t)__cvta_generic_to_shared(sm.hist), span = rem < 32 ? (1u << rem) - 1u : ~0u;
#pragma unroll
        for (int j = 0; j < UPT; ++j) {
            const uint32_t d = (uint32_t)key[j] - (uint32_t)K;   // keys below K wrap; the pass's range is cut at span
            const uint32_t in = (FULL || j * T + tid < k.n) && key[j] >= K && d <= span;
            asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p red.shared.add.u32 [%1], 1; }" :: "r"(in), "r"(hist + (d >> sh) * 4u) : "memory");
        }
        __syncthreads();
        if (warp == 0) {
            // a lane owns kOwn neighbouring digits; suffix sums over the lanes, then over the owner's bins
            constexpr uint32_t kOwn = kBins / 32;
            uint32_t h[kOwn], s = 0;
#pragma unroll
            for (uint32_t i = 0; i < kOwn; ++i) { h[i] = sm.hist[kOwn * lane + i]; s += h[i]; }
            uint32_t suf = s;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t v = __shfl_down_sync(0xFFFFFFFFu, suf, off);
                if (lane + off < 32) suf += v;
            }
            const uint32_t reach = __ballot_sync(0xFFFFFFFFu, suf >= need);    // never empty: the counts add up to >= need
            if (lane == 31u - __clz(reach)) {
                uint32_t higher = suf - s;
#pragma unroll
                for (int i = kOwn - 1; i >= 0; --i) {
                    if (higher + h[i] >= need) {
                        sm.K = (int32_t)((uint32_t)K + ((kOwn * lane + i) << sh));
                        sm.need = need - higher;
                        sm.equal = h[i];
                        break;
                    }
                    higher += h[i];
                }
            }
        }
        __syncthreads();
        K = sm.K; need = sm.need; equal = sm.equal;
        rem = sh;
        if (pass == 0 && rem > 0 && equal <= kListCap) {
            // The first digit's bin usually holds a few keys: they go to a shared list and each is ranked against
            // the others, which settles the remaining bits at once.
            uint32_t least = ~0u;
#pragma unroll
            for (int j = 0; j < UPT; ++j)
                if (FULL || j * T + tid < k.n) least = min(least, (uint32_t)key[j] - (uint32_t)K);
            if (least >> rem == 0u) {
#pragma unroll
                for (int j = 0; j < UPT; ++j)
                    if ((FULL || j * T + tid < k.n) && ((uint32_t)key[j] - (uint32_t)K) >> rem == 0u)
                        sm.list[atomicAdd(&sm.cnt[1], 1u)] = key[j];
            }
            __syncthreads();
            for (uint32_t c = tid; c < equal; c += T) {
                const int32_t v = sm.list[c];
                uint32_t above = 0, same = 0;
                for (uint32_t i = 0; i < equal; ++i) {
                    const int32_t x = sm.list[i];
                    above += x > v ? 1u : 0u;
                    same += x == v ? 1u : 0u;
                }
                if (above < need && need <= above + same) {   // v is the need-th largest; equal keys write the same
                    sm.K = v; sm.need = need - above; sm.equal = same;
                }
            }
            __syncthreads();
            K = sm.K; need = sm.need; equal = sm.equal;
            rem = 0;
        }
    }
    const uint32_t take = need;                              // ties to admit, lowest unit index first
    const bool rank_ties = equal != take;                    // and when all keys from the bound up are equal
    uint32_t* row = k.out + (size_t)t * k.W32;
    if (!rank_ties) {                                        // the usual case, kept apart so that its loop stays small
        uint32_t word = 0;                                   // lane j keeps and stores round j's word
#pragma unroll
        for (int j = 0; j < UPT; ++j) {
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, (FULL || j * T + tid < k.n) && key[j] >= K);
            if (lane == (uint32_t)j) word = bits;
        }
        const uint32_t i = lane * T + (tid & ~31u);
        if (lane < UPT && (FULL || i < k.n)) {
            uint32_t* const to = row + ((gbase + i) >> 5);
            const uint32_t sh = (gbase + i) & 31u;
            if (k.aligned) {
                *to = word;
            } else {                                         // its bits in two words of the row, which groups share
                if (word << sh) atomicOr(to, word << sh);
                if (sh && word >> (32u - sh)) atomicOr(to + 1, word >> (32u - sh));
            }
        }
        return;
    }
    if (tid == 0) sm.run = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < UPT; ++j) {
        const uint32_t i = j * T + tid;
        const bool ok = FULL || i < k.n;
        const bool tie = ok && key[j] == K;
        // units of round j are consecutive over the CTA, so index order = (round, thread) order
        const uint32_t tb = __ballot_sync(0xFFFFFFFFu, tie);
        if (lane == 0) sm.warp[warp] = __popc(tb);
        __syncthreads();
        uint32_t before = sm.run;
        for (uint32_t w = 0; w < warp; ++w) before += sm.warp[w];
        before += __popc(tb & ((1u << lane) - 1u));
        const bool pick = (ok && key[j] > K) || (tie && before < take);
        __syncthreads();
        if (tid == 0) { uint32_t s = 0; for (uint32_t w = 0; w < (T >> 5); ++w) s += sm.warp[w]; sm.run += s; }
        __syncthreads();
        if (k.aligned) {
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, pick);
            if (lane == 0 && (FULL || j * T + (tid & ~31u) < k.n)) row[(gbase + j * T + tid) >> 5] = bits;
        } else if (pick) {
            atomicOr(row + ((gbase + i) >> 5), 1u << ((gbase + i) & 31));
        }
    }
}

// ceil(k / warps), if the lanes' largest keys can bound the k-th largest that way, else 0. From 25 of 32 lanes on the
// bound lies so low that it would keep a third of the keys.
__host__ __device__ __forceinline__ uint32_t select_want(uint32_t topk, uint32_t threads)
{
    const uint32_t warps = threads / 32, want = (topk + warps - 1) / warps;
    return want <= 24u ? want : 0u;
}

// importance of unit u at step t given its state at t-1 (Q16.16). The 64-bit sum of the two 32x32 products is
// shifted and then cut to 32 bits (the range check on the host keeps the true value inside them).
template <bool BURST>
__device__ __forceinline__ int32_t next_state(const TraceK& k, uint32_t u, uint32_t t, int32_t x)
{
    const int32_t e = noise_q16(k.keys, u, t);
    const int64_t acc = t == 0 ? (int64_t)k.sigma_q * e : (int64_t)k.rho_q * x + (int64_t)k.c_q * e;
    int32_t xn = (int32_t)(acc >> 16);
    if (BURST && k.burst_thr) {
        uint32_t r[4];
        philox4x32_10(u, t, 0u, TAG_BURST, k.keys, r);
        if (r[0] < k.burst_thr) xn += k.burst_jump;
    }
    return xn;
}

// Fused form: one CTA per group walks the steps; used when the score matrix would not fit the scratch budget.
// Two CTAs per SM (at most 32 registers per thread): one CTA's barriers in the search hide behind the other's work.
// GROW: units have birth steps; one that is not there yet gets kNoKey and is never picked.
template <int UPT, bool GROW>
__global__ void __launch_bounds__(1024, 2)
trace_kernel(const TraceK k)
{
    __shared__ SelectSmem sm;
    const uint32_t g = blockIdx.x, T = blockDim.x, tid = threadIdx.x;
    const uint32_t gbase = g * k.n;
    int32_t x[UPT], b[UPT];
#pragma unroll
    for (int j = 0; j < UPT; ++j) {
        const uint32_t i = j * T + tid;
        x[j] = 0;
        b[j] = (i < k.n && k.base) ? __ldg(k.base + gbase + i) : 0;
    }
    // the group reads at the steps of its layer, one per token
    const uint32_t layer = g / k.per_layer;
    uint32_t born[GROW ? UPT : 1];
    if (GROW) {
#pragma unroll
        for (int j = 0; j < (GROW ? UPT : 1); ++j) {
            const uint32_t i = j * T + tid;
            born[j] = i < k.n ? __ldg(k.birth + gbase + i) : 0u;
        }
    }
    const uint32_t want = UPT >= 8 ? select_want(k.topk, T) : 0u;
    for (uint32_t tok = 0, t = layer; t < k.steps; ++tok, t += k.layers) {
        select_reset(sm);
        int32_t key[UPT];
        uint32_t here = 0;
#pragma unroll
        for (int j = 0; j < UPT; ++j) {
            const uint32_t i = j * T + tid;
            key[j] = kNoKey;
            if (i < k.n) {
                x[j] = next_state<true>(k, gbase + i, tok, x[j]);
                if (!GROW || born[GROW ? j : 0] <= t) {
                    key[j] = x[j] + b[j];
                    ++here;
                }
            }
        }
        __syncthreads();
        uint32_t topk = k.topk;
        if (GROW) topk = min(topk, block_sum(here, &sm.cnt[0]));
        select_step<UPT>(key, k, want, topk, gbase, t, sm);
        __syncthreads();
    }
}

// Two-pass form, pass 1: scores [steps][U]. The random draws of a (unit, step) pair depend on nothing else, only the
// AR(1) recurrence is sequential in time. A CTA owns 32 consecutive units and walks the steps in segments: all its
// threads draw the segment's noise (and burst decisions) into shared memory, then one warp, a lane per unit, runs
// the recurrence over the segment and writes 128 contiguous bytes per step. 256 threads: while the one warp runs
// the recurrence the others wait, so smaller CTAs waste less (640 x 4096 units x 64 steps: 0.95 ms with 512, 0.85 with 256).
constexpr uint32_t kScoreSeg = 256, kScoreThreads = 256;

__global__ void __launch_bounds__(kScoreThreads)
trace_scores_kernel(const TraceK k, uint32_t U, int32_t* __restrict__ scores)
{
    __shared__ int32_t draw[kScoreSeg][32];              // noise << 1 | burst
    const uint32_t u0 = blockIdx.x * 32, tid = threadIdx.x;
    const uint32_t ul = tid & 31, u = u0 + ul;
    int32_t x = 0, b = 0;
    if (tid < 32 && u < U && k.base) b = __ldg(k.base + u);
    for (uint32_t t0 = 0; t0 < k.steps; t0 += kScoreSeg) {
        const uint32_t len = min(kScoreSeg, k.steps - t0);
        for (uint32_t tt = tid >> 5; tt < len; tt += kScoreThreads / 32) {
            if (u < U) {
                int32_t d = noise_q16(k.keys, u, t0 + tt) * 2;
                if (k.burst_thr) {
                    uint32_t r[4];
                    philox4x32_10(u, t0 + tt, 0u, TAG_BURST, k.keys, r);
                    d |= r[0] < k.burst_thr ? 1 : 0;
                }
                draw[tt][ul] = d;
            }
        }
        __syncthreads();
        if (tid < 32 && u < U) {
            for (uint32_t tt = 0; tt < len; ++tt) {
                const int32_t d = draw[tt][ul], e = d >> 1;
                const uint32_t t = t0 + tt;
                const int64_t acc = t == 0 ? (int64_t)k.sigma_q * e : (int64_t)k.rho_q * x + (int64_t)k.c_q * e;
                x = (int32_t)(acc >> 16);
                if (d & 1) x += k.burst_jump;
                scores[(size_t)t * U + u] = x + b;
            }
        }
        __syncthreads();
    }
}

// Pass 1 for traces of many units: a thread per unit walks the steps, draws and recurrence together, and the threads
// of a warp write 128 contiguous bytes per step. No shared memory and no barrier; the draws of later steps do not
// depend on the state, so the loop, unrolled four times, overlaps their Philox chains with the
// recurrence. It needs about a
// thousand units per SM to fill the machine, which is why fewer units take the segmented kernel above.
template <bool BURST>
__global__ void __launch_bounds__(256)
trace_scores_unit_kernel(const TraceK k, uint32_t U, int32_t* __restrict__ scores)
{
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= U) return;
    const int32_t b = k.base ? __ldg(k.base + u) : 0;
    int32_t x = 0;
#pragma unroll 4
    for (uint32_t t = 0; t < k.steps; ++t) {
        x = next_state<BURST>(k, u, t, x);
        scores[(size_t)t * U + u] = x + b;
    }
}

// Two-pass form, pass 2: the top-k selections of different steps are independent: one CTA per (group, step).
template <int UPT, bool FULL>
__global__ void __launch_bounds__(512, 3)
trace_select_kernel(const TraceK k, uint32_t want, uint32_t U, const int32_t* __restrict__ scores)
{
    __shared__ SelectSmem sm;
    const uint32_t g = blockIdx.x, t = blockIdx.y, T = blockDim.x, tid = threadIdx.x;
    const uint32_t gbase = g * k.n;
    select_reset(sm);
    int32_t key[UPT];
    const int32_t* from = scores + (size_t)t * U + gbase + tid;
#pragma unroll
    for (int j = 0; j < UPT; ++j) key[j] = (FULL || j * T + tid < k.n) ? __ldcs(from + j * T) : kNoKey;
    __syncthreads();
    select_step<UPT, FULL>(key, k, want, k.topk, gbase, t, sm);
}

}  // namespace

}  // namespace kvp

using namespace kvp;

extern "C" int kvp_trace_generate(const kvp_trace_params* tp, uint32_t* access_bitmaps, void* stream)
{
    if (!tp || !access_bitmaps || !tp->groups || !tp->units_per_group || !tp->steps || (tp->flags & ~KVP_TRACE_SINGLE_PASS))
        return KVP_ERR_ARG;
    if (!tp->topk || tp->topk > tp->units_per_group) return KVP_ERR_ARG;
    if (tp->reserved || (tp->layers > 1 && tp->groups % tp->layers)) return KVP_ERR_ARG;
    if (tp->rho_q < 0 || tp->rho_q > 65536 || tp->c_q < 0 || tp->c_q > (1 << 20) || tp->sigma_q < 0 ||
        tp->sigma_q > (1 << 20))
        return KVP_ERR_ARG;
    const uint64_t U64 = (uint64_t)tp->groups * tp->units_per_group;
    if (U64 >= (1ull << 26) || tp->units_per_group > 8192 || tp->steps > 32768) return KVP_ERR_RANGE;
    // |score| must stay below 2^31: bound |x_t| by its worst case, step by step (|base| <= 2^29 is the caller's)
    {
        const int64_t emax = (((int64_t)262140 * 80265) >> 16) + 1;
        const int64_t jump = tp->burst_thr ? (tp->burst_jump < 0 ? -(int64_t)tp->burst_jump : tp->burst_jump) : 0;
        int64_t bound = (((int64_t)tp->sigma_q * emax) >> 16) + 1 + jump;
        for (uint32_t t = 1; t < tp->steps && bound < (1ll << 30); ++t)
            bound = (((int64_t)tp->rho_q * bound + (int64_t)tp->c_q * emax) >> 16) + 1 + jump;
        if (bound >= (1ll << 30)) return KVP_ERR_RANGE;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    TraceK k;
    k.groups = tp->groups; k.n = tp->units_per_group; k.steps = tp->steps; k.topk = tp->topk;
    k.W32 = (uint32_t)((U64 + 31) / 32);
    k.keys = philox_keys((uint32_t)tp->seed, (uint32_t)(tp->seed >> 32));
    k.rho_q = tp->rho_q; k.c_q = tp->c_q; k.sigma_q = tp->sigma_q; k.burst_jump = tp->burst_jump;
    k.burst_thr = tp->burst_thr; k.base = tp->base; k.out = access_bitmaps;
    k.aligned = tp->units_per_group % 32 == 0;
    k.layers = tp->layers ? tp->layers : 1u;
    k.per_layer = tp->groups / k.layers;
    k.birth = tp->birth;
    const bool layered = k.layers > 1 || k.birth;        // rows of other layers' steps stay zero
    if (!k.aligned || layered) KVP_CUDA(cudaMemsetAsync(access_bitmaps, 0, (size_t)tp->steps * k.W32 * 4, st));
    const uint32_t n = tp->units_per_group;
    const int upt = n <= 1024 ? 1 : n <= 2048 ? 2 : n <= 4096 ? 4 : 8;
    uint32_t T = (n + upt - 1) / upt;
    T = (T + 31) / 32 * 32;
    // Two passes (scores, then one CTA per (group, step)) whenever the score matrix fits a 1 GiB scratch: the work
    // then comes in tens of thousands of equal pieces, while the fused kernel has only `groups` CTAs that walk the
    // steps one after the other (measured: 0.84 vs 0.89 ms on 256 groups of 2048, 1.85 vs 2.11 ms on 640 of 4096,
    // 0.05 vs 2.1 ms on one group of 256). One launch with CTAs of both kinds, selecting from the chunk of steps before, was
    // slower than two after each other (1.10 against 0.99 ms on 640 of 4096): the kinds crowd each other out of registers and
    // instruction cache.
    const size_t score_bytes = (size_t)U64 * tp->steps * 4;
    if (score_bytes <= ((size_t)1 << 30) && !(tp->flags & KVP_TRACE_SINGLE_PASS) && !layered) {
        int32_t* scores = nullptr;
        int dev = 0;
        KVP_CUDA(cudaGetDevice(&dev));
        int prc = retain_in_pool(dev, score_bytes);          // the next call gets the block back from the pool
        if (prc) return prc;
        KVP_CUDA(cudaMallocAsync(&scores, score_bytes, st));
        const uint32_t U = (uint32_t)U64;
        if (U >= 148u * 1024u) {
            if (k.burst_thr) trace_scores_unit_kernel<true><<<(U + 255) / 256, 256, 0, st>>>(k, U, scores);
            else trace_scores_unit_kernel<false><<<(U + 255) / 256, 256, 0, st>>>(k, U, scores);
        } else {
            trace_scores_kernel<<<(U + 31) / 32, kScoreThreads, 0, st>>>(k, U, scores);
        }
        dim3 grid(tp->groups, tp->steps);
        // Small CTAs with many units per thread: a selection is a chain of barriers and a serial histogram walk, so
        // what counts is how many of them an SM overlaps, and a key has little to do (with sixteen keys per thread 294 us, with
        // eight 330 on 640 groups of 4096 units x 64 steps; 240 with sixteen and registers for three times 512 threads).
        int su = 1;
        while (su < 16 && (n + su - 1) / su > 128) su *= 2;
        const uint32_t ST = ((n + su - 1) / su + 31) / 32 * 32, want = select_want(k.topk, ST);
        const bool full = (uint64_t)su * ST == n;             // every slot of the CTA holds a unit
#define KVP_SELECT(UPT)                                                                     \
    if (full) trace_select_kernel<UPT, true><<<grid, ST, 0, st>>>(k, want, U, scores);      \
    else trace_select_kernel<UPT, false><<<grid, ST, 0, st>>>(k, want, U, scores)
        switch (su) {
            case 1: KVP_SELECT(1); break;
            case 2: KVP_SELECT(2); break;
            case 4: KVP_SELECT(4); break;
            case 8: KVP_SELECT(8); break;
            default: KVP_SELECT(16); break;
        }
#undef KVP_SELECT
        cudaError_t le = cudaGetLastError();
        KVP_CUDA(cudaFreeAsync(scores, st));
        KVP_CUDA(le);
        return KVP_OK;
    }
    if (k.birth) {
        switch (upt) {
            case 1: trace_kernel<1, true><<<tp->groups, T, 0, st>>>(k); break;
            case 2: trace_kernel<2, true><<<tp->groups, T, 0, st>>>(k); break;
            case 4: trace_kernel<4, true><<<tp->groups, T, 0, st>>>(k); break;
            default: trace_kernel<8, true><<<tp->groups, T, 0, st>>>(k); break;
        }
    } else {
        switch (upt) {
            case 1: trace_kernel<1, false><<<tp->groups, T, 0, st>>>(k); break;
            case 2: trace_kernel<2, false><<<tp->groups, T, 0, st>>>(k); break;
            case 4: trace_kernel<4, false><<<tp->groups, T, 0, st>>>(k); break;
            default: trace_kernel<8, false><<<tp->groups, T, 0, st>>>(k); break;
        }
    }
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}
