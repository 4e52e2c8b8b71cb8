// Layout kernels: bit-matrix transposes between the step-major API layout and the time-packed layout
// the annealer works on, pad-bit cleaning, per-unit access counts and the static initial placements.
#include "kvp_common.cuh"

namespace kvp {

namespace {

// 32 x 32 bit transpose in a warp's registers: lane l holds row l, afterwards lane l holds column l. Five rounds in which
// lanes l and l ^ j exchange the blocks of j x j bits on their side of the diagonal; a rotation serves both shift directions.
struct WarpTranspose {
    uint32_t mask[5];        // the bits a lane keeps in round i (j = 16 >> i)
    int rot[5];
    __device__ __forceinline__ WarpTranspose()
    {
        const uint32_t lane = threadIdx.x & 31;
        const uint32_t low[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int j = 16 >> i;
            mask[i] = lane & j ? ~low[i] : low[i];
            rot[i] = lane & j ? 32 - j : j;
        }
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const
    {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, 16 >> i);
            x = (x & mask[i]) | (__funnelshift_l(y, y, rot[i]) & ~mask[i]);
        }
        return x;
    }
};

// in: [rows][in_words] words, bit c of row r = bit (c & 31) of in[r][c >> 5].
// out: [cols][out_words], bit r of row c. Bits beyond `rows` in the last out word are 0.
//
// A CTA transposes tiles of 32 * RB rows x WB words: RB words of output side by side, WB words of input, so that both sides
// move whole 32-byte sectors also where the rows of one side are only a few words long. Bound by memory: 8 MB in and out
// (1056 x 131,072 bits) took 64 and 106 us with 32 ballots per 32 words and a word per sector on the output side.
// Strides in shared memory are odd, so lanes that walk rows or columns meet different banks.
//
// OPEN (problem construction): the input is the access bitmap as the caller passed it. The kernel also writes its copy
// with clean pad bits, adds up the accesses of every row (one shared counter per row, flushed once per CTA: grid.y is
// kept to what fills the machine, each CTA walking several tiles) and of every column (added where a column is more than
// one CTA's tile, which `ucnt_add` says). Five passes over the bitmap before: 186 us for 640 x 4096 units x 64 steps.
struct OpenArgs {
    uint32_t* copy;
    uint32_t* row_count;
    uint32_t* ucnt;
    uint32_t pad_mask;
    bool ucnt_add;
};

template <int LRB, int LWB, bool OPEN>
__global__ void __launch_bounds__(256)
bit_transpose_kernel(const uint32_t* in, uint32_t rows, uint32_t in_words, uint32_t cols,
                     uint32_t* __restrict__ out, uint32_t out_words, const OpenArgs open, const ChosenInput chosen)
{
    if (chosen.index) in = *chosen.valid == ~0ull ? chosen.otherwise : in + (size_t)*chosen.index * rows * in_words;
    constexpr uint32_t RB = 1u << LRB, WB = 1u << LWB, IS = WB | 1u, OS = RB | 1u;
    __shared__ uint32_t tin[RB * 32 * IS], tout[WB * 32 * OS];
    __shared__ uint32_t s_rows[OPEN ? RB * 32 : 1];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t r0 = blockIdx.x * RB * 32;                    // row tiles can be millions: they go in x
    const WarpTranspose transpose;
    if (OPEN)
        for (uint32_t r = tid; r < RB * 32; r += 256) s_rows[r] = 0u;
    for (uint32_t w0 = blockIdx.y * WB; w0 < in_words; w0 += gridDim.y * WB) {
#pragma unroll
        for (uint32_t n = 0; n < RB * WB / 8; ++n) {
            const uint32_t i = n * 256 + tid, r = i >> LWB, w = i & (WB - 1);
            uint32_t v = 0u;
            if (r0 + r < rows && w0 + w < in_words) {
                const size_t at = (size_t)(r0 + r) * in_words + w0 + w;
                v = __ldg(in + at);
                if (OPEN) {
                    if (w0 + w == in_words - 1) v &= open.pad_mask;
                    open.copy[at] = v;
                }
            }
            tin[r * IS + w] = v;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t n = 0; n < RB * WB / 8; ++n) {
            const uint32_t q = n * 8 + warp, b = q >> LWB, w = q & (WB - 1);
            tout[(w * 32 + lane) * OS + b] = transpose(tin[(b * 32 + lane) * IS + w]);
        }
        if (OPEN) {
            constexpr uint32_t R = RB * 32, PARTS = R < 256 ? 256 / R : 1, SPAN = WB / PARTS ? WB / PARTS : 1;
            const uint32_t r = tid % R, part = tid / R;
            if (part * SPAN < WB) {
                uint32_t n = 0;
#pragma unroll
                for (uint32_t w = 0; w < SPAN; ++w) n += __popc(tin[r * IS + part * SPAN + w]);
                if (n) atomicAdd(s_rows + r, n);
            }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t n = 0; n < RB * WB / 8; ++n) {
            const uint32_t i = n * 256 + tid, c = i >> LRB, b = i & (RB - 1);
            const uint32_t col = w0 * 32 + c, word = blockIdx.x * RB + b;
            if (col < cols && word < out_words) out[(size_t)col * out_words + word] = tout[c * OS + b];
        }
        if (OPEN) {
            for (uint32_t c = tid; c < WB * 32 && w0 * 32 + c < cols; c += 256) {
                uint32_t n = 0;
#pragma unroll
                for (uint32_t b = 0; b < RB; ++b) n += __popc(tout[c * OS + b]);
                if (!open.ucnt_add) open.ucnt[w0 * 32 + c] = n;
                else if (n) atomicAdd(open.ucnt + w0 * 32 + c, n);
            }
        }
        __syncthreads();
    }
    if (OPEN)
        for (uint32_t r = tid; r < RB * 32; r += 256)
            if (s_rows[r]) atomicAdd(open.row_count + r0 + r, s_rows[r]);
}

__global__ void clean_copy_kernel(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, size_t total,
                                  uint32_t W32, uint32_t pad_mask)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t v = in[i];
        if (i % W32 == W32 - 1) v &= pad_mask;
        out[i] = v;
    }
}

// Per-step constants of the cost function. in: [S] HBM writes of the step, then [S] external ones, or null for none.
__global__ void stepc_kernel(StepC* __restrict__ stepc, const uint32_t* __restrict__ in, const uint32_t* __restrict__ a,
                             uint32_t S, const CostK K)
{
    const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const uint32_t h = in ? in[s] : 0u, e = in ? in[S + s] : 0u;
    stepc[s] = make_uint4(K.kh * h, K.kk * e, K.kd * e, K.ke * a[s]);
}

// The `cap` most accessed units, ties to the lower index, in three launches that each read the counts once. What bounds them
// is their launch latency (2.6M units: 52 us with a CTA per 1024 units and a launch of its own for the threshold).
//
// First, a histogram of the counts (bins 0..S). Few bins and millions of units: every CTA counts its units in shared
// memory (when the bins fit) and adds only its non-empty bins to the global histogram. The last CTA then finds the
// threshold: sel = {threshold count, number of ties to take}, and with it the row's accesses over all steps (hits).
constexpr uint32_t kHistBins = 8192;
__global__ void __launch_bounds__(1024)
static_threshold_kernel(const uint32_t* __restrict__ ucnt, uint32_t U, uint32_t S, uint32_t cap, uint32_t* __restrict__ hist,
                        uint32_t* __restrict__ sel, uint32_t* __restrict__ ticket, unsigned long long* __restrict__ hits)
{
    __shared__ uint32_t local[kHistBins];
    __shared__ uint32_t s_thr, s_take, s_found, s_last;
    __shared__ uint32_t s_warp[32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, bins = S + 1;
    const bool staged = bins <= kHistBins;
    if (staged) {
        for (uint32_t b = threadIdx.x; b < bins; b += blockDim.x) local[b] = 0u;
        __syncthreads();
    }
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < U; u += gridDim.x * blockDim.x)
        atomicAdd((staged ? local : hist) + ucnt[u], 1u);
    __syncthreads();
    if (staged)
        for (uint32_t b = threadIdx.x; b < bins; b += blockDim.x)
            if (local[b]) atomicAdd(hist + b, local[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        s_thr = S + 1; s_take = 0; s_found = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // counts run 0..S; descend, 1024 counts at a time (thread i looks at count top - i), until the capacity is reached
    if (cap != 0) {
        uint32_t above = 0;                               // units with a count above this chunk
        unsigned long long got = 0;                       // accesses of the units this thread's counts contribute
        for (int64_t top = S; top >= 0; top -= 1024) {
            const int64_t c = top - (int64_t)threadIdx.x;
            const uint32_t h = c >= 0 ? __ldcg(hist + c) : 0u;
            uint32_t incl = h;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= (uint32_t)off) incl += v;
            }
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            uint32_t before = 0, total = 0;
            for (uint32_t w = 0; w < 32; ++w) {
                const uint32_t v = s_warp[w];
                before += w < warp ? v : 0u;
                total += v;
            }
            incl += before + above;
            const uint32_t excl = incl - h;
            if (c > 0 && excl < cap) got += (unsigned long long)c * (min(incl, cap) - excl);
            if (c >= 0 && excl < cap && incl >= cap) { s_thr = (uint32_t)c; s_take = cap - excl; s_found = 1; }   // one thread at most
            __syncthreads();
            if (s_found) break;
            above += total;
            __syncthreads();
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) got += __shfl_xor_sync(0xFFFFFFFFu, got, off);
        if (lane == 0 && got) atomicAdd(hits, got);
    }
    if (threadIdx.x == 0) { sel[0] = s_thr; sel[1] = s_take; }
}

// Second, every CTA counts the ties (units whose count equals the threshold) of its chunk: 32 warps, each with `span`
// consecutive units (a multiple of 32).
__global__ void __launch_bounds__(1024)
static_ties_kernel(const uint32_t* __restrict__ ucnt, const uint32_t* __restrict__ sel, uint32_t U, uint32_t span,
                   uint32_t* __restrict__ ties)
{
    __shared__ uint32_t s_n;
    if (threadIdx.x == 0) s_n = 0u;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, thr = sel[0], u0 = (blockIdx.x * 32 + (threadIdx.x >> 5)) * span;
    uint32_t n = 0;
#pragma unroll 4
    for (uint32_t i = lane; i < span; i += 32) n += u0 + i < U && ucnt[u0 + i] == thr ? 1u : 0u;
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    if (lane == 0 && n) atomicAdd(&s_n, n);
    __syncthreads();
    if (threadIdx.x == 0) ties[blockIdx.x] = s_n;
}

// Third, every CTA takes its units above the threshold and as many of its ties as are left after the ties of the CTAs
// before it (ties go to the lower index).
__global__ void __launch_bounds__(1024)
static_pick_kernel(const uint32_t* __restrict__ ucnt, const uint32_t* __restrict__ sel, const uint32_t* __restrict__ ties,
                   uint32_t U, uint32_t span, uint32_t* __restrict__ row, uint32_t W32)
{
    __shared__ uint32_t s_warp[32], s_ties[32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t thr = sel[0], take = sel[1], u0 = (blockIdx.x * 32 + warp) * span;
    uint32_t mine = 0, n = 0;
    for (uint32_t j = threadIdx.x; j < blockIdx.x; j += 1024) mine += ties[j];
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
#pragma unroll 4
    for (uint32_t i = lane; i < span; i += 32) n += u0 + i < U && ucnt[u0 + i] == thr ? 1u : 0u;
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    if (lane == 0) { s_warp[warp] = mine; s_ties[warp] = n; }
    __syncthreads();
    uint32_t before = __reduce_add_sync(0xFFFFFFFFu, s_warp[lane] + (lane < warp ? s_ties[lane] : 0u));
#pragma unroll 4
    for (uint32_t i = 0; i < span; i += 32) {
        const uint32_t u = u0 + i + lane;
        const uint32_t c = u < U ? ucnt[u] : 0u;
        const bool tie = u < U && c == thr;
        const uint32_t tie_bits = __ballot_sync(0xFFFFFFFFu, tie);
        const bool pick = u < U && (c > thr || (tie && before + __popc(tie_bits & ((1u << lane) - 1u)) < take));
        const uint32_t bits = __ballot_sync(0xFFFFFFFFu, pick);
        before += __popc(tie_bits);
        if (lane == 0 && (u >> 5) < W32) row[u >> 5] = bits;
    }
}

__global__ void static_first_kernel(uint32_t* __restrict__ row, uint32_t W32, uint32_t cap)
{
    const uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= W32) return;
    const uint32_t lo = w * 32;
    row[w] = cap >= lo + 32 ? 0xFFFFFFFFu : (cap > lo ? (1u << (cap - lo)) - 1u : 0u);
}

// every row of sched equals `row`; with births (L not null) cut to the units that exist at the step
__device__ __forceinline__ void broadcast_row(const uint32_t* __restrict__ row, uint32_t W32, size_t total, const uint32_t* __restrict__ L,
                                              uint32_t* __restrict__ sched)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
        sched[i] = __ldg(row + i % W32) & (L ? __ldg(L + i) : ~0u);
}
__global__ void broadcast_row_kernel(const uint32_t* __restrict__ row, uint32_t W32, size_t total, uint32_t* __restrict__ sched)
{
    broadcast_row(row, W32, total, nullptr, sched);
}

// The same and its time-packed columns: a unit's bits are set from the step on at which it exists.
__global__ void initial_schedule_kernel(const uint32_t* __restrict__ row, uint32_t U, uint32_t S, uint32_t W32, uint32_t S32,
                                        const uint32_t* __restrict__ L, const uint32_t* __restrict__ birth,
                                        uint32_t* __restrict__ sched, uint32_t* __restrict__ Pcol)
{
    broadcast_row(row, W32, (size_t)S * W32, L, sched);
    const size_t total = (size_t)U * S32;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const uint32_t u = (uint32_t)(i / S32), j = (uint32_t)(i % S32);
        const uint32_t on = (__ldg(row + (u >> 5)) >> (u & 31)) & 1u;
        uint32_t valid = (j + 1) * 32 <= S ? 0xFFFFFFFFu : ((1u << (S - j * 32)) - 1u);
        if (birth) {
            const uint32_t b = __ldg(birth + u);
            valid &= b <= j * 32 ? ~0u : b >= (j + 1) * 32 ? 0u : ~0u << (b - j * 32);
        }
        Pcol[i] = on ? valid : 0u;
    }
}

// Growing cache: row s of L has bit u set iff unit u exists at step s (birth[u] <= s). A thread keeps the births of its
// word's 32 units in registers and walks kAliveSteps steps; two instructions per bit (131,072 units x 1056 steps: 489 us
// with the births read again for every word).
constexpr uint32_t kAliveSteps = 32;
__global__ void __launch_bounds__(128)
alive_rows_kernel(const uint32_t* __restrict__ birth, uint32_t U, uint32_t S, uint32_t W32, uint32_t* __restrict__ L)
{
    const uint32_t s0 = blockIdx.y * kAliveSteps, s1 = min(s0 + kAliveSteps, S);
    for (uint32_t w = blockIdx.x * 128 + threadIdx.x; w < W32; w += gridDim.x * 128) {
        uint32_t b[32];
#pragma unroll
        for (uint32_t i = 0; i < 32; ++i) b[i] = w * 32 + i < U ? __ldg(birth + w * 32 + i) : ~0u;
        for (uint32_t s = s0; s < s1; ++s) {
            uint32_t bits = 0;
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) bits |= b[i] <= s ? 1u << i : 0u;
            L[(size_t)s * W32 + w] = bits;
        }
    }
}

// Births per step, and the checks of kvp_set_births: flag bit 0 = a birth beyond the horizon, bit 1 = a unit
// that is accessed before it exists.
__global__ void birth_stats_kernel(const uint32_t* __restrict__ birth, uint32_t U, uint32_t S,
                                   const uint32_t* __restrict__ Acol, uint32_t S32, uint32_t* __restrict__ nb,
                                   uint32_t* __restrict__ flag)
{
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= U) return;
    const uint32_t b = birth[u];
    if (b >= S) { atomicOr(flag, 1u); return; }
    if (b == 0) return;
    atomicAdd(nb + b, 1u);
    uint32_t early = 0;
    for (uint32_t j = 0; j < (b >> 5); ++j) early |= __ldg(Acol + (size_t)u * S32 + j);
    if (b & 31u) early |= __ldg(Acol + (size_t)u * S32 + (b >> 5)) & ((1u << (b & 31u)) - 1u);
    if (early) atomicOr(flag, 2u);
}

// every unit born in a step is first counted as written to DRAM (see step_cost_g)
__global__ void stepc_births_kernel(StepC* __restrict__ stepc, const uint32_t* __restrict__ nb, uint32_t S, uint32_t kk,
                                    uint32_t kd)
{
    const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    StepC c = stepc[s];
    c.y += kk * nb[s];
    c.z += kd * nb[s];
    stepc[s] = c;
}

__global__ void and_rows_kernel(uint32_t* __restrict__ sched, const uint32_t* __restrict__ L, size_t total)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
        sched[i] &= __ldg(L + i);
}

inline uint32_t grid_for(size_t total, uint32_t block)
{
    size_t g = (total + block - 1) / block;
    return (uint32_t)(g > 148 * 16 ? 148 * 16 : (g ? g : 1));
}

}  // namespace

template <int LRB, int LWB, bool OPEN>
static int launch_transpose(const uint32_t* in, uint32_t rows, uint32_t in_words, uint32_t cols, uint32_t* out, uint32_t out_words,
                            const OpenArgs& open, const ChosenInput& chosen, uint32_t most_y, cudaStream_t st)
{
    uint32_t y = (in_words + (1u << LWB) - 1) >> LWB;
    if (y > most_y) y = most_y;
    dim3 grid((out_words + (1u << LRB) - 1) >> LRB, y);
    bit_transpose_kernel<LRB, LWB, OPEN><<<grid, 256, 0, st>>>(in, rows, in_words, cols, out, out_words, open, chosen);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

// Tiles follow the short side: short rows in (a few steps' words per unit) take many rows, short rows out many words.
int launch_bit_transpose(const uint32_t* in, uint32_t rows, uint32_t in_words, uint32_t cols, uint32_t* out,
                         uint32_t out_words, cudaStream_t st, const ChosenInput& chosen)
{
#define KVP_TRANSPOSE(LRB, LWB) launch_transpose<LRB, LWB, false>(in, rows, in_words, cols, out, out_words, OpenArgs(), chosen, 32768, st)
    if (in_words <= 2) return KVP_TRANSPOSE(5, 1);
    if (in_words <= 4) return KVP_TRANSPOSE(4, 2);
    if (out_words <= 2) return KVP_TRANSPOSE(1, 5);
    if (out_words <= 4) return KVP_TRANSPOSE(2, 4);
    return KVP_TRANSPOSE(3, 3);
#undef KVP_TRANSPOSE
}

// p->dA, p->dAcol, p->d_a and p->d_ucnt from the caller's access bitmap; d_a and d_ucnt come zeroed.
int launch_open(const kvp_problem* p, const uint32_t* access, cudaStream_t st)
{
    OpenArgs open;
    open.copy = p->dA; open.row_count = p->d_a; open.ucnt = p->d_ucnt; open.pad_mask = p->pad_mask;
    open.ucnt_add = p->S32 > 8;
    const uint32_t fill = 148 * 8;                       // CTAs that fill the machine: eight of 256 threads per SM
#define KVP_OPEN(LRB, LWB, most) launch_transpose<LRB, LWB, true>(access, p->S, p->W32, p->U, p->dAcol, p->S32, open, ChosenInput(), most, st)
    if (p->S32 <= 2) return KVP_OPEN(1, 5, fill);
    if (p->S32 <= 4) return KVP_OPEN(2, 4, fill);
    const uint32_t tiles = (p->S32 + 7) / 8;
    return KVP_OPEN(3, 3, (fill + tiles - 1) / tiles);
#undef KVP_OPEN
}

int launch_clean_copy(const uint32_t* in, uint32_t* out, uint32_t S, uint32_t W32, uint32_t pad_mask, cudaStream_t st)
{
    const size_t total = (size_t)S * W32;
    clean_copy_kernel<<<grid_for(total, 256), 256, 0, st>>>(in, out, total, W32, pad_mask);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_stepc(StepC* stepc, const uint32_t* writes, const uint32_t* a, uint32_t S, const CostK& K, cudaStream_t st)
{
    stepc_kernel<<<(S + 255) / 256, 256, 0, st>>>(stepc, writes, a, S, K);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

// chunks of the tie count: 32 warps of 32 units, of 256 where there are enough units to fill the machine that way
static uint32_t static_span(const kvp_problem* p) { return p->U >= 148u * 8192u ? 256u : 32u; }

size_t static_freq_words(const kvp_problem* p)
{
    const uint32_t chunk = 32u * static_span(p);
    return (size_t)((p->S + 2 + 3) & ~3u) + 4 + (p->W32 * 32 + chunk - 1) / chunk;
}

// scratch: static_freq_words, of which the first S + 2 are zero: the histogram (S + 1 bins), the ticket of the first kernel,
// the selection (2 words) and the tie counts of the chunks. hits (zero before): the accesses of the row's units over all steps
int launch_static_freq_row(const kvp_problem* p, uint32_t* scratch, uint32_t* row, unsigned long long* hits, cudaStream_t st)
{
    uint32_t* hist = scratch;
    uint32_t* sel = hist + ((p->S + 2 + 3) & ~3u);
    uint32_t* ties = sel + 4;
    const uint32_t span = static_span(p), chunks = (p->W32 * 32 + 32 * span - 1) / (32 * span);
    uint32_t hgrid = (p->U + 8191) / 8192;
    if (hgrid > 148) hgrid = 148;
    static_threshold_kernel<<<hgrid, 1024, 0, st>>>(p->d_ucnt, p->U, p->S, p->cap, hist, sel, hist + p->S + 1, hits);
    KVP_CUDA(cudaGetLastError());
    static_ties_kernel<<<chunks, 1024, 0, st>>>(p->d_ucnt, sel, p->U, span, ties);
    KVP_CUDA(cudaGetLastError());
    static_pick_kernel<<<chunks, 1024, 0, st>>>(p->d_ucnt, sel, ties, p->U, span, row, p->W32);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_static_first_row(const kvp_problem* p, uint32_t* row, cudaStream_t st)
{
    static_first_kernel<<<(p->W32 + 255) / 256, 256, 0, st>>>(row, p->W32, p->cap);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_broadcast_row(const uint32_t* row, uint32_t S, uint32_t W32, uint32_t* sched, cudaStream_t st)
{
    const size_t total = (size_t)S * W32;
    broadcast_row_kernel<<<grid_for(total, 256), 256, 0, st>>>(row, W32, total, sched);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_initial_schedule(const kvp_problem* p, const uint32_t* row, uint32_t* sched, uint32_t* Pcol, cudaStream_t st)
{
    initial_schedule_kernel<<<grid_for((size_t)p->U * p->S32, 256), 256, 0, st>>>(row, p->U, p->S, p->W32, p->S32, p->dL, p->d_birth,
                                                                                 sched, Pcol);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_alive_rows(const uint32_t* birth, uint32_t U, uint32_t S, uint32_t W32, uint32_t* L, cudaStream_t st)
{
    const uint32_t x = (W32 + 127) / 128;
    dim3 grid(x < 4096u ? x : 4096u, (S + kAliveSteps - 1) / kAliveSteps);
    alive_rows_kernel<<<grid, 128, 0, st>>>(birth, U, S, W32, L);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_birth_stats(const uint32_t* birth, uint32_t U, uint32_t S, const uint32_t* Acol, uint32_t S32, uint32_t* nb,
                       uint32_t* flag, cudaStream_t st)
{
    birth_stats_kernel<<<(U + 255) / 256, 256, 0, st>>>(birth, U, S, Acol, S32, nb, flag);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_stepc_births(StepC* stepc, const uint32_t* nb, uint32_t S, uint32_t kk, uint32_t kd, cudaStream_t st)
{
    stepc_births_kernel<<<(S + 255) / 256, 256, 0, st>>>(stepc, nb, S, kk, kd);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

int launch_and_rows(uint32_t* sched, const uint32_t* L, size_t total, cudaStream_t st)
{
    and_rows_kernel<<<grid_for(total, 256), 256, 0, st>>>(sched, L, total);
    KVP_CUDA(cudaGetLastError());
    return KVP_OK;
}

}  // namespace kvp
