// The acceptance table of kvp.h: quantised Metropolis thresholds. Pure host arithmetic (C++, no device code).
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <thread>
#include <vector>

#include "../../include/kvp.h"

namespace {

typedef double v4d __attribute__((vector_size(32)));
typedef int64_t v4l __attribute__((vector_size(32)));
typedef uint32_t v4u __attribute__((vector_size(16)));

// One threshold as it is defined: floor(2^32 exp(-x/C)), capped. Entries whose exponent is beyond 22.5 > ln(2^32) are
// zero whatever the last bits of exp() are.
uint32_t accept_entry(uint32_t q, double bin, double C)
{
    const double x = ((double)q + 0.5) * bin;
    if (x / C > 22.5) return 0u;
    const double thr = 4294967296.0 * exp(-x / C);
    return thr >= 4294967295.0 ? 0xFFFFFFFFu : (uint32_t)thr;
}

// One row of the table. The thresholds of a row are a geometric sequence, so after every eighth of exp() calls per 256
// entries each entry is the one eight before it times a constant. The sequence and the formula differ by less than 1e-4
// (31 multiplications and an exp() on either side: a relative error below 2e-14 of at most 2^32), so an entry farther
// than 1e-3 from a whole number has the formula's floor; the others, two in a thousand, are computed by the formula.
// 1.4 us a row; with exp() for every entry 6.9 us, which made the table a quarter of a small annealing call.
#if defined(__x86_64__)
__attribute__((target_clones("avx2", "default")))
#endif
void accept_row(double C, uint32_t shift, uint32_t* row)
{
    const double bin = (double)(1ull << shift);
    const double r8 = exp(-8.0 * bin / C);
    const double m = 6755399441055744.0;                         // 1.5 * 2^52: adding it rounds to a whole number
    const v4d magic = {m, m, m, m}, zero = {0.0, 0.0, 0.0, 0.0}, half = {0.5, 0.5, 0.5, 0.5}, edge = {1e-3, 1e-3, 1e-3, 1e-3};
    const v4d ratio = {r8, r8, r8, r8};
    for (uint32_t q0 = 0; q0 < KVP_TABLE_Q; q0 += 256) {
        v4d v[2];
        for (int i = 0; i < 8; ++i) v[i >> 2][i & 3] = 4294967296.0 * exp(-(((double)(q0 + i) + 0.5) * bin) / C);
        if (v[0][0] < 0.5) {                                     // below one from here on
            memset(row + q0, 0, (KVP_TABLE_Q - q0) * sizeof(uint32_t));
            break;
        }
        for (uint32_t q = q0; q < q0 + 256; q += 8) {
            v4l risky = {0, 0, 0, 0};
            for (int h = 0; h < 2; ++h) {
                const v4d t = v[h] + magic, d = v[h] - (t - magic);
                v4l w;
                memcpy(&w, &t, sizeof w);
                w += d < zero;                                   // rounded up: one less (a true lane is -1)
                const v4l small = v[h] < half;
                w &= ~small;
                risky |= (d < edge) & (d > -edge) & ~small;
                const v4u n = __builtin_convertvector(w, v4u);
                memcpy(row + q + 4 * h, &n, sizeof n);
                v[h] *= ratio;
            }
            if (risky[0] | risky[1] | risky[2] | risky[3])
                for (int i = 0; i < 8; ++i) row[q + i] = accept_entry(q + i, bin, C);
        }
    }
}

// the rows rows[i0..i1) of the acceptance table
void accept_rows(const double* temps, const uint32_t* shifts, const uint32_t* rows, uint32_t i0, uint32_t i1, uint32_t* table)
{
    for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t j = rows[i];
        accept_row(temps[j] >= 1.0 ? temps[j] : 1.0, shifts[j], table + (size_t)j * KVP_TABLE_Q);   // also maps NaN to 1
    }
}

}  // namespace

extern "C" int kvp_accept_table(const double* temps, uint32_t levels, uint32_t* table, uint32_t* shifts)
try {
    if (!temps || !table || !shifts || !levels) return KVP_ERR_ARG;
    // A level whose (clamped) temperature equals that of the level before it has the same row: a ladder that has
    // cooled below one tick repeats its last row, often for a third of its levels. Only the others are computed.
    std::vector<uint32_t> rows;
    rows.reserve(levels);
    double prev = 0.0;
    for (uint32_t j = 0; j < levels; ++j) {
        const double C = temps[j] >= 1.0 ? temps[j] : 1.0;
        uint32_t sh = 0;
        while ((double)KVP_TABLE_Q * (double)(1ull << sh) < 23.0 * C)
            if (++sh > 40) return KVP_ERR_RANGE;
        shifts[j] = sh;
        if (j == 0 || C != prev) rows.push_back(j);
        prev = C;
    }
    const uint32_t nrows = (uint32_t)rows.size();
    // A ladder of 64 levels takes less time (0.09 ms) than a few threads take to start; long ladders are shared out.
    uint32_t nthr = nrows >= 256 ? std::min<uint32_t>(8u, std::max(1u, std::thread::hardware_concurrency())) : 1u;
    if (nthr > 1) {
        std::vector<std::thread> pool;
        const uint32_t per = (nrows + nthr - 1) / nthr;
        try {
            for (uint32_t t = 1; t < nthr && t * per < nrows; ++t)
                pool.emplace_back(accept_rows, temps, shifts, rows.data(), t * per, std::min(nrows, (t + 1) * per), table);
        } catch (...) {                                        // no thread to be had: this one does the rest
            const uint32_t done = (uint32_t)pool.size() + 1;
            accept_rows(temps, shifts, rows.data(), std::min(nrows, done * per), nrows, table);
        }
        accept_rows(temps, shifts, rows.data(), 0, std::min(nrows, per), table);
        for (auto& th : pool) th.join();
    } else {
        accept_rows(temps, shifts, rows.data(), 0, nrows, table);
    }
    for (uint32_t j = 1, i = 1; j < levels; ++j) {             // the repeated rows, each from the row before it
        if (i < nrows && rows[i] == j) { ++i; continue; }
        memcpy(table + (size_t)j * KVP_TABLE_Q, table + (size_t)(j - 1) * KVP_TABLE_Q, KVP_TABLE_Q * sizeof(uint32_t));
    }
    return KVP_OK;
} catch (const std::bad_alloc&) {
    return KVP_ERR_NOMEM;
}
