// Shapes and shared-memory sizes of the recovery kernel k_omp (sgc_omp.cu): plain integer arithmetic for host and device, which
// a C++ compiler without CUDA takes as well, so that it can be checked over every size the library accepts.
#pragma once

#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define SGC_HD __host__ __device__
#else
#define SGC_HD
#endif

namespace sgc {

constexpr int kRescoreCap = 16;                       // candidates rescored in fp64 per iteration and residual
constexpr int kOmpBlock = 512;                        // threads per block of k_omp
constexpr long long kOmpDynBytes = 196 * 1024;        // dynamic shared memory of every launch (one block per SM)
constexpr long long kOmpCorrLeast = 40 * 1024;        // ... of which partial sums and norms of the correlation take at least this
constexpr double kOmpOneWork = 1.2e6;                 // k * d up to which one cluster of 16 serves the lock-step recovery
constexpr double kOmpPairCols = 1000.0;               // columns per pick from which pairs do

// both residuals as operands of the correlation
SGC_HD inline size_t frag_bytes(int k) { return (size_t)((k + 15) / 16) * 128; }

// blocks of a group (the books of one recovery) in clusters of cl
SGC_HD constexpr int group_blocks(int cl) { return cl == 16 ? 8 : cl; }

// row slices: an even number of rows per block (a generated word holds two rows)
SGC_HD inline int slice_rows(int k, int gs) { return 2 * ((k + 2 * gs - 1) / (2 * gs)); }
SGC_HD inline int even(int n) { return (n + 1) & ~1; }

// a slot of the exchange: products with q_l and the residual (by l), then ||a||^2, ||r||^2, and two values per further candidate
SGC_HD inline int exchange_stride(int s) { return even(s + 2 + 2 * kRescoreCap); }

// dynamic shared memory of a bookkeeping block, in doubles: residual slice | partial sums | exchanged sums | exchange slots
SGC_HD inline size_t book_doubles(int k, int s, int gs, bool two) {
    const int R = slice_rows(k, gs);
    return (size_t)R + (R > kOmpBlock ? R : kOmpBlock) + even(s + 4) + (size_t)(two ? 2 : 1) * gs * exchange_stride(s) + 2 * gs;
}

// What fits beside the fixed buffers of a launch in clusters of cl (mode 1: lock-step).
struct OmpBudget {
    bool fits;                         // false: the fixed buffers alone are too large, this form cannot serve the state
    int q_cols;                        // columns of q that a bookkeeping block keeps in shared memory
    int book_correlates;               // the bookkeeping blocks correlate, too
    int z_words;                       // 32-bit words that the correlation may use for sums, norms and generated entries
};
inline OmpBudget omp_budget(int cl, int k, int s, int mode) {
    const int gs = group_blocks(cl);
    const long long pb = (long long)frag_bytes(k), bb = (long long)(book_doubles(k, s, gs, cl == 16) * sizeof(double));
    const long long col = (long long)slice_rows(k, gs) * (long long)sizeof(double);
    OmpBudget b = {false, 0, 0, 0};
    // bookkeeping blocks correlate as well in lock-step, as far as both fit (one cluster: there are no others)
    b.book_correlates = (cl == 16 || (mode == 1 && bb + pb + kOmpCorrLeast <= kOmpDynBytes)) ? 1 : 0;
    long long room = kOmpDynBytes - bb - (b.book_correlates ? pb : 0);
    b.fits = b.book_correlates ? room >= kOmpCorrLeast : (room >= 0 && kOmpDynBytes - pb >= kOmpCorrLeast);
    if (!b.fits) return b;
    long long q = b.book_correlates ? (room - kOmpCorrLeast) / 2 : room;
    if (q > col * s) q = col * s;
    b.q_cols = (int)(q / col);
    room = b.book_correlates ? room - b.q_cols * col : kOmpDynBytes - pb;
    b.z_words = (int)(room / 4) - 8;
    return b;
}

// The share of block blk of nblk in the correlation of n columns, and where its sums, norms and generated entries lie (word offsets
// in the z_words of shared memory that it has).
struct CorrPlan { uint32_t e0; int cnt, tiles, ks, kblocks; bool cached, norms; size_t part_off, inv_off, col_off, z_off; };

SGC_HD inline CorrPlan corr_plan(uint32_t n, int k, int z_words, int blk, int nblk) {
    CorrPlan c;
    const uint64_t per = ((uint64_t)n + nblk - 1) / nblk, e0 = per * blk;      // (up to 2^32 - 1 columns)
    c.e0 = e0 < n ? (uint32_t)e0 : n;
    c.cnt = (int)(n - c.e0 < per ? n - c.e0 : per);
    const int tiles = (int)((per + 15) / 16);                         // the same plan in every block
    c.kblocks = (k + 15) / 16;
    int best = 1; float cost = 3e38f;
    for (int ks = 1; ks <= 16 && ks <= c.kblocks && tiles * ks <= 64; ks <<= 1) {
        const float rounds = (float)((tiles * ks + kOmpBlock / 32 - 1) / (kOmpBlock / 32));
        const float t = rounds * ((float)((c.kblocks + ks - 1) / ks) + 3.0f);
        if (t < cost * 0.99f) { cost = t; best = ks; }
    }
    c.ks = best;
    c.tiles = tiles;
    // partial sums of split tiles, norms, generated entries
    c.part_off = 0;
    c.inv_off = best > 1 ? (size_t)tiles * best * 32 : 0;
    c.norms = c.inv_off + (size_t)tiles * 32 <= (size_t)z_words;      // norms, and the columns themselves (lists)
    c.col_off = c.inv_off + (size_t)tiles * 16;
    c.z_off = (c.inv_off + (c.norms ? (size_t)tiles * 32 : 0) + 3) & ~(size_t)3;
    c.cached = c.norms && c.z_off + (size_t)tiles * c.kblocks * 128 <= (size_t)z_words;
    return c;
}

// Which cluster shape (16, 2 or 8; one: a cluster of 16 can be resident; groups: the device holds three clusters of 8 at a time, two
// for the books and one that correlates; a small partition of a GPU does not, and pairs serve everything there): the one-cluster form while a pick's correlation takes
// 16 SMs no longer than the grid barriers cost the others; pairs (all 148 SMs correlate, two blocks keep each recovery's books)
// when the correlation of a pick (k d) dwarfs its bookkeeping (k s), whatever k is; groups of 8 (120 SMs, the most that
// clusters of 8 can occupy) otherwise and for lists.  The first two only where their buffers fit: with k in the ten thousands and a
// handful of columns the one cluster has no room for the books beside the operands, with many rows and picks the pairs have none.
// Step in groups of 8 / in pairs, us: d = 500000, k = 210, s = 30: 2187 / 1832; 65000, 350, 50: 1312 / 1126; 10000, 200, 8:
// 143 / 136;  60000, 512, 64 (940 columns per pick): 1692 / 1694;  60000, 1024, 64: 2359 / 2521;  25000, 1400, 200: 7708 / 13020.
inline int omp_shape(long long d, int k, int s, int mode, bool one, bool groups) {
    if (mode == 1) {
        if (one && (double)k * (double)d <= kOmpOneWork && omp_budget(16, k, s, mode).fits) return 16;
        const OmpBudget pair = omp_budget(2, k, s, mode);
        if (pair.fits && pair.book_correlates && (double)d >= kOmpPairCols * s) return 2;
    }
    return groups ? 8 : 2;
}

}  // namespace sgc
