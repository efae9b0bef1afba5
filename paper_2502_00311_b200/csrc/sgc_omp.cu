// a4, the picks: orthogonal matching pursuit (Appendix B, Algorithm 3) on a set of columns -- all d of them (lock-step) or a
// short candidate list (speculation, to be confirmed by the screening pass of sgc_pass.cu).
//
// Both recoveries (M^ and V^) advance together, one pick each per iteration.  Algorithm 3 is carried in its orthogonal
// form: q_j is the picked column made orthogonal to the earlier ones (c^(j)_l = <q_l, a_new>, gamma_j = 1 / ||a_new - sum c_l q_l||,
// the printed inverse-Cholesky factor is the inverse of the triangular matrix with entries c and 1 / gamma), a_j = <q_j, r>,
// r <- r - a_j q_j.  The coefficients x are one back-substitution at the end of the step (k_finish in sgc_recover.cu).
// Everything but the first screen of a pick is fp64.
//
// One kernel, k_omp<CL>, launched as clusters of CL blocks.  Two groups of GS blocks keep the books, one group per
// recovery; the rows of A (k) are split over the blocks of a group, which hold their slice of r and of the q_l in shared
// memory and combine partial sums through distributed shared memory: a pick costs a group two or three cluster barriers
// (0.28 us each) instead of the chain of a dozen block barriers and L2 round trips that one block needs for it.  All other
// blocks (in lock-step: all blocks) correlate the columns with the current residuals.  An iteration is
//     correlate | grid barrier | decide in fp64, update q, r | grid barrier
// What an iteration takes: see the table at k_omp.
//
// Lists of up to kGramList columns (the steady state of a run with a stable support) need no iteration of that kind: with
// the Gram matrix G of the list at hand, block m runs all picks of recovery m on it alone (gram_picks), and the whole grid
// then forms the residuals of all picks at once (gram_rows, gram_emit).
#include <mutex>

#include <cooperative_groups.h>

#include "sgc_omp.cuh"

namespace cg = cooperative_groups;

namespace sgc {
namespace {

constexpr int kT = kOmpBlock;
constexpr int kWarps = kT / 32;
constexpr int kRescanCap = 64;
constexpr double kPivot = 1e-10;                      // a new column whose orthogonal part is below this share is dependent

// the best column seen (lowest index on ties), and the largest score among all others (what is dropped: the caller can tell
// whether a dropped column could still have mattered)
struct Top {
    float s1, s2; uint32_t i1;
    __device__ __forceinline__ void init() { s1 = s2 = -1.0f; i1 = kNoColumn; }
    __device__ __forceinline__ void push(float s, uint32_t i) {
        if (better(s, i, s1, i1)) { s2 = s1; s1 = s; i1 = i; }
        else s2 = fmaxf(s2, s);
    }
};

__device__ __forceinline__ unsigned int score_key(float s) { return s >= 0.0f ? __float_as_uint(s) + 1u : 0u; }
__device__ __forceinline__ float key_score(unsigned int k) { return k ? __uint_as_float(k - 1u) : -1.0f; }

// best column and second-best score over the lanes of a warp (every lane returns the result); columns of different lanes differ
__device__ __forceinline__ void warp_merge(Top& t) {
    const unsigned int mine = score_key(t.s1), best = __reduce_max_sync(0xffffffffu, mine);
    const uint32_t idx = __reduce_min_sync(0xffffffffu, (best != 0u && mine == best) ? t.i1 : kNoColumn);
    const bool holder = best != 0u && mine == best && t.i1 == idx;
    const unsigned int second = __reduce_max_sync(0xffffffffu, holder ? score_key(t.s2) : mine);
    t.s1 = key_score(best); t.i1 = idx; t.s2 = key_score(second);
}

__device__ __forceinline__ bool in_list(const uint32_t* lam, int n, uint32_t col) {
    for (int q = 0; q < n; ++q) if (lam[q] == col) return true;
    return false;
}

// shared memory of k_omp that has a fixed size
struct OmpSmem {
    unsigned int wkey[kWarps], wkey2[kWarps], floor_key[2];
    float npart[64][16];
    double wsum[kWarps];
    Top wtop[2][kWarps];
    uint32_t cidx[kRescoreCap];
    uint32_t rbuf[kRescanCap];
    int rescan_blk[8]; uint32_t rescan_col[8];
    int nc, peer_nc, rescan_n, rbuf_n;
    __align__(16) uint32_t sup[2][kMaxS];
};

// ------------------------------------------------------------------------------------------------
// correlation: columns e0 .. e0 + cnt of a set (col_list, or the identity) against both residuals
// ------------------------------------------------------------------------------------------------
// Warp = 16 columns at a time, mma.m16n8k16: a generated row pair of a column is exactly one register of the A operand, and
// the B operand holds both residuals, each as two binary16 numbers (value and remainder, 22 bits), so that the products
// are summed in fp32 by the tensor cores and a row pair costs its 13 generator instructions and little else (26 with the
// conversions and multiply-adds done one by one).  This is the legacy matrix instruction on purpose: N is 4, so a tcgen05 tile
// would be idle but for one in sixty columns, and the generator bounds it anyway.  A tile's rows are split over several warps when the block has fewer tiles than warps.  When the generated entries
// of the block's columns fit its shared memory they are kept from the first iteration on, as operand registers: an iteration
// then reads 16 bytes per lane and 16 rows instead of regenerating them.  The norms are summed in the first iteration.
// membership in a support staged in shared memory (padded with kNoColumn to a multiple of 4)
__device__ __forceinline__ bool in_support4(const uint32_t* sup, int n, uint32_t col) {
    bool hit = false;
    for (int q = 0; q < n; q += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(sup + q);
        hit |= v.x == col || v.y == col || v.z == col || v.w == col;
    }
    return hit;
}

// The threads of the block tell one another the second best score that each has seen: a column below any of these can be
// neither the block's best nor its second best, so that after the first few columns hardly any gets further than one compare.  (One at
// the bound goes on: of equal scores, those of a zero residual, the lowest column has to win.)
// (A column of the support scores rounding noise: the look-up is needed only for what passes.)
__device__ __forceinline__ void offer(OmpSmem& sh, Top& best, const int* picks, int m, float score, uint32_t col) {
    if (!(score > best.s2) || score_key(score) < *reinterpret_cast<volatile unsigned int*>(&sh.floor_key[m])) return;
    if (in_support4(sh.sup[m], picks[m], col)) return;
    const float before = best.s2;
    best.push(score, col);
    if (best.s2 > before && best.s2 >= 0.0f) atomicMax(&sh.floor_key[m], score_key(best.s2));
}

__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_half(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// The residuals as B operands: for each 16 rows, lane (g, t) with g < 4 holds rows 2t, 2t + 1 and 2t + 8, 2t + 9 of column g: 0 and
// 1 value and remainder of the M^ residual, 2 and 3 of V^'s.  Each residual is scaled by a power of two (largest entry in
// [2^10, 2^11)); a score is homogeneous in it, and back[m] undoes it.
__device__ void stage_residuals(const OmpArgs& a, OmpSmem& sh, uint2* frag, float* back, const int* picks) {
    constexpr int kHold = 4;                                          // row pairs per thread fetched once (k <= 4096)
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, k = a.k;
    const float4* r = reinterpret_cast<const float4*>(a.r32);         // (padded by two rows: a pair may be read whole)
    const int items = (k + 15) / 16 * 8;                              // row pairs: (16-row block, which half, t)
    auto fetch = [&](int it) -> float4 {
        const int pair = (it >> 3) * 8 + (it & 1) * 4 + ((it >> 1) & 3);
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (2 * pair < k) v = __ldcg(r + pair);
        if (2 * pair + 1 >= k) v.z = v.w = 0.0f;
        return v;
    };
    float4 v[kHold];
#pragma unroll
    for (int u = 0; u < kHold; ++u) v[u] = t + u * kT < items ? fetch(t + u * kT) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const uint32_t l0 = t < picks[0] ? __ldcg(a.lam + t) : kNoColumn, l1 = t < picks[1] ? __ldcg(a.lam + a.s + t) : kNoColumn;
    unsigned int m0 = 0u, m1 = 0u;
    auto widest = [&](const float4& f) {
        m0 = max(m0, max(__float_as_uint(f.x) & 0x7FFFFFFFu, __float_as_uint(f.z) & 0x7FFFFFFFu));
        m1 = max(m1, max(__float_as_uint(f.y) & 0x7FFFFFFFu, __float_as_uint(f.w) & 0x7FFFFFFFu));
    };
#pragma unroll
    for (int u = 0; u < kHold; ++u) widest(v[u]);
    for (int it = t + kHold * kT; it < items; it += kT) widest(fetch(it));
    sh.sup[0][t] = l0; sh.sup[1][t] = l1;
    for (int e = kT + t; e < kMaxS; e += kT) {
        if (e < ((picks[0] + 3) & ~3)) sh.sup[0][e] = e < picks[0] ? __ldcg(a.lam + e) : kNoColumn;
        if (e < ((picks[1] + 3) & ~3)) sh.sup[1][e] = e < picks[1] ? __ldcg(a.lam + a.s + e) : kNoColumn;
    }
    m0 = __reduce_max_sync(0xffffffffu, m0); m1 = __reduce_max_sync(0xffffffffu, m1);
    if (lane == 0) { sh.wkey[warp] = m0; sh.wkey2[warp] = m1; }
    if (t < 2) sh.floor_key[t] = 0u;
    __syncthreads();
    m0 = __reduce_max_sync(0xffffffffu, lane < kWarps ? sh.wkey[lane] : 0u);
    m1 = __reduce_max_sync(0xffffffffu, lane < kWarps ? sh.wkey2[lane] : 0u);
    // 2^10 <= largest * scale < 2^11 (exponent field e: scale 2^(137 - e)); tiny or zero residuals get the largest scale
    int e0 = (int)(m0 >> 23), e1 = (int)(m1 >> 23);
    e0 = e0 < 20 ? 20 : (e0 > 250 ? 250 : e0); e1 = e1 < 20 ? 20 : (e1 > 250 ? 250 : e1);
    const float s0 = __uint_as_float((unsigned int)(264 - e0) << 23), s1 = __uint_as_float((unsigned int)(264 - e1) << 23);
    back[0] = __uint_as_float((unsigned int)(e0 - 10) << 23); back[1] = __uint_as_float((unsigned int)(e1 - 10) << 23);
    auto put = [&](int it, const float4& f) {
        const int kb = it >> 3, q = (it >> 1) & 3, which = it & 1;    // which: rows 2q.. or 2q + 8..
        const float a0 = f.x * s0, a1 = f.z * s0, b0 = f.y * s1, b1 = f.w * s1;
        const uint32_t ah = pack_half(a0, a1), bh = pack_half(b0, b1);
        const float2 af = half2_bits_to_float2(ah), bf = half2_bits_to_float2(bh);
        uint32_t* w = reinterpret_cast<uint32_t*>(frag + (size_t)kb * 16) + which;
        w[2 * (0 * 4 + q)] = ah;
        w[2 * (1 * 4 + q)] = pack_half(a0 - af.x, a1 - af.y);
        w[2 * (2 * 4 + q)] = bh;
        w[2 * (3 * 4 + q)] = pack_half(b0 - bf.x, b1 - bf.y);
    };
#pragma unroll
    for (int u = 0; u < kHold; ++u) if (t + u * kT < items) put(t + u * kT, v[u]);
    for (int it = t + kHold * kT; it < items; it += kT) put(it, fetch(it));
}

// Tiles of a block from which they are streamed: four per warp, two rounds of two (rows are split over warps up to here).  From 64
// instead of 128 tiles, steps: d = 200000, k = 210, s = 30: 1001 -> 919 us;  250000, 64, 9: 258 -> 236 us.
constexpr int kStreamTiles = 64;

// The columns of a block in lock-step when they are too many to keep: a warp takes 32 columns a round.  Each lane works out the
// key of one of them, and the two tiles' eight generated words overlap one another.  The norms (HAVE: those kept from the first
// iteration, inv_s) are the diagonals of two more products with the tile itself as B operand (lane (g, t) holds the very words
// that B wants of columns g and g + 8), which saves the conversions and multiply-adds; their accumulators are emptied into a sum
// every kNormBlocks blocks of rows, so that a norm is as exact as one summed entry by entry.  A column that cannot pass the
// block's second best score so far costs one compare and no division.  Issue slots bound it: 16 rows of 2e6 columns take 10 us
// (3.2e12 entries/s; the generator alone allows 5.1e12), and what a column costs whatever k is another 16 us.  Per pick, d = 2e6,
// k = 42: 96 -> 55 us;  1.2e6, 224: 110 -> 88;  5e5, 700: 140 -> 105.
constexpr int kNormBlocks = 16;
template <bool HAVE>
__device__ __forceinline__ void correlate_stream(const OmpArgs& a, OmpSmem& sh, const CorrPlan& c, const uint2* frag, float* inv_s,
                                                 const float (&back)[2], const int* picks, Top& best) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    const int diag = g * 4 + (g >> 1);                                // lane of column g's own norm, element g & 1 of its pair
    const bool odd = g & 1;
    const float bq = q == 0 ? back[0] : back[1];
    for (int base = warp * 32; base < c.cnt; base += 32 * kWarps) {
        const ColKey key = column_key(a.seed_lo, a.seed_hi, (uint32_t)(c.e0 + base + lane));
        uint32_t h[4], st[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t mk = __shfl_sync(0xffffffffu, key.mk, g + 8 * u);
            h[u] = __shfl_sync(0xffffffffu, key.ck, g + 8 * u) + (uint32_t)q * mk;
            st[u] = 4u * mk;
        }
        float acc0[4] = {0.0f, 0.0f, 0.0f, 0.0f}, acc1[4] = {0.0f, 0.0f, 0.0f, 0.0f}, n[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        // rows 2q, 2q + 1 (lo) and 2q + 8, 2q + 9 (hi) of columns g + 8 u
        auto words = [&](uint32_t (&lo)[4], uint32_t (&hi)[4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                lo[u] = z_pair_from_word(h[u]); h[u] += st[u];
                hi[u] = z_pair_from_word(h[u]); h[u] += st[u];
            }
        };
        if (HAVE) {
            // (rows beyond k meet zeros of the residuals)
#pragma unroll 2
            for (int kb = 0; kb < c.kblocks; ++kb) {
                const uint2 b = lane < 16 ? frag[(size_t)kb * 16 + lane] : make_uint2(0u, 0u);
                uint32_t lo[4], hi[4];
                words(lo, hi);
                mma_16816(acc0, lo[0], lo[1], hi[0], hi[1], b.x, b.y);
                mma_16816(acc1, lo[2], lo[3], hi[2], hi[3], b.x, b.y);
            }
        } else {
            for (int kg = 0; kg < c.kblocks; kg += kNormBlocks) {
                const int kend = kg + kNormBlocks < c.kblocks ? kg + kNormBlocks : c.kblocks;
                float na[4] = {0.0f, 0.0f, 0.0f, 0.0f}, nb[4] = {0.0f, 0.0f, 0.0f, 0.0f}, nc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, nd[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
                for (int kb = kg; kb < kend; ++kb) {
                    const uint2 b = lane < 16 ? frag[(size_t)kb * 16 + lane] : make_uint2(0u, 0u);
                    uint32_t lo[4], hi[4];
                    words(lo, hi);
                    if (kb == c.kblocks - 1) {                        // rows beyond k do not count
                        const int r0 = kb * 16 + 2 * q, r1 = r0 + 8;
                        const uint32_t m0 = r0 >= a.k ? 0u : r0 + 1 >= a.k ? 0xFFFFu : 0xFFFFFFFFu;
                        const uint32_t m1 = r1 >= a.k ? 0u : r1 + 1 >= a.k ? 0xFFFFu : 0xFFFFFFFFu;
#pragma unroll
                        for (int u = 0; u < 4; ++u) { lo[u] &= m0; hi[u] &= m1; }
                    }
                    mma_16816(acc0, lo[0], lo[1], hi[0], hi[1], b.x, b.y);
                    mma_16816(acc1, lo[2], lo[3], hi[2], hi[3], b.x, b.y);
                    mma_16816(na, lo[0], lo[1], hi[0], hi[1], lo[0], hi[0]);
                    mma_16816(nb, lo[0], lo[1], hi[0], hi[1], lo[1], hi[1]);
                    mma_16816(nc, lo[2], lo[3], hi[2], hi[3], lo[2], hi[2]);
                    mma_16816(nd, lo[2], lo[3], hi[2], hi[3], lo[3], hi[3]);
                }
                n[0] += odd ? na[1] : na[0]; n[1] += odd ? nb[3] : nb[2];
                n[2] += odd ? nc[1] : nc[0]; n[3] += odd ? nd[3] : nd[2];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) n[u] = __shfl_sync(0xffffffffu, n[u], diag);
            if (c.norms) {                                            // (room for whole tiles; an odd one may end the block's columns)
                const float nq = q == 0 ? n[0] : q == 1 ? n[1] : q == 2 ? n[2] : n[3];
                if (base + 8 * q < c.tiles * 16) inv_s[base + g + 8 * q] = nq > 0.0f ? 1.0f / nq : 0.0f;
            }
        }
        if (q < 2) {
            // lane (g, 0): M^ products (value part and remainder part); lane (g, 1): V^'s
            const float e[4] = {(acc0[0] + acc0[1]) * bq, (acc0[2] + acc0[3]) * bq, (acc1[0] + acc1[1]) * bq, (acc1[2] + acc1[3]) * bq};
            // (a hair below the bound: offer() decides exactly)
            const float bound = fmaxf(best.s2, key_score(*reinterpret_cast<volatile unsigned int*>(&sh.floor_key[q]))) * 0.999999f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = base + g + 8 * u;
                if (HAVE) {
                    const float score = i < c.cnt ? e[u] * e[u] * inv_s[i] : -1.0f;
                    if (score >= bound && i < c.cnt) offer(sh, best, picks, q, score, (uint32_t)(c.e0 + i));
                } else if (e[u] * e[u] >= bound * n[u] && i < c.cnt)
                    offer(sh, best, picks, q, e[u] * e[u] * (n[u] > 0.0f ? 1.0f / n[u] : 0.0f), (uint32_t)(c.e0 + i));
            }
        }
        __syncwarp();
    }
}

__device__ void correlate(const OmpArgs& a, OmpSmem& sh, const CorrPlan& c, const uint32_t* col_list, uint2* frag, float* mem,
                          bool filled, const int* picks, int blk, int nblk) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, q = lane & 3;
    float back[2];
    stage_residuals(a, sh, frag, back, picks);
    __syncthreads();
    float* part = mem + c.part_off;
    float* inv_s = mem + c.inv_off;
    uint32_t* col_s = reinterpret_cast<uint32_t*>(mem + c.col_off);
    uint4* zc = reinterpret_cast<uint4*>(mem + c.z_off);
    const bool have = filled && c.norms, read = filled && c.cached;
    Top best;                                                         // of residual q & 1
    best.init();
    const bool stream = col_list == nullptr && !c.cached && c.tiles > kStreamTiles;
    if (stream && have) correlate_stream<true>(a, sh, c, frag, inv_s, back, picks, best);
    else if (stream) correlate_stream<false>(a, sh, c, frag, inv_s, back, picks, best);
    const int ks_log = 31 - __clz(c.ks), units = stream ? 0 : c.tiles * c.ks, kper = (c.kblocks + c.ks - 1) / c.ks;
    for (int u = warp; u < units; u += kWarps) {
        const int tile = u >> ks_log, part_k = u & (c.ks - 1);
        const int kb0 = part_k * kper, kb1 = kb0 + kper < c.kblocks ? kb0 + kper : c.kblocks;
        const int i0 = tile * 16 + g, i1 = i0 + 8;
        const bool ok0 = i0 < c.cnt, ok1 = i1 < c.cnt;
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        float n0 = 0.0f, n1 = 0.0f;
        // lane l < 16 looks up column l of the tile (and works out its key); the others get theirs from it
        uint32_t col_l = kNoColumn;
        {
            const int il = tile * 16 + (lane & 15);
            if (il < c.cnt) col_l = col_list ? (have ? col_s[il] : col_list[c.e0 + il]) : (uint32_t)(c.e0 + il);
            if (c.norms && !have && part_k == 0 && lane < 16) col_s[il] = col_l;
        }
        const uint32_t col0 = __shfl_sync(0xffffffffu, col_l, g), col1 = __shfl_sync(0xffffffffu, col_l, g + 8);
        const uint2* fb = frag + lane;
        uint4* zt = zc + (size_t)tile * c.kblocks * 32 + lane;
        if (read) {
#pragma unroll 4
            for (int kb = kb0; kb < kb1; ++kb) {
                const uint4 z = zt[(size_t)kb * 32];
                const uint2 b = lane < 16 ? fb[(size_t)kb * 16] : make_uint2(0u, 0u);
                mma_16816(acc, z.x, z.y, z.z, z.w, b.x, b.y);
            }
        } else {
            const ColKey key = column_key(a.seed_lo, a.seed_hi, col_l);
            ColKey k0, k1;
            k0.ck = __shfl_sync(0xffffffffu, key.ck, g); k0.mk = __shfl_sync(0xffffffffu, key.mk, g);
            k1.ck = __shfl_sync(0xffffffffu, key.ck, g + 8); k1.mk = __shfl_sync(0xffffffffu, key.mk, g + 8);
            uint32_t h00 = k0.ck + (uint32_t)(kb0 * 8 + q) * k0.mk, h01 = h00 + 4u * k0.mk;
            uint32_t h10 = k1.ck + (uint32_t)(kb0 * 8 + q) * k1.mk, h11 = h10 + 4u * k1.mk;
            const uint32_t st0 = 8u * k0.mk, st1 = 8u * k1.mk;
            if (have) {
#pragma unroll 2
                for (int kb = kb0; kb < kb1; ++kb) {
                    const uint2 b = lane < 16 ? fb[(size_t)kb * 16] : make_uint2(0u, 0u);
                    const uint32_t z00 = z_pair_from_word(h00), z10 = z_pair_from_word(h10), z01 = z_pair_from_word(h01), z11 = z_pair_from_word(h11);
                    h00 += st0; h01 += st0; h10 += st1; h11 += st1;
                    mma_16816(acc, z00, z10, z01, z11, b.x, b.y);
                }
            } else {
#pragma unroll 1
                for (int kb = kb0; kb < kb1; ++kb) {
                    const uint2 b = lane < 16 ? fb[(size_t)kb * 16] : make_uint2(0u, 0u);
                    uint32_t z[4] = {z_pair_from_word(h00), z_pair_from_word(h10), z_pair_from_word(h01), z_pair_from_word(h11)};
                    h00 += st0; h01 += st0; h10 += st1; h11 += st1;
                    if (kb == c.kblocks - 1) {                         // rows beyond k do not count
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int row = kb * 16 + 2 * q + (e & 2 ? 8 : 0);
                            if (row >= a.k) z[e] = 0u;
                            else if (row + 1 >= a.k) z[e] &= 0xFFFFu;
                        }
                    }
                    mma_16816(acc, z[0], z[1], z[2], z[3], b.x, b.y);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f = half2_bits_to_float2(z[e]);
                        float& n2 = (e & 1) ? n1 : n0;
                        n2 = __fmaf_rn(f.x, f.x, n2); n2 = __fmaf_rn(f.y, f.y, n2);
                    }
                    if (c.cached) zt[(size_t)kb * 32] = make_uint4(z[0], z[1], z[2], z[3]);
                }
                n0 += __shfl_xor_sync(0xffffffffu, n0, 1); n0 += __shfl_xor_sync(0xffffffffu, n0, 2);
                n1 += __shfl_xor_sync(0xffffffffu, n1, 1); n1 += __shfl_xor_sync(0xffffffffu, n1, 2);
            }
        }
        // lane (g, 0): M^ products of columns g and g + 8 (value part and remainder part); lane (g, 1): V^'s
        const float d0 = acc[0] + acc[1], d1 = acc[2] + acc[3];
        if (c.ks > 1) {
            float* dst = part + (size_t)u * 32;
            if (q < 2) { dst[g * 2 + q] = d0; dst[(g + 8) * 2 + q] = d1; }
            if (!have && q == 2) { sh.npart[u & 63][g] = n0; sh.npart[u & 63][g + 8] = n1; }
        } else {
            float v0, v1;
            if (have) { v0 = ok0 ? inv_s[i0] : 0.0f; v1 = ok1 ? inv_s[i1] : 0.0f; }
            else {
                v0 = n0 > 0.0f ? 1.0f / n0 : 0.0f; v1 = n1 > 0.0f ? 1.0f / n1 : 0.0f;
                if (c.norms && q == 0) { inv_s[i0] = v0; inv_s[i1] = v1; }
            }
            if (q < 2) {
                const float bq = q == 0 ? back[0] : back[1];
                const float e0 = d0 * bq, e1 = d1 * bq;
                if (ok0) offer(sh, best, picks, q, e0 * e0 * v0, col0);
                if (ok1) offer(sh, best, picks, q, e1 * e1 * v1, col1);
            }
        }
    }
    if (c.ks > 1) {
        __syncthreads();
        // thread = (column, residual): the sums over the row parts
        for (int e = t; e < c.tiles * 32; e += kT) {
            const int idx = e >> 1, m = e & 1, tile = idx >> 4;
            float d = 0.0f, n2 = 0.0f;
            for (int p = 0; p < c.ks; ++p) {
                d += part[(size_t)(tile * c.ks + p) * 32 + (idx & 15) * 2 + m];
                if (!have) n2 += sh.npart[tile * c.ks + p][idx & 15];
            }
            float inv;
            if (have) inv = inv_s[idx];
            else { inv = n2 > 0.0f ? 1.0f / n2 : 0.0f; if (c.norms && m == 0) inv_s[idx] = inv; }
            if (idx < c.cnt) {
                const float f = d * (m == 0 ? back[0] : back[1]);
                offer(sh, best, picks, m, f * f * inv, col_list ? (c.norms ? col_s[idx] : col_list[c.e0 + idx]) : (uint32_t)(c.e0 + idx));
            }
        }
        // (kT is even: a thread has met one residual only, that of its own parity)
    }
    const int mine = c.ks > 1 ? (t & 1) : (q < 2 ? q : -1);
    Top none, m0 = best, m1 = best;
    none.init();
    if (mine != 0) m0 = none;
    if (mine != 1) m1 = none;
    warp_merge(m0);
    warp_merge(m1);
    if (lane == 0) { sh.wtop[0][warp] = m0; sh.wtop[1][warp] = m1; }
    __syncthreads();
    if (warp < 2) {
        Top m = none;
        if (lane < kWarps) m = sh.wtop[warp][lane];
        warp_merge(m);
        if (lane == 0) {
            // best column, its score, and the best score that this block did not forward
            a.corr_cand[(size_t)warp * nblk + blk] = make_float4(m.s1, __uint_as_float(m.i1), m.s2, 0.0f);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// bookkeeping: one group of GS blocks per recovery, block g owns rows [row0, row0 + R) of A
// ------------------------------------------------------------------------------------------------
template <int CL> struct Group { static constexpr int GS = group_blocks(CL); };

// dynamic shared memory of a bookkeeping block, in doubles: residual slice | partial sums | exchanged sums | exchange slots | q
struct BookMem {
    double *rr, *part, *cs, *x0, *x1, *xrn, *qs;
    int R, P, row0, rows;                                  // slice length, parts per row in the update, first row, rows owned
};
__device__ BookMem book_mem(const OmpArgs& a, double* base, int gs, int g, bool two) {
    BookMem b;
    b.R = slice_rows(a.k, gs);
    b.row0 = g * b.R;
    b.rows = b.row0 >= a.k ? 0 : (a.k - b.row0 < b.R ? a.k - b.row0 : b.R);
    b.P = b.R >= kT ? 1 : kT / b.R;
    b.rr = base; b.part = b.rr + b.R;
    b.cs = b.part + (b.R > kT ? b.R : kT);
    b.x0 = b.cs + even(a.s + 4);
    b.x1 = two ? b.x0 + (size_t)gs * exchange_stride(a.s) : b.x0;
    b.xrn = b.x1 + (size_t)gs * exchange_stride(a.s);
    b.qs = b.xrn + 2 * gs;
    return b;
}

// rows 2 p, 2 p + 1 of a column in this slice, scaled by sigma (rows beyond k are zero)
__device__ __forceinline__ double2 column_rows(const OmpArgs& a, const BookMem& b, const ColKey& key, int p) {
    const int row = b.row0 + 2 * p;
    const float2 z = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)(row >> 1) * key.mk));
    return make_double2(row < a.k ? a.sigma * (double)z.x : 0.0, row + 1 < a.k ? a.sigma * (double)z.y : 0.0);
}

// q_l of this slice: in shared memory for the first q_cols, in global memory beyond
__device__ __forceinline__ const double* q_slice(const OmpArgs& a, const BookMem& b, int m, int l) {
    return l < a.q_cols ? b.qs + (size_t)l * b.R : a.q + ((size_t)m * a.s + l) * a.k + b.row0;
}

template <int N>
__device__ __forceinline__ void warp_sums(double (&v)[N]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < N; ++u) v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
    }
}

constexpr int kLanePairs = 4;                              // row pairs of a column that a lane generates at a time (256 rows per warp)

// Partial products of column `col` over this slice with q_0 .. q_(j-1) and the residual, and (full) its squared norm and the
// residual's, sent to slot g of the exchange buffer of every block of the group.  Warp = V vectors at a time (as many as it takes
// to keep all warps busy: the sums of a vector over the lanes are most of the work); every warp generates the slice of the column
// for itself (a few words per lane), which saves a barrier.
template <int GS, int V>
__device__ __forceinline__ void send_vectors(cg::cluster_group& cluster, const OmpArgs& a, const BookMem& b, int m, int j, const ColKey& key,
                                             double* xbuf, int rank0, int g) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pairs = b.R / 2, xstride = exchange_stride(a.s);
    const bool vec = (a.k & 1) == 0 || j <= a.q_cols;
    for (int l0 = warp; l0 <= j; l0 += V * kWarps) {
        double acc[V];
        const double* v[V];
        bool live[V];
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const int l = l0 + u * kWarps;
            acc[u] = 0.0;
            live[u] = l <= j;
            v[u] = l < j ? q_slice(a, b, m, l) : b.rr;
        }
        for (int p0 = lane; p0 < pairs; p0 += 32 * kLanePairs) {
            double2 x[kLanePairs];
#pragma unroll
            for (int i = 0; i < kLanePairs; ++i) x[i] = p0 + 32 * i < pairs ? column_rows(a, b, key, p0 + 32 * i) : make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < V; ++u) {
                if (!live[u]) continue;
#pragma unroll
                for (int i = 0; i < kLanePairs; ++i) {
                    const int r = 2 * (p0 + 32 * i);
                    if (r >= b.rows) continue;
                    if (vec) {
                        const double2 y = *reinterpret_cast<const double2*>(v[u] + r);       // (an odd last row: shared memory, zero beyond)
                        acc[u] = fma(y.x, x[i].x, acc[u]); acc[u] = fma(y.y, x[i].y, acc[u]);
                    } else {
                        acc[u] = fma(v[u][r], x[i].x, acc[u]);
                        if (r + 1 < b.rows) acc[u] = fma(v[u][r + 1], x[i].y, acc[u]);
                    }
                }
            }
        }
        warp_sums(acc);
        if (lane < GS) {
            double* dst = cluster.map_shared_rank(xbuf, rank0 + lane) + (size_t)g * xstride;
#pragma unroll
            for (int u = 0; u < V; ++u) if (live[u]) dst[l0 + u * kWarps] = acc[u];
        }
    }
}
template <int GS>
__device__ void send_products(cg::cluster_group& cluster, const OmpArgs& a, const BookMem& b, int m, int j, uint32_t col, bool full,
                              double* xbuf, int rank0, int g) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pairs = b.R / 2, xstride = exchange_stride(a.s);
    const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
    if (full && warp == kWarps - 1) {
        double acc[2] = {0.0, 0.0};
        for (int p = lane; p < pairs; p += 32) {
            const double2 x = column_rows(a, b, key, p), y = *reinterpret_cast<const double2*>(b.rr + 2 * p);
            acc[0] = fma(x.x, x.x, acc[0]); acc[0] = fma(x.y, x.y, acc[0]);
            acc[1] = fma(y.x, y.x, acc[1]); acc[1] = fma(y.y, y.y, acc[1]);
        }
        warp_sums(acc);
        if (lane < GS) {
            double* dst = cluster.map_shared_rank(xbuf, rank0 + lane) + (size_t)g * xstride;
            dst[a.s] = acc[0]; dst[a.s + 1] = acc[1];
        }
    }
    if (j < kWarps) send_vectors<GS, 1>(cluster, a, b, m, j, key, xbuf, rank0, g);
    else if (j < 2 * kWarps) send_vectors<GS, 2>(cluster, a, b, m, j, key, xbuf, rank0, g);
    else send_vectors<GS, 4>(cluster, a, b, m, j, key, xbuf, rank0, g);
}

// a further candidate: its product with the residual and its squared norm (warp = one candidate)
template <int GS>
__device__ void send_candidate(cg::cluster_group& cluster, const OmpArgs& a, const BookMem& b, uint32_t col, int e, double* xbuf, int rank0, int g) {
    const int lane = threadIdx.x & 31, pairs = b.R / 2;
    const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
    double acc[2] = {0.0, 0.0};
    for (int p = lane; p < pairs; p += 32) {
        const double2 x = column_rows(a, b, key, p), y = *reinterpret_cast<const double2*>(b.rr + 2 * p);
        acc[0] = fma(x.x, y.x, acc[0]); acc[0] = fma(x.y, y.y, acc[0]);
        acc[1] = fma(x.x, x.x, acc[1]); acc[1] = fma(x.y, x.y, acc[1]);
    }
    warp_sums(acc);
    if (lane < GS) {
        double* dst = cluster.map_shared_rank(xbuf, rank0 + lane) + (size_t)g * exchange_stride(a.s) + a.s + 2 + 2 * (e - 1);
        dst[0] = acc[0]; dst[1] = acc[1];
    }
}

// squared norm of the residual slice, sent to slot g of xrn of every block of the group (one warp)
template <int GS>
__device__ void send_norm(cg::cluster_group& cluster, const BookMem& b, int rank0, int g) {
    if (threadIdx.x >= 32) return;
    double acc[1] = {0.0};
    for (int r = threadIdx.x; r < b.R; r += 32) acc[0] = fma(b.rr[r], b.rr[r], acc[0]);
    warp_sums(acc);
    if (threadIdx.x < GS) cluster.map_shared_rank(b.xrn, rank0 + threadIdx.x)[g] = acc[0];
}

// the residual of this slice as row n of the screened batch (scaled binary16, and fp64 for the resolve kernel)
__device__ void emit_row(const OmpArgs& a, const BookMem& b, size_t n, double rn, int g) {
    const double sc = residual_scale(rn);
    for (int r = threadIdx.x; r < b.rows; r += kT) {
        a.rt[n * a.kp + b.row0 + r] = half_rn_bits(b.rr[r] * sc);
        a.rhist[n * a.k + b.row0 + r] = b.rr[r];
    }
    if (g == 0 && threadIdx.x == 0) a.inv_scale[n] = (float)(1.0 / sc);
}

// Block `blk` of the screen forwarded its best column for residual m, but another scored inside the rescoring window as well.
// Its columns are screened again here and every free one inside the window (with a little slack: the sums run in another order)
// that was not forwarded is noted, so that all of them reach the fp64 decision.  Lock-step (col_list == nullptr): thread = column;
// a block's share of a list is a few columns of as many rows: warp = column.
__device__ void rescan_block(const OmpArgs& a, OmpSmem& sh, const uint32_t* col_list, unsigned int n_cols, int m, int j, int blk, int nblk,
                             float thr, uint32_t forwarded) {
    const CorrPlan c = corr_plan(n_cols, a.k, a.z_words, blk, nblk);
    const float2* r = reinterpret_cast<const float2*>(a.r32);
    auto note = [&](uint32_t col, float acc, float n2) {
        const float sc = n2 > 0.0f ? acc * acc / n2 : 0.0f;
        if (sc >= thr * 0.9999f && col != forwarded && !in_list(a.lam + (size_t)m * a.s, j, col)) {
            const int slot = atomicAdd(&sh.rbuf_n, 1);
            if (slot < kRescanCap) sh.rbuf[slot] = col;
        }
    };
    if (col_list != nullptr) {
        const int lane = threadIdx.x & 31;
        for (int idx = threadIdx.x >> 5; idx < c.cnt; idx += kWarps) {
            const uint32_t col = col_list[c.e0 + idx];
            const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
            float acc = 0.0f, n2 = 0.0f;
            for (int p = lane; 2 * p < a.k; p += 32) {
                const float4 rr = __ldcg(reinterpret_cast<const float4*>(r) + p);        // (padded by two rows)
                const float2 z = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)p * key.mk));
                acc = __fmaf_rn(z.x, m ? rr.y : rr.x, acc); n2 = __fmaf_rn(z.x, z.x, n2);
                if (2 * p + 1 < a.k) { acc = __fmaf_rn(z.y, m ? rr.w : rr.z, acc); n2 = __fmaf_rn(z.y, z.y, n2); }
            }
            for (int o = 16; o > 0; o >>= 1) { acc += __shfl_xor_sync(0xffffffffu, acc, o); n2 += __shfl_xor_sync(0xffffffffu, n2, o); }
            if (lane == 0) note(col, acc, n2);
        }
        __syncthreads();
        return;
    }
    for (int idx = threadIdx.x; idx < c.cnt; idx += kT) {
        const uint32_t col = c.e0 + (uint32_t)idx;
        const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
        uint32_t h = key.ck;
        float acc = 0.0f, n2 = 0.0f;
        for (int row = 0; row < a.k; row += 2) {
            const float2 r0 = __ldcg(r + row), r1 = row + 1 < a.k ? __ldcg(r + row + 1) : make_float2(0.0f, 0.0f);
            const float2 z = half2_bits_to_float2(z_pair_from_word(h));
            h += key.mk;
            acc = __fmaf_rn(z.x, m ? r0.y : r0.x, acc); n2 = __fmaf_rn(z.x, z.x, n2);
            if (row + 1 < a.k) { acc = __fmaf_rn(z.y, m ? r1.y : r1.x, acc); n2 = __fmaf_rn(z.y, z.y, n2); }
        }
        note(col, acc, n2);
    }
    __syncthreads();
}

// The screened candidates of pick j: everything within 2e-3 (relative, squared scores) of the best fp32 score, the best one
// first; every block of a group finds the same list.  Returns their number; *first: the best one (a list of more than one is in
// sh.cidx); *inexact: not every column inside the window is in it (list mode: the screening pass then judges the list's members as
// it does all others).  col_list, n_cols: the columns that the blocks share, all of them (nullptr) or a list's.  Every warp reads all
// blocks' entries: the usual case of one candidate needs no barrier.
__device__ int gather_candidates(const OmpArgs& a, OmpSmem& sh, int m, int j, int nblk, const uint32_t* col_list, unsigned int n_cols,
                                 uint32_t* first, bool* inexact) {
    constexpr int kPer = kCorrBlocks / 32;
    const int t = threadIdx.x, lane = t & 31;
    const float4* cc = a.corr_cand + (size_t)m * nblk;
    float4 c[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int e = u * 32 + lane;
        c[u] = e < nblk ? __ldcg(cc + e) : make_float4(-1.0f, __uint_as_float(kNoColumn), -1.0f, 0.0f);
    }
    unsigned int key = 0u;
#pragma unroll
    for (int u = 0; u < kPer; ++u) if (__float_as_uint(c[u].y) != kNoColumn) key = max(key, score_key(c[u].x));
    key = __reduce_max_sync(0xffffffffu, key);
    if (key == 0u) return 0;
    const float mx = key_score(key);
    const float thr = mx - 2e-3f * fabsf(mx);
    int total = 0;
    bool kept = false;
    uint32_t best = kNoColumn;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const bool in = __float_as_uint(c[u].y) != kNoColumn && c[u].x >= thr;
        total += __popc(__ballot_sync(0xffffffffu, in));
        if (in && score_key(c[u].x) == key) best = min(best, __float_as_uint(c[u].y));
        kept = kept || (c[u].z >= 0.0f && c[u].z >= thr);
    }
    best = __reduce_min_sync(0xffffffffu, best);
    kept = __any_sync(0xffffffffu, kept);
    *first = best;
    if (total == 1 && !kept) return 1;
    // several candidates, or columns that a block kept to itself
    __syncthreads();
    if (t == 0) { sh.nc = 0; sh.rescan_n = 0; sh.rbuf_n = 0; }
    __syncthreads();
    if (t < 32) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const uint32_t idx = __float_as_uint(c[u].y);
            const bool in = idx != kNoColumn && c[u].x >= thr && idx != best;
            const unsigned int b = __ballot_sync(0xffffffffu, in);
            const int slot = 1 + sh.nc + __popc(b & ((1u << lane) - 1u));
            if (in && slot < kRescoreCap) sh.cidx[slot] = idx;
            __syncwarp();
            if (lane == 0) sh.nc += __popc(b);
            __syncwarp();
            if (c[u].z >= 0.0f && c[u].z >= thr) {
                const int q = atomicAdd(&sh.rescan_n, 1);
                if (q < 8) { sh.rescan_blk[q] = u * 32 + lane; sh.rescan_col[q] = idx; }
            }
        }
        if (lane == 0) sh.cidx[0] = best;
    }
    __syncthreads();
    if (kept) {
        const int n_blk = sh.rescan_n < 8 ? sh.rescan_n : 8;
        for (int q = 0; q < n_blk; ++q) rescan_block(a, sh, col_list, n_cols, m, j, sh.rescan_blk[q], nblk, thr, sh.rescan_col[q]);
        const bool over = sh.rescan_n > 8 || sh.rbuf_n > kRescanCap || total + sh.rbuf_n > kRescoreCap;
        if (over) *inexact = true;
        if (t == 0) {
            if (over && col_list == nullptr) atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_CANDIDATE_OVERFLOW);
            if (!over)
                // ascending order, so that every block of the group has the same list whatever order the atomics gave
                for (int e = 0; e < sh.rbuf_n; ++e) {
                    int lo = e;
                    for (int q = e + 1; q < sh.rbuf_n; ++q) if (sh.rbuf[q] < sh.rbuf[lo]) lo = q;
                    const uint32_t v = sh.rbuf[lo]; sh.rbuf[lo] = sh.rbuf[e]; sh.rbuf[e] = v;
                    sh.cidx[total + e] = v;
                }
        }
        if (!over) total += sh.rbuf_n;
    }
    if (total > kRescoreCap) {
        if (t == 0) atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_CANDIDATE_OVERFLOW);
        total = kRescoreCap;
        *inexact = true;
    }
    __syncthreads();
    return total;
}

// ------------------------------------------------------------------------------------------------
// the Gram path: lists of up to kGramList columns
// ------------------------------------------------------------------------------------------------
constexpr int kRowBatch = 2 * kWarps;                 // rows of A per step of gram_rows: two per warp

// the list's columns as binary16 (zlist) and p0 = Z_C^T y for both residuals: block = column
__device__ void gram_prepare(const OmpArgs& a, OmpSmem& sh, int n) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, k = a.k;
    __shared__ double red2[2][kWarps];
    for (int b = blockIdx.x; b < n; b += gridDim.x) {
        const ColKey key = column_key(a.seed_lo, a.seed_hi, a.cand_list[b]);
        uint32_t* dst = reinterpret_cast<uint32_t*>(a.zlist + (size_t)b * a.kp);
        double dm = 0.0, dv = 0.0;
        for (int p = t; 2 * p < k; p += kT) {
            uint32_t z2 = z_pair_from_word(key.ck + (uint32_t)p * key.mk);
            if (2 * p + 1 >= k) z2 &= 0xFFFFu;
            dst[p] = z2;
            const float2 z = half2_bits_to_float2(z2);
            dm += (double)z.x * a.y64[2 * p]; dv += (double)z.x * a.y64[k + 2 * p];
            if (2 * p + 1 < k) { dm += (double)z.y * a.y64[2 * p + 1]; dv += (double)z.y * a.y64[k + 2 * p + 1]; }
        }
        dm = warp_sum(dm); dv = warp_sum(dv);
        __syncthreads();
        if (lane == 0) { red2[0][warp] = dm; red2[1][warp] = dv; }
        __syncthreads();
        if (t < 2) {
            double s = 0.0;
            for (int w = 0; w < kWarps; ++w) s += red2[t][w];
            a.p0[t * kGramList + b] = s;
        }
    }
}

// G = Z_C^T Z_C: warp = one pair of columns (products of two binary16 numbers are exact in fp32, sums in fp64)
__device__ void gram_matrix(const OmpArgs& a, int n) {
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * kWarps + (threadIdx.x >> 5), nw = gridDim.x * kWarps;
    const int vecs = a.kp >> 3;
    for (int e = gw; e < n * n; e += nw) {
        const int b = e / n, c = e % n;
        if (c < b) continue;
        const uint4* pb = reinterpret_cast<const uint4*>(a.zlist + (size_t)b * a.kp);
        const uint4* pc = reinterpret_cast<const uint4*>(a.zlist + (size_t)c * a.kp);
        double acc = 0.0;
#pragma unroll 2
        for (int v = lane; v < vecs; v += 32) {
            const uint4 x = __ldcg(pb + v), y = __ldcg(pc + v);
            const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, yw[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 fa = half2_bits_to_float2(xw[q]), fb = half2_bits_to_float2(yw[q]);
                acc += (double)(fa.x * fb.x);
                acc += (double)(fa.y * fb.y);
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) { a.gram[(size_t)b * kGramList + c] = acc; a.gram[(size_t)c * kGramList + b] = acc; }
    }
}

// All picks of recovery m on the Gram matrix, one block.  Thread i owns list member i: its correlation p_i = <z_i, r> and
// its products w_l(i) = <q_l, z_i> with the orthogonal vectors of the picks so far (shared memory, global memory when they do
// not fit).  A pick reads c_l = sigma w_l(pick) and updates
//     w_j(i) = gamma (sigma G(pick, i) - sum_l c_l w_l(i)),    p_i -= a_j w_j(i):
// one block barrier per pick and j fp64 multiply-adds per member.  64 picks on 64 columns: 270 us with the k-free form of
// the printed recurrences (F kept, p recomputed from x), 40 us this way.
//
// fin, vc, fc: what the control block said of both recoveries before this phase, read by the whole grid ahead of a grid barrier.
// Both blocks look both recoveries up in the list and have to come to the same answer, while each moves its own recovery's words on
// as it goes: neither may read the other's here.
__device__ void gram_picks(const OmpArgs& a, int m, int n, double* dyn, const int (&fin)[2], const int (&vc)[2], const uint32_t (&fc)[2]) {
    __shared__ unsigned int khi[2][8], klo[2][8];
    __shared__ uint32_t kcol[2][8];
    __shared__ int kidx[2][8];
    __shared__ double ps[2][kGramList], gd[kGramList];
    __shared__ int li[kGramList + 1];
    __shared__ int found;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, s = a.s;
    for (int c = t; c < a.half_n; c += kT) {
        a.rep_count[m * a.half_n + c] = 0u;
        a.tau[m * a.half_n + c] = __int_as_float(0x7f800000);
    }
    const int v0 = m ? vc[1] : vc[0];
    const uint32_t forced0 = m ? fc[1] : fc[0];
    const int base = v0 + (forced0 != kNoColumn ? 1 : 0);
    int end = base + a.half_n < s ? base + a.half_n : s;
    if (end > n + 1) end = n + 1;
    const double sigma = a.sigma, sig2 = sigma * sigma;
    const bool member = t < n;
    const uint32_t my_col = member ? a.cand_list[t] : kNoColumn;
    double* ac = a.acoef + (size_t)m * s;
    double* gm = a.gam + (size_t)m * s;
    double* crow = a.crow + (size_t)m * s * s;
    double* ccol = a.ccol + (size_t)m * s * s;
    uint32_t* lam = a.lam + (size_t)m * s;
    // w in shared memory when it fits, then G
    const size_t room = kOmpDynBytes / sizeof(double);
    const bool w_sm = (size_t)n * end <= room;
    double* W = w_sm ? dyn : a.wgram + (size_t)m * kGramList * s;
    const bool g_sm = w_sm && (size_t)n * end + (size_t)n * n <= room;
    double* Gs = dyn + (size_t)n * end;
    if (g_sm)
        for (int e = t; e < n * n; e += kT) Gs[e] = __ldcg(a.gram + (size_t)(e / n) * kGramList + e % n);
    double p = 0.0;
    bool taken = false;
    if (t == 0) found = 0;
    __syncthreads();
    double my_g = 1.0;
    int want = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (fin[u]) continue;
        const int vu = vc[u];
        const uint32_t fu = fc[u];
        want += vu + (fu != kNoColumn ? 1 : 0);
        if (!member) continue;
        for (int l = 0; l < vu; ++l) if (a.lam[(size_t)u * s + l] == my_col) { if (u == m) li[l] = t; atomicAdd(&found, 1); }
        if (fu != kNoColumn && my_col == fu) { if (u == m) li[vu] = t; atomicAdd(&found, 1); }
    }
    if (member) {
        p = __ldcg(a.p0 + m * kGramList + t);
        my_g = __ldcg(a.gram + (size_t)t * kGramList + t);
        gd[t] = my_g;
    }
    __syncthreads();
    if (found != want) {                                              // a pick is missing from the list: the other path serves
        if (t == 0) a.ctl->gram_ok = 0;
        return;
    }
    if (m ? fin[1] : fin[0]) return;
    const double inv_g = my_g > 0.0 ? 1.0 / my_g : 0.0;
    int hi = base, extra = 0, dep = 0;
    const int nw = (n + 31) >> 5;                                     // the warps that hold members go on by themselves
    if (warp >= nw) return;
    auto meet = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nw * 32) : "memory"); };
    for (int j = 0; j < end; ++j) {
        const int par = j & 1;
        const bool given = j < base;                                  // a confirmed pick (j < v0) or the prescribed one
        if (member) ps[par][t] = p;
        int q;
        if (given) {
            meet();
            q = li[j];
        } else {
            // "Select": argmax of p_i^2 / g_ii over the free list members, lowest column index on ties
            {
                const double sc = (member && !taken && my_g > 0.0) ? p * p * inv_g : -1.0;
                const unsigned long long bits = sc >= 0.0 ? (unsigned long long)__double_as_longlong(sc) + 1ull : 0ull;
                const unsigned int h = __reduce_max_sync(0xffffffffu, (unsigned int)(bits >> 32));
                const bool e1 = (unsigned int)(bits >> 32) == h;
                const unsigned int l = __reduce_max_sync(0xffffffffu, e1 ? (unsigned int)bits : 0u);
                const bool e2 = e1 && (unsigned int)bits == l && bits != 0ull;
                const uint32_t c = __reduce_min_sync(0xffffffffu, e2 ? my_col : kNoColumn);
                const unsigned int who = __ballot_sync(0xffffffffu, e2 && my_col == c);
                if (lane == 0) { khi[par][warp] = h; klo[par][warp] = l; kcol[par][warp] = c; kidx[par][warp] = who ? warp * 32 + __ffs(who) - 1 : -1; }
            }
            meet();
            const unsigned int h0 = lane < nw ? khi[par][lane] : 0u, l0 = lane < nw ? klo[par][lane] : 0u;
            const uint32_t c0 = lane < nw ? kcol[par][lane] : kNoColumn;
            const unsigned int h = __reduce_max_sync(0xffffffffu, h0);
            const unsigned int l = __reduce_max_sync(0xffffffffu, h0 == h ? l0 : 0u);
            const bool e = h0 == h && l0 == l && c0 != kNoColumn;
            const uint32_t c = __reduce_min_sync(0xffffffffu, e ? c0 : kNoColumn);
            const unsigned int who = __ballot_sync(0xffffffffu, e && c0 == c);
            if (who == 0u) { extra = 1; break; }                      // every list member is in the support already
            q = kidx[par][__ffs(who) - 1];
        }
        const double pq = ps[par][q], gqq = gd[q];
        double acc0 = 0.0, acc1 = 0.0, sq0 = 0.0, sq1 = 0.0;
        const int ti = member ? t : 0;
        {
            int l = 0;
#pragma unroll 4
            for (; l + 1 < j; l += 2) {
                const double c0 = sigma * W[(size_t)l * n + q], c1 = sigma * W[(size_t)(l + 1) * n + q];
                acc0 = fma(c0, W[(size_t)l * n + ti], acc0); sq0 = fma(c0, c0, sq0);
                acc1 = fma(c1, W[(size_t)(l + 1) * n + ti], acc1); sq1 = fma(c1, c1, sq1);
            }
            if (l < j) { const double c0 = sigma * W[(size_t)l * n + q]; acc0 = fma(c0, W[(size_t)l * n + ti], acc0); sq0 = fma(c0, c0, sq0); }
        }
        const double gnn = sig2 * gqq, piv = gnn - (sq0 + sq1);
        if (t == 0 && !given) {
            lam[j] = a.cand_list[q];
            a.pick_score[(size_t)m * s + j] = fabs(pq) / sqrt(gqq);
        }
        if (!(piv > kPivot * gnn)) {
            // dependent column: a speculative one is screened and ends the recovery if confirmed; a prescribed one ends it now
            if (given) {
                if (t == 0) {
                    lam[j] = a.cand_list[q];
                    a.cnt->stopped[m] = 1;
                    atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_DEPENDENT_COLUMN);
                    a.cnt->done[m] = j; a.ctl->v[m] = j; a.ctl->finished[m] = 1; a.ctl->forced[m] = kNoColumn;
                }
                hi = j;
            } else { dep = 1; hi = j + 1; }
            break;
        }
        const double gamma = rsqrt(piv);
        const double aj = gamma * sigma * pq;
        if (member) {
            const double gq = g_sm ? Gs[q * n + t] : __ldcg(a.gram + (size_t)q * kGramList + t);
            const double w = gamma * (sigma * gq - (acc0 + acc1));
            W[(size_t)j * n + t] = w;
            p -= aj * w;
            if (t == q) taken = true;
        }
        for (int l = t; l < j; l += nw * 32) {
            const double c = sigma * W[(size_t)l * n + q];
            crow[(size_t)j * s + l] = c; ccol[(size_t)l * s + j] = c;
        }
        if (t == 0) {
            ac[j] = aj; gm[j] = gamma;
            if (given && j == v0) {
                lam[j] = forced0;
                a.cnt->done[m] = j + 1; a.ctl->v[m] = j + 1; a.ctl->forced[m] = kNoColumn;
            }
        }
        hi = j + 1;
    }
    if (t == 0 && !a.ctl->finished[m]) {
        a.ctl->base[m] = base;
        a.ctl->hi[m] = hi < base ? base : hi;
        a.ctl->extra[m] = extra;
        a.ctl->dep[m] = dep;
        a.ctl->list_exact[m] = 1;
    }
}

// q_l and the residuals r_l of all picks, two rows of A per warp: lane owns the picks lane, lane + 32, ... and carries
// sum_{l < pick} c^(pick)_l q_l[row] for them; q_l follows from its owner's sum, one shuffle per pick.
__device__ void gram_rows(const OmpArgs& a, double* dyn) {
    volatile SpecCtl* ctl = a.ctl;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, k = a.k, s = a.s;
    const int batches = (k + kRowBatch - 1) / kRowBatch;
    int staged = -1, L = 0;
    double* nrm = dyn;                                                // [kWarps][L + 1]
    double* zt = nrm + kWarps * (kGramList + 1);                      // [L][kRowBatch]
    double* gs = zt + (size_t)kGramList * kRowBatch;                  // gamma, a
    double* as = gs + kGramList;
    double* ct = as + kGramList;                                      // [L][L] when it fits
    const size_t ct_room = kOmpDynBytes / sizeof(double) - (size_t)(ct - dyn);
    bool ct_sm = false;
    for (int item = blockIdx.x; item < 2 * batches; item += gridDim.x) {
        const int m = item & 1, batch = item >> 1;
        if (ctl->finished[m]) continue;
        const int base = ctl->base[m];
        if (staged != m) {
            __syncthreads();
            L = ctl->hi[m] - (ctl->dep[m] ? 1 : 0);                   // a dependent pick leaves no new vector behind
            ct_sm = (size_t)L * L <= ct_room;
            for (int l = t; l < L; l += kT) { gs[l] = __ldcg(a.gam + (size_t)m * s + l); as[l] = __ldcg(a.acoef + (size_t)m * s + l); }
            if (ct_sm)
                for (int e = t; e < L * L; e += kT) {
                    const int l = e / L, j = e % L;
                    ct[e] = j > l ? __ldcg(a.ccol + (size_t)m * s * s + (size_t)l * s + j) : 0.0;
                }
            staged = m;
        }
        __syncthreads();
        for (int e = t; e < L * (kRowBatch / 2); e += kT) {
            const int l = e / (kRowBatch / 2), p = e % (kRowBatch / 2), row = batch * kRowBatch + 2 * p;
            const ColKey key = column_key(a.seed_lo, a.seed_hi, a.lam[(size_t)m * s + l]);
            const float2 z = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)(row >> 1) * key.mk));
            zt[l * kRowBatch + 2 * p] = a.sigma * (double)z.x;
            zt[l * kRowBatch + 2 * p + 1] = a.sigma * (double)z.y;
        }
        __syncthreads();
        const int row = batch * kRowBatch + 2 * warp;
        const bool ok0 = row < k, ok1 = row + 1 < k;
        double r0 = ok0 ? a.y64[(size_t)m * k + row] : 0.0, r1 = ok1 ? a.y64[(size_t)m * k + row + 1] : 0.0;
        double acc0[kGramList / 32], acc1[kGramList / 32];
#pragma unroll
        for (int u = 0; u < kGramList / 32; ++u) acc0[u] = acc1[u] = 0.0;
        double* qg = a.q + (size_t)m * s * k;
        double* rh = a.rhist + (size_t)m * a.half_n * k;
        const double* cg_ = a.ccol + (size_t)m * s * s;
        const int U = (L + 31) >> 5;
#pragma unroll
        for (int u0 = 0; u0 < kGramList / 32; ++u0) {
            if (u0 >= U) break;
            const int n_here = L - u0 * 32 < 32 ? L - u0 * 32 : 32;
            double kq0 = 0.0, kq1 = 0.0, kr0 = 0.0, kr1 = 0.0;
            for (int ll = 0; ll < n_here; ++ll) {
                const int l = u0 * 32 + ll;
                const double v0 = __shfl_sync(0xffffffffu, acc0[u0], ll), v1 = __shfl_sync(0xffffffffu, acc1[u0], ll);
                const double2 z = *reinterpret_cast<const double2*>(zt + l * kRowBatch + 2 * warp);
                const double q0 = gs[l] * (z.x - v0), q1 = gs[l] * (z.y - v1);
                if (lane == ll) { kq0 = q0; kq1 = q1; kr0 = r0; kr1 = r1; }
                r0 -= as[l] * q0; r1 -= as[l] * q1;
#pragma unroll
                for (int u = u0; u < kGramList / 32; ++u) {
                    if (u < U) {
                        const int j = u * 32 + lane;
                        const double c = j < L ? (ct_sm ? ct[l * L + j] : (j > l ? __ldcg(cg_ + (size_t)l * s + j) : 0.0)) : 0.0;
                        acc0[u] = fma(c, q0, acc0[u]); acc1[u] = fma(c, q1, acc1[u]);
                    }
                }
            }
            const int l = u0 * 32 + lane, c = l - base;
            if (lane < n_here) {
                nrm[warp * (kGramList + 1) + l] = (ok0 ? kr0 * kr0 : 0.0) + (ok1 ? kr1 * kr1 : 0.0);
                const bool vec = (k & 1) == 0;
                if (vec && ok1) {
                    *reinterpret_cast<double2*>(qg + (size_t)l * k + row) = make_double2(kq0, kq1);
                    if (c >= 0 && c < a.half_n) *reinterpret_cast<double2*>(rh + (size_t)c * k + row) = make_double2(kr0, kr1);
                } else {
                    if (ok0) { qg[(size_t)l * k + row] = kq0; if (c >= 0 && c < a.half_n) rh[(size_t)c * k + row] = kr0; }
                    if (ok1) { qg[(size_t)l * k + row + 1] = kq1; if (c >= 0 && c < a.half_n) rh[(size_t)c * k + row + 1] = kr1; }
                }
            }
        }
        if (lane == 0) {                                              // the residual after the last pick
            nrm[warp * (kGramList + 1) + L] = (ok0 ? r0 * r0 : 0.0) + (ok1 ? r1 * r1 : 0.0);
            const int c = L - base;
            if (c >= 0 && c < a.half_n) { if (ok0) rh[(size_t)c * k + row] = r0; if (ok1) rh[(size_t)c * k + row + 1] = r1; }
        }
        __syncthreads();
        for (int l = t; l <= L; l += kT) {
            double v = 0.0;
            for (int w = 0; w < kWarps; ++w) v += nrm[w * (kGramList + 1) + l];
            a.pnorm[((size_t)m * batches + batch) * (kGramList + 1) + l] = v;
        }
    }
}

// norms, thresholds and the scaled binary16 rows of the screened residuals: block = residual
__device__ void gram_emit(const OmpArgs& a, OmpSmem& sh) {
    volatile SpecCtl* ctl = a.ctl;
    const int t = threadIdx.x, k = a.k, s = a.s;
    const int batches = (k + kRowBatch - 1) / kRowBatch;
    for (int item = blockIdx.x; item < 2 * (a.half_n + 1); item += gridDim.x) {
        const int m = item & 1, c = item >> 1;
        if (ctl->finished[m]) continue;
        const int base = ctl->base[m], hi = ctl->hi[m], extra = ctl->extra[m], dep = ctl->dep[m];
        const int j = base + c;
        if (j > hi || (dep && j == hi)) continue;
        const bool screened = c < a.half_n && (j < hi || extra);
        const size_t nrow = (size_t)m * a.half_n + c;
        double v = 0.0;
        for (int b = t; b < batches; b += kT) v += __ldcg(a.pnorm + ((size_t)m * batches + b) * (kGramList + 1) + j);
        v = warp_sum(v);
        __syncthreads();
        if ((t & 31) == 0) sh.wsum[t >> 5] = v;
        __syncthreads();
        double rn = 0.0;
        for (int w = 0; w < kWarps; ++w) rn += sh.wsum[w];
        rn = sqrt(rn);
        if (t == 0) {
            if (j == 0) a.ctl->ynorm[m] = rn;
            else a.rnorm[(size_t)m * s + j - 1] = rn;
        }
        if (!screened) continue;
        const double sc = residual_scale(rn);
        const double* src = a.rhist + nrow * k;
        uint16_t* dst = a.rt + nrow * a.kp;
        for (int row = t; row < k; row += kT) dst[row] = half_rn_bits(__ldcg(src + row) * sc);
        if (t == 0) {
            a.inv_scale[nrow] = (float)(1.0 / sc);
            const double tau = j < hi ? report_threshold(a, rn, a.pick_score[(size_t)m * s + j]) : a.z_harvest * rn / sqrt((double)k);
            a.tau[nrow] = (float)(tau * sc);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// the kernel.  mode 0: speculate on the candidate list; mode 1: lock-step over all columns.
//   CL = 16: one cluster is the whole grid (both groups of 8 in it): every barrier is a cluster barrier
//   CL = 8, 2: clusters 0 and 1 keep the books of M^ and V^
// Bound by the generator where the columns are many (correlate_stream), else by latency: barriers, and for each pick the chain
// best score -> exact scores -> products with the q_l -> new q, r.  us per pick, one block per recovery and a grid barrier after
// every phase (the Cholesky form) / this form:
//   lock-step  d = 4096, k = 256: 50 / 11;  50304, 128: 34 / 15;  31820, 1024: 140 / 27;  110000, 210: 46 / 22;  1.2e6, 224: 128 / 88;
//              2e6, 42: 63 / 55
//   the books of a pick alone  k = 1024: 16 / 5.5;  k = 2048: 40 / 7
// ------------------------------------------------------------------------------------------------
template <int CL>
__global__ void __launch_bounds__(kT, 1) k_omp(OmpArgs a, int mode) {
    constexpr int GS = Group<CL>::GS;
    constexpr bool kOneCluster = CL == 16;
    cg::grid_group grid = cg::this_grid();
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char dyn_raw[];
    __shared__ OmpSmem sh;
    double* dyn = reinterpret_cast<double*>(dyn_raw);
    const int t = threadIdx.x;
    volatile SpecCtl* ctl = a.ctl;
    const int k = a.k, s = a.s;
    auto barrier = [&]() { if (kOneCluster) cluster.sync(); else grid.sync(); };
    // ---- gate: identical in every block, because nothing below changes the control block before the first barrier
    const int fin[2] = {ctl->finished[0], ctl->finished[1]};
    const int vc[2] = {ctl->v[0], ctl->v[1]};                            // confirmed picks
    const uint32_t fc[2] = {ctl->forced[0], ctl->forced[1]};             // confirmed winner for pick vc, if any
    if (mode == 0) {
        if (!ctl->round_active || ctl->fallback) return;
        if (a.mini && (ctl->mini_done || ctl->n_cand <= kGramList || (a.wide_count[0] == 0u && a.wide_count[1] == 0u))) return;
        if (ctl->n_cand <= kGramList && ctl->gram_ok && a.zlist != nullptr) {
            const int n = ctl->n_cand;
            const bool todo = ctl->gram_version != ctl->list_version;
            gram_prepare(a, sh, n);
            barrier();
            if (todo) {
                gram_matrix(a, n);
                if (blockIdx.x == 0 && t == 0) a.ctl->gram_version = ctl->list_version;
                barrier();
            }
            if (blockIdx.x < 2) gram_picks(a, (int)blockIdx.x, n, dyn, fin, vc, fc);
            barrier();
            if (ctl->gram_ok) {
                gram_rows(a, dyn);
                barrier();
                gram_emit(a, sh);
                return;
            }
        }
    }
    if (mode == 1 && fin[0] && fin[1]) return;
    const int n_cand = ctl->n_cand;
    const int base[2] = {vc[0] + (fc[0] != kNoColumn ? 1 : 0), vc[1] + (fc[1] != kNoColumn ? 1 : 0)};
    // where this kernel starts: the speculation resumes after the tentative picks (those confirmed against the wide
    // lists only), lock-step after the confirmed ones.  The first pick may be prescribed: confirmed (final) or imposed
    // by a list pass (still speculative).
    int v0[2]; uint32_t first_col[2]; bool first_final[2];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const int tv = ctl->tv[m];
        v0[m] = (mode == 0 && tv > vc[m]) ? tv : vc[m];
        first_final[m] = v0[m] == vc[m] && fc[m] != kNoColumn;
        uint32_t first = kNoColumn;
        if (first_final[m]) first = fc[m];
        else if (mode == 0 && v0[m] == tv) first = ctl->tforced[m];
        first_col[m] = first;
    }
    const bool restart_wide = mode == 0 && !a.mini && a.wide_count != nullptr && ctl->rounds == 0;
    barrier();
    // ---- roles
    const int rank = (int)cluster.block_rank();
    const int cid = (int)blockIdx.x / CL;
    const int mb = kOneCluster ? rank / GS : cid;                        // recovery whose books this block keeps (0, 1)
    const bool book = kOneCluster || cid < 2;
    const int g = kOneCluster ? rank % GS : rank, rank0 = kOneCluster ? mb * GS : 0;
    const bool all_correlate = kOneCluster || (mode == 1 && a.book_correlates);
    const int nblk = all_correlate ? (int)gridDim.x : (int)gridDim.x - 2 * CL;
    const int cblk = all_correlate ? (int)blockIdx.x : (int)blockIdx.x - 2 * CL;
    const bool corr = cblk >= 0;
    const unsigned int n_cols = mode == 0 ? (unsigned int)n_cand : (unsigned int)a.d;
    // ---- shared memory: residuals as operands | books | columns of q | the correlation's sums, norms and generated entries
    const size_t pb = corr ? frag_bytes(k) : 0;
    const size_t bb = book ? (book_doubles(k, s, GS, kOneCluster) + (size_t)a.q_cols * slice_rows(k, GS)) * sizeof(double) : 0;
    uint2* frag = reinterpret_cast<uint2*>(dyn_raw);
    const BookMem bk = book_mem(a, reinterpret_cast<double*>(dyn_raw + pb), GS, g, kOneCluster);
    float* corr_mem = reinterpret_cast<float*>(dyn_raw + ((pb + bb + 15) & ~(size_t)15));
    const int xstride = exchange_stride(s);
    // the first full pass of a step starts the wide lists afresh; later ones add what their residuals bring (the lists then
    // cover the whole path of this step, which is where the next step's path runs, too)
    if (restart_wide) {
        if (blockIdx.x == 0 && t == 0) a.wide_count[0] = a.wide_count[1] = 0u;
        const size_t words = 2 * (((size_t)a.d + 31) / 32);              // both streams' bitmaps
        for (size_t w = (size_t)blockIdx.x * kT + t; w < words; w += (size_t)gridDim.x * kT) a.wide_bits[w] = 0u;
    }
    // ---- the books at the first pick: r = y - sum a_l q_l over the picks made so far
    double cur_rnorm = 0.0;                                              // ||r|| of the residual the next pick is made from
    int hi = 0, extra = 0, dep = 0;
    bool inexact = false;
    int pend = -1;                                                       // pick whose residual's norm is still spread over the group
    if (book) {
        const int m = mb;
        if (!fin[m]) {
            const double* y = a.y64 + (size_t)m * k + bk.row0;
            for (int r = t; r < bk.R; r += kT) {
                double v = r < bk.rows ? y[r] : 0.0;
                if (r < bk.rows)
                    for (int l = 0; l < v0[m]; ++l) {
                        const double q = __ldcg(a.q + ((size_t)m * s + l) * k + bk.row0 + r);
                        if (l < a.q_cols) bk.qs[(size_t)l * bk.R + r] = q;
                        v -= __ldcg(a.acoef + (size_t)m * s + l) * q;
                    }
                bk.rr[r] = v;
                if (r < bk.rows) a.r32[2 * (bk.row0 + r) + m] = (float)v;
            }
            if ((k & 1) && bk.rows < bk.R) for (int l = t; l < a.q_cols; l += kT) bk.qs[(size_t)l * bk.R + bk.rows] = 0.0;
            __syncthreads();
            send_norm<GS>(cluster, bk, rank0, g);
        }
        cluster.sync();
        if (!fin[m]) {
            for (int p = 0; p < GS; ++p) cur_rnorm += bk.xrn[p];
            cur_rnorm = sqrt(cur_rnorm);
            hi = v0[m] > base[m] ? v0[m] : base[m];
            if (g == 0 && t == 0) {
                if (v0[m] == 0) a.ctl->ynorm[m] = cur_rnorm;
                a.ctl->stop[m] = 0;
            }
            const int c0 = v0[m] - base[m];
            if (mode == 0 && !first_final[m] && c0 >= 0 && c0 < a.half_n) emit_row(a, bk, (size_t)m * a.half_n + c0, cur_rnorm, g);
        } else if (g == 0 && t == 0) a.ctl->stop[m] = 1;
        if (mode == 0 && g == 0) {
            const int keep = fin[m] ? 0 : (v0[m] - base[m] > 0 ? v0[m] - base[m] : 0);   // rows of earlier tentative picks stay
            for (int c = t; c < a.half_n; c += kT) {
                a.rep_count[m * a.half_n + c] = 0u;
                if (c >= keep) {
                    a.tau[m * a.half_n + c] = __int_as_float(0x7f800000);
                    a.wide_tau[m * a.half_n + c] = __int_as_float(0x7f800000);
                }
            }
        }
    }
    CorrPlan plan = corr_plan(n_cols, k, a.z_words, corr ? cblk : 0, nblk);
    bool filled = false;
    barrier();
    for (int i = 0;; ++i) {
        int jm[2], picks[2];
        bool act[2], need_corr = false;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            jm[m] = v0[m] + i;
            act[m] = !fin[m] && jm[m] < s && !ctl->stop[m];
            if (mode == 0 && (jm[m] - base[m] >= a.half_n || i >= a.depth)) act[m] = false;
            picks[m] = jm[m] < s ? jm[m] : s;
            if (act[m] && !(i == 0 && first_col[m] != kNoColumn)) need_corr = true;
        }
        if (!act[0] && !act[1]) break;
        if (need_corr && corr) {
            correlate(a, sh, plan, mode == 0 ? a.cand_list : nullptr, frag, corr_mem, filled, picks, cblk, nblk);
            filled = true;
        }
        barrier();
        const bool active = book && act[mb];
        const int m = mb, j = active ? jm[mb] : 0;
        const bool speculative = mode == 0 && !(i == 0 && active && first_final[mb]);
        const int c = active ? j - base[mb] : 0;                      // -1 for a confirmed prescribed pick
        int nc = 0;
        uint32_t col = kNoColumn;
        // ---- 1. candidates, their exact scores, the products of the best one with the q_l, ||r||
        if (active) {
            if (i == 0 && first_col[mb] != kNoColumn) { col = first_col[mb]; nc = 1; }
            else nc = gather_candidates(a, sh, m, j, nblk, mode == 0 ? a.cand_list : nullptr, n_cols, &col, &inexact);
            if (nc > 0) {
                send_products<GS>(cluster, a, bk, m, j, col, true, bk.x0, rank0, g);
                for (int e = 1 + (t >> 5); e < nc; e += kWarps) send_candidate<GS>(cluster, a, bk, sh.cidx[e], e, bk.x0, rank0, g);
            } else if (pend >= 0) send_norm<GS>(cluster, bk, rank0, g);
        }
        if (kOneCluster && t == 0) *cluster.map_shared_rank(&sh.peer_nc, rank ^ GS) = nc;
        if (book) cluster.sync();
        // ---- 2. the winner: largest <a, r>^2 / ||a||^2, lowest index on ties
        bool again = false;
        if (active) {
            if (nc > 0) {
                for (int l = t; l < j + 3; l += kT) {
                    const int at = l <= j ? l : s + (l - j - 1);
                    double v = 0.0;
#pragma unroll
                    for (int p = 0; p < GS; ++p) v += bk.x0[(size_t)p * xstride + at];
                    bk.cs[l] = v;
                }
                __syncthreads();
            }
            if (pend >= 0) {
                double rn2 = 0.0;
                if (nc > 0) rn2 = bk.cs[j + 2];
                else for (int p = 0; p < GS; ++p) rn2 += bk.xrn[p];
                cur_rnorm = sqrt(rn2);
            }
        }
        double dot = 0.0, n2 = 1.0;
        if (active && nc > 0) {
            dot = bk.cs[j]; n2 = bk.cs[j + 1];
            if (nc > 1) {
                double best = n2 > 0.0 ? dot * dot / n2 : 0.0;
                uint32_t bi = col;
                int win = 0;
                for (int e = 1; e < nc; ++e) {
                    double ed = 0.0, en = 0.0;
                    for (int p = 0; p < GS; ++p) {
                        ed += bk.x0[(size_t)p * xstride + s + 2 + 2 * (e - 1)];
                        en += bk.x0[(size_t)p * xstride + s + 3 + 2 * (e - 1)];
                    }
                    const double sc = en > 0.0 ? ed * ed / en : 0.0;
                    const uint32_t idx = sh.cidx[e];
                    if (sc > best || (sc == best && idx < bi)) { best = sc; bi = idx; win = e; dot = ed; n2 = en; }
                }
                again = win != 0;                                      // the same in every block of the group
                col = bi;
            }
        }
        const bool more = kOneCluster ? (nc > 1 || sh.peer_nc > 1) : nc > 1;     // the same in every block of the cluster
        if (more) {
            if (!kOneCluster) cluster.sync();                           // everybody has read the exchange buffer
            if (again) send_products<GS>(cluster, a, bk, m, j, col, false, bk.x1, rank0, g);
            cluster.sync();
            if (again) {
                for (int l = t; l < j; l += kT) {
                    double v = 0.0;
                    for (int p = 0; p < GS; ++p) v += bk.x1[(size_t)p * xstride + l];
                    bk.cs[l] = v;
                }
                __syncthreads();
            }
        }
        // ---- 3. gamma, a_j; q_j and the new residual of this slice
        if (active) {
            int rc = nc == 0 ? 1 : 0;
            // the residual of the previous pick, whose norm has just come together, is a row of the screened batch
            if (pend >= 0) {
                if (g == 0 && t == 0) a.rnorm[(size_t)m * s + pend] = cur_rnorm;
                if (mode == 0 && c >= 0 && c < a.half_n) emit_row(a, bk, (size_t)m * a.half_n + c, cur_rnorm, g);
                pend = -1;
            }
            if (nc > 0) {
                double csq = 0.0;
                for (int l = t & 31; l < j; l += 32) csq = fma(bk.cs[l], bk.cs[l], csq);
                csq = warp_sum(csq);
                const double piv = n2 - csq;
                if (!(piv > kPivot * n2)) rc = 2;
                else {
                    const double gamma = rsqrt(piv), aj = gamma * dot;
                    const int R = bk.R, P = bk.P < (j + 3) / 4 ? bk.P : (j + 3) / 4 > 0 ? (j + 3) / 4 : 1;      // at least four vectors per part
                    const int r0 = P == 1 ? t : t % R, h = P == 1 ? 0 : t / R;
                    if (h < P)
                        for (int r = r0; r < bk.rows; r += P == 1 ? kT : R) {                       // (P > 1: one row per thread)
                            double va = 0.0, vb = 0.0;
                            int l = h;
#pragma unroll 4
                            for (; l + P < j; l += 2 * P) {
                                va = fma(bk.cs[l], q_slice(a, bk, m, l)[r], va);
                                vb = fma(bk.cs[l + P], q_slice(a, bk, m, l + P)[r], vb);
                            }
                            if (l < j) va = fma(bk.cs[l], q_slice(a, bk, m, l)[r], va);
                            bk.part[h * R + r] = va + vb;
                        }
                    __syncthreads();
                    const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
                    for (int r = t; r < bk.rows; r += kT) {
                        double v = 0.0;
                        for (int e = 0; e < P; ++e) v += bk.part[e * R + r];
                        const double q = gamma * (a.sigma * (double)z_at(key, (uint32_t)(bk.row0 + r)) - v);
                        a.q[((size_t)m * s + j) * k + bk.row0 + r] = q;
                        if (j < a.q_cols) bk.qs[(size_t)j * R + r] = q;
                        const double rv = bk.rr[r] - aj * q;
                        bk.rr[r] = rv;
                        a.r32[2 * (bk.row0 + r) + m] = (float)rv;
                    }
                    if (g == 0) {
                        for (int l = t; l < j; l += kT) {
                            a.crow[((size_t)m * s + j) * s + l] = bk.cs[l];
                            a.ccol[((size_t)m * s + l) * s + j] = bk.cs[l];
                        }
                        if (t == 0) {
                            a.gam[(size_t)m * s + j] = gamma; a.acoef[(size_t)m * s + j] = aj; a.lam[(size_t)m * s + j] = col;
                            // a prescribed column, if there was one, is consumed with this pick
                            if (!speculative) { a.cnt->done[m] = j + 1; a.ctl->v[m] = j + 1; a.ctl->forced[m] = kNoColumn; }
                        }
                    }
                    pend = j;
                }
            }
            if (nc > 0 && speculative && g == 0 && t == kT - 32) {         // (a warp with little else to do)
                const double psc = fabs(dot) * rsqrt(n2);
                a.pick_score[(size_t)m * s + j] = psc;
                a.tau[m * a.half_n + c] = (float)(report_threshold(a, cur_rnorm, psc) * residual_scale(cur_rnorm));
                a.wide_tau[m * a.half_n + c] = wide_threshold(a, c, cur_rnorm);
                a.lam[(size_t)m * s + j] = col;
            }
            // what ends this recovery's run of picks
            if (rc == 0) hi = j + 1;
            else if (speculative) {
                // no candidate left: the current residual is screened without a pick; dependent column: the
                // pick is screened, and the recovery stops there if the pick is confirmed
                if (rc == 1) {
                    extra = 1;
                    if (g == 0 && t == 0) {
                        a.tau[m * a.half_n + c] = (float)(a.z_harvest * cur_rnorm / sqrt((double)k) * residual_scale(cur_rnorm));
                        a.wide_tau[m * a.half_n + c] = wide_threshold(a, c, cur_rnorm);
                    }
                } else { dep = 1; hi = j + 1; }
                if (g == 0 && t == 0) a.ctl->stop[m] = 1;
            } else if (g == 0 && t == 0) {
                // a confirmed pick cannot be made: this recovery ends with j picks
                a.cnt->stopped[m] = 1;
                atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_DEPENDENT_COLUMN);
                a.cnt->done[m] = j;
                a.ctl->v[m] = j;
                a.ctl->finished[m] = 1;
                a.ctl->stop[m] = 1;
            }
        }
        barrier();
    }
    // the norm of the last residual
    if (book) {
        if (pend >= 0) send_norm<GS>(cluster, bk, rank0, g);
        cluster.sync();
        if (pend >= 0 && g == 0 && t == 0) {
            double rn2 = 0.0;
            for (int p = 0; p < GS; ++p) rn2 += bk.xrn[p];
            a.rnorm[(size_t)mb * s + pend] = sqrt(rn2);
        }
    }
    if (book && g == 0 && t == 0 && !fin[mb]) {
        const int m = mb;
        if (mode == 0) {
            a.ctl->base[m] = base[m];
            a.ctl->hi[m] = hi < base[m] ? base[m] : hi;
            a.ctl->extra[m] = extra;
            a.ctl->dep[m] = dep;
            a.ctl->list_exact[m] = inexact ? 0 : 1;
        } else if (!a.ctl->finished[m]) {
            a.cnt->done[m] = a.ctl->v[m];
            a.ctl->finished[m] = 1;
        }
    }
}

}  // namespace

namespace {

template <int CL>
cudaError_t omp_opt_in() {
    cudaError_t e = cudaFuncSetAttribute(k_omp<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOmpDynBytes);
    if (e == cudaSuccess && CL > 8) e = cudaFuncSetAttribute(k_omp<CL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

struct OmpLaunch {
    cudaLaunchConfig_t cfg; cudaLaunchAttribute attr[2];
    OmpLaunch(int cl, int grid, cudaStream_t stream) : cfg{} {
        cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kOmpDynBytes; cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cl; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeCooperative;
        attr[1].val.cooperative = 1;
        cfg.attrs = attr; cfg.numAttrs = cl == 16 ? 1 : 2;            // one cluster is resident as a whole or not at all
    }
};

template <int CL>
cudaError_t resident_clusters(int* out) {
    OmpLaunch l(CL, CL, 0);
    l.cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(out, k_omp<CL>, &l.cfg);
}

template <int CL>
cudaError_t omp_launch(OmpArgs a, int mode, int grid, cudaStream_t stream) {
    const OmpBudget b = omp_budget(CL, a.k, a.s, mode);
    if (!b.fits) return cudaErrorInvalidConfiguration;
    a.q_cols = b.q_cols; a.book_correlates = b.book_correlates; a.z_words = b.z_words;
    OmpLaunch l(CL, grid, stream);
    return cudaLaunchKernelEx(&l.cfg, k_omp<CL>, a, mode);
}

}  // namespace

cudaError_t omp_configure(sgc_state* st) {
    // How many clusters a device holds is a property of the device: asked once for each (the three questions would otherwise be
    // most of what the creation of a small state takes, and chunked optimizers create hundreds)
    struct Resident { int n2, n8, n16; bool known; };
    constexpr int kDevices = 64;
    static std::mutex lock;
    static Resident table[kDevices];
    cudaError_t e = omp_opt_in<2>();
    if (e == cudaSuccess) e = omp_opt_in<8>();
    if (e != cudaSuccess) return e;
    const bool clusters16 = omp_opt_in<16>() == cudaSuccess;
    if (!clusters16) cudaGetLastError();
    Resident r = {};
    const bool listed = st->device >= 0 && st->device < kDevices;
    if (listed) { std::lock_guard<std::mutex> hold(lock); r = table[st->device]; }
    if (!r.known) {
        e = resident_clusters<2>(&r.n2);
        if (e == cudaSuccess) e = resident_clusters<8>(&r.n8);
        if (e != cudaSuccess) return e;
        if (!clusters16 || resident_clusters<16>(&r.n16) != cudaSuccess) { r.n16 = 0; cudaGetLastError(); }
        r.known = true;
        if (listed) { std::lock_guard<std::mutex> hold(lock); table[st->device] = r; }
    }
    int n2 = r.n2, n8 = r.n8;
    const int n16 = r.n16;
    if (2 * n2 > kCorrBlocks) n2 = kCorrBlocks / 2;
    if (8 * n8 > kCorrBlocks) n8 = kCorrBlocks / 8;
    st->omp_grid2 = 2 * n2; st->omp_grid8 = n8 >= 3 ? 8 * n8 : 0; st->omp_one = n16 >= 1 ? 1 : 0;
    return n2 >= 3 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

cudaError_t launch_omp(sgc_state* st, const OmpArgs& a, int mode, cudaStream_t stream) {
    switch (omp_shape(st->d, a.k, a.s, mode, st->omp_one != 0, st->omp_grid8 != 0)) {
        case 16: return omp_launch<16>(a, mode, 16, stream);
        case 2: return omp_launch<2>(a, mode, st->omp_grid2, stream);
        default: return omp_launch<8>(a, mode, st->omp_grid8, stream);
    }
}

}  // namespace sgc
