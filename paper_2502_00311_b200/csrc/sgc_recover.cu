// a4 + a5: x^M = OMP_A(M^), x^V = OMP_A(V^) (Eq. 7; Appendix B Algorithm 3), then
// N = alpha x^M / (sqrt(x^V) + eps) and W <- W - lr N (Eq. 8, Eq. 3; Algorithm 2).
//
// Algorithm 3 needs, for every pick, the argmax of |<A_i, r>| / ||A_i|| over all d columns ("Projection" and
// "Select"), and A is regenerated rather than stored, so one such argmax costs k*d generated entries.  Two ways
// of getting the picks are implemented; both produce exactly the picks of Algorithm 3.
//
// Lock-step (k_omp of sgc_omp.cu, mode 1): one pass over all columns per pick, both residuals (M^ and V^) against every
//   generated entry; fp32 screen, fp64 decision among the near-maximal candidates.
//
// Speculative (rounds of k_omp mode 0, the tensor-core screening pass, k_resolve): OMP first runs on a short
//   candidate list only (the supports of the previous step plus harvested columns), which costs next to
//   nothing, and records the residual before every pick.  ONE pass over all d columns then correlates A with
//   all those residuals at once (sgc_pass.cu) and reports every column whose score comes within the rounding
//   margin of the speculated pick's.  k_resolve walks the picks in order: a pick without a challenger, or one
//   that wins the fp64 rescoring against its challengers, is the true argmax; at the first pick that loses,
//   the global winner (known from the same pass) is forced, the columns reported for that residual join the
//   candidate list and the next round continues from there.  Every round fixes at least one more pick; what is
//   still open after the enqueued rounds, or after any overflow, is finished in lock-step.
//
// k_begin opens a step's recovery; k_finish closes it: coefficients, Eq. (8) on the common support, candidate-list upkeep.
// Several states that share A are recovered together (launch_recover_group): their residuals sit side by
// side in one screened batch, so one pass serves them all.
#include <cuda_fp16.h>
#include <math.h>

#include "sgc_omp.cuh"

namespace sgc {
namespace {

// deterministic block sum (kOmpThreads threads); every thread receives the result.  red: 32 doubles.
__device__ double block_sum(double v, double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = (lane < kOmpThreads / 32) ? red[lane] : 0.0;
    t = warp_sum(t);
    return t;
}

// Challengers of one pick that the walk rescores (3 us each at k = 16384) before it gives the step up to lock-step, where a pick
// costs a generation of all columns.  The margin grows with k: with 16384 rows and kept entries of nearly equal size more than the 16
// that the other kernels have room for come within it (d = 65600, s = 250: half of the steps were given up, 41 -> 110 to 170 ms).
constexpr int kResolveCap = 256;

// shared memory of the resolve kernel's walk
struct BookSmem {
    double red[32];
    double best_dot, best_n2, best_score;
    uint32_t best_idx;
    uint32_t cand_idx[kResolveCap];
    int n_cand;
    unsigned int smax_bits;
};

// exact score of one column against a residual: dot = <Z_i, r>, n2 = ||Z_i||^2 (fp64), for every thread
__device__ void rescore_column(const OmpArgs& a, BookSmem& sh, uint32_t idx, const double* r, double* dot_out, double* n2_out) {
    const ColKey key = column_key(a.seed_lo, a.seed_hi, idx);
    double dot = 0.0, n2 = 0.0;
    for (int row = 2 * threadIdx.x; row < a.k; row += 2 * kOmpThreads) {            // one generated word = two rows
        const float2 zz = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)(row >> 1) * key.mk));
        dot += (double)zz.x * r[row];
        n2 += (double)zz.x * (double)zz.x;
        if (row + 1 < a.k) {
            dot += (double)zz.y * r[row + 1];
            n2 += (double)zz.y * (double)zz.y;
        }
    }
    *dot_out = block_sum(dot, sh.red);
    *n2_out = block_sum(n2, sh.red);
}

// fp64 argmax of |<A_i, r>| / ||A_i|| among sh.cand_idx[0..nc), lowest index on ties -> sh.best_*
__device__ void rescore_candidates(const OmpArgs& a, BookSmem& sh, int nc, const double* r) {
    if (threadIdx.x == 0) { sh.best_score = -1.0; sh.best_idx = kNoColumn; sh.best_dot = 0.0; sh.best_n2 = 1.0; }
    __syncthreads();
    for (int c = 0; c < nc; ++c) {
        const uint32_t idx = sh.cand_idx[c];
        double dot, n2;
        rescore_column(a, sh, idx, r, &dot, &n2);
        if (threadIdx.x == 0) {
            const double sc = n2 > 0.0 ? dot * dot / n2 : 0.0;
            if (sc > sh.best_score || (sc == sh.best_score && idx < sh.best_idx)) {
                sh.best_score = sc; sh.best_idx = idx; sh.best_dot = dot; sh.best_n2 = n2;
            }
        }
        __syncthreads();
    }
}
// ------------------------------------------------------------------------------------------------
// resolve: confirm or refute the speculated picks with the reports of the screening pass
// ------------------------------------------------------------------------------------------------
struct ResolveArgs {
    OmpArgs o;
    const uint2* rep; int rep_cap;
    unsigned int* cand_bits; uint32_t* cand_list;
    const uint32_t* kept_ring;
    int mini;                              // 1: the reports come from a list pass (two-level screening)
    const unsigned int* wide_count;
};

// <z, r> and ||z||^2 of a column, as one warp sums them
__device__ __forceinline__ void warp_products(const OmpArgs& a, uint32_t col, const double* r, double* dot_out, double* n2_out) {
    const int lane = threadIdx.x & 31;
    const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
    double dot = 0.0, n2 = 0.0;
#pragma unroll 4
    for (int p = lane; 2 * p < a.k; p += 32) {
        const float2 z = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)p * key.mk));
        const bool two = 2 * p + 1 < a.k;
        const double r0 = r[2 * p], r1 = two ? r[2 * p + 1] : 0.0, z1 = two ? (double)z.y : 0.0;
        dot = fma((double)z.x, r0, dot); dot = fma(z1, r1, dot);
        n2 = fma((double)z.x, (double)z.x, n2); n2 = fma(z1, z1, n2);
    }
    *dot_out = warp_sum(dot); *n2_out = warp_sum(n2);
}
constexpr int kSweepCap = 8;                           // challengers per pick that the sweep rescores

__device__ __forceinline__ bool in_support(const uint32_t* lam, int n, uint32_t col) {
    for (int q = 0; q < n; ++q) if (lam[q] == col) return true;
    return false;
}

// Collects into sh.cand_idx[start..] the reported columns of one residual that are not in the first n_sup picks,
// differ from `skip`, and score within `window` of the best such report, provided that best reaches `floor_sc`.
// Returns the number of candidates (start included), or -1 on overflow.
__device__ int collect_challengers(BookSmem& sh, const uint2* rep, unsigned int count, const uint32_t* lam, int n_sup,
                                   uint32_t skip, float floor_sc, float window, int start) {
    __syncthreads();
    if (threadIdx.x == 0) { sh.smax_bits = 0u; sh.n_cand = start; }
    __syncthreads();
    for (unsigned int e = threadIdx.x; e < count; e += kOmpThreads) {
        const uint2 rp = rep[e];
        const float sc = __uint_as_float(rp.y);
        if (sc >= floor_sc && rp.x != skip && !in_support(lam, n_sup, rp.x)) atomicMax(&sh.smax_bits, rp.y);   // scores are >= 0
    }
    __syncthreads();
    const unsigned int smax_bits = sh.smax_bits;
    if (smax_bits == 0u) return start;
    const float lo = __uint_as_float(smax_bits) - window;
    for (unsigned int e = threadIdx.x; e < count; e += kOmpThreads) {
        const uint2 rp = rep[e];
        const float sc = __uint_as_float(rp.y);
        if (sc >= floor_sc && sc >= lo && rp.x != skip && !in_support(lam, n_sup, rp.x)) {
            const int slot = atomicAdd(&sh.n_cand, 1);
            if (slot < kResolveCap) sh.cand_idx[slot] = rp.x;
        }
    }
    __syncthreads();
    const int n = sh.n_cand;
    return n > kResolveCap ? -1 : n;
}

// appends the columns `cols` that the list does not hold yet; n_s is the running length (shared memory)
__device__ void cand_append(const uint32_t* cols, int n_cols, int* n_s, uint32_t* cand_list, unsigned int* cand_bits) {
    for (int e = threadIdx.x; e < n_cols; e += blockDim.x) {
        const uint32_t col = cols[e];
        if (col == kNoColumn) continue;
        const unsigned int bit = 1u << (col & 31u);
        if (atomicOr(&cand_bits[col >> 5], bit) & bit) continue;
        const int slot = atomicAdd(n_s, 1);
        if (slot < kCandCap) cand_list[slot] = col;
        else atomicAnd(&cand_bits[col >> 5], ~bit);
    }
}

// Cuts the candidate list back to what is certain to matter when `incoming` more columns would let it outgrow kCandKeep:
// the ring of kept index sets and the picks made so far (columns harvested for earlier residuals have lost most of
// their value: the residual has moved on).
__device__ void make_room(const ResolveArgs& ra, int incoming) {
    volatile SpecCtl* ctl = ra.o.ctl;
    __shared__ int n_s;
    __syncthreads();
    const int n0 = ctl->n_cand;
    if (n0 + incoming <= kCandKeep) return;
    for (int e = threadIdx.x; e < n0; e += kOmpThreads) {
        const uint32_t col = ra.cand_list[e];
        atomicAnd(&ra.cand_bits[col >> 5], ~(1u << (col & 31u)));
    }
    if (threadIdx.x == 0) n_s = 0;
    __syncthreads();
    cand_append(ra.kept_ring, ctl->hist_count * ra.o.s, &n_s, ra.cand_list, ra.cand_bits);
    __syncthreads();
    for (int m = 0; m < 2; ++m) {
        cand_append(ra.o.lam + (size_t)m * ra.o.s, ctl->finished[m] ? ra.o.cnt->done[m] : ctl->hi[m], &n_s, ra.cand_list,
                    ra.cand_bits);
        __syncthreads();
    }
    if (threadIdx.x == 0) { ctl->n_cand = n_s < kCandCap ? n_s : kCandCap; ctl->list_version = ctl->list_version + 1; }
    __syncthreads();
}

// the reported columns of one residual that score at least `floor_sc` join the candidate list (the forced winner first)
__device__ void harvest(const ResolveArgs& ra, BookSmem& sh, const uint2* rep, unsigned int count, uint32_t first,
                        float floor_sc = 0.0f) {
    volatile SpecCtl* ctl = ra.o.ctl;
    __shared__ int n_s;
    __syncthreads();
    if (threadIdx.x == 0) n_s = ctl->n_cand;
    __syncthreads();
    if (first != kNoColumn) cand_append(&first, 1, &n_s, ra.cand_list, ra.cand_bits);
    __syncthreads();
    for (unsigned int e = threadIdx.x; e < count; e += kOmpThreads) {
        const uint2 rp = rep[e];
        if (__uint_as_float(rp.y) < floor_sc) continue;
        const uint32_t col = rp.x;
        const unsigned int bit = 1u << (col & 31u);
        if (atomicOr(&ra.cand_bits[col >> 5], bit) & bit) continue;
        const int slot = atomicAdd(&n_s, 1);
        if (slot < kCandCap) ra.cand_list[slot] = col;
        else atomicAnd(&ra.cand_bits[col >> 5], ~bit);
    }
    __syncthreads();
    if (threadIdx.x == 0) { ctl->n_cand = n_s < kCandCap ? n_s : kCandCap; ctl->list_version = ctl->list_version + 1; }
    __syncthreads();
}

// Full mode (reports of a pass over all d columns): confirms the speculated picks in order; the first refuted pick of a
// stream gets its true winner, which becomes final.  Mini mode (reports of a list pass over the wide lists): the same
// walk, but what it establishes is tentative -- tv / tforced tell the next speculation where to resume, while v, forced,
// the round count and everything a finished recovery records are left alone; the next full pass decides on all of it.
__global__ void __launch_bounds__(kOmpThreads, 1) k_resolve(ResolveArgs ra) {
    const OmpArgs& a = ra.o;
    __shared__ BookSmem sh;
    __shared__ int give_up, any_failed;
    volatile SpecCtl* ctl = a.ctl;
    const bool mini = ra.mini != 0;
    if (!ctl->round_active) return;
    if (ctl->fallback || ctl->pass_error) {
        // a wait inside the screening pass ran out: its reports are void, the remaining picks are made in lock-step
        if (threadIdx.x == 0) {
            if (ctl->pass_error) atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_TIMEOUT);
            ctl->fallback = 1; ctl->round_active = 0;
        }
        return;
    }
    if (mini) {
        if (ctl->mini_done || ctl->n_cand <= kGramList) return;
        if (ra.wide_count[0] == 0u && ra.wide_count[1] == 0u) {
            if (threadIdx.x == 0) ctl->mini_done = 1;
            return;
        }
    }
    const int s = a.s;
    // Sweep: every block takes its share of the report lists (warp per residual), rescores the challengers within the margin and
    // notes which picks one of them may beat; the walk below only stops at those (it rescored all of them one after the other before:
    // 116 us on average for a round of d = 3e6, k = 700, s = 100).  Nothing of the control block changes before the walk.
    {
        const int gw = blockIdx.x * (kOmpThreads / 32) + (threadIdx.x >> 5), nw = gridDim.x * (kOmpThreads / 32);
        for (int m = 0; m < 2; ++m) {
            if (ctl->finished[m]) continue;
            const int base = ctl->base[m], hi = ctl->hi[m];
            const int lo = (mini && ctl->tv[m] > base) ? ctl->tv[m] : base;
            for (int j = lo + gw; j < hi; j += nw) {
                const int n = m * a.half_n + (j - base);
                const unsigned int count = a.rep_count[n];
                bool hit = count > (unsigned int)ra.rep_cap;             // an overflowed list: the walk gives up there
                if (!hit) {
                    const uint32_t pick = a.lam[(size_t)m * s + j];
                    const double ps = a.pick_score[(size_t)m * s + j];
                    const double rn = j == 0 ? ctl->ynorm[m] : a.rnorm[(size_t)m * s + j - 1];
                    const float floor_sc = (float)ps - (float)screen_margin(rn, ps, a.k);
                    const bool skip_members = ctl->list_exact[m] != 0;
                    const uint2* list = ra.rep + (size_t)n * ra.rep_cap;
                    const int lane = threadIdx.x & 31;
                    // Whether a challenger reaches the pick is asked of this residual for both, as the walk does, in another order of the sums:
                    // what comes within 1e-9 of the pick (ties among it) is left to the walk.  (pick_score would not do: on the Gram
                    // path it comes from a recursion whose error is relative to ||y||, some 1e-8 of the score once ||r|| is at 1e-7 of ||y||.)
                    const double* res = a.rhist + (size_t)n * a.k;
                    double pd = 0.0, pn2 = 0.0;                          // the pick's products, from the first challenger on
                    int met = 0;                                         // challengers so far, the same in every lane
                    for (unsigned int e0 = 0; e0 < count && !hit; e0 += 8 * 32) {
                        uint2 rp8[8];                                    // eight reports in flight per lane
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const unsigned int e = e0 + 32u * u + lane;
                            rp8[u] = e < count ? list[e] : make_uint2(pick, 0u);
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const uint2 rp = rp8[u];
                            bool in = __uint_as_float(rp.y) >= floor_sc && rp.x != pick;
                            // a list member lost the exact comparison against the pick during the speculation (or is in the support)
                            if (in && skip_members && ((ra.cand_bits[rp.x >> 5] >> (rp.x & 31u)) & 1u)) in = false;
                            if (in && in_support(a.lam + (size_t)m * s, j, rp.x)) in = false;
                            for (unsigned int who = __ballot_sync(0xffffffffu, in); who && !hit; who &= who - 1u) {
                                const uint32_t col = __shfl_sync(0xffffffffu, rp.x, __ffs(who) - 1);
                                double dot, n2;
                                if (++met > kSweepCap) { hit = true; break; }
                                if (met == 1) warp_products(a, pick, res, &pd, &pn2);
                                warp_products(a, col, res, &dot, &n2);
                                hit = dot * dot * pn2 >= pd * pd * n2 * (1.0 - 1e-9);
                            }
                        }
                    }
                }
                if ((threadIdx.x & 31) == 0) a.ctl->contested[n] = hit ? 1 : 0;
            }
        }
    }
    // the block that finishes its share last walks the picks (ticket counter, nobody waits)
    __shared__ int last_block;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int ticket = atomicAdd(&a.ctl->resolve_ticket, 1u);
        last_block = ticket == gridDim.x - 1 ? 1 : 0;
        if (last_block) a.ctl->resolve_ticket = 0u;
    }
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    __shared__ int contested[kPassMaxN];
    for (int n = threadIdx.x; n < kPassMaxN; n += kOmpThreads) contested[n] = ctl->contested[n];
    if (threadIdx.x == 0) {
        give_up = 0; any_failed = 0;
        if (mini) ctl->list_rounds = ctl->list_rounds + 1;
        else {
            ctl->rounds = ctl->rounds + 1;
            // width of the pass whose reports are being resolved (ctl->narrow still names it)
            ctl->pass_rows = ctl->pass_rows + (ctl->narrow ? a.rows_narrow : a.rows_wide);
        }
    }
    __syncthreads();
    for (int m = 0; m < 2; ++m) {
        if (ctl->finished[m]) continue;
        const int base = ctl->base[m], hi = ctl->hi[m], extra = ctl->extra[m], dep = ctl->dep[m];
        const uint32_t* lam = a.lam + (size_t)m * s;
        const int lo = (mini && ctl->tv[m] > base) ? ctl->tv[m] : base;
        int v = lo;
        uint32_t forced = kNoColumn;
        bool failed = false, bad = false;
        for (int j = lo; j < hi && !failed && !bad; ++j) {
            const int n = m * a.half_n + (j - base);
            if (!contested[n]) { v = j + 1; continue; }           // nobody comes close: the pick is the argmax
            const unsigned int count = a.rep_count[n];
            if (count > (unsigned int)ra.rep_cap) { bad = true; break; }
            const uint32_t pick = lam[j];
            const double ps = a.pick_score[(size_t)m * s + j];
            const double rn = j == 0 ? ctl->ynorm[m] : a.rnorm[(size_t)m * s + j - 1];
            const float margin = (float)screen_margin(rn, ps, a.k);
            if (threadIdx.x == 0) sh.cand_idx[0] = pick;
            const int nc = collect_challengers(sh, ra.rep + (size_t)n * ra.rep_cap, count, lam, j, pick, (float)ps - margin,
                                               2.0f * margin, 1);
            if (nc < 0) { bad = true; break; }
            if (nc == 1) { v = j + 1; continue; }                 // nobody comes close: the pick is the argmax
            rescore_candidates(a, sh, nc, a.rhist + (size_t)n * a.k);       // the residual this pick was made from
            if (sh.best_idx == pick) { v = j + 1; continue; }
            forced = sh.best_idx; v = j; failed = true;
            if (!mini && threadIdx.x == 0) ctl->refuted = ctl->refuted + 1;
            make_room(ra, (int)count + 1 + ((hi - j) / kLookAhead) * 1024);
            harvest(ra, sh, ra.rep + (size_t)n * ra.rep_cap, count, forced);
            // look ahead: the later residuals of this speculation are off the true path by a pick or a few, yet close
            // to it, so the columns that come near their picks are the likely picks of the next round
            for (int jj = j + kLookAhead; jj < hi; jj += kLookAhead) {
                const int nn = m * a.half_n + (jj - base);
                const unsigned int cc = a.rep_count[nn];
                if (cc > (unsigned int)ra.rep_cap) continue;
                harvest(ra, sh, ra.rep + (size_t)nn * ra.rep_cap, cc, kNoColumn,
                        (float)(kLookAheadShare * a.pick_score[(size_t)m * s + jj]));        // reports hold unscaled scores
            }

        }
        if (mini) {
            // tentative outcome only
            if (!failed && !bad) v = dep ? hi - 1 : hi;
            __syncthreads();
            if (threadIdx.x == 0) {
                ctl->tv[m] = v;
                ctl->tforced[m] = forced;
                if (failed) { any_failed = 1; ctl->list_refuted = ctl->list_refuted + 1; }
                if (bad) give_up = 1;
            }
            __syncthreads();
            continue;
        }
        if (!failed && !bad) {
            if (dep) {
                // the dependent pick was the true argmax: Algorithm 3 cannot extend the support, this recovery ends
                v = hi - 1;
                if (threadIdx.x == 0) {
                    a.cnt->stopped[m] = 1; a.cnt->done[m] = v; ctl->finished[m] = 1;
                    atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_DEPENDENT_COLUMN);
                }
            } else if (hi >= s) {
                v = s;
                if (threadIdx.x == 0) { a.cnt->done[m] = s; ctl->finished[m] = 1; }
            } else if (extra) {
                // residual screened without a pick: its best reported column is the next pick
                const int n = m * a.half_n + (hi - base);
                const unsigned int count = a.rep_count[n];
                const double rn = hi == 0 ? ctl->ynorm[m] : a.rnorm[(size_t)m * s + hi - 1];
                const float margin = (float)screen_margin(rn, 8.0 * rn / sqrt((double)a.k), a.k);    // scores near the noise maximum
                int nc = -1;
                if (count >= 1u && count <= (unsigned int)ra.rep_cap)
                    nc = collect_challengers(sh, ra.rep + (size_t)n * ra.rep_cap, count, lam, hi, kNoColumn, 0.0f, 2.0f * margin, 0);
                if (nc <= 0) bad = true;
                else {
                    rescore_candidates(a, sh, nc, a.rhist + (size_t)n * a.k);
                    forced = sh.best_idx; v = hi;
                    make_room(ra, (int)count + 1);
                    harvest(ra, sh, ra.rep + (size_t)n * ra.rep_cap, count, forced);
                }
            } else {
                v = hi;                                           // the pass had no room for more residuals
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            ctl->v[m] = v;
            ctl->forced[m] = forced;
            ctl->tv[m] = v;
            ctl->tforced[m] = kNoColumn;
            if (bad) give_up = 1;
        }
        __syncthreads();
    }
    if (mini) {
        // list passes rest until the next full pass once every screened window is full and nothing in it was refuted, or
        // when the reports overflowed (the full pass has to sort that out)
        if (threadIdx.x == 0 && give_up) ctl->mini_done = 1;
        if (threadIdx.x == 0 && !any_failed && !give_up) {
            bool full = true;
            for (int m = 0; m < 2; ++m) {
                if (ctl->finished[m]) continue;
                const int base = ctl->base[m], hi = ctl->hi[m];
                if (!(hi - base >= a.half_n || hi >= s || ctl->dep[m] || ctl->extra[m])) full = false;
            }
            if (full) ctl->mini_done = 1;
        }
        return;
    }
    if (threadIdx.x == 0) {
        ctl->mini_done = 0;
        if (give_up) {
            ctl->fallback = 1; ctl->round_active = 0;
            atomicOr(&a.cnt->status, (unsigned int)SGC_STATUS_CANDIDATE_OVERFLOW);
        } else if (ctl->finished[0] && ctl->finished[1]) {
            ctl->round_active = 0;
        }
        ctl->narrow = (ctl->finished[1] && !ctl->finished[0]) ? 1 : 0;     // the rows of a pass start with the first stream's
        const int r = ctl->rounds - 1;
        if (r >= 0 && r < kMaxRounds) { ctl->trace[r][0] = ctl->v[0]; ctl->trace[r][1] = ctl->v[1]; ctl->trace[r][2] = ctl->n_cand; }
    }
}
// start of the recovery of one step.  keep_list (a state that speculates, in this step or in others): after Sparsify_s, M^ and V^ are combinations of the columns
// kept in this and in earlier steps (Eq. 4, 5), so the indices just kept are candidates, and they enter the ring of recent
// index sets.
__global__ void __launch_bounds__(kOmpThreads, 1)
k_begin(SpecCtl* ctl, int speculate, int keep_list, float* wide_tau, int shared, const uint32_t* sel_idx, int s, uint32_t* kept_ring, int hist_slots,
        uint32_t* cand_list, unsigned int* cand_bits) {
    __shared__ int n_s;
    const int t = threadIdx.x;
    // no wide list unless a long-list speculation asks for one
    if (wide_tau != nullptr && t < kPassMaxN) wide_tau[t] = __int_as_float(0x7f800000);
    if (t < kMaxRounds) ctl->trace[t][0] = ctl->trace[t][1] = ctl->trace[t][2] = 0;
    const int n0 = ctl->n_cand, version = ctl->list_version;
    const int slot = keep_list ? ctl->hist_next % hist_slots : 0;
    if (t == 0) n_s = n0;
    __syncthreads();
    if (keep_list) {
        for (int e = t; e < s; e += kOmpThreads) kept_ring[(size_t)slot * s + e] = sel_idx[e];
        cand_append(sel_idx, s, &n_s, cand_list, cand_bits);
    }
    __syncthreads();
    if (t == 0) {
        ctl->tv[0] = ctl->tv[1] = 0;
        ctl->tforced[0] = ctl->tforced[1] = kNoColumn;
        ctl->mini_done = 0; ctl->list_rounds = 0; ctl->list_refuted = 0; ctl->refuted = 0;
        ctl->round_active = speculate; ctl->fallback = speculate ? 0 : 1;
        ctl->v[0] = ctl->v[1] = 0;
        ctl->forced[0] = ctl->forced[1] = kNoColumn;
        ctl->finished[0] = 0;
        ctl->finished[1] = shared ? 1 : 0;          // shared support: the second stream makes no picks of its own
        ctl->narrow = shared ? 1 : 0;
        ctl->stop[0] = ctl->stop[1] = 0;
        ctl->rounds = 0; ctl->pass_error = 0; ctl->pass_rows = 0;
        ctl->gram_ok = 1;
        if (keep_list) {
            const int n_new = n_s < kCandCap ? n_s : kCandCap;
            // a version of 0 means a fresh state: no Gram matrix yet
            if (n_new != n0) { ctl->n_cand = n_new; ctl->list_version = version + 1; }
            else if (version == 0) ctl->list_version = 1;
            ctl->hist_next = (slot + 1) % hist_slots;
            if (ctl->hist_count < hist_slots) ctl->hist_count = ctl->hist_count + 1;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// the end of a step: coefficients, opt-in variants, Eq. (8), scatter, candidate-list upkeep
// ------------------------------------------------------------------------------------------------
struct FinishArgs {
    OmpArgs o;
    double* x; float* W; uint32_t* upd_idx; double* upd_val;
    double alpha, eps, lr, tol;
    int shared, speculate, keep_list;
    uint32_t* cand_list; unsigned int* cand_bits; const uint32_t* kept_ring; int* rounds_out;
};
constexpr size_t kFinishDynBytes = 160 * 1024;
constexpr int kFinishAhead = 8;                       // row entries per lane fetched ahead of their use

// x = the least-squares coefficients on the first n picks: x_j = gamma_j (a_j - sum_{l > j} c^(l)_j x_l), last pick first.  One
// warp; acc holds a on entry and x on return.  rows: c^(j)_l at [j * stride + l].
__device__ void back_substitute(double* acc, const double* gam, const double* rows, size_t stride, int n) {
    const int lane = threadIdx.x & 31;
    double next[kFinishAhead];
#pragma unroll
    for (int u = 0; u < kFinishAhead; ++u) { const int l = u * 32 + lane; next[u] = (n > 0 && l < n - 1) ? rows[(size_t)(n - 1) * stride + l] : 0.0; }
    double gn = n > 0 ? gam[n - 1] : 0.0;
    for (int j = n - 1; j >= 0; --j) {
        double row[kFinishAhead];
        const double gj = gn;
#pragma unroll
        for (int u = 0; u < kFinishAhead; ++u) {
            const int l = u * 32 + lane;
            row[u] = next[u];
            next[u] = (j > 0 && l < j - 1) ? rows[(size_t)(j - 1) * stride + l] : 0.0;
        }
        if (j > 0) gn = gam[j - 1];
        __syncwarp();
        const double xj = gj * acc[j];
        __syncwarp();
        if (lane == 0) acc[j] = xj;
#pragma unroll
        for (int u = 0; u < kFinishAhead; ++u) { const int l = u * 32 + lane; if (l < j) acc[l] = fma(-row[u], xj, acc[l]); }
        for (int l = kFinishAhead * 32 + lane; l < j; l += 32) acc[l] = fma(-rows[(size_t)j * stride + l], xj, acc[l]);
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kOmpThreads, 1) k_finish(FinishArgs f) {
    extern __shared__ double rows_s[];
    __shared__ double acc[2][kMaxS], gam_s[2][kMaxS];
    __shared__ uint32_t lam_s[2][kMaxS], vidx[kMaxS];
    __shared__ double red[32];
    __shared__ int cut, n_mis, n_neg, n_s;
    const OmpArgs& a = f.o;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, k = a.k, s = a.s;
    Counters* cnt = a.cnt;
    int n[2] = {cnt->done[0], cnt->done[1]};
    // ---- opt-in variants (remark after Eq. (8): both recoveries have their non-zeros at the same positions)
    //   tol > 0: a recovery is cut after the first pick that left ||r|| <= tol ||y||.  OMP is greedy, so the picks before the
    //            cut are those an early-stopping run makes, and the leading block of the recurrences gives the fit on them.
    //   shared:  the second stream made no picks; x^V is the least-squares fit of V^ on the support of the first stream:
    //            its coefficients in the orthogonal basis are <q_l, V^>.
    if (f.tol > 0.0) {
        for (int m = 0; m < (f.shared ? 1 : 2); ++m) {
            const double* y = a.y64 + (size_t)m * k;
            double yn2 = 0.0;
            for (int row = t; row < k; row += kOmpThreads) yn2 += y[row] * y[row];
            yn2 = block_sum(yn2, red);
            if (t == 0) {
                const double bound = f.tol * sqrt(yn2);
                cut = n[m];
                for (int j = 0; j < n[m]; ++j) if (a.rnorm[(size_t)m * s + j] <= bound) { cut = j + 1; break; }
                cnt->done[m] = cut;
            }
            __syncthreads();
            for (int i = cut + t; i < s; i += kOmpThreads) a.rnorm[(size_t)m * s + i] = 0.0;
            n[m] = cut;
            __syncthreads();
        }
    }
    for (int l = t; l < n[0]; l += kOmpThreads) { acc[0][l] = a.acoef[l]; gam_s[0][l] = a.gam[l]; lam_s[0][l] = a.lam[l]; }
    if (f.shared) {
        n[1] = n[0];
        for (int l = warp; l < n[0]; l += kOmpThreads / 32) {
            const double* q = a.q + (size_t)l * k;
            double u = 0.0;
            for (int row = lane; row < k; row += 32) u = fma(q[row], a.y64[(size_t)k + row], u);
            u = warp_sum(u);
            if (lane == 0) { acc[1][l] = u; gam_s[1][l] = a.gam[l]; }
        }
        for (int l = t; l < s; l += kOmpThreads) {
            const uint32_t v = l < n[0] ? a.lam[l] : kNoColumn;
            lam_s[1][l] = v; a.lam[s + l] = v;
            a.rnorm[s + l] = 0.0;
        }
        if (t == 0) cnt->done[1] = n[1];
    } else {
        for (int l = t; l < n[1]; l += kOmpThreads) { acc[1][l] = a.acoef[s + l]; gam_s[1][l] = a.gam[s + l]; lam_s[1][l] = a.lam[s + l]; }
    }
    // ---- coefficients: one warp per recovery; the triangular factors come into shared memory when they fit
    {
        const size_t need0 = (size_t)n[0] * n[0], need1 = f.shared ? 0 : (size_t)n[1] * n[1];
        const bool staged = (need0 + need1) * sizeof(double) <= kFinishDynBytes;
        if (staged) {
            for (int e = t; e < (int)need0; e += kOmpThreads) { const int j = e / n[0], l = e - j * n[0]; if (l < j) rows_s[e] = a.crow[(size_t)j * s + l]; }
            for (int e = t; e < (int)need1; e += kOmpThreads) { const int j = e / n[1], l = e - j * n[1]; if (l < j) rows_s[need0 + e] = a.crow[((size_t)s + j) * s + l]; }
        }
        __syncthreads();
        if (warp < 2) {
            const double* g0 = a.crow + (f.shared ? 0 : (size_t)warp * s * s);
            const double* s0 = rows_s + (f.shared ? 0 : warp * need0);
            back_substitute(acc[warp], gam_s[warp], staged ? s0 : g0, staged ? (size_t)n[warp] : (size_t)s, n[warp]);
        }
    }
    if (t == 0) { n_mis = 0; n_neg = 0; }
    __syncthreads();
    // ---- records: coefficients; unpicked slots read as "none"
    for (int i = t; i < 2 * s; i += kOmpThreads) {
        const int m = i >= s ? 1 : 0, l = i - m * s;
        f.x[i] = l < n[m] ? acc[m][l] : 0.0;
        if (l >= n[m]) a.lam[i] = kNoColumn;
    }
    // ---- Eq. (8) on the common support, where x^V > 0
    bool upd = false;
    double val = 0.0;
    const uint32_t mine = t < n[0] ? lam_s[0][t] : kNoColumn;
    if (t < n[0]) {
        int hit = -1;
        for (int b = 0; b < n[1]; ++b) if (lam_s[1][b] == mine) { hit = b; break; }
        if (hit < 0) atomicAdd(&n_mis, 1);
        else {
            const double xv = acc[1][hit];
            if (!(xv > 0.0)) atomicAdd(&n_neg, 1);
            else { val = f.lr * (f.alpha * acc[0][t] / (sqrt(xv) + f.eps)); upd = true; }
        }
    }
    vidx[t] = upd ? mine : kNoColumn;
    const int n_upd = __syncthreads_count(upd ? 1 : 0);
    if (upd) {
        int rank = 0;
        for (int b = 0; b < n[0]; ++b) rank += vidx[b] < mine ? 1 : 0;
        f.upd_idx[rank] = mine;
        f.upd_val[rank] = val;
        f.W[mine] = (float)((double)f.W[mine] - val);
    }
    if (t == 0) {
        cnt->n_upd = n_upd; cnt->mismatch = n_mis; cnt->negv = n_neg;
        unsigned int bits = 0;
        if (n_mis > 0 || n[0] != n[1]) bits |= (unsigned int)SGC_STATUS_SUPPORT_MISMATCH;
        if (n_neg > 0) bits |= (unsigned int)SGC_STATUS_NEGATIVE_V;
        if (bits) atomicOr(&cnt->status, bits);
    }
    if (!f.keep_list) return;
    // ---- the supports found stay (or become) candidates of the next step
    SpecCtl* ctl = a.ctl;
    // how many rounds this step took (the enqueued rounds if even they were not enough): sizes the next step's launches
    // bit 8: a list pass refuted a pick (the wide lists earned their keep); bit 9: a full pass refuted a pick; bits 10, 11: how
    // many speculating steps in a row were refuted, that is, needed more passes than the residuals of s picks fill (at most 3)
    if (t == 0 && f.speculate) {
        // (list passes that refute nothing count against a state of one pass alone: the next step then does without them)
        const int room = a.depth < a.half_n ? a.depth : a.half_n, fewest = (s + room - 1) / room;
        const bool confirmed = !ctl->fallback && ctl->refuted == 0 && ctl->rounds <= fewest && ctl->list_refuted == 0 &&
                               (fewest > 1 || ctl->list_rounds == 0);
        const int streak = confirmed ? 0 : (ctl->inexact_streak < 3 ? ctl->inexact_streak + 1 : 3);
        ctl->inexact_streak = streak;
        *f.rounds_out = (ctl->fallback ? kMaxRounds : ctl->rounds) | (ctl->list_refuted > 0 ? 256 : 0) | (ctl->refuted > 0 ? 512 : 0) |
                        (streak << 10);
    }
    int nl = ctl->n_cand;
    // rebuild from the supports and the ring of kept index sets when the list has outgrown its bound, or when it holds
    // far more than those although a single round confirmed every pick (harvested columns of an earlier cold start)
    const int n_hist = ctl->hist_count * s;
    const bool rebuild = nl > kCandKeep || (ctl->rounds <= 1 && !ctl->fallback && nl > 4 * s + n_hist);
    if (rebuild) {
        for (int e = t; e < nl; e += kOmpThreads) {
            const uint32_t col = f.cand_list[e];
            atomicAnd(&f.cand_bits[col >> 5], ~(1u << (col & 31u)));
        }
        nl = 0;
    }
    if (t == 0) n_s = nl;
    __syncthreads();
    for (int m = 0; m < 2; ++m) {
        cand_append(lam_s[m], n[m], &n_s, f.cand_list, f.cand_bits);
        __syncthreads();
    }
    if (rebuild) cand_append(f.kept_ring, n_hist, &n_s, f.cand_list, f.cand_bits);
    __syncthreads();
    if (t == 0) {
        const int n_new = n_s < kCandCap ? n_s : kCandCap;
        if (n_new != ctl->n_cand || nl == 0) ctl->list_version = ctl->list_version + 1;     // rebuilt or extended
        ctl->n_cand = n_new;
    }
}

// z with d * P(|N(0,1)| > z) = target (bisection on erfc)
double normal_tail_threshold_impl(double d, double target) {
    double p = target / d;
    if (p > 0.5) p = 0.5;
    double lo = 0.0, hi = 12.0;
    for (int i = 0; i < 80; ++i) {
        const double mid = 0.5 * (lo + hi);
        if (erfc(mid / sqrt(2.0)) > p) lo = mid; else hi = mid;
    }
    return 0.5 * (lo + hi);
}

OmpArgs make_args(const sgc_state* st) {
    OmpArgs a;
    memset(&a, 0, sizeof(a));
    a.seed_lo = (uint32_t)(st->seed & 0xFFFFFFFFu); a.seed_hi = (uint32_t)(st->seed >> 32);
    a.d = (unsigned long long)st->d; a.k = st->k; a.s = st->s; a.kp = st->kp;
    a.sigma = (double)(float)(1.0 / sqrt((double)st->k));
    a.half_n = st->pass_n / 2;
    a.rows_wide = st->pass_n; a.rows_narrow = st->pass_n_half;
    a.z_harvest = st->z_harvest; a.z_floor = st->z_floor;
    a.corr_cand = st->corr_cand; a.y64 = st->y64; a.r32 = reinterpret_cast<float*>(st->r32);
    a.lam = st->lam; a.q = st->q_basis; a.crow = st->F; a.ccol = st->ccol; a.gam = st->gam; a.acoef = st->acoef; a.rnorm = st->rnorm;
    a.cnt = st->cnt; a.ctl = st->ctl;
    a.rt = st->rt; a.tau = st->tau; a.inv_scale = st->inv_scale; a.rep_count = st->rep_count; a.pick_score = st->pick_score;
    a.rhist = st->rhist;
    a.cand_list = st->cand_list;
    a.zlist = st->zlist; a.gram = st->gram; a.p0 = st->p0; a.wgram = st->wgram; a.pnorm = st->pnorm;
    a.wide_tau = st->wide_tau; a.z_wide = st->z_wide; a.wide_every = st->wide_every; a.wide_count = nullptr; a.wide_bits = st->wide_bits; a.mini = 0;
    a.depth = 1 << 30;
    return a;
}

}  // namespace

double normal_tail_threshold(double d, double target) { return normal_tail_threshold_impl(d, target); }

cudaError_t configure_recover(sgc_state* st) {
    cudaError_t e = omp_configure(st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFinishDynBytes);
    if (e != cudaSuccess) return e;
    int coop = 0;
    e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, st->device);
    if (e != cudaSuccess) return e;
    if (!coop) return cudaErrorNotSupported;
    // the tensor-core pass works on whole 64-row chunks of A: rows beyond k are zero in the residuals
    st->kp = (st->k + 63) / 64 * 64;
    int half = st->s < 128 ? st->s : 128;
    half = (half + 15) / 16 * 16;
    st->pass_n = 2 * half;
    // shared-support variant: only the first stream has residuals to screen, a pass half as wide does
    st->pass_n_half = ((st->pass_n / 2 + 31) / 32) * 32;
    st->z_harvest = normal_tail_threshold_impl((double)st->d, 3072.0);
    st->z_harvest_few = normal_tail_threshold_impl((double)st->d, 256.0);
    st->z_floor = normal_tail_threshold_impl((double)st->d, 6144.0);
    st->z_wide = normal_tail_threshold_impl((double)st->d, 100000.0);
    // How often a screened residual feeds the wide lists: a pick takes 25-30 / k of the residual's energy, so the scores of the
    // columns drift the faster the smaller k is.  Mean step (full passes per step) at every 8th / 4th / 2nd residual, 4096 x 11008:
    // k = 256, s = 16: 16.2 (2.80) / 14.7 (2.45) / 14.1 ms (2.25); k = 2048, s = 128: 125 (3.50) / 117 (3.19) / 119 ms (3.19);
    // k = 4096, s = 256: 247 (2.55) / 259 (2.60) / 263 ms (2.60): denser feeding makes the lists longer.
    st->wide_every = st->k < 512 ? 2 : st->k <= 2048 ? 4 : 8;
    return cudaSuccess;
}

cudaError_t finish_recover_setup(sgc_state* st, cudaStream_t stream) {
    cudaError_t e = pass_configure(kPassMaxN);
    for (int g = 1; g <= kPassMaxN / st->pass_n && e == cudaSuccess; ++g)      // one map per number of states in a batch
        e = pass_encode_map(st->tmap[g - 1], st->rt, g * st->pass_n, st->kp);
    if (e != cudaSuccess) return e;
    e = pass_encode_map(st->tmap_half, st->rt, st->pass_n_half, st->kp);
    if (e != cudaSuccess) return e;
    return launch_inv_norms(st->seed, (uint64_t)st->d, st->k, st->inv_norm, stream);     // column norms: a property of (seed, k)
}

// Whether the next step of a state speculates.  Requested modes are obeyed.  SGC_MODE_AUTO compares estimates (us, from the
// timings below): in lock-step every pick costs its bookkeeping and barriers and one correlation of all columns; a
// speculation that one pass confirms costs that pass and little per pick; one that is refuted every few picks costs list
// correlations, list passes and resolving.  Which of the two a state meets is known once it has speculated for two steps; before,
// the sizes tell: steps of d = 129344, k = 512, s = 33 (k = 1.32 s ln d) are confirmed by one pass, those of 1721085, 384, 26
// (1.03) and 2^24, 1024, 64 (0.96) are not.
//   lock-step, us per pick:  d = 65000, k = 350: 22;  200000, 210: 30;  270000, 300: 41;  1200000, 224: 88;  500000, 700: 105
//                                                                                             (11 + k d / 2.8e6)
//   refuted speculation:     some 56 s / k rounds (at most one for every four picks), each a full pass, its launches and as many picks as are speculated ahead: ms per step
//                            d = 400400, k = 1024, s = 128: 6.6;  1e6, 448, 60: 4.2;  3001000, 700, 100: 12.2;  5e6, 192, 24: 3.9
//                                                                   ((1 + 56 s / k) (250 + k d / 3.3e6 + 17 per speculated pick));
//                            with list passes 1876582, 960, 123: 168 us per pick;  7.3e6, 576, 73: 230      (100 + k d / 2.0e7)
//   confirmed speculation, us per step: d = 143488, k = 1600, s = 25: 370 (with the launches; 140 + k d / 3.3e6 per pass, + 1.2 s)
// A state that has come to prefer lock-step tries a speculating step now and then: its gradients may have changed.
constexpr int kRetrySteps = 32;
constexpr double kFewRoundsWork = 3.0e8;              // k * d up to which a pick in lock-step costs at most 120 us
// k * d from which list passes are cheaper than full ones (ms per step with / without them: d = 400400, k = 1024, s = 128: 11.2 / 6.6;  1e6, 448, 60:
// 7.8 / 3.9;  5e6, 192, 24: 5.6 / 3.8;  3e6, 700, 100: 14.8 / 12.2;  3.2e6, 576, 73: 9.8 / 9.0;  7.3e6, 576, 73: 16.9 / 18.4).  A state that is told to
// speculate whatever its size gets them from the smaller bound on.
constexpr double kTwoLevelWork = 3.0e9, kTwoLevelWorkForced = 1.0e8;
// Picks that a refuted state below that bound speculates ahead of a full pass: a pick takes 25-30 / k of the residual's energy, so a speculation
// of noise columns holds for some k / 55 picks, and what follows the first refuted pick is thrown away (it was most of such a step:
// 17 us per pick).  ms per step at depth 16 / 24 / 32 / 48 / all that a pass has room for:  1e6, 448, 60: 4.0 / 4.4 / 4.9 / 5.9 / 6.5;  400400, 1024, 128:
// 7.2 / 7.0 / 6.6 / 8.0 / 9.7;  522992, 1036, 148: 10.4 / 9.4 / 9.1 / 11.0 / 13.3;  5e6, 192, 24: 3.8 / 4.0 / 4.0 / 4.0 / 4.0 (at 12: 3.5).
static int refuted_depth(const sgc_state* st) {
    const int depth = st->k / 32 > 12 ? st->k / 32 : 12, least = (st->s + 7) / 8;      // (at most eight rounds of picks that all hold)
    return depth > least ? depth : least;
}
static bool was_refuted(const sgc_state* st) { return ((*reinterpret_cast<volatile int*>(st->h_rounds) >> 10) & 3) != 0; }

// passes over all columns that a step takes when nothing is refuted: a pass has room for pass_n / 2 residuals per recovery
static int fewest_passes(const sgc_state* st) { return (st->s + st->pass_n / 2 - 1) / (st->pass_n / 2); }

static bool prefers_speculation(const sgc_state* st) {
    const double kd = (double)st->k * (double)st->d, s = (double)st->s;
    const double lock = s * (11.0 + kd / 2.8e6);
    const int seen = *reinterpret_cast<volatile int*>(st->h_rounds);
    const bool refuted = (seen & 255) != 0 ? ((seen >> 10) & 3) >= 2 : (double)st->k < 1.2 * s * log((double)st->d);
    const double passes = (double)fewest_passes(st);
    const double rounds = 1.0 + (56.0 * s / (double)st->k < 0.25 * s ? 56.0 * s / (double)st->k : 0.25 * s);
    const double ahead = (double)(st->s < refuted_depth(st) ? st->s : refuted_depth(st));
    const double again = kd < kTwoLevelWork ? rounds * (250.0 + kd / 3.3e6 + 17.0 * ahead) : s * (100.0 + kd / 2.0e7);
    const double spec = refuted ? again : passes * (140.0 + kd / 3.3e6) + 1.2 * s;
    return spec < lock;
}

bool will_speculate(const sgc_state* st) {
    if (st->mode != SGC_MODE_AUTO) return st->mode == SGC_MODE_SPECULATIVE;
    return st->d >= kSpecMinD && (prefers_speculation(st) || st->lock_steps >= kRetrySteps);
}

// the same, and counts the lock-step steps since the last speculating one (only a state that has speculated and turned away
// tries again)
static bool wants_speculation(sgc_state* st) {
    const bool yes = will_speculate(st);
    if (yes) st->lock_steps = 0;
    else if ((*reinterpret_cast<volatile int*>(st->h_rounds) & 255) != 0) st->lock_steps += 1;
    return yes;
}

// the candidate list is kept up in lock-step steps as well, so that a later speculation does not start cold
static bool keeps_list(const sgc_state* st) { return st->spec_ready && st->mode != SGC_MODE_LOCKSTEP; }

// Recovery (a4 + a5) of n states that share (d, k, s, seed), hence A.  The states' screened residuals are laid out side by
// side in the screening buffers of the first state of each batch (a batch = as many states as fit kPassMaxN columns), so
// one pass over A serves a whole batch; everything else runs per state.  n = 1 is the plain sgc_step.
static cudaError_t recover_batches(sgc_state* const* sts, float* const* weights, int n, cudaStream_t stream, int* launches) {
    sgc_state* st0 = sts[0];
    bool speculate = true;
    for (int i = 0; i < n; ++i)
        speculate = wants_speculation(sts[i]) && sts[i]->spec_ready && speculate;
    const int per_batch = speculate ? kPassMaxN / st0->pass_n : 1;
    std::vector<OmpArgs> args((size_t)n);
    cudaError_t e = cudaSuccess;
    int n_rounds = 0;
    int mini_rounds = 0;          // rounds that get list passes: the likely ones; the spare rounds behind them stay cheap to enqueue
    for (int i = 0; i < n; ++i) {
        sgc_state* st = sts[i];
        sgc_state* lead = sts[i - i % per_batch];
        const int slot = i % per_batch;
        OmpArgs a = make_args(st);
        // this state's slice of the batch's screening buffers
        a.rt = lead->rt + (size_t)slot * st->pass_n * st->kp;
        a.tau = lead->tau + slot * st->pass_n;
        a.inv_scale = lead->inv_scale + slot * st->pass_n;
        a.rep_count = lead->rep_count + slot * st->pass_n;
        // a state whose picks one pass confirms, step after step, needs no candidates from it: fewer columns are reported
        // and swept by the resolve kernel
        const int seen = *reinterpret_cast<volatile int*>(st->h_rounds);
        if (st->mode == SGC_MODE_AUTO && (seen & 255) == 1 && (seen >> 10) == 0) a.z_harvest = st->z_harvest_few;
        if (was_refuted(st) && (double)st->k * (double)st->d < kTwoLevelWork) a.depth = refuted_depth(st);
        args[i] = a;
        {
            PhaseTimer timer(st, stream, kPhaseBook, 1);
            k_begin<<<1, kOmpThreads, 0, stream>>>(st->ctl, speculate ? 1 : 0, keeps_list(st) ? 1 : 0, st->wide_tau, st->shared_support, st->sel_idx, st->s,
                                                   st->kept_ring, st->hist_slots, st->cand_list, st->cand_bits);
            *launches += 1;
        }
        // rounds to enqueue: twice what the last finished step needed plus slack (read from pinned memory without
        // synchronising; a stale value only changes how much is enqueued); what they leave open is done in lock-step
        const int hint = speculate ? *reinterpret_cast<volatile int*>(st->h_rounds) : 0;
        const int last = hint & 255;
        int want = last <= 0 ? 8 : 2 * last + 3;
        // a state whose steps one pass confirms, and for which finishing in lock-step would cost little: one spare round (each
        // costs three launches, 12 us, of a step of 300)
        const bool smooth = st->mode == SGC_MODE_AUTO && last == 1 && (hint >> 10) == 0;
        if (smooth && (double)st->k * (double)st->d <= kFewRoundsWork) want = 2;
        if (last > 0 && last + 2 > mini_rounds) mini_rounds = last + 2;
        if (last <= 0) mini_rounds = kMaxRounds;
        if (st->max_rounds > 0 && want > st->max_rounds) want = st->max_rounds;
        if (want > n_rounds) n_rounds = want;
        // two-level screening pays where steps need several full passes (recovery picks columns outside the kept sets);
        // it is dropped again when a step needed one pass and its list passes refuted nothing.  Several passes that refute nothing
        // because s picks do not fit one are no reason for it
        const bool contested = (hint >> 10) != 0;
        const double least = st->mode == SGC_MODE_SPECULATIVE ? kTwoLevelWorkForced : kTwoLevelWork;
        if (last >= 3 && contested && (double)st->k * (double)st->d >= least) st->two_level = true;
        else if (last == 1 && !(hint & 256)) st->two_level = false;
    }
    if (n_rounds > kMaxRounds) n_rounds = kMaxRounds;
    const bool two_level = speculate && n == 1 && st0->two_level;
    // A state whose two streams fill a pass of more than kPassFastRows rows, and whose last step had a pick refuted: the
    // refuted stream needs several rounds anyway, and the rows of a speculation beyond its first refuted pick are wasted.
    // Such a step screens half as many residuals per stream and round, in the pass of half the width at half the cost;
    // the stream that is confirmed without contest rides along in two rounds instead of one.
    const bool compact = speculate && n == 1 && st0->pass_n > kPassFastRows && st0->pass_n_half <= kPassFastRows &&
                         (*reinterpret_cast<volatile int*>(st0->h_rounds) & 512) != 0;
    if (compact) {
        args[0].half_n = st0->pass_n_half / 2;
        args[0].rows_wide = args[0].rows_narrow = st0->pass_n_half;
        n_rounds = n_rounds + 1 < kMaxRounds ? n_rounds + 1 : kMaxRounds;
        if (st0->max_rounds > 0 && n_rounds > st0->max_rounds) n_rounds = st0->max_rounds;
    }
    PassWide wide;
    if (two_level) {
        args[0].wide_count = st0->wide_count;
        wide.tau = st0->wide_tau; wide.list = st0->wide_list; wide.count = st0->wide_count; wide.bits = st0->wide_bits;
        wide.cap = kWideCap; wide.half_n = args[0].half_n; wide.ctl = st0->ctl; wide.list_pass = false;
    }
    if (speculate) {
        for (int round = 0; round < n_rounds && e == cudaSuccess; ++round) {
            // list passes first: speculate a few picks ahead, screen the wide lists only, keep what they confirm as
            // tentative picks; every kernel of this loop returns at once when there is nothing (more) to do
            for (int mini = 0; two_level && round < mini_rounds && mini < kMiniRounds && e == cudaSuccess; ++mini) {
                sgc_state* st = st0;
                {
                    PhaseTimer timer(st, stream, kPhaseCorr, 1);
                    OmpArgs am = args[0];
                    am.mini = 1; am.depth = st->k < kMiniShallowK ? kMiniDepth / 2 : kMiniDepth;
                    e = launch_omp(st, am, 0, stream);
                    *launches += 1;
                }
                if (e != cudaSuccess) break;
                {
                    PhaseTimer timer(st, stream, kPhasePass, 1);
                    const int* gates[kPassMaxBatch] = {&st->ctl->round_active};
                    int* errors[kPassMaxBatch] = {&st->ctl->pass_error};
                    PassWide lp = wide;
                    lp.list_pass = true;
                    const bool two_widths = !compact && st->pass_n_half < st->pass_n;   // the width that ctl->narrow names runs
                    if (compact)
                        e = launch_pass(st->tmap_half, st->seed, (uint64_t)st->d, st->kp, st->pass_n_half, st->tau, st->inv_scale,
                                        st->inv_norm, st->rep_count, st->rep, kRepCap, gates, errors, st->sm_count, stream, &lp,
                                        nullptr, 0, st->wait_limit_ns);
                    else
                    e = launch_pass(st->tmap[0], st->seed, (uint64_t)st->d, st->kp, st->pass_n, st->tau, st->inv_scale,
                                    st->inv_norm, st->rep_count, st->rep, kRepCap, gates, errors, st->sm_count, stream, &lp,
                                    two_widths ? &st->ctl->narrow : nullptr, 0, st->wait_limit_ns);
                    if (two_widths && e == cudaSuccess) {
                        e = launch_pass(st->tmap_half, st->seed, (uint64_t)st->d, st->kp, st->pass_n_half, st->tau,
                                        st->inv_scale, st->inv_norm, st->rep_count, st->rep, kRepCap, gates, errors,
                                        st->sm_count, stream, &lp, &st->ctl->narrow, 1, st->wait_limit_ns);
                        *launches += 1;
                    }
                    *launches += 1;
                }
                if (e != cudaSuccess) break;
                ResolveArgs ra;
                ra.o = args[0];
                ra.rep = st->rep; ra.rep_cap = kRepCap; ra.cand_bits = st->cand_bits; ra.cand_list = st->cand_list;
                ra.kept_ring = st->kept_ring; ra.mini = 1; ra.wide_count = st->wide_count;
                PhaseTimer timer(st, stream, kPhaseBook, 1);
                k_resolve<<<kResolveBlocks, kOmpThreads, 0, stream>>>(ra);
                *launches += 1;
            }
            for (int b0 = 0; b0 < n && e == cudaSuccess; b0 += per_batch) {
                const int nb = n - b0 < per_batch ? n - b0 : per_batch;
                for (int i = b0; i < b0 + nb && e == cudaSuccess; ++i) {
                    sgc_state* st = sts[i];
                    const OmpArgs& a = args[i];
                    PhaseTimer timer(st, stream, kPhaseCorr, 1);
                    e = launch_omp(st, a, 0, stream);
                    *launches += 1;
                }
                if (e != cudaSuccess) break;
                sgc_state* lead = sts[b0];
                {
                    PhaseTimer timer(lead, stream, kPhasePass, 1);
                    const int* gates[kPassMaxBatch];
                    int* errors[kPassMaxBatch];
                    for (int q = 0; q < kPassMaxBatch; ++q) {
                        gates[q] = q < nb ? &sts[b0 + q]->ctl->round_active : nullptr;
                        errors[q] = q < nb ? &sts[b0 + q]->ctl->pass_error : nullptr;
                    }
                    // a state on its own: once only its first stream has residuals left (the second recovery is complete, or
                    // the shared-support variant is on), the pass half as wide serves the round; ctl->narrow names the width
                    const bool two_widths = n == 1 && !compact && lead->pass_n_half < lead->pass_n;
                    if (compact)
                        e = launch_pass(lead->tmap_half, lead->seed, (uint64_t)lead->d, lead->kp, lead->pass_n_half, lead->tau,
                                        lead->inv_scale, lead->inv_norm, lead->rep_count, lead->rep, kRepCap, gates, errors,
                                        lead->sm_count, stream, two_level ? &wide : nullptr, nullptr, 0, lead->wait_limit_ns);
                    else
                    e = launch_pass(lead->tmap[nb - 1], lead->seed, (uint64_t)lead->d, lead->kp, nb * lead->pass_n, lead->tau,
                                    lead->inv_scale, lead->inv_norm, lead->rep_count, lead->rep, kRepCap, gates, errors,
                                    lead->sm_count, stream, two_level ? &wide : nullptr,
                                    two_widths ? &lead->ctl->narrow : nullptr, 0, lead->wait_limit_ns);
                    if (two_widths && e == cudaSuccess) {
                        e = launch_pass(lead->tmap_half, lead->seed, (uint64_t)lead->d, lead->kp, lead->pass_n_half, lead->tau,
                                        lead->inv_scale, lead->inv_norm, lead->rep_count, lead->rep, kRepCap, gates, errors,
                                        lead->sm_count, stream, two_level ? &wide : nullptr, &lead->ctl->narrow, 1,
                                        lead->wait_limit_ns);
                        *launches += 1;
                    }
                    *launches += 1;
                }
                for (int i = b0; i < b0 + nb && e == cudaSuccess; ++i) {
                    sgc_state* st = sts[i];
                    ResolveArgs ra;
                    ra.o = args[i];
                    ra.rep = lead->rep + (size_t)(i - b0) * st->pass_n * kRepCap;
                    ra.rep_cap = kRepCap; ra.cand_bits = st->cand_bits; ra.cand_list = st->cand_list;
                    ra.kept_ring = st->kept_ring; ra.mini = 0; ra.wide_count = st->wide_count;
                    PhaseTimer timer(st, stream, kPhaseBook, 1);
                    k_resolve<<<kResolveBlocks, kOmpThreads, 0, stream>>>(ra);
                    *launches += 1;
                }
            }
        }
        if (e != cudaSuccess) return e;
    }
    for (int i = 0; i < n; ++i) {
        sgc_state* st = sts[i];
        {
            PhaseTimer timer(st, stream, kPhaseCorr, 1);
            e = launch_omp(st, args[i], 1, stream);
            *launches += 1;
        }
        if (e != cudaSuccess) return e;
        PhaseTimer timer(st, stream, kPhaseScatter, 1);
        FinishArgs f;
        f.o = args[i];
        f.x = st->x; f.W = weights[i]; f.upd_idx = st->upd_idx; f.upd_val = st->upd_val;
        f.alpha = (double)st->alpha; f.eps = (double)st->eps; f.lr = (double)st->lr; f.tol = st->residual_tol;
        f.shared = st->shared_support; f.speculate = speculate ? 1 : 0; f.keep_list = keeps_list(st) ? 1 : 0;
        f.cand_list = st->cand_list; f.cand_bits = st->cand_bits; f.kept_ring = st->kept_ring; f.rounds_out = st->d_rounds;
        k_finish<<<1, kOmpThreads, kFinishDynBytes, stream>>>(f);
        *launches += 1;
    }
    return cudaGetLastError();
}

// Which states of a group share passes.  One pass serves a batch of states only while it has room for all their residuals
// (kPassMaxN rows), and the two-level screening -- what keeps the number of passes over all d columns down when the
// recovery picks columns outside the kept sets -- is a single-state scheme.  So a state goes alone when a batch could hold
// nothing beside it, or when its last step needed three or more passes over all columns (the signal that switches its two-level
// screening on, from k d = kTwoLevelWork on; smaller states go by the same rule, and make their rounds alone without it); the others
// are batched.  The result does not depend on the split.
cudaError_t launch_recover_group(sgc_state* const* sts, float* const* weights, int n, cudaStream_t stream, int* launches) {
    if (n == 1) return recover_batches(sts, weights, 1, stream, launches);
    std::vector<sgc_state*> together;
    std::vector<float*> together_w;
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < n && e == cudaSuccess; ++i) {
        sgc_state* st = sts[i];
        const bool speculates = st->spec_ready && will_speculate(st);
        const int last = speculates ? (*reinterpret_cast<volatile int*>(st->h_rounds) & 255) : 0;
        const bool alone = !speculates || (kPassMaxN / st->pass_n < 2 || st->two_level || last >= 3);
        if (alone) e = recover_batches(&sts[i], &weights[i], 1, stream, launches);
        else { together.push_back(st); together_w.push_back(weights[i]); }
    }
    if (e == cudaSuccess && !together.empty())
        e = recover_batches(together.data(), together_w.data(), (int)together.size(), stream, launches);
    return e;
}

cudaError_t launch_recover(sgc_state* st, float* weight, cudaStream_t stream, int* launches) {
    return recover_batches(&st, &weight, 1, stream, launches);
}

}  // namespace sgc