// The recoveries of the batched chunk path (sgc_chunked.cu) in one launch, for chunks whose matrix A is too large for the shared memory
// of a cluster but not for that of the whole GPU: one block per SM keeps its share of the columns (K-major, 128-byte swizzle,
// generated once), and an iteration of Algorithm 3 for all recoveries is
//     scores: the residuals (binary16, one row each) pass by 128 at a time as the M operand of tcgen05.mma, the block's columns are
//             the N operand (up to 256 at a time); a thread owns one residual and notes the columns that reach its threshold;
//             what the block noted joins the recoveries' report lists          | grid barrier
//     books:  every block decides for its recoveries in fp64 among the reported columns within twice the scores' error bound of the
//             best, updates q and r and writes the new residual row            | grid barrier
// What the reports cannot settle (none, too many, a window that reaches below the threshold, a wait that expired) is settled by going
// through all columns in fp64.  Scores only say which columns the fp64 decision looks at: rounding a residual to one binary16 number is
// part of the bound that its window is made of, where the general form's fp32 route (which scores value and remainder) has 2e-3 of the best.
// Bound by latency: an iteration of 512 recoveries over 65536 columns, k = 112, takes 23 us (54 in six launches, which generated A twice): scores 11,
// of which the products take 4 and the comparisons are issue slots; books 7; the two grid barriers 4.  Step: 874 -> 424 us.
#include <cooperative_groups.h>

#include "sgc_chunk_book.cuh"

namespace cg = cooperative_groups;

namespace sgc {
namespace {

constexpr int kGT = 32 * kClusterWarps;                // threads that score and keep books; one more warp issues the matrix operations
constexpr int kAccCols = 256;                         // tensor-memory columns of an accumulator buffer (two of them)
constexpr unsigned long long kGridWaitNs = 2000000000ull;

struct GridHead {
    unsigned long long full[2], empty[2], rows[2], drain;        // accumulators complete, and read; residual rows in place
    uint32_t tmem;
    int abort_flag;
    unsigned int n_queue;
};
static_assert(sizeof(GridHead) <= kGridHead, "barriers");

__device__ __forceinline__ uint32_t swizzled(uint32_t row, uint32_t piece) { return row * 128u + ((piece ^ (row & 7u)) << 4); }

// the block's columns: [column block of 256][64-row chunk][column][64 rows], and 1 / ||Z_i|| (0 beyond the chunk).  Thread = column.
__device__ __forceinline__ void grid_columns(const ChunkArgs& a, const GridPlan& p, unsigned char* sm, long long col0) {
    float* inv = reinterpret_cast<float*>(sm + p.off_inv);
    for (int c = threadIdx.x; c < p.cols; c += kGT + 32) {
        const int nb = c / kAccCols, in = c % kAccCols, width = p.cols - nb * kAccCols < kAccCols ? p.cols - nb * kAccCols : kAccCols;
        unsigned char* block = sm + (size_t)nb * kAccCols * p.kc * 128;
        const ColKey key = column_key(a.seed_lo, a.seed_hi, (uint32_t)(col0 + c));
        uint32_t h = key.ck;
        float n2 = 0.0f;
        for (int piece = 0; piece < p.kc * 8; ++piece) {               // eight rows
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = piece * 8 + 2 * e;
                w[e] = z_pair_from_word(h);
                h += key.mk;
                if (row >= a.k) w[e] = 0u;
                else if (row + 1 >= a.k) w[e] &= 0xFFFFu;
                const float2 f = half2_bits_to_float2(w[e]);
                n2 = __fmaf_rn(f.x, f.x, n2); n2 = __fmaf_rn(f.y, f.y, n2);
            }
            *reinterpret_cast<uint4*>(block + (size_t)(piece >> 3) * width * 128 + swizzled((uint32_t)in, (uint32_t)(piece & 7))) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
        inv[c] = col0 + c < a.dc && n2 > 0.0f ? 1.0f / sqrtf(n2) : 0.0f;
    }
}

// residual rows of tile mt: sixteen bytes per thread and piece.  KC: 64-row chunks of A
template <int KC>
__device__ __forceinline__ void fetch_rows(const ChunkArgs& a, int mt, uint4 (&v)[2 * KC]) {
    const uint4* src = reinterpret_cast<const uint4*>(a.rt + (size_t)mt * 128 * (KC * 64)) + threadIdx.x;
#pragma unroll
    for (int i = 0; i < 2 * KC; ++i) v[i] = __ldcg(src + i * kGT);     // (other blocks wrote them)
}
template <int KC>
__device__ __forceinline__ void store_rows(unsigned char* dst, const uint4 (&v)[2 * KC]) {
#pragma unroll
    for (int i = 0; i < 2 * KC; ++i) {
        const int at = threadIdx.x + i * kGT, row = at / (KC * 8), piece = at % (KC * 8);
        *reinterpret_cast<uint4*>(dst + (size_t)(piece >> 3) * 16384 + swizzled((uint32_t)row, (uint32_t)(piece & 7))) = v[i];
    }
    fence_async_smem();
}

// Largest |v_i| w_i of 16 accumulators.  Products that are not negative are ordered like their bits, and the integer maximum takes three
// operands: one and a half instructions per score instead of two.
__device__ __forceinline__ unsigned int peak_bits16(const uint32_t* v, const float* w) {
    int p[2] = {0, 0};
    const float4* w4 = reinterpret_cast<const float4*>(w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 x = w4[i];
        p[0] = __vimax3_s32(p[0], __float_as_int(fabsf(__uint_as_float(v[4 * i])) * x.x), __float_as_int(fabsf(__uint_as_float(v[4 * i + 1])) * x.y));
        p[1] = __vimax3_s32(p[1], __float_as_int(fabsf(__uint_as_float(v[4 * i + 2])) * x.z), __float_as_int(fabsf(__uint_as_float(v[4 * i + 3])) * x.w));
    }
    return (unsigned int)max(p[0], p[1]);
}
// which of 16 accumulators reach tau (weights: 1 / ||Z_i||, zero beyond the chunk)
__device__ __forceinline__ unsigned int hits16(const uint32_t* v, const float* w, float tau) {
    unsigned int h = 0u;
    const float4* w4 = reinterpret_cast<const float4*>(w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 x = w4[i];
        h |= fabsf(__uint_as_float(v[4 * i])) * x.x >= tau ? 1u << (4 * i) : 0u;
        h |= fabsf(__uint_as_float(v[4 * i + 1])) * x.y >= tau ? 2u << (4 * i) : 0u;
        h |= fabsf(__uint_as_float(v[4 * i + 2])) * x.z >= tau ? 4u << (4 * i) : 0u;
        h |= fabsf(__uint_as_float(v[4 * i + 3])) * x.w >= tau ? 8u << (4 * i) : 0u;
    }
    return h;
}

// ---- scores ------------------------------------------------------------------------------------------------
// One warp issues the products, a tile of residual rows and a block of columns at a time, into two accumulator buffers by turns; the
// other sixteen bring the next rows into place and compare, each at its own pace: a warp that notes a report takes 0.3 us longer
// than the others, and with block-wide barriers between the steps every step took as long as its slowest warp.  done_steps, done_tiles: how many
// steps and row tiles this launch has behind it.  False: a wait expired.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
    return mbar_test(bar, parity) || block_wait_slow(bar, parity, abort_flag, limit_ns);
}
template <int KC>
__device__ __forceinline__ bool grid_scores(const ChunkArgs& a, const GridPlan& p, unsigned char* sm, GridHead* head, uint32_t tmem, long long col0, uint32_t done_steps,
                            uint32_t done_tiles) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const unsigned long long limit_ns = a.wait_ns ? a.wait_ns : kGridWaitNs;
    const uint32_t full = smem_u32(&head->full[0]), empty = smem_u32(&head->empty[0]), ready = smem_u32(&head->rows[0]);
    const bool pair = p.row_bufs == 2;
    uint32_t step = done_steps;
    bool ok = true;
    if (warp == kClusterWarps) {
        if (lane == 0) {
            // (descriptors differ only in their start address, in units of 16 bytes: the low word)
            const uint64_t desc_hi = umma_desc(0) & 0xFFFFFFFF00000000ull;
            const uint32_t rows0 = (uint32_t)umma_desc(smem_u32(sm + p.off_rows)), cols0 = (uint32_t)umma_desc(smem_u32(sm));
            for (int mt = 0; ok && mt < p.mt; ++mt) {
                const uint32_t tile = done_tiles + mt, rb = pair ? tile & 1u : 0u, turn = pair ? tile >> 1 : tile;
                if (!bar_wait(ready + 8u * rb, turn & 1u, &head->abort_flag, limit_ns)) { ok = false; break; }
                for (int nb = 0; nb < p.nb; ++nb, ++step) {
                    const uint32_t buf = step & 1u;
                    if (!bar_wait(empty + 8u * buf, ((step >> 1) & 1u) ^ 1u, &head->abort_flag, limit_ns)) { ok = false; break; }
                    tc_fence_after();
                    const int width = p.cols - nb * kAccCols < kAccCols ? p.cols - nb * kAccCols : kAccCols;
                    const uint32_t idesc = umma_idesc(width), acc = tmem + buf * kAccCols, chunk = (uint32_t)width * 8u;
                    uint32_t lo_r = rows0 + rb * KC * 1024u, lo_c = cols0 + (uint32_t)nb * kAccCols * KC * 8u;
                    for (int kc = 0; kc < KC; ++kc, lo_r += 1024u, lo_c += chunk) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            if (kc * 4 + kk >= p.ks) break;
                            umma_f16(acc, desc_hi | (uint64_t)(lo_r + 2 * kk), desc_hi | (uint64_t)(lo_c + 2 * kk), idesc, (kc | kk) != 0 ? 1u : 0u);
                        }
                    }
                    umma_commit(full + 8u * buf);
                }
            }
        }
    } else {
        const int quad = warp & 3, part = warp >> 2;
        const float* inv = reinterpret_cast<const float*>(sm + p.off_inv);
        uint32_t* queue = reinterpret_cast<uint32_t*>(sm + p.off_queue);
        uint4 held[2 * KC];
        auto put = [&](int mt) {
            const uint32_t tile = done_tiles + mt, rb = pair ? tile & 1u : 0u;
            store_rows<KC>(sm + p.off_rows + (size_t)rb * KC * 16384, held);
            __syncwarp();
            if (lane == 0) mbar_arrive(ready + 8u * rb);
        };
        auto note = [&](int row, uint32_t col, float sc) {
            const unsigned int e = atomicAdd(&head->n_queue, 1u);
            if (e < (unsigned int)kGridQueue) { queue[3 * e] = (uint32_t)row; queue[3 * e + 1] = col; queue[3 * e + 2] = __float_as_uint(sc); }
            else {
                const unsigned int slot = atomicAdd(&a.rep_count[row], 1u);
                if (slot < (unsigned int)kChunkRepCap) a.rep[(size_t)row * kChunkRepCap + slot] = make_uint2(col, __float_as_uint(sc));
            }
        };
        fetch_rows<KC>(a, 0, held);
        float tau = __ldcg(a.tau + quad * 32 + lane), tau_next = tau;
        put(0);
        for (int mt = 0; ok && mt < p.mt; ++mt) {
            tau = tau_next;
            if (mt + 1 < p.mt) { fetch_rows<KC>(a, mt + 1, held); tau_next = __ldcg(a.tau + (mt + 1) * 128 + quad * 32 + lane); }
            const int n_res = mt * 128 + quad * 32 + lane;
            for (int nb = 0; nb < p.nb; ++nb, ++step) {
                const uint32_t buf = step & 1u;
                if (!__all_sync(0xffffffffu, bar_wait(full + 8u * buf, (step >> 1) & 1u, &head->abort_flag, limit_ns))) { ok = false; break; }
                tc_fence_after();
                // the next rows: their place was last read by the products of two tiles ago (of this tile where there is one place)
                if (mt + 1 < p.mt && nb == (pair ? 0 : p.nb - 1)) put(mt + 1);
                const int width = p.cols - nb * kAccCols < kAccCols ? p.cols - nb * kAccCols : kAccCols;
                // a quarter of the block's columns per warp, 32 at a time
                const int c_end = (part + 1) * 64 < width ? (part + 1) * 64 : width;
#pragma unroll 1
                for (int c0 = part * 64; c0 < c_end; c0 += 32) {
                    const float* w = inv + nb * kAccCols + c0;
                    uint32_t v[32];
                    tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + buf * kAccCols + c0, v);
                    const bool two = c0 + 16 < c_end;                 // (the last sixteen may be beyond the block's columns)
                    const float peak = __uint_as_float(max(peak_bits16(&v[0], w), two ? peak_bits16(&v[16], w + 16) : 0u));
                    if (!__any_sync(0xffffffffu, peak >= tau)) continue;
                    const unsigned int hits = hits16(&v[0], w, tau) | (two ? hits16(&v[16], w + 16, tau) << 16 : 0u);
                    const uint32_t first = (uint32_t)(col0 + nb * kAccCols + c0);
                    if (!__any_sync(0xffffffffu, (hits & (hits - 1u)) != 0u)) {
                        if (hits) note(n_res, first + __ffs(hits) - 1, peak);                  // (the only one is the largest)
                    } else
                        for (unsigned int any = __reduce_or_sync(0xffffffffu, hits); any; any &= any - 1u) {
                            const int i = __ffs(any) - 1;
                            const float sc = fabsf(tmem_ld1(tmem + ((uint32_t)(quad * 32) << 16) + buf * kAccCols + c0 + i)) * w[i];
                            if (hits >> i & 1u) note(n_res, first + i, sc);
                        }
                }
                __syncwarp();
                tc_fence_before();
                if (lane == 0) mbar_arrive(empty + 8u * buf);
            }
        }
    }
    __syncwarp();
    ok = __syncthreads_and(ok ? 1 : 0) != 0;
    const unsigned int n = head->n_queue < (unsigned int)kGridQueue ? head->n_queue : (unsigned int)kGridQueue;
    const uint32_t* queue = reinterpret_cast<const uint32_t*>(sm + p.off_queue);
    if (ok)
        for (unsigned int e = t; e < n; e += kGT + 32) {
            const uint32_t row = queue[3 * e];
            const unsigned int slot = atomicAdd(&a.rep_count[row], 1u);
            if (slot < (unsigned int)kChunkRepCap) a.rep[(size_t)row * kChunkRepCap + slot] = make_uint2(queue[3 * e + 1], queue[3 * e + 2]);
        }
    return ok;
}

// ---- books -------------------------------------------------------------------------------------------------
// The column that recovery rec picks next (kNoColumn: none left), the same in every thread of the team; scores_void: nothing was reported.
__device__ __forceinline__ uint32_t grid_decide(const ChunkArgs& a, ChunkBook& bk, const double* r, int rec, int j, const Team& tm, bool scores_void) {
    const double rn = bk.rn;
    if (!isfinite(rn)) return kNoColumn;
    if (rn == 0.0) {
        // a zero residual: all scores are equal, and the lowest free column it is (one of the first j + 1)
        const unsigned int who = __ballot_sync(0xffffffffu, tm.lane <= j && tm.lane < a.dc && !in_picks(bk.lam, j, (uint32_t)tm.lane));
        return who ? (uint32_t)(__ffs(who) - 1) : kNoColumn;
    }
    // (the first report of every thread is fetched with the count, whatever that will be)
    const uint2* rp = a.rep + (size_t)rec * kChunkRepCap;
    uint2 mine = make_uint2(kNoColumn, 0u);
    unsigned int count = 0u;
    if (!scores_void) { count = __ldcg(a.rep_count + rec); mine = __ldcg(rp + tm.t); }
    bool settled = count > 0u && count <= (unsigned int)kChunkRepCap;
    int nc = 0;
    if (settled) {
        if (tm.t == 0) bk.nc = 0;
        // (scores are not negative: ordered like their bits; columns of the support score rounding noise, but so does everything
        // else once a residual has fallen to that)
        unsigned int best = tm.t < (int)count && !in_picks(bk.lam, j, mine.x) ? mine.y : 0u;
        for (unsigned int e = tm.t + 32 * tm.warps; e < count; e += 32 * tm.warps) {
            const uint2 v = __ldcg(rp + e);
            if (v.y > best && !in_picks(bk.lam, j, v.x)) best = v.y;
        }
        best = __reduce_max_sync(0xffffffffu, best);
        if (tm.lane == 0) bk.bi[tm.warp] = best;
        tm.meet();
        for (int w = 0; w < tm.warps; ++w) best = max(best, bk.bi[w]);
        // (in the units of the row; twice the bound on what a score is off by, rounded up)
        const float smax = __uint_as_float(best);
        const float lo = smax - 2.00001f * (((float)kScreenMargin + (float)a.kp64 * (float)kScreenAccMargin) * bk.row_norm + (float)kScreenNormMargin * smax);
        // the window must stay above the report threshold, or a column inside it may not have been reported
        settled = best != 0u && lo > bk.row_tau * 1.001f;
        if (settled) {
            for (unsigned int e = tm.t; e < count; e += 32 * tm.warps) {
                const uint2 v = e == (unsigned int)tm.t ? mine : __ldcg(rp + e);
                if (__uint_as_float(v.y) < lo || in_picks(bk.lam, j, v.x)) continue;
                const int slot = atomicAdd(&bk.nc, 1);
                if (slot < kListed) bk.cidx[slot] = v.x;
            }
            tm.meet();
            nc = bk.nc;
            settled = nc <= kListed;
        }
    }
    if (!settled) {
        BestColumn b;
        scan_columns(a, bk, r, tm, j, 0, a.dc, b);
        tm.meet();
        return join_columns(bk, tm, b);
    }
    return nc == 1 ? bk.cidx[0] : best_candidate(a, bk, r, tm, nc);
}

// the residual of recovery rec as a row of the screened matrix, with its threshold and an empty list; a recovery that has ended
// screens nothing
__device__ __forceinline__ void grid_row(const ChunkArgs& a, ChunkBook& bk, const double* r, int rec, double rn, bool ended, const Team& tm) {
    const double sc = residual_scale(rn);
    const bool screened = !ended && rn > 0.0 && isfinite(rn);
    if (screened) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(a.rt + (size_t)rec * a.kp64);
        for (int i = tm.t; 2 * i < a.k; i += 32 * tm.warps)
            dst[i] = (uint32_t)half_rn_bits(r[2 * i] * sc) | (uint32_t)half_rn_bits(r[2 * i + 1] * sc) << 16;
    }
    if (tm.t == 0) {
        a.tau[rec] = screened ? (float)(a.z_rep * rn / sqrt((double)a.k) * sc) : __int_as_float(0x7f800000);
        a.rep_count[rec] = 0u;
        bk.rn = rn; bk.row_norm = (float)(rn * sc); bk.row_tau = (float)(a.z_rep * rn / sqrt((double)a.k) * sc);
    }
}

template <int KC>
__global__ void __launch_bounds__(kGT + 32, 1) k_chunk_grid(const __grid_constant__ ChunkArgs a, const __grid_constant__ GridPlan p) {
    extern __shared__ unsigned char raw[];
    const uint32_t pad = (1024u - (smem_u32(raw) & 1023u)) & 1023u;
    unsigned char* sm = raw + pad;
    cg::grid_group grid = cg::this_grid();
    GridHead* head = reinterpret_cast<GridHead*>(sm + p.off_head);
    const int t = threadIdx.x, warp = t >> 5;
    const long long col0 = (long long)blockIdx.x * p.cols;
    if (t == 0) {
        head->abort_flag = 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&head->full[b]), 1);
            mbar_init(smem_u32(&head->empty[b]), kClusterWarps);
            mbar_init(smem_u32(&head->rows[b]), kClusterWarps);
        }
        mbar_init(smem_u32(&head->drain), 1);
        head->n_queue = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
        if (blockIdx.x == 0) a.flags[1] = 0;                          // (nobody writes it before the first grid barrier)
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&head->tmem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    grid_columns(a, p, sm, col0);
    fence_async_smem();
    for (size_t e = t; e < (p.bytes - p.off_r) / 8; e += kGT + 32) reinterpret_cast<unsigned long long*>(sm + p.off_r)[e] = 0ull;      // (rows beyond k)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = head->tmem;
    Team tm;
    tm.warps = p.gw; tm.id = warp / p.gw; tm.warp = warp % p.gw; tm.lane = t & 31; tm.t = tm.warp * 32 + tm.lane;
    const int teams = kClusterWarps / p.gw, n_rec = warp < kClusterWarps ? 2 * a.c : 0;      // (the last warp keeps no books)
    // recovery blockIdx.x + own * (number of blocks): chunk rec / 2, moment rec & 1
    auto book_of = [&](int own) -> ChunkBook& { return *reinterpret_cast<ChunkBook*>(sm + p.off_book + (size_t)own * kClusterBook); };
    auto r_of = [&](int own) { return reinterpret_cast<double*>(sm + p.off_r) + (size_t)own * p.kq; };
    double* xs = reinterpret_cast<double*>(sm + p.off_x) + (size_t)(warp < kClusterWarps ? tm.id : 0) * p.kq;
    for (int own = tm.id; (int)blockIdx.x + own * (int)gridDim.x < n_rec; own += teams) {
        const int rec = (int)blockIdx.x + own * (int)gridDim.x, m = rec & 1;
        ChunkBook& bk = book_of(own);
        double* r = r_of(own);
        if (tm.t == 0) { bk.stopped = 0; bk.ref = a.table[rec >> 1]; }
        tm.meet();
        double part = 0.0;
        for (int i = tm.t; i < a.k; i += 32 * tm.warps) {
            const double v = bk.ref.r64[(size_t)m * a.k + i];
            r[i] = v;
            part = fma(v, v, part);
        }
        const double rn2 = team_sum(bk, part, tm, a.k);
        grid_row(a, bk, r, rec, sqrt(rn2), false, tm);
    }
    grid.sync();
    bool ok = true, scores_void = false;
    for (int j = 0; j < a.s; ++j) {
        if (!scores_void) {
            ok = grid_scores<KC>(a, p, sm, head, tmem, col0, (uint32_t)(j * p.mt * p.nb), (uint32_t)(j * p.mt));
            if (!ok && t == 0) atomicExch(&a.flags[1], 1);            // all blocks go on without scores
            grid.sync();
            if (t == 0) head->n_queue = 0u;                           // (read before that barrier, written again after the next)
            scores_void = *reinterpret_cast<volatile int*>(a.flags + 1) != 0;
        }
        for (int own = tm.id; (int)blockIdx.x + own * (int)gridDim.x < n_rec; own += teams) {
            const int rec = (int)blockIdx.x + own * (int)gridDim.x, m = rec & 1;
            ChunkBook& bk = book_of(own);
            if (bk.stopped) continue;
            const ChunkRef& ref = bk.ref;
            double* r = r_of(own);
            if (scores_void && tm.t == 0) atomicOr(&ref.cnt->status, (unsigned int)SGC_STATUS_TIMEOUT);
            uint32_t col = grid_decide(a, bk, r, rec, j, tm, scores_void);
            double gamma = 0.0, aj = 0.0, rn2 = 0.0;
            if (col == kNoColumn) { if (tm.t == 0) { ref.cnt->stopped[m] = 1; ref.cnt->done[m] = j; } }
            else if (!extend_basis<false>(a, bk, ref, r, ref.qb + (size_t)m * a.s * a.k, a.k, xs, m, j, col, tm, &gamma, &aj, &rn2)) col = kNoColumn;
            if (j + 1 < a.s) grid_row(a, bk, r, rec, sqrt(rn2), col == kNoColumn, tm);
            tm.meet();
            if (tm.warp == tm.warps - 1) {
                if (col == kNoColumn) { if (tm.lane == 0) bk.stopped = 1; }
                else record_pick(a, bk, ref, m, j, col, gamma, aj, rn2, tm.lane);
            }
            tm.meet();
        }
        if (j + 1 < a.s) {
            if (scores_void) __syncthreads();
            else grid.sync();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (!ok) {
        // Nothing is issued any more; the matrix operations in flight are waited for (a commit arrives once all of them have completed).
        if (t == kGT) {
            umma_commit(smem_u32(&head->drain));
            const unsigned long long t0 = global_ns();
            while (!mbar_try(smem_u32(&head->drain), 0u) && global_ns() - t0 < 2000000ull) __nanosleep(1000);
        }
        __syncthreads();
    }
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

}  // namespace

template <int KC>
static cudaError_t grid_opt_in(bool* fits) {
    int blocks = 0;
    cudaError_t e = cudaFuncSetAttribute(k_chunk_grid<KC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGridSmem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_chunk_grid<KC>, kGT + 32, kGridSmem);
    *fits = e == cudaSuccess && blocks >= 1;
    return e;
}

cudaError_t chunk_grid_configure(int device, int kc, bool* fits) {
    int coop = 0;
    cudaError_t e = kc == 1 ? grid_opt_in<1>(fits) : kc == 2 ? grid_opt_in<2>(fits) : kc == 3 ? grid_opt_in<3>(fits) : grid_opt_in<4>(fits);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device);
    *fits = *fits && e == cudaSuccess && coop != 0;
    return e;
}

cudaError_t launch_chunk_grid(const ChunkArgs& a, const GridPlan& p, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.blocks); cfg.blockDim = dim3(kGT + 32); cfg.dynamicSmemBytes = p.bytes + 1024; cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    switch (p.kc) {
        case 1: return cudaLaunchKernelEx(&cfg, k_chunk_grid<1>, a, p);
        case 2: return cudaLaunchKernelEx(&cfg, k_chunk_grid<2>, a, p);
        case 3: return cudaLaunchKernelEx(&cfg, k_chunk_grid<3>, a, p);
        default: return cudaLaunchKernelEx(&cfg, k_chunk_grid<4>, a, p);
    }
}

}  // namespace sgc
