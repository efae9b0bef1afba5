// The recoveries of the batched chunk path (sgc_chunked.cu) in one launch: all iterations of Algorithm 3 inside thread-block
// clusters, for chunks whose matrix A (k_c x d/c) fits the shared memory of a cluster.
//
// Every cluster holds all columns of A, generated once, as operands of mma.m16n8k16 (its blocks split the columns) and makes the
// picks of some chunks.  An iteration is
//     correlate: every block scores its columns against the residuals of all the cluster's recoveries and sends its best two per
//                recovery to the block that keeps that recovery's books
//     books:     that block decides in fp64, updates q and r (orthogonal form, see sgc_omp.cu) and sends the new residual, as an
//                operand, to every block
// The recoveries of different clusters have nothing to say to one another, so nothing is grid-wide, and nothing but the records
// leaves the SMs.  What is sent goes by st.async, which counts its bytes on a barrier in the receiver's shared memory: a
// block waits for what it needs and for nothing else (a cluster-wide barrier of 16 blocks takes 0.6 us, and an iteration needs two).
// Latency bounds it: 5.6 us per pick for one vector of 4096 (k = 256; three cluster barriers and L2 trips of the lock-step kernel: 11), 9.0 us for 10 recoveries per
// cluster of 8 blocks over 2048 columns (k = 217; two launches: 17); scoring takes a quarter to a third, bound by shared-memory reads of the operands.
// Every wait is bounded; on expiry the block marks its chunks, leaves the loops, gives what is still on its way time to land, meets the
// others, and makes the picks that its recoveries lack by itself, going through all columns in fp64.
#include <mutex>

#include <cooperative_groups.h>

#include "sgc_chunk_book.cuh"
#include "sgc_tcgen05.cuh"

namespace cg = cooperative_groups;

namespace sgc {
namespace {

constexpr int kCT = 32 * kClusterWarps;
constexpr unsigned long long kClusterWaitNs = 2000000000ull;      // bound of every wait, unless the caller sets another
constexpr float kWindow = 2e-3f;                      // relative: what comes this close to the best score is decided in fp64

// the first bytes of the dynamic shared memory
struct ClusterHead {
    unsigned long long bar_cand, bar_res;             // candidates of this block's recoveries; residuals of all of the cluster's
    int abort_flag;
};
static_assert(sizeof(ClusterHead) <= kClusterHead, "barriers");

__device__ __forceinline__ uint32_t peer_at(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void send_16(uint32_t dst, uint32_t bar, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(dst), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
// ---- the block's columns as operands, with 1 / ||Z_i|| (0 beyond the chunk) ----------------------------------
__device__ __forceinline__ void generate_columns(const ChunkArgs& a, const ChunkPlan& p, unsigned char* cols, unsigned char* norms, long long col0) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    uint4* zt = reinterpret_cast<uint4*>(cols);
    float* inv = reinterpret_cast<float*>(norms);
    for (int tile = warp; tile < p.tiles; tile += kClusterWarps) {
        const long long first = col0 + tile * 16;
        const ColKey key = column_key(a.seed_lo, a.seed_hi, (uint32_t)(first + (lane & 15)));
        const uint32_t ck0 = __shfl_sync(0xffffffffu, key.ck, g), mk0 = __shfl_sync(0xffffffffu, key.mk, g);
        const uint32_t ck1 = __shfl_sync(0xffffffffu, key.ck, g + 8), mk1 = __shfl_sync(0xffffffffu, key.mk, g + 8);
        float n0 = 0.0f, n1 = 0.0f;
        for (int kb = 0; kb < p.kb; ++kb) {
            const uint32_t h0 = ck0 + (uint32_t)(kb * 8 + q) * mk0, h1 = ck1 + (uint32_t)(kb * 8 + q) * mk1;
            uint32_t z[4] = {z_pair_from_word(h0), z_pair_from_word(h1), z_pair_from_word(h0 + 4u * mk0), z_pair_from_word(h1 + 4u * mk1)};
#pragma unroll
            for (int e = 0; e < 4; ++e) {                              // rows beyond k do not count
                const int row = kb * 16 + 2 * q + (e & 2 ? 8 : 0);
                if (row >= a.k) z[e] = 0u;
                else if (row + 1 >= a.k) z[e] &= 0xFFFFu;
                const float2 f = half2_bits_to_float2(z[e]);
                float& n = (e & 1) ? n1 : n0;
                n = __fmaf_rn(f.x, f.x, n); n = __fmaf_rn(f.y, f.y, n);
            }
            zt[(size_t)(tile * p.kb + kb) * 32 + lane] = make_uint4(z[0], z[1], z[2], z[3]);
        }
        n0 += __shfl_xor_sync(0xffffffffu, n0, 1); n0 += __shfl_xor_sync(0xffffffffu, n0, 2);
        n1 += __shfl_xor_sync(0xffffffffu, n1, 1); n1 += __shfl_xor_sync(0xffffffffu, n1, 2);
        if (q == 0) {
            inv[tile * 16 + g] = first + g < a.dc && n0 > 0.0f ? 1.0f / sqrtf(n0) : 0.0f;
            inv[tile * 16 + g + 8] = first + g + 8 < a.dc && n1 > 0.0f ? 1.0f / sqrtf(n1) : 0.0f;
        }
    }
}

// ---- correlate ---------------------------------------------------------------------------------------------
// A warp's column tiles (TT at a time) against NB tiles of four recoveries, each residual as value and remainder in binary16 (columns
// 2 i and 2 i + 1 of the B operand), sums in fp32.  Scores are compared as keys: the score's bits with the lowest ten replaced by the
// column's place in the warp's share (relative error 2^-13, an eighth of the window that the books decide in fp64; the lowest column
// has the largest code), so that the best two follow from integer minima and maxima.
// A residual as an operand: [recovery][16-row block][q] of 16 bytes, the rows 2q, 2q + 1, 2q + 8, 2q + 9 as values and then as
// remainders; recoveries lie an odd number of 64 bytes apart, so that a warp's read meets every bank once.
template <int NB, int TT>
__device__ __forceinline__ void correlate_tiles(const ChunkPlan& p, const unsigned char* sm, float4* tops, long long col0, int slot, int nt0, int nt1,
                                                int n_rec) {
    constexpr int AC = NB * TT <= 2 ? 2 : 1;                          // few products: two chains each
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const uint4* zt = reinterpret_cast<const uint4*>(sm + kClusterHead) + lane;
    const float* inv = reinterpret_cast<const float*>(sm + p.off_inv);
    const unsigned char* rf = sm + p.off_frag + (size_t)(4 * nt0 + (g >> 1)) * p.rec_bytes + q * 16 + (g & 1) * 8;
    unsigned int k1[NB], k2[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) k1[i] = k2[i] = 0u;
    unsigned int code = 1023u - (unsigned int)g;
    for (int t0 = slot; t0 < p.tiles; t0 += TT * p.slots, code -= 16u * TT) {
        float acc[AC][TT][NB][4];
#pragma unroll
        for (int c = 0; c < AC; ++c)
#pragma unroll
            for (int u = 0; u < TT; ++u)
#pragma unroll
                for (int i = 0; i < NB; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[c][u][i][e] = 0.0f;
        const uint4* z[TT];
#pragma unroll
        for (int u = 0; u < TT; ++u) {
            const int tile = t0 + u * p.slots;
            z[u] = zt + (size_t)(tile < p.tiles ? tile : t0) * p.kb * 32;
        }
        auto step = [&](int kb, int c) {
            uint4 x[TT];
#pragma unroll
            for (int u = 0; u < TT; ++u) x[u] = z[u][kb * 32];
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const uint2 b = *reinterpret_cast<const uint2*>(rf + (size_t)(4 * i) * p.rec_bytes + kb * 64);
#pragma unroll
                for (int u = 0; u < TT; ++u) mma_16816(acc[c][u][i], x[u], b.x, b.y);
            }
        };
        int kb = 0;
#pragma unroll 2
        for (; kb + 1 < p.kb; kb += 2) { step(kb, 0); step(kb + 1, AC - 1); }
        if (kb < p.kb) step(kb, 0);
#pragma unroll
        for (int u = 0; u < TT; ++u) {
            const int tile = t0 + u * p.slots;
            if (u > 0 && tile >= p.tiles) break;
            const float v0 = inv[tile * 16 + g], v1 = inv[tile * 16 + g + 8];
            const unsigned int c0 = v0 > 0.0f ? code - 16u * u : 0u, c1 = v1 > 0.0f ? code - 16u * u - 8u : 0u;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                float d0 = acc[0][u][i][0] + acc[0][u][i][1], d1 = acc[0][u][i][2] + acc[0][u][i][3];
                if (AC > 1) { d0 += acc[AC - 1][u][i][0] + acc[AC - 1][u][i][1]; d1 += acc[AC - 1][u][i][2] + acc[AC - 1][u][i][3]; }
                const unsigned int x0 = (__float_as_uint(fabsf(d0) * v0) & ~1023u) | c0;
                const unsigned int x1 = (__float_as_uint(fabsf(d1) * v1) & ~1023u) | c1;
                k2[i] = max(k2[i], min(k1[i], x0)); k1[i] = max(k1[i], x0);
                k2[i] = max(k2[i], min(k1[i], x1)); k1[i] = max(k1[i], x1);
            }
        }
    }
    // the eight lanes of a recovery (same q) join their best two; k3: the largest key that may be left out (a lane has not kept its
    // third, which its second bounds)
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        unsigned int k3 = k2[i];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            const unsigned int o1 = __shfl_xor_sync(0xffffffffu, k1[i], o), o2 = __shfl_xor_sync(0xffffffffu, k2[i], o);
            const unsigned int o3 = __shfl_xor_sync(0xffffffffu, k3, o);
            k3 = max(max(k3, o3), max(min(k2[i], o1), min(k1[i], o2)));
            k2[i] = max(max(k2[i], o2), min(k1[i], o1));
            k1[i] = max(k1[i], o1);
        }
        const int rec = 4 * (nt0 + i) + q;
        if (g == 0 && nt0 + i < nt1 && rec < n_rec) {
            auto column = [&](unsigned int key) -> uint32_t {
                const int at = 1023 - (int)(key & 1023u);
                return (uint32_t)(col0 + (slot + p.slots * (at >> 4)) * 16 + (at & 15));
            };
            const float s1 = __uint_as_float(k1[i] & ~1023u), s2 = __uint_as_float(k2[i] & ~1023u), s3 = __uint_as_float(k3 & ~1023u);
            const uint32_t mark = (k3 & 1023u) && s3 > 0.0f && s3 >= s1 * (1.0f - kKeyWindow) ? kThirdMark : 0u;
            const uint32_t i1 = k1[i] & 1023u ? column(k1[i]) | mark : kNoColumn, i2 = k2[i] & 1023u ? column(k2[i]) : kNoColumn;
            tops[rec * p.slots + slot] = make_float4(s1, __uint_as_float(i1), s2, __uint_as_float(i2));
        }
    }
}

// scores of the block's columns; its best two per recovery go to the block that keeps the recovery's books.  A first candidate's mark: the
// block may hold more columns as good as these.
__device__ __forceinline__ void correlate_columns(const ChunkPlan& p, unsigned char* sm, int rank, long long col0, int n_rec) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4* tops = reinterpret_cast<float4*>(sm + p.off_top);
    {
        const int slot = warp & (p.slots - 1), part = warp >> p.slots_log, share = kClusterWarps >> p.slots_log;
        const int nt = (n_rec + 3) >> 2, per = (nt + share - 1) >> (4 - p.slots_log);
        const int n0 = part * per, n1 = n0 + per < nt ? n0 + per : nt;
        for (int n = n0; n < n1; n += 4) {
            if (p.tiles <= p.slots) {
                if (n1 - n >= 4) correlate_tiles<4, 1>(p, sm, tops, col0, slot, n, n1, n_rec);
                else if (n1 - n == 3) correlate_tiles<3, 1>(p, sm, tops, col0, slot, n, n1, n_rec);
                else if (n1 - n == 2) correlate_tiles<2, 1>(p, sm, tops, col0, slot, n, n1, n_rec);
                else correlate_tiles<1, 1>(p, sm, tops, col0, slot, n, n1, n_rec);
            }
            else if (n1 - n >= 4) correlate_tiles<4, 2>(p, sm, tops, col0, slot, n, n1, n_rec);
            else if (n1 - n == 3) correlate_tiles<3, 2>(p, sm, tops, col0, slot, n, n1, n_rec);
            else if (n1 - n == 2) correlate_tiles<2, 2>(p, sm, tops, col0, slot, n, n1, n_rec);
            else correlate_tiles<1, 2>(p, sm, tops, col0, slot, n, n1, n_rec);
        }
    }
    __syncthreads();
    // half a warp per recovery joins what the warps found
    const uint32_t ents = smem_u32(sm + p.off_ent), bar = smem_u32(&reinterpret_cast<ClusterHead*>(sm)->bar_cand);
    for (int r0 = 2 * warp; r0 < n_rec; r0 += 2 * kClusterWarps) {
        const int rec = r0 + (lane >> 4), e = lane & 15;
        const bool real = rec < n_rec && e < p.slots;
        const float4 f = real ? tops[rec * p.slots + e] : make_float4(-1.0f, __uint_as_float(kNoColumn), -1.0f, __uint_as_float(kNoColumn));
        const uint32_t w1 = __float_as_uint(f.y);
        uint32_t i1 = w1, i2 = __float_as_uint(f.w);
        float s1 = w1 != kNoColumn ? f.x : -1.0f, s2 = i2 != kNoColumn ? f.z : -1.0f, s3 = -1.0f;
        if (w1 != kNoColumn && (w1 & kThirdMark)) { s3 = s1; i1 = w1 & ~kThirdMark; }      // (s3: bound of what is left out)
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const float t1 = __shfl_xor_sync(0xffffffffu, s1, o), t2 = __shfl_xor_sync(0xffffffffu, s2, o), t3 = __shfl_xor_sync(0xffffffffu, s3, o);
            const uint32_t c1 = __shfl_xor_sync(0xffffffffu, i1, o), c2 = __shfl_xor_sync(0xffffffffu, i2, o);
            const bool first = s1 > t1 || (s1 == t1 && i1 <= c1);
            const float lo = first ? t1 : s1, lo2 = first ? s2 : t2, rest = first ? t2 : s2;      // loser's best; winner's second; loser's second
            const uint32_t lo_i = first ? c1 : i1, lo2_i = first ? i2 : c2;
            const bool second = lo > lo2 || (lo == lo2 && lo_i <= lo2_i);
            s3 = fmaxf(fmaxf(s3, t3), second ? fmaxf(lo2, rest) : lo);
            s1 = first ? s1 : t1; i1 = first ? i1 : c1;
            s2 = second ? lo : lo2; i2 = second ? lo_i : lo2_i;
        }
        if (e == 0 && rec < n_rec) {
            if (i1 != kNoColumn && s3 > 0.0f && s3 >= s1 * (1.0f - kWindow)) i1 |= kThirdMark;
            const int owner = rec & (p.cl - 1), own = rec >> p.cl_log;
            send_16(peer_at(ents, owner) + (uint32_t)(own * p.cl + rank) * 16u, peer_at(bar, owner), __float_as_uint(s1), i1, __float_as_uint(s2), i2);
        }
    }
}

// ---- books -------------------------------------------------------------------------------------------------
// What hardly any pick needs: near-ties, columns of the support among the best, a zero residual.  Returns the column to pick
// (kNoColumn: none left), the same in every thread of the team.  j: picks made so far.
__device__ __noinline__ uint32_t decide(const ChunkArgs& a, const ChunkPlan& p, ChunkBook& bk, const float4* ents, const double* r, const Team& tm, int j) {
    const int n_ent = p.cl, lane = tm.lane;
    tm.meet();
    if (tm.warp == 0) {
        const float4 f = lane < n_ent ? ents[lane] : make_float4(-1.0f, __uint_as_float(kNoColumn), -1.0f, __uint_as_float(kNoColumn));
        const uint32_t w1 = __float_as_uint(f.y), i1 = w1 & ~kThirdMark, i2 = __float_as_uint(f.w);
        const bool v1 = w1 != kNoColumn, v2 = i2 != kNoColumn, mark = v1 && w1 != i1;
        const bool t1 = v1 && in_picks(bk.lam, j, i1), t2 = v2 && in_picks(bk.lam, j, i2);
        const unsigned int best = __reduce_max_sync(0xffffffffu, max(v1 && !t1 ? order_key(f.x) : 0u, v2 && !t2 ? order_key(f.z) : 0u));
        const float mx = order_score(best), thr = mx - kWindow * fabsf(mx);
        int n = 0;
        unsigned int redo = 0u;
        if (mx == 0.0f) {
            // a zero residual: all scores are equal, and the lowest free column it is (one of the first j + 1)
            const unsigned int who = __ballot_sync(0xffffffffu, lane <= j && lane < a.dc && !in_picks(bk.lam, j, (uint32_t)lane));
            if (who != 0u) { n = 1; if (lane == 0) bk.cidx[0] = (uint32_t)(__ffs(who) - 1); }
        } else {
            const bool in1 = v1 && !t1 && f.x >= thr && mx > 0.0f, in2 = v2 && !t2 && f.z >= thr && mx > 0.0f;
            const unsigned int b1 = __ballot_sync(0xffffffffu, in1), b2 = __ballot_sync(0xffffffffu, in2), below = (1u << lane) - 1u;
            const int n1 = __popc(b1), at1 = __popc(b1 & below), at2 = n1 + __popc(b2 & below);
            n = n1 + __popc(b2);
            if (in1 && at1 < kListed) bk.cidx[at1] = i1;
            if (in2 && at2 < kListed) bk.cidx[at2] = i2;
            // the block may hold more: a mark, or columns of the support in the places of its best
            redo = __ballot_sync(0xffffffffu, (mark && f.x >= thr) || ((t1 || t2) && f.z >= 0.0f && f.z >= thr));
            if (n > kListed) { n = 0; redo = (1u << n_ent) - 1u; }    // too many to list: all columns once more
        }
        if (lane == 0) { bk.nc = n; bk.redo = redo; }
    }
    tm.meet();
    int nc = bk.nc;
    if (bk.redo != 0u) {
        // the best free one of those blocks' columns joins the candidates
        BestColumn b;
        for (unsigned int left = bk.redo; left; left &= left - 1u) {
            const long long first = (long long)(__ffs(left) - 1) * p.cols;
            scan_columns(a, bk, r, tm, j, first, first + p.cols, b);
        }
        const uint32_t bi = join_columns(bk, tm, b);
        if (bi != kNoColumn) { if (tm.t == 0) bk.cidx[nc] = bi; ++nc; }
        tm.meet();
    }
    return best_candidate(a, bk, r, tm, nc);
}

// power of two that brings a residual of squared norm rn2 to [2^9, 2^10)
__device__ __forceinline__ double operand_scale(double rn2) {
    const int e = (int)((unsigned long long)__double_as_longlong(rn2) >> 52);          // (a square is not negative)
    if (e < 64 || e >= 2047) return 0.125;
    return __longlong_as_double((long long)(1023 + 9 - ((e - 1023) >> 1)) << 52);
}

// the residual as value and remainder into every block's operands: thread = 16 bytes for some of the blocks.  rec: its place in the cluster
__device__ __forceinline__ void send_residual(const ChunkPlan& p, unsigned char* sm, int rec, const double* r, double rn2, const Team& tm) {
    const double scale = operand_scale(rn2);
    const uint32_t frag = smem_u32(sm + p.off_frag) + (uint32_t)(rec * p.rec_bytes), bar = smem_u32(&reinterpret_cast<ClusterHead*>(sm)->bar_res);
    const int quads = 4 * p.kb, pad = 1 << p.quads_log;
    // (quads, rounded up to a power of two) x blocks
    for (int i = tm.t; i < pad * p.cl; i += 32 * tm.warps) {
        const int at = i & (pad - 1), b = i >> p.quads_log;
        if (at >= quads) continue;
        const double* v = r + (at >> 2) * 16 + (at & 3) * 2;
        const double2 lo = *reinterpret_cast<const double2*>(v), hi = *reinterpret_cast<const double2*>(v + 8);
        const float x0 = (float)(lo.x * scale), x1 = (float)(lo.y * scale), x2 = (float)(hi.x * scale), x3 = (float)(hi.y * scale);
        const __half2 h0 = __floats2half2_rn(x0, x1), h1 = __floats2half2_rn(x2, x3);
        const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
        const __half2 l0 = __floats2half2_rn(x0 - f0.x, x1 - f0.y), l1 = __floats2half2_rn(x2 - f1.x, x3 - f1.y);
        send_16(peer_at(frag, b) + (uint32_t)at * 16u, peer_at(bar, b), *reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1),
                *reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
    }
}

// pick j of recovery m of a chunk.  SHARED: its q_l are in shared memory, p.kq rows apart and zero beyond k (else in the chunk's
// records, k apart)
template <bool SHARED>
__device__ __forceinline__ void make_pick(const ChunkArgs& a, const ChunkPlan& p, unsigned char* sm, int rec, int m, int own, int j, const Team& tm) {
    ChunkBook& bk = *reinterpret_cast<ChunkBook*>(sm + p.off_book + (size_t)own * kClusterBook);
    const ChunkRef& ref = bk.ref;
    double* xs = reinterpret_cast<double*>(sm + p.off_x) + (size_t)tm.id * p.kq;       // the column
    const int lane = tm.lane, s = a.s, k = a.k;
    double* r = reinterpret_cast<double*>(sm + p.off_r) + (size_t)own * p.kq;
    double* qs = SHARED ? reinterpret_cast<double*>(sm + p.off_q) + (size_t)own * s * p.kq : ref.qb + (size_t)m * s * k;
    const int qstride = SHARED ? p.kq : k;
    const float4* ents = reinterpret_cast<const float4*>(sm + p.off_ent) + (size_t)own * p.cl;
    uint32_t col = kNoColumn;
    if (!bk.stopped) {
        // the usual case, one candidate and nothing close: every warp finds it by itself
        const float4 f = lane < p.cl ? ents[lane] : make_float4(-1.0f, __uint_as_float(kNoColumn), -1.0f, __uint_as_float(kNoColumn));
        const uint32_t w1 = __float_as_uint(f.y);
        const uint32_t held = lane < j ? bk.lam[lane] : kNoColumn;
        const unsigned int best = __reduce_max_sync(0xffffffffu, w1 != kNoColumn ? order_key(f.x) : 0u);
        const float mx = order_score(best), thr = mx - kWindow * fabsf(mx);
        const bool in = w1 != kNoColumn && f.x >= thr;
        const unsigned int who = __ballot_sync(0xffffffffu, in);
        const bool close = __any_sync(0xffffffffu, in && ((w1 & kThirdMark) || f.z >= thr));
        col = __shfl_sync(0xffffffffu, w1, who ? __ffs(who) - 1 : 0);
        const bool again = __any_sync(0xffffffffu, held == col);
        if (__popc(who) != 1 || close || again || !(mx > 0.0f)) col = decide(a, p, bk, ents, r, tm, j);
        if (col == kNoColumn && tm.t == 0) { ref.cnt->stopped[m] = 1; ref.cnt->done[m] = j; }      // no column left to pick (d/c = iterations made)
    }
    double rn2 = 1.0, gamma = 0.0, aj = 0.0;
    if (col != kNoColumn) {
        if (!extend_basis<SHARED>(a, bk, ref, r, qs, qstride, xs, m, j, col, tm, &gamma, &aj, &rn2)) col = kNoColumn;
    }
    // (a recovery that has ended still sends what the others wait for)
    if (j + 1 < s) send_residual(p, sm, rec, r, rn2, tm);
    // the records, while the others read what was sent
    if (tm.warp == tm.warps - 1) {
        if (col == kNoColumn) { if (lane == 0) bk.stopped = 1; }
        else record_pick(a, bk, ref, m, j, col, gamma, aj, rn2, lane);
    }
}

// books of a recovery as its chunk's first kernel left it; returns the squared norm of its residual, to all of the team
__device__ __forceinline__ double open_books(const ChunkArgs& a, ChunkBook& bk, const ChunkRef& ref, double* r, int m, const Team& tm) {
    double part = 0.0;
    for (int i = tm.t; i < a.k; i += 32 * tm.warps) {
        const double v = ref.r64[(size_t)m * a.k + i];
        r[i] = v;
        part = fma(v, v, part);
    }
    if (tm.t == 0) { bk.stopped = 0; bk.ref = ref; }
    return team_sum(bk, part, tm, a.k);
}

// A wait has expired at pick j0 of the batch that starts with chunk c0: this block goes on without the others.  Its recoveries go through all
// columns in fp64, which decides as the kernel does (of equal scores the lowest column), from pick j0 on, and those of the batches behind it
// from their first.  (Rare: one copy of the code for vectors in shared and in global memory.)
__device__ __noinline__ void finish_alone(const ChunkArgs& a, const ChunkPlan& p, unsigned char* sm, int rank, int c0, int last, int j0, const Team tm) {
    const int teams = kClusterWarps / p.gw;
    double* xs = reinterpret_cast<double*>(sm + p.off_x) + (size_t)tm.id * p.kq;
    for (bool open = true; c0 < last; c0 += p.batch, j0 = 0, open = false) {
        const int n_rec = 2 * (last - c0 < p.batch ? last - c0 : p.batch);
        for (int own = tm.id; own * p.cl + rank < n_rec; own += teams) {
            const int rec = own * p.cl + rank, m = rec & 1;
            ChunkBook& bk = *reinterpret_cast<ChunkBook*>(sm + p.off_book + (size_t)own * kClusterBook);
            double* r = reinterpret_cast<double*>(sm + p.off_r) + (size_t)own * p.kq;
            if (!open) open_books(a, bk, chunk_ref(a, c0 + (rec >> 1)), r, m, tm);
            const ChunkRef& ref = bk.ref;
            double* qs = p.q_shared ? reinterpret_cast<double*>(sm + p.off_q) + (size_t)own * a.s * p.kq : ref.qb + (size_t)m * a.s * a.k;
            const int qstride = p.q_shared ? p.kq : a.k;
            for (int j = j0; j < a.s && !bk.stopped; ++j) {
                BestColumn b;
                scan_columns(a, bk, r, tm, j, 0, a.dc, b);
                uint32_t col = join_columns(bk, tm, b);
                double gamma = 0.0, aj = 0.0, rn2 = 0.0;
                if (col == kNoColumn) { if (tm.t == 0) { ref.cnt->stopped[m] = 1; ref.cnt->done[m] = j; } }
                else if (!extend_basis<false>(a, bk, ref, r, qs, qstride, xs, m, j, col, tm, &gamma, &aj, &rn2)) col = kNoColumn;
                tm.meet();
                if (tm.warp == tm.warps - 1) {
                    if (col == kNoColumn) { if (tm.lane == 0) bk.stopped = 1; }
                    else record_pick(a, bk, ref, m, j, col, gamma, aj, rn2, tm.lane);
                }
                tm.meet();
            }
        }
    }
}

// ---- the kernel --------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kCT, 1) k_chunk_cluster(const __grid_constant__ ChunkArgs a, const __grid_constant__ ChunkPlan p) {
    extern __shared__ __align__(16) unsigned char sm[];
    cg::cluster_group cluster = cg::this_cluster();
    ClusterHead* head = reinterpret_cast<ClusterHead*>(sm);
    const int rank = (int)blockIdx.x & (p.cl - 1), cid = (int)blockIdx.x >> p.cl_log;
    const int t = threadIdx.x, warp = t >> 5;
    const long long col0 = (long long)rank * p.cols;
    const uint32_t bar_cand = smem_u32(&head->bar_cand), bar_res = smem_u32(&head->bar_res);
    if (t == 0) {
        head->abort_flag = 0;
        mbar_init(bar_cand, 1); mbar_init(bar_res, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    generate_columns(a, p, sm + kClusterHead, sm + p.off_inv, col0);   // (needs nothing of the kernel before)
    for (size_t e = t; e < (p.off_top - p.off_frag) / 4; e += kCT) reinterpret_cast<uint32_t*>(sm + p.off_frag)[e] = 0u;
    for (size_t e = t; e < (p.bytes - p.off_r) / 4; e += kCT) reinterpret_cast<uint32_t*>(sm + p.off_r)[e] = 0u;      // (rows beyond k)
    after_previous_kernel(1);
    cluster.sync();
    Team tm;
    tm.warps = p.gw; tm.id = warp / p.gw; tm.warp = warp % p.gw; tm.lane = t & 31; tm.t = tm.warp * 32 + tm.lane;
    const int teams = kClusterWarps / p.gw;
    const int first = cid * p.per_cluster, last = first + p.per_cluster < a.c ? first + p.per_cluster : a.c;
    const unsigned long long limit_ns = a.wait_ns ? a.wait_ns : kClusterWaitNs;
    uint32_t ph_cand = 0, ph_res = 0;
    bool ok = true;
    int c_left = first, j_left = 0;                                   // where a wait expired: first chunk of the batch, picks made
    for (int c0 = first; ok && c0 < last; c0 += p.batch) {
        // recovery rec of the batch: chunk c0 + rec / 2, moment rec & 1; kept by block rec % cl as its rec / cl-th
        const int n_rec = 2 * (last - c0 < p.batch ? last - c0 : p.batch);
        const int n_own = rank < n_rec ? ((n_rec - 1 - rank) >> p.cl_log) + 1 : 0;
        const uint32_t res_bytes = (uint32_t)(n_rec * p.kb * 64), cand_bytes = (uint32_t)(n_own * p.cl * 16);
        if (t == 0) mbar_arrive_expect_tx(bar_res, res_bytes);
        // (the last pick of a batch sends nothing that anybody waits for: a team's last warp may still be writing its records, for which it
        // reads the books that are set up anew here, and a recovery that has just ended may still have to say so)
        if (c0 > first) __syncthreads();
        for (int own = tm.id; own < n_own; own += teams) {
            const int rec = own * p.cl + rank, m = rec & 1;
            const ChunkRef& ref = chunk_ref(a, c0 + (rec >> 1));
            ChunkBook& bk = *reinterpret_cast<ChunkBook*>(sm + p.off_book + (size_t)own * kClusterBook);
            double* r = reinterpret_cast<double*>(sm + p.off_r) + (size_t)own * p.kq;
            send_residual(p, sm, rec, r, open_books(a, bk, ref, r, m, tm), tm);
        }
        int j = 0;
        for (; j < a.s; ++j) {
            if (t == 0 && n_own > 0) mbar_arrive_expect_tx(bar_cand, cand_bytes);
            if (!(ok = block_wait(bar_res, ph_res & 1u, &head->abort_flag, limit_ns))) break;
            ++ph_res;
            if (t == 0 && j + 1 < a.s) mbar_arrive_expect_tx(bar_res, res_bytes);
            correlate_columns(p, sm, rank, col0, n_rec);
            if (n_own == 0) continue;
            if (!(ok = block_wait(bar_cand, ph_cand & 1u, &head->abort_flag, limit_ns))) break;
            ++ph_cand;
            for (int own = tm.id; own < n_own; own += teams) {
                const int rec = own * p.cl + rank;
                if (p.q_shared) make_pick<true>(a, p, sm, rec, rec & 1, own, j, tm);
                else make_pick<false>(a, p, sm, rec, rec & 1, own, j, tm);
            }
        }
        if (!ok) {
            c_left = c0; j_left = j;
            for (int ch = c0 + t; ch < last; ch += kCT) atomicOr(&chunk_ref(a, ch).cnt->status, (unsigned int)SGC_STATUS_TIMEOUT);
        }
    }
    // after an expired wait: what was sent, by this block and to it, may still be on its way; it lands in microseconds
    auto settle = [] { const unsigned long long t0 = global_ns(); while (global_ns() - t0 < 200000ull) __nanosleep(1000); };
    if (!ok) settle();
    cluster.sync();
    if (!ok) {
        settle();
        finish_alone(a, p, sm, rank, c_left, last, j_left, tm);
    }
}

struct ClusterLaunch {
    cudaLaunchConfig_t cfg; cudaLaunchAttribute attr[2];
    ClusterLaunch(int cl, int clusters, size_t smem, cudaStream_t stream) : cfg{} {
        cfg.gridDim = dim3((unsigned)(cl * clusters)); cfg.blockDim = dim3(kCT); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cl; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
    }
};

}  // namespace

// How many clusters of each shape the device holds at a time with all the shared memory that a plan may ask for: a property of the
// device, asked once for each.
cudaError_t chunk_cluster_configure(int device, int (&resident)[kChunkShapes]) {
    struct Resident { int n[kChunkShapes]; bool known; };
    constexpr int kDevices = 64;
    static std::mutex lock;
    static Resident table[kDevices];
    const bool listed = device >= 0 && device < kDevices;
    Resident r = {};
    if (listed) { std::lock_guard<std::mutex> hold(lock); r = table[device]; }
    if (!r.known) {
        cudaError_t e = cudaFuncSetAttribute(k_chunk_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmem);
        if (e != cudaSuccess) return e;
        const bool wide = cudaFuncSetAttribute(k_chunk_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (!wide) cudaGetLastError();
        for (int i = 0; i < kChunkShapes; ++i) {
            if ((1 << i) > 8 && !wide) continue;
            ClusterLaunch l(1 << i, 1, kClusterSmem, 0);
            if (cudaOccupancyMaxActiveClusters(&r.n[i], k_chunk_cluster, &l.cfg) != cudaSuccess) { r.n[i] = 0; cudaGetLastError(); }
        }
        r.known = true;
        if (listed) { std::lock_guard<std::mutex> hold(lock); table[device] = r; }
    }
    for (int i = 0; i < kChunkShapes; ++i) resident[i] = r.n[i];
    return cudaSuccess;
}

cudaError_t launch_chunk_cluster(const ChunkArgs& a, const ChunkPlan& p, bool overlap, cudaStream_t stream) {
    ClusterLaunch l(p.cl, p.clusters, p.bytes, stream);
    l.cfg.numAttrs = overlap ? 2 : 1;
    return cudaLaunchKernelEx(&l.cfg, k_chunk_cluster, a, p);
}

}  // namespace sgc
