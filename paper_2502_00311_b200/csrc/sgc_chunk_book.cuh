// The books of one recovery of a small problem: what a few warps ("team") do with a picked column, and with the rare picks that the
// screening scores leave open.  Shared by the kernels that make all picks of chunks in one launch.  Not part of the C ABI.
#pragma once

#include "sgc_chunked.cuh"
#include "sgc_tcgen05.cuh"

namespace sgc {

constexpr int kListed = 16;                           // candidates that the fp64 decision takes without going through the columns again

// what a block keeps of a recovery, besides its residual and the q_l
struct ChunkBook {
    double cs[kChunkMaxS + 2];                        // <q_l, a>, then <r, a> and ||a||^2 behind the last
    double red[kClusterWarps];
    double bs[kClusterWarps];                         // best of the columns that were gone through again, per warp
    double cdot[kListed + 1], cn2[kListed + 1];
    uint32_t cidx[kListed + 1], bi[kClusterWarps];
    uint32_t lam[kChunkMaxS];
    ChunkRef ref;                                     // where its records go
    double rn;                                        // whole-GPU form: norm of the residual ...
    float row_norm, row_tau;                          // ... and, in the units of its row, that norm and the report threshold
    int nc, stopped;
    unsigned int redo;                                // blocks whose columns are gone through again
};
static_assert(sizeof(ChunkBook) <= kClusterBook, "a recovery's records");

// The whole block waits for a barrier and agrees on whether the wait expired.  The waits acquire at the scope of the block, as those on TMA
// loads do, also where another block of the cluster has sent what is waited for: it lies in this block's own shared memory, of which there is
// one copy, the barrier counts bytes that have been written there, and blocks exchange nothing through global memory while the kernel runs,
// which is all that the cluster's scope would add (it empties the SM's L1: with one acquire of that scope behind every wait 111 instead of 109 us at
// 64 x 64, k = 256, and 457 instead of 442 for the projected 4096 x 4096; polled with it 105 instead of 94 us).  Where the caller wants waits to expire (a limit under a
// millisecond) the barrier is polled without the hardware's own pause.
static __device__ __noinline__ bool block_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
    const bool brief = limit_ns < 1000000ull;
    unsigned long long t0 = 0;
    for (uint32_t i = 0;; ++i) {
        if (brief ? mbar_test(bar, parity) : mbar_try(bar, parity)) return true;
        if (brief || (i & 63u) == 63u) {
            if (*abort_flag) return false;
            const unsigned long long t = global_ns();
            if (t0 == 0) t0 = t;
            else if (t - t0 > limit_ns) { *abort_flag = 1; return false; }
        }
    }
}
__device__ __forceinline__ bool block_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
    bool ok = mbar_test(bar, parity);
    if (!ok) ok = block_wait_slow(bar, parity, abort_flag, limit_ns);
    return __syncthreads_and(ok ? 1 : 0) != 0;
}

// the warps that work on one recovery
struct Team {
    int id, warps, warp, lane, t;
    __device__ __forceinline__ void meet() const {
        if (warps == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + id), "r"(warps * 32) : "memory");
    }
};

__device__ __forceinline__ bool in_picks(const uint32_t* lam, int n, uint32_t col) {
    bool hit = false;
#pragma unroll 4
    for (int l = 0; l < n; ++l) hit |= lam[l] == col;
    return hit;
}

__device__ __forceinline__ unsigned int order_key(float s) { return s >= 0.0f ? __float_as_uint(s) + 1u : 0u; }
__device__ __forceinline__ float order_score(unsigned int k) { return k ? __uint_as_float(k - 1u) : -1.0f; }

// rows 2 p, 2 p + 1 of a column (rows beyond k are zero)
__device__ __forceinline__ double2 pair_rows(const ChunkArgs& a, const ColKey& key, int p) {
    const float2 z = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)p * key.mk));
    return make_double2(2 * p < a.k ? (double)z.x : 0.0, 2 * p + 1 < a.k ? (double)z.y : 0.0);
}

// best free column seen by this thread, fp64 scores, lowest column on ties
struct BestColumn { double score = -1.0; uint32_t col = kNoColumn; };

// columns first .. last of the chunk against the residual: thread = column
__device__ __forceinline__ void scan_columns(const ChunkArgs& a, const ChunkBook& bk, const double* r, const Team& tm, int j, long long first, long long last,
                                             BestColumn& b) {
    if (last > a.dc) last = a.dc;
    for (long long col = first + tm.t; col < last; col += 32 * tm.warps) {
        if (in_picks(bk.lam, j, (uint32_t)col)) continue;
        const ColKey key = column_key(a.seed_lo, a.seed_hi, (uint32_t)col);
        double dot = 0.0, n2 = 0.0;
        for (int q = 0; 2 * q < a.k; ++q) {
            const double2 x = pair_rows(a, key, q);
            dot = fma(x.x, r[2 * q], dot); n2 = fma(x.x, x.x, n2);
            dot = fma(x.y, r[2 * q + 1], dot); n2 = fma(x.y, x.y, n2);
        }
        const double sc = n2 > 0.0 ? dot * dot / n2 : 0.0;
        if (sc > b.score || (sc == b.score && (uint32_t)col < b.col)) { b.score = sc; b.col = (uint32_t)col; }
    }
}
// the best over the team, for all of it
__device__ __forceinline__ uint32_t join_columns(ChunkBook& bk, const Team& tm, const BestColumn& b) {
    double best = b.score;
    uint32_t bi = b.col;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double so = __shfl_xor_sync(0xffffffffu, best, o);
        const uint32_t io = __shfl_xor_sync(0xffffffffu, bi, o);
        if (so > best || (so == best && io < bi)) { best = so; bi = io; }
    }
    if (tm.lane == 0) { bk.bs[tm.warp] = best; bk.bi[tm.warp] = bi; }
    tm.meet();
    for (int w = 0; w < tm.warps; ++w) {
        const double so = bk.bs[w];
        const uint32_t io = bk.bi[w];
        if (so > best || (so == best && io < bi)) { best = so; bi = io; }
    }
    return bi;
}

// the winner of the nc candidates in bk.cidx: exact scores, lowest column on ties
__device__ __forceinline__ uint32_t best_candidate(const ChunkArgs& a, ChunkBook& bk, const double* r, const Team& tm, int nc) {
    const int lane = tm.lane;
    if (nc == 0) return kNoColumn;
    if (nc == 1) return bk.cidx[0];
    // exact scores, warp = candidate
    for (int c = tm.warp; c < nc; c += tm.warps) {
        const ColKey key = column_key(a.seed_lo, a.seed_hi, bk.cidx[c]);
        double dot = 0.0, n2 = 0.0;
        for (int q = lane; 2 * q < a.k; q += 32) {
            const double2 x = pair_rows(a, key, q);
            dot = fma(x.x, r[2 * q], dot); n2 = fma(x.x, x.x, n2);
            dot = fma(x.y, r[2 * q + 1], dot); n2 = fma(x.y, x.y, n2);
        }
        dot = warp_sum_d(dot); n2 = warp_sum_d(n2);
        if (lane == 0) { bk.cdot[c] = dot; bk.cn2[c] = n2; }
    }
    tm.meet();
    double best = -1.0;
    uint32_t win = kNoColumn;
    for (int c = 0; c < nc; ++c) {
        const double sc = bk.cn2[c] > 0.0 ? bk.cdot[c] * bk.cdot[c] / bk.cn2[c] : 0.0;
        const uint32_t col = bk.cidx[c];
        if (sc > best || (sc == best && col < win)) { best = sc; win = col; }
    }
    return win;
}

// sum over the team of what its threads hold, for all of them; only the first `rows` threads hold anything
__device__ __forceinline__ double team_sum(ChunkBook& bk, double part, const Team& tm, int rows) {
    const int busy = (rows + 31) / 32 < tm.warps ? (rows + 31) / 32 : tm.warps;
    if (tm.warp < busy) {
        part = warp_sum_d(part);
        if (tm.warps > 1 && tm.lane == 0) bk.red[tm.warp] = part;
    }
    tm.meet();                                                        // (and everything that the team wrote before is visible)
    if (tm.warps == 1) return part;
    double v0 = 0.0, v1 = 0.0;
#pragma unroll
    for (int w = 0; w < kChunkMaxK / 32; w += 2) { if (w < busy) v0 += bk.red[w]; if (w + 1 < busy) v1 += bk.red[w + 1]; }
    return v0 + v1;
}

// Column `col` becomes pick j of recovery m: c_l = <q_l, a>, gamma, a_j, the new q and residual, its squared norm.  False: the column
// depends on the earlier ones, this recovery ends.  SHARED: the q_l are in shared memory, qstride rows apart and zero beyond k, (else in the chunk's
// records, k apart).  xs: room for a column, zero beyond k.
template <bool SHARED>
__device__ __forceinline__ bool extend_basis(const ChunkArgs& a, ChunkBook& bk, const ChunkRef& ref, double* r, double* qs, int qstride, double* xs, int m,
                                             int j, uint32_t col, const Team& tm, double* gamma_out, double* aj_out, double* rn2_out) {
    const int lane = tm.lane, k = a.k;
    // ---- products of the column with the q_l and the residual, and its norm: warp = two vectors at a time
    {
        const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
        for (int i = tm.t; 2 * i < k; i += 32 * tm.warps) {
            const double2 z = pair_rows(a, key, i);
            *reinterpret_cast<double2*>(xs + 2 * i) = make_double2(a.sigma * z.x, a.sigma * z.y);
        }
    }
    tm.meet();
    {
        double2 x[kChunkMaxK / 64];
#pragma unroll
        for (int u = 0; u < kChunkMaxK / 64; ++u) x[u] = 64 * u < k ? *reinterpret_cast<const double2*>(xs + 2 * (lane + 32 * u)) : make_double2(0.0, 0.0);
        if (tm.warp == tm.warps - 1) {
            double n0 = 0.0, n1 = 0.0;
#pragma unroll
            for (int u = 0; u < kChunkMaxK / 64; ++u) { n0 = fma(x[u].x, x[u].x, n0); n1 = fma(x[u].y, x[u].y, n1); }
            n0 = warp_sum_d(n0 + n1);
            if (lane == 0) bk.cs[j + 1] = n0;
        }
        // (vectors in global memory: more of them at a time, for the latency)
        constexpr int V = SHARED ? 2 : 4;
        for (int l0 = tm.warp; l0 <= j; l0 += V * tm.warps) {
            double c[V];
            const double* v[V];
#pragma unroll
            for (int e = 0; e < V; ++e) { const int l = l0 + e * tm.warps; c[e] = 0.0; v[e] = l < j ? qs + (size_t)l * qstride : r; }
#pragma unroll
            for (int u = 0; u < kChunkMaxK / 64; ++u) {
                if (64 * u >= k) break;
                const int i = 2 * (lane + 32 * u);
                double2 y[V];
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    if (SHARED) y[e] = *reinterpret_cast<const double2*>(v[e] + i);
                    else y[e] = make_double2(i < k ? v[e][i] : 0.0, i + 1 < k ? v[e][i + 1] : 0.0);
                }
#pragma unroll
                for (int e = 0; e < V; ++e) { c[e] = fma(y[e].x, x[u].x, c[e]); c[e] = fma(y[e].y, x[u].y, c[e]); }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int e = 0; e < V; ++e) c[e] += __shfl_xor_sync(0xffffffffu, c[e], o);
            }
            if (lane == 0) {
#pragma unroll
                for (int e = 0; e < V; ++e) if (l0 + e * tm.warps <= j) bk.cs[l0 + e * tm.warps] = c[e];
            }
        }
    }
    tm.meet();
    const double mine = lane < j ? bk.cs[lane] : 0.0, dot = bk.cs[j], n2 = bk.cs[j + 1];
    const double piv = n2 - warp_sum_d(mine * mine);
    if (!(piv > 1e-10 * n2)) {                                    // dependent column: this recovery ends with j picks
        if (tm.t == 0) {
            ref.cnt->stopped[m] = 1; ref.cnt->done[m] = j;
            atomicOr(&ref.cnt->status, (unsigned int)SGC_STATUS_DEPENDENT_COLUMN);
        }
        return false;
    }
    {
        const double gamma = rsqrt(piv), aj = gamma * dot;
        double part = 0.0;
        for (int row = tm.t; row < k; row += 32 * tm.warps) {
            const double x = xs[row];
            double v0 = 0.0, v1 = 0.0;
            int l = 0;
#pragma unroll 1
            for (; l + 8 <= j; l += 8) {
                double y[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) y[e] = qs[(l + e) * qstride + row];
#pragma unroll
                for (int e = 0; e < 8; e += 2) { v0 = fma(bk.cs[l + e], y[e], v0); v1 = fma(bk.cs[l + e + 1], y[e + 1], v1); }
            }
            for (; l + 1 < j; l += 2) { v0 = fma(bk.cs[l], qs[l * qstride + row], v0); v1 = fma(bk.cs[l + 1], qs[(l + 1) * qstride + row], v1); }
            if (l < j) v0 = fma(bk.cs[l], qs[l * qstride + row], v0);
            const double q = gamma * (x - (v0 + v1));
            qs[j * qstride + row] = q;
            const double rv = r[row] - aj * q;
            r[row] = rv;
            part = fma(rv, rv, part);
        }
        *rn2_out = team_sum(bk, part, tm, k);
        *gamma_out = gamma; *aj_out = aj;
    }
    return true;
}

// the records of pick j (one warp)
__device__ __forceinline__ void record_pick(const ChunkArgs& a, ChunkBook& bk, const ChunkRef& ref, int m, int j, uint32_t col, double gamma, double aj,
                                            double rn2, int lane) {
    const int s = a.s;
    if (lane < j) ref.crow[((size_t)m * s + j) * s + lane] = bk.cs[lane];
    if (lane == 0) {
        bk.lam[j] = col;
        ref.gam[(size_t)m * s + j] = gamma; ref.acoef[(size_t)m * s + j] = aj; ref.lam[(size_t)m * s + j] = col;
        ref.rnorm[(size_t)m * s + j] = sqrt(rn2);
        ref.cnt->done[m] = j + 1;
    }
}

}  // namespace sgc
