// MESGC (Section 4.4) with small per-chunk problems: c chunks of one flat vector, each an SGC problem of its own
// (own M, V; s_c <= 32 kept entries, k_c <= 256 rows), all sharing the matrix A (k_c x d/c) named by one seed.
// Run chunk by chunk this costs ~25 launches per chunk; here the whole step of all chunks takes three launches where A fits the
// shared memory of a thread-block cluster (sgc_chunk_cluster.cu) or of the GPU (sgc_chunk_grid.cu), and 2 + 2 s_c in the general form:
//   k_chunk_front    block (or cluster) = chunk: exact top-s_c of the chunk (a1), p = A g~, q = A g~^2 and the k-space Adam
//                    moments (a2 + a3), residuals r = y for both moments
//   per OMP iteration (Algorithm 3, all 2c recoveries in lock-step, which is where the shared A pays: a column of A is
//   generated once and meets the residuals of every chunk):
//     k_chunk_corr   columns of A as the A operand of mma.m16n8k16, four residuals as two binary16 numbers each as the B
//                    operand: scores |<A_i,r>| / ||A_i||, best two columns of the block's range per residual
//     k_chunk_pick   block = one recovery: fp64 rescoring of the columns within 2e-3 of the best score, lowest
//                    index on ties, then Algorithm 3 in the orthogonal form of sgc_omp.cu: c_l = <q_l, a>, q, a_j, r
//   k_chunk_scatter  block = chunk: coefficients, Eq. (8) on the common support, weight update (a5)
// Every record lands in the chunk's own state, so sgc_get works per chunk exactly as after sgc_step.
#include <algorithm>
#include <new>
#include <utility>
#include <vector>

#include <cooperative_groups.h>

#include "sgc_chunked.cuh"

namespace cg = cooperative_groups;

namespace sgc {
namespace {

constexpr int kFrontThreads = 512;
// ---- residuals as operands of k_chunk_corr ----------------------------------------------------------------
// Position of row `row` in a residual's operand: for each 16 rows, lane q of a column group holds rows 2q, 2q + 1 and 2q + 8, 2q + 9
// as two registers of the B operand of mma.m16n8k16.
__device__ __forceinline__ int frag_place(int row) {
    const int r = row & 15;
    return (row & ~15) + ((r & 7) >> 1) * 4 + (r >> 3) * 2 + (r & 1);
}
// one entry (scale: a power of two that brings the residual's norm into [2^9, 2^10)): the value and what it leaves
__device__ __forceinline__ void frag_write(const ChunkArgs& a, int res, int row, double v, double scale) {
    const float x = (float)(v * scale);
    const __half h = __float2half_rn(x);
    const __half l = __float2half_rn(x - __half2float(h));
    uint16_t* f = a.frag + (size_t)res * 2 * a.kf + frag_place(row);
    f[0] = __half_as_ushort(h);
    f[a.kf] = __half_as_ushort(l);
}
// ---- a1 + a2 + a3, one block or cluster of blocks per chunk -----------------------------------------------
// Top-s of the chunk by the key (|g| bits << 32) | ~index (unique; lowest index wins equal magnitudes).  One read of the
// chunk gives every thread the largest magnitude of its strided share; with e = ceil(s / warps), the smallest over the warps of
// a warp's e-th largest thread maximum is a bound that at least s elements reach.  Only the shares whose maximum
// reaches it are read again (from L2, a share per warp and trip), and the few elements that do are ranked.  Registers hold one
// word per thread whatever s is (keeping the s largest of every share in registers and sorting in one thread took 146 us for
// 256 chunks of 65536 floats at s = 16).  More survivors than can be ranked at once (many equal magnitudes) send the block
// through s sweeps of "largest key below the last one" instead.  Long chunks in small number are split over a cluster, so
// that the SMs are all reading.
constexpr int kFrontCap = 2048;
constexpr int kFrontRank = 256;                  // survivors ranked all against all
constexpr int kFrontMaxSplit = 8;

__device__ __forceinline__ unsigned long long front_key(float g, uint32_t i) {
    return ((unsigned long long)(__float_as_uint(g) & 0x7FFFFFFFu) << 32) | (uint32_t)(~i);
}
__device__ __forceinline__ unsigned int mag4(const float4& f) {
    return max(max(__float_as_uint(f.x) & 0x7FFFFFFFu, __float_as_uint(f.y) & 0x7FFFFFFFu),
               max(__float_as_uint(f.z) & 0x7FFFFFFFu, __float_as_uint(f.w) & 0x7FFFFFFFu));
}

// largest 64-bit value over the block (kFrontThreads threads); part: one word per warp
__device__ unsigned long long front_max(unsigned long long v, unsigned long long* part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) { const unsigned long long t = __shfl_xor_sync(0xffffffffu, v, o); v = t > v ? t : v; }
    __syncthreads();
    if (lane == 0) part[warp] = v;
    __syncthreads();
    v = 0ull;
#pragma unroll
    for (int w = 0; w < kFrontThreads / 32; ++w) v = part[w] > v ? part[w] : v;
    return v;
}

__global__ void __launch_bounds__(kFrontThreads, 2)
k_chunk_front(ChunkArgs a, const float* __restrict__ grad, double b1, double b2, double c1, double c2) {
    __shared__ unsigned long long list[kFrontCap];
    __shared__ unsigned long long part[kFrontThreads / 32];
    __shared__ unsigned int wtau[kFrontMaxSplit * kFrontThreads / 32];
    __shared__ unsigned long long sel_key[kChunkMaxS];
    __shared__ ColKey keys[kChunkMaxS];
    __shared__ float vals[kChunkMaxS];
    __shared__ double norms[2][kFrontThreads / 32];
    __shared__ int n_list;
    cg::cluster_group cluster = cg::this_cluster();
    const int split = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();      // split: a power of two
    // every block of the cluster has to run before another writes to its shared memory: announced here, waited for after the read
    cg::cluster_group::arrival_token started;
    if (split > 1) started = cluster.barrier_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");                 // (only the launch overlaps the kernel before)
    if (a.early_front) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int ch = blockIdx.x / split, s = a.s, k = a.k, t = threadIdx.x;
    const ChunkRef ref = chunk_ref(a, ch);
    const float* g = grad + (size_t)ch * a.dc;
    const float4* g4 = reinterpret_cast<const float4*>(g);
    const int lane = t & 31, warp = t >> 5, stride = split * kFrontThreads;
    const int nvec = (int)(a.dc >> 2);                               // chunks start on 16-byte boundaries
    const int v_first = rank * kFrontThreads + t;
    unsigned int top = 0u;
    {
        int v = v_first;
        for (; v + 7 * stride < nvec; v += 8 * stride) {
            float4 f[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) f[u] = g4[v + u * stride];
#pragma unroll
            for (int u = 0; u < 8; ++u) top = max(top, mag4(f[u]));
        }
        for (; v < nvec; v += stride) top = max(top, mag4(g4[v]));
    }
    // (a vector on its own may have any length)
    const int tail = (int)(a.dc & 3);
    const bool has_tail = rank == 0 && t < tail;
    const float tail_g = has_tail ? g[4 * (long long)nvec + t] : 0.0f;
    const unsigned int tail_mag = __float_as_uint(tail_g) & 0x7FFFFFFFu;
    top = max(top, tail_mag);
    const int warps = split * (kFrontThreads / 32);
    if (t == 0) n_list = 0;
    {
        // the warp's e-th largest thread maximum (equal ones count one by one), told to every block of the cluster
        const int e = (s + warps - 1) / warps;
        unsigned int m = 0u;
        bool out = false;
        for (int q = 0; q < e; ++q) {
            m = __reduce_max_sync(0xffffffffu, out ? 0u : top);
            const unsigned int who = __ballot_sync(0xffffffffu, !out && top == m);
            if (who != 0u && lane == __ffs(who) - 1) out = true;
        }
        if (split > 1) cluster.barrier_wait(std::move(started));
        if (lane < split) *cluster.map_shared_rank(&wtau[rank * (kFrontThreads / 32) + warp], lane) = m;
    }
    if (split > 1) cluster.sync(); else __syncthreads();
    unsigned int tau = 0xFFFFFFFFu;
    for (int w = lane; w < warps; w += 32) tau = min(tau, wtau[w]);
    tau = __reduce_min_sync(0xffffffffu, tau);
    int* count = cluster.map_shared_rank(&n_list, 0);
    unsigned long long* dst = cluster.map_shared_rank(list, 0);
    if (tau == 0u) tau = 1u;                                          // (fewer than s shares with a non-zero: zeros are added below)
    unsigned int redo = __ballot_sync(0xffffffffu, top >= tau);
    while (redo) {
        const int owner = __ffs(redo) - 1;
        redo &= redo - 1u;
        for (int v0 = rank * kFrontThreads + warp * 32 + owner; v0 < nvec; v0 += 32 * stride) {
            const long long v = (long long)v0 + (long long)lane * stride;
            if (v >= nvec) continue;
            const float4 f = g4[v];
            if (mag4(f) < tau) continue;
            const float x[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if ((__float_as_uint(x[u]) & 0x7FFFFFFFu) >= tau) {
                    const int slot = atomicAdd(count, 1);
                    if (slot < kFrontCap) dst[slot] = front_key(x[u], (uint32_t)(4 * v + u));
                }
        }
    }
    if (has_tail && tail_mag >= tau) {
        const int slot = atomicAdd(count, 1);
        if (slot < kFrontCap) dst[slot] = front_key(tail_g, (uint32_t)(4 * (long long)nvec + t));
    }
    if (split > 1) { cluster.sync(); if (rank != 0) return; }          // (nobody reads this block's memory after this)
    __syncthreads();
    int n = n_list;
    if (n < s) {
        // fewer than s non-zeros: the first zeros of the chunk are kept as well, and those that are missing lie among its first
        // s + n entries (a bound of zero let everything through: 1024 x 1024 zeros cost 160 us)
        if (t < s + n && t < a.dc && (__float_as_uint(g[t]) & 0x7FFFFFFFu) == 0u) list[atomicAdd(&n_list, 1)] = front_key(0.0f, (uint32_t)t);
        __syncthreads();
        n = n_list;
    }
    if (n <= kFrontRank) {
        // rank of every survivor among the others: the s largest
        if (t < n) {
            const unsigned long long mine = list[t];
            int r = 0;
            for (int q = 0; q < n; ++q) r += list[q] > mine ? 1 : 0;
            if (r < s) sel_key[r] = mine;
        }
    } else {
        unsigned long long last = ~0ull;
        for (int r = 0; r < s; ++r) {
            unsigned long long m = 0ull;                              // no real key is 0
            if (n <= kFrontCap) { for (int q = t; q < n; q += kFrontThreads) { const unsigned long long v = list[q]; if (v < last && v > m) m = v; } }
            else {
                if (has_tail) { const unsigned long long key = front_key(tail_g, (uint32_t)(4 * (long long)nvec + t)); if (key < last) m = key; }
                for (int v = t; v < nvec; v += kFrontThreads) {
                    const float4 f = g4[v];
                    const float x[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) { const unsigned long long key = front_key(x[u], (uint32_t)(4 * v + u)); if (key < last && key > m) m = key; }
                }
            }
            last = front_max(m, part);
            if (t == 0) sel_key[r] = last;
        }
    }
    __syncthreads();
    if (t < s) {
        // ascending index order, as the records of sgc_step have it
        const unsigned long long mine = sel_key[t];
        const uint32_t idx = ~(uint32_t)mine;
        int r = 0;
        for (int q = 0; q < s; ++q) r += (uint32_t)(~(uint32_t)sel_key[q]) < idx ? 1 : 0;
        const float val = g[idx];
        ref.sel_idx[r] = idx; ref.sel_val[r] = val;
        keys[r] = column_key(a.seed_lo, a.seed_hi, idx);
        vals[r] = val;
        if ((mine >> 32) >= 0x7F800000ull) atomicOr(&ref.cnt->status, (unsigned int)SGC_STATUS_NONFINITE_INPUT);
    }
    if (t == 0) {
        ref.cnt->done[0] = ref.cnt->done[1] = 0;
        ref.cnt->stopped[0] = ref.cnt->stopped[1] = 0;
        ref.cnt->n_upd = ref.cnt->mismatch = ref.cnt->negv = 0;
        ref.ctl->round_active = 0; ref.ctl->fallback = 1; ref.ctl->rounds = 0; ref.ctl->list_rounds = 0;
    }
    __syncthreads();
    // a2 + a3: thread = row; fp64 sums in ascending column order (the arithmetic of the one-state kernel, term by term)
    static_assert(kChunkMaxK <= kFrontThreads, "one row per thread");
    double mh = 0.0, vh = 0.0;
    if (t < k) {
        const int row = t;
        double accp = 0.0, accq = 0.0;
        for (int i = 0; i < s; ++i) {
            const double av = a.sigma * (double)z_at(keys[i], (uint32_t)row);
            const double gv = (double)vals[i];
            accp = accp + av * gv;
            accq = accq + av * (gv * gv);
        }
        ref.p[row] = accp;
        ref.q[row] = accq;
        const float m = (float)(b1 * (double)ref.M[row] + (1.0 - b1) * accp);
        const float v = (float)(b2 * (double)ref.V[row] + (1.0 - b2) * accq);
        ref.M[row] = m;
        ref.V[row] = v;
        mh = (double)m / c1; vh = (double)v / c2;                    // bias-corrected temporaries; state stays uncorrected
        ref.y64[row] = mh; ref.y64[k + row] = vh;
        ref.r64[row] = mh; ref.r64[k + row] = vh;
    }
    if (a.frag != nullptr) {
        double m2 = warp_sum_d(mh * mh), v2 = warp_sum_d(vh * vh);
        if (lane == 0) { norms[0][warp] = m2; norms[1][warp] = v2; }
        __syncthreads();
        m2 = v2 = 0.0;
#pragma unroll
        for (int w = 0; w < kFrontThreads / 32; ++w) { m2 += norms[0][w]; v2 += norms[1][w]; }
        const double sm = frag_scale(sqrt(m2)), sv = frag_scale(sqrt(v2));
        if (t < k) { frag_write(a, 2 * ch, t, mh, sm); frag_write(a, 2 * ch + 1, t, vh, sv); }
        if (t == 0) { a.back[2 * ch] = (float)(1.0 / sm); a.back[2 * ch + 1] = (float)(1.0 / sv); }
    }
}

// ---- phase A of one OMP iteration: every column of A against the residuals of all recoveries ------------------
// grid = (column splits, groups of recoveries).  The block walks its columns a tile at a time: its warps generate the tile in the
// register layout of mma.m16n8k16's A operand (a row pair of a column is one register) into shared memory, with 1 / ||Z_i||,
// and every warp multiplies it with the residuals it holds as B operands: NT tiles of four recoveries, each residual as two
// binary16 numbers (value and remainder, 22 bits, scaled by a power of two), sums in fp32.  A lane ends up with the scores of
// one recovery for two columns of every 16; only the best two columns per recovery leave the block.  (The legacy matrix instruction on purpose: with 2c residuals of k_c
// rows the tensor work is small, what bounds the kernel is generating, comparing and the launch itself, and an operand in
// registers needs no hand-off.  With one multiply-add per instruction it took 37 us at k_c = 8, 512 recoveries, 65536
// columns, and 22 us per iteration at k_c = 217, 128 recoveries, 2048 columns.)
__host__ __device__ constexpr int corr_threads(int kp) { return kp <= 32 ? 512 : 256; }              // (registers hold the residuals)
__host__ __device__ constexpr int corr_kb(int kp) { return kp / 16 > 0 ? kp / 16 : 1; }              // 16-row blocks
__host__ __device__ constexpr int corr_nt(int kp) { return kp == 64 ? 8 : (kp <= 128 ? 4 : 2); }     // tiles of four recoveries per warp
__host__ __device__ constexpr int corr_group(int kp) { return corr_threads(kp) / 32 * 4 * corr_nt(kp); }   // recoveries per block
static_assert(corr_group(8) == chunk_corr_group(8) && corr_group(32) == chunk_corr_group(32) && corr_group(64) == chunk_corr_group(64) &&
              corr_group(128) == chunk_corr_group(128) && corr_group(256) == chunk_corr_group(256), "the estimates count the same groups");
__host__ __device__ constexpr int corr_tile(int kp) { return kp <= 16 ? 256 : kp == 32 ? 128 : kp == 64 ? 64 : 32; }   // columns generated at a time
constexpr int kCorrSuper = 512;                                                                      // columns that a key can tell apart

// launch configuration of such a kernel
struct ChainedLaunch {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    ChainedLaunch(dim3 grid, dim3 block, size_t smem, cudaStream_t stream) : cfg{} {
        cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
    }
};

// the two best columns of a recovery, and a bound on the score of all others
struct Best2 {
    float s1, s2, s3; uint32_t i1, i2;
    __device__ __forceinline__ void push(float s, uint32_t i) {      // i != i1, i2; lower index first on ties
        if (s > s1 || (s == s1 && i < i1)) { s3 = fmaxf(s3, s2); s2 = s1; i2 = i1; s1 = s; i1 = i; }
        else if (s > s2 || (s == s2 && i < i2)) { s3 = fmaxf(s3, s2); s2 = s; i2 = i; }
        else s3 = fmaxf(s3, s);
    }
};

// 1 / ||Z|| of a column and the code that its keys carry
__device__ __forceinline__ float2 corr_norm(float n2, int code, bool real) {
    return make_float2(real && n2 > 0.0f ? 1.0f / sqrtf(n2) : 0.0f, __uint_as_float(real ? (unsigned int)code : 0u));
}

// gate != nullptr: the launch is a fallback of the tensor-core route and returns at once unless *gate names this
// iteration (a.epoch): the word holds the epoch of the last iteration that left a recovery unresolved.
template <int KP>
__global__ void __launch_bounds__(corr_threads(KP)) k_chunk_corr(ChunkArgs a, int iter, const int* gate) {
    constexpr int KB = corr_kb(KP), NT = corr_nt(KP), TC = corr_tile(KP), TILES = TC / 16, WARPS = corr_threads(KP) / 32;
    extern __shared__ uint4 smem4[];
    uint4* zt = smem4;                                                // [TILES][KB][32] A operands
    float2* inv = reinterpret_cast<float2*>(zt + TILES * KB * 32);    // [TC] 1 / ||Z_i||, code of the column
    float* n2p = reinterpret_cast<float*>(inv + TC);                  // [KB][TC] partial ||Z_i||^2
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    const long long col0 = (long long)blockIdx.x * a.cols_per_split;
    long long col1 = col0 + a.cols_per_split;
    if (col1 > a.dc) col1 = a.dc;
    // code: see the keys below (columns beyond this block's range get code 0 and 1 / ||Z|| = 0)
    // (unit of work: 16 columns, 16 rows)
    auto generate = [&](long long tile0, int code0) {
        const int units = (int)(col1 - tile0 < TC ? (col1 - tile0 + 15) / 16 : TILES) * KB;
        for (int u = warp; u < units; u += WARPS) {
            const int tl = u / KB, kb = u % KB;
            // a column's key is worked out by one lane (lanes 0-15) and handed to the four that use it
            const ColKey key = column_key(a.seed_lo, a.seed_hi, (uint32_t)(tile0 + tl * 16 + (lane & 15)));
            const uint32_t ck0 = __shfl_sync(0xffffffffu, key.ck, g), mk0 = __shfl_sync(0xffffffffu, key.mk, g);
            const uint32_t ck1 = __shfl_sync(0xffffffffu, key.ck, g + 8), mk1 = __shfl_sync(0xffffffffu, key.mk, g + 8);
            const uint32_t h0 = ck0 + (uint32_t)(kb * 8 + q) * mk0, h1 = ck1 + (uint32_t)(kb * 8 + q) * mk1;
            uint32_t z[4] = {z_pair_from_word(h0), z_pair_from_word(h1), 0u, 0u};
            if (KP > 8) { z[2] = z_pair_from_word(h0 + 4u * mk0); z[3] = z_pair_from_word(h1 + 4u * mk1); }
            float n[2] = {0.0f, 0.0f};
#pragma unroll
            for (int e = 0; e < (KP > 8 ? 4 : 2); ++e) {              // rows beyond k do not count
                const int row = kb * 16 + 2 * q + (e & 2 ? 8 : 0);
                if (row >= a.k) z[e] = 0u;
                else if (row + 1 >= a.k) z[e] &= 0xFFFFu;
                const float2 f = half2_bits_to_float2(z[e]);
                n[e & 1] = __fmaf_rn(f.x, f.x, n[e & 1]); n[e & 1] = __fmaf_rn(f.y, f.y, n[e & 1]);
            }
            zt[(size_t)u * 32 + lane] = make_uint4(z[0], z[1], z[2], z[3]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                n[e] += __shfl_xor_sync(0xffffffffu, n[e], 1); n[e] += __shfl_xor_sync(0xffffffffu, n[e], 2);
                const int c = tl * 16 + g + 8 * e;
                if (q == 0) {
                    if (KB > 1) n2p[kb * TC + c] = n[e];
                    else inv[c] = corr_norm(n[e], code0 - c, tile0 + c < col1);
                }
            }
        }
    };
    if (gate == nullptr) generate(col0, kCorrSuper);                              // the first tile needs nothing of the kernels before
    after_previous_kernel(a.early);
    if (gate != nullptr) {
        if (*gate != a.epoch0 + iter) return;
        generate(col0, kCorrSuper);
    }
    // residuals as B operands: n = g of a tile is value (g even) or remainder (g odd) of recovery 4 tile + g / 2.  (Recoveries
    // that have stopped are scored like the others; k_chunk_pick does not look at them.)
    const int res0 = blockIdx.y * corr_group(KP) + warp * NT * 4;
    uint2 bf[NT][KB];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int res = res0 + 4 * i + (g >> 1);
        const uint2* src = reinterpret_cast<const uint2*>(a.frag + ((size_t)(res < 2 * a.c ? res : 0) * 2 + (g & 1)) * (16 * KB)) + q;
#pragma unroll
        for (int kb = 0; kb < KB; ++kb) bf[i][kb] = src[4 * kb];
    }
    // lane g of a recovery's eight holds every eighth column of its support, for the check at the end
    constexpr int kHeld = kChunkMaxS / 8;
    uint32_t held[NT][kHeld];
    if (NT <= 4) {
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const int mine = res0 + 4 * i + q;
            const uint32_t* sup = a.lam + (size_t)(mine < 2 * a.c ? mine : 0) * a.s;
#pragma unroll
            for (int h = 0; h < kHeld; ++h) held[i][h] = g + 8 * h < iter ? sup[g + 8 * h] : kNoColumn;
        }
    }
    // Scores are compared as keys: the score's bits with the lowest ten replaced by a code of the column (relative error 2^-13, an
    // eighth of the window that k_chunk_pick rescores), so that the best two follow from three integer minima and maxima, without
    // a branch.  Columns of a recovery's support score rounding noise; should one be among the best two all the same (hardly any
    // columns left), the block goes through its columns again and leaves them out.  A zero residual scores zero everywhere: what it
    // is handed does not matter.
    Best2 best[NT];
    bool exclude = false;
    for (;;) {
#pragma unroll
        for (int i = 0; i < NT; ++i) { best[i].s1 = best[i].s2 = best[i].s3 = -1.0f; best[i].i1 = best[i].i2 = kNoColumn; }
        for (long long super = col0; super < col1; super += kCorrSuper) {
            unsigned int k1[NT], k2[NT];
#pragma unroll
            for (int i = 0; i < NT; ++i) k1[i] = k2[i] = 0u;
            const long long super1 = super + kCorrSuper < col1 ? super + kCorrSuper : col1;
            for (long long tile0 = super; tile0 < super1; tile0 += TC) {
                const int code0 = (int)(kCorrSuper - (tile0 - super));
                if (tile0 != col0 || exclude) { __syncthreads(); generate(tile0, code0); }
                __syncthreads();
                if (KB > 1) {
                    if (threadIdx.x < TC) {
                        float n2 = 0.0f;
#pragma unroll
                        for (int kb = 0; kb < KB; ++kb) n2 += n2p[kb * TC + threadIdx.x];
                        inv[threadIdx.x] = corr_norm(n2, code0 - (int)threadIdx.x, tile0 + threadIdx.x < col1);
                    }
                    __syncthreads();
                }
#pragma unroll 1
                for (int tl = 0; tl < TILES && tile0 + tl * 16 < col1; ++tl) {
                    float acc[NT][4];
#pragma unroll
                    for (int i = 0; i < NT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.0f;
#pragma unroll
                    for (int kb = 0; kb < KB; ++kb) {
                        const uint4 x = zt[(size_t)(tl * KB + kb) * 32 + lane];
#pragma unroll
                        for (int i = 0; i < NT; ++i) mma_16816(acc[i], x, bf[i][kb].x, bf[i][kb].y);
                    }
                    const float2 v0 = inv[tl * 16 + g], v1 = inv[tl * 16 + g + 8];
#pragma unroll
                    for (int i = 0; i < NT; ++i) {
                        unsigned int x0 = (__float_as_uint(fabsf(acc[i][0] + acc[i][1]) * v0.x) & ~1023u) | __float_as_uint(v0.y);
                        unsigned int x1 = (__float_as_uint(fabsf(acc[i][2] + acc[i][3]) * v1.x) & ~1023u) | __float_as_uint(v1.y);
                        if (exclude) {
                            const int mine = res0 + 4 * i + q;
                            const uint32_t* sup = a.lam + (size_t)(mine < 2 * a.c ? mine : 0) * a.s;
                            const uint32_t c0 = (uint32_t)(tile0 + tl * 16 + g);
                            for (int l = 0; l < iter; ++l) { if (sup[l] == c0) x0 = 0u; if (sup[l] == c0 + 8u) x1 = 0u; }
                        }
                        k2[i] = max(k2[i], min(k1[i], x0)); k1[i] = max(k1[i], x0);
                        k2[i] = max(k2[i], min(k1[i], x1)); k1[i] = max(k1[i], x1);
                    }
                }
            }
            // the eight lanes of a recovery (same q) join their best two; k3: the largest key that may be left out (a lane has not kept
            // its third, which its second bounds)
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                unsigned int k3 = k2[i];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    const unsigned int t1 = __shfl_xor_sync(0xffffffffu, k1[i], o), t2 = __shfl_xor_sync(0xffffffffu, k2[i], o);
                    const unsigned int t3 = __shfl_xor_sync(0xffffffffu, k3, o);
                    k3 = max(max(k3, t3), max(min(k2[i], t1), min(k1[i], t2)));
                    k2[i] = max(max(k2[i], t2), min(k1[i], t1));
                    k1[i] = max(k1[i], t1);
                }
                if (k1[i]) best[i].push(__uint_as_float(k1[i] & ~1023u), (uint32_t)(super + kCorrSuper - (k1[i] & 1023u)));
                if (k2[i]) best[i].push(__uint_as_float(k2[i] & ~1023u), (uint32_t)(super + kCorrSuper - (k2[i] & 1023u)));
                best[i].s3 = fmaxf(best[i].s3, __uint_as_float(k3 & ~1023u));
            }
        }
        if (exclude || iter == 0) break;
        bool taken = false;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            if (best[i].s1 == 0.0f) continue;                         // a zero residual: k_chunk_pick knows what to do
            if (NT <= 4) {
#pragma unroll
                for (int h = 0; h < kHeld; ++h)
                    taken = taken || (held[i][h] != kNoColumn && (held[i][h] == best[i].i1 || held[i][h] == best[i].i2));
            } else {
                const int mine = res0 + 4 * i + q;
                const uint32_t* sup = a.lam + (size_t)(mine < 2 * a.c ? mine : 0) * a.s;
                for (int l = g; l < iter; l += 8) { const uint32_t v = sup[l]; taken = taken || v == best[i].i1 || v == best[i].i2; }
            }
        }
        if (!__syncthreads_or(taken ? 1 : 0)) break;
        exclude = true;
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int mine = res0 + 4 * i + q;
        if (g == 0 && mine < 2 * a.c) {
            const float back = a.back[mine];
            float4* out = reinterpret_cast<float4*>(a.cand + ((size_t)mine * a.splits + blockIdx.x) * 2);
            const bool third = best[i].s3 > 0.0f && best[i].s3 >= best[i].s1 * (1.0f - kKeyWindow);
            *out = make_float4(best[i].i1 != kNoColumn ? best[i].s1 * back : -1.0f, __uint_as_float(third ? best[i].i1 | kThirdMark : best[i].i1),
                               best[i].i2 != kNoColumn ? best[i].s2 * back : -1.0f, __uint_as_float(best[i].i2));
        }
    }
}

// ---- phase B of one OMP iteration: one block per recovery ---------------------------------------------------------
// Argmax among the columns that phase A left within 2e-3 (relative) of the best score, decided on fp64 scores
// <Z_i, r>^2 / ||Z_i||^2 with the lowest index winning ties; then Algorithm 3 (Appendix B) in its orthogonal form for the new
// column a: c_l = <q_l, a>, gamma = 1 / ||a - sum c_l q_l|| (a squared norm below 1e-10 ||a||^2 ends this recovery),
// q = gamma (a - sum c_l q_l), a_j = gamma <a, r>, r <- r - a_j q.  The coefficients x follow once, at the end of the step.
// The orthogonal vectors q_l of the earlier picks are fetched into shared memory in one trip, before anything else; a pick is
// then four block barriers and j + 1 multiply-adds per row, all fp64, with no conversion in a loop (the inverse-Cholesky form
// on the stored binary16 columns took 10 to 24 us per pick at k_c = 217).
constexpr int kPickMaxThreads = 256;

struct PickSmem {
    double cs[kChunkMaxS];
    double cdot[kRescoreCap], cn2[kRescoreCap];
    double red[kPickMaxThreads / 32];
    float fred[kPickMaxThreads / 32];
    uint32_t cidx[kRescoreCap];
    int redo[8];
    int n_c, n_redo;
};

// dynamic shared memory: residual r [k], q [j][k]
__device__ __forceinline__ double* pick_mem() {
    extern __shared__ __align__(16) double pick_dyn_mem[];
    return pick_dyn_mem;
}
size_t pick_dyn_bytes(int s, int k) { return (size_t)s * k * sizeof(double); }
int pick_threads(int k) { return k <= 64 ? 64 : (k <= 128 ? 128 : kPickMaxThreads); }      // one row per thread

// the vectors of the earlier picks and the residual: independent loads, one trip to global memory.  A block-wide barrier has to
// follow before pick_finish reads them.
__device__ __forceinline__ void pick_stage(const ChunkArgs& a, const ChunkRef& ref, int m, int j) {
    const int k = a.k;
    double* r = pick_mem();
    double* q = r + k;
    const double* src = ref.qb + (size_t)m * a.s * k;
    for (int e = threadIdx.x; e < j * k; e += blockDim.x) q[e] = src[e];
    const double* rg = ref.r64 + (size_t)m * k;
    for (int row = threadIdx.x; row < k; row += blockDim.x) r[row] = rg[row];
}

// largest value over the block; every thread receives it
__device__ __forceinline__ float pick_max(PickSmem& sh, float v) {
    const unsigned int key = v >= 0.0f ? __float_as_uint(v) + 1u : 0u;
    const unsigned int w = __reduce_max_sync(0xffffffffu, key);
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) sh.fred[threadIdx.x >> 5] = __uint_as_float(w);
    __syncthreads();
    const unsigned int m = __reduce_max_sync(0xffffffffu, lane < warps ? __float_as_uint(sh.fred[lane]) : 0u);
    return m ? __uint_as_float(m - 1u) : -1.0f;
}

constexpr int kPickRows = kChunkMaxK / 32;            // rows of a column per lane

// this warp's copy of a column (scaled by sigma; rows beyond k are zero): lane holds the rows lane, lane + 32, ... (a generated word
// serves two rows, so it is worked out twice; in exchange the reads of the q_l are consecutive)
__device__ __forceinline__ void pick_column(const ChunkArgs& a, uint32_t col, double (&x)[kPickRows]) {
    const ColKey key = column_key(a.seed_lo, a.seed_hi, col);
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < kPickRows; ++u) {
        const int row = lane + 32 * u;
        x[u] = row < a.k ? a.sigma * (double)z_at(key, (uint32_t)row) : 0.0;
    }
}
// this lane's part of <v, x>
__device__ __forceinline__ double pick_dot(const ChunkArgs& a, const double* v, const double (&x)[kPickRows]) {
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
#pragma unroll
    for (int u = 0; u < kPickRows; ++u) if (lane + 32 * u < a.k) acc = fma(v[lane + 32 * u], x[u], acc);
    return acc;
}
// c_l = <q_l, a> for all earlier picks: warp = two vectors at a time
__device__ __forceinline__ void pick_products(const ChunkArgs& a, PickSmem& sh, const double* qs, int j, const double (&x)[kPickRows]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    for (int l = warp; l < j; l += 2 * warps) {
        const int l2 = l + warps < j ? l + warps : l;
        double c0 = pick_dot(a, qs + (size_t)l * a.k, x), c1 = pick_dot(a, qs + (size_t)l2 * a.k, x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { c0 += __shfl_xor_sync(0xffffffffu, c0, o); c1 += __shfl_xor_sync(0xffffffffu, c1, o); }
        if (lane == 0) { sh.cs[l] = c0; sh.cs[l2] = l2 != l ? c1 : c0; }
    }
}

// the decision among the nc candidates in sh.cidx and the update of the recovery `res` with the winner as pick j
// (all threads of the block; nc is the same in every thread; pick_stage has run for this recovery)
__device__ void pick_finish(const ChunkArgs& a, const ChunkRef& ref, PickSmem& sh, int res, int j, int nc) {
    const int m = res & 1, t = threadIdx.x, lane = t & 31, warp = t >> 5, warps = blockDim.x >> 5, k = a.k, s = a.s;
    if (nc == 0) {                                                   // no column left to pick (d/c = iterations made)
        if (t == 0) { ref.cnt->stopped[m] = 1; ref.cnt->done[m] = j; }
        return;
    }
    double* r = pick_mem();
    double* qs = r + k;
    __syncthreads();                                                 // the staged state and the candidates are complete
    double x[kPickRows];
    // exact scores (warp = one candidate, the last warp takes the first), and the products of the first candidate with the q_l
    for (int c = (warps - 1) - warp; c < nc; c += warps) {
        pick_column(a, sh.cidx[c], x);
        double dot = pick_dot(a, r, x), n2 = 0.0;
#pragma unroll
        for (int u = 0; u < kPickRows; ++u) n2 = fma(x[u], x[u], n2);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { dot += __shfl_xor_sync(0xffffffffu, dot, o); n2 += __shfl_xor_sync(0xffffffffu, n2, o); }
        if (lane == 0) { sh.cdot[c] = dot; sh.cn2[c] = n2; }
    }
    if (warp < j) { pick_column(a, sh.cidx[0], x); pick_products(a, sh, qs, j, x); }
    __syncthreads();
    int win = 0;
    {
        double best = -1.0;
        for (int c = 0; c < nc; ++c) {
            const double sc = sh.cn2[c] > 0.0 ? sh.cdot[c] * sh.cdot[c] / sh.cn2[c] : 0.0;
            if (sc > best || (sc == best && sh.cidx[c] < sh.cidx[win])) { best = sc; win = c; }
        }
    }
    const uint32_t col = sh.cidx[win];
    const double dot = sh.cdot[win], n2 = sh.cn2[win];
    if (win != 0 && j > 0) {
        __syncthreads();                                             // (a slow warp may still be reading sums of the first candidate)
        if (warp < j) { pick_column(a, col, x); pick_products(a, sh, qs, j, x); }
        __syncthreads();
    }
    double csq = lane < j ? sh.cs[lane] * sh.cs[lane] : 0.0;         // (j < 32)
    csq = warp_sum_d(csq);
    const double piv = n2 - csq;
    if (!(piv > 1e-10 * n2)) {                                       // dependent column: this recovery ends with j picks
        if (t == 0) {
            ref.cnt->stopped[m] = 1; ref.cnt->done[m] = j;
            atomicOr(&ref.cnt->status, (unsigned int)SGC_STATUS_DEPENDENT_COLUMN);
        }
        return;
    }
    const double gamma = rsqrt(piv), aj = gamma * dot;
    double rv = 0.0;                                                 // row t of the new residual (pick_threads: at least k threads)
    if (t < k) {
        const int row = t;
        double v0 = 0.0, v1 = 0.0;
        int l = 0;
#pragma unroll 4
        for (; l + 1 < j; l += 2) { v0 = fma(sh.cs[l], qs[l * k + row], v0); v1 = fma(sh.cs[l + 1], qs[(l + 1) * k + row], v1); }
        if (l < j) v0 = fma(sh.cs[l], qs[l * k + row], v0);
        const double q = gamma * (a.sigma * (double)z_at(column_key(a.seed_lo, a.seed_hi, col), (uint32_t)row) - (v0 + v1));
        ref.qb[((size_t)m * s + j) * k + row] = q;
        rv = r[row] - aj * q;
        ref.r64[(size_t)m * k + row] = rv;
    }
    if (t < j) ref.crow[((size_t)m * s + j) * s + t] = sh.cs[t];
    if (t == 0) {
        a.lam[(size_t)res * s + j] = col;
        ref.gam[(size_t)m * s + j] = gamma; ref.acoef[(size_t)m * s + j] = aj; ref.lam[(size_t)m * s + j] = col;
        ref.cnt->done[m] = j + 1;
    }
    const double part = warp_sum_d(rv * rv);
    if (lane == 0) sh.red[warp] = part;
    __syncthreads();
    double rn2 = 0.0;
    for (int w = 0; w < warps; ++w) rn2 += sh.red[w];
    const double rn = sqrt(rn2), sc = frag_scale(rn);
    if (t < k) frag_write(a, res, t, rv, sc);
    if (t == 0) { ref.rnorm[(size_t)m * s + j] = rn; a.back[res] = (float)(1.0 / sc); }
}

// What hardly any pick needs, out of the way of the others.  thr = 0: a zero residual; all scores are equal, and the lowest free
// column it is (one of the first j + 1).  Otherwise: the columns of the splits in sh->redo once more, whose third key came too close;
// every free column with score >= thr that its split did not forward joins the candidates (fp64, thread = column; once in some 10^5
// picks of a noisy recovery).
__device__ __noinline__ void pick_rare(PickSmem* sh, const Cand* fwd, uint32_t seed_lo, uint32_t seed_hi, int k, uint32_t dc,
                                       uint32_t cols_per_split, const uint32_t* sup, int j, double thr) {
    auto taken = [&](uint32_t col) { bool v = false; for (int l = 0; l < j; ++l) v = v || sup[l] == col; return v; };
    if (thr == 0.0) {
        if (threadIdx.x < 32) {
            const unsigned int who = __ballot_sync(0xffffffffu, (int)threadIdx.x <= j && threadIdx.x < dc && !taken(threadIdx.x));
            if (threadIdx.x == 0 && who != 0u) { sh->cidx[0] = (uint32_t)(__ffs(who) - 1); sh->n_c = 1; }
        }
        __syncthreads();
        return;
    }
    const double* r = pick_mem();
    const int n_redo = sh->n_redo < 8 ? sh->n_redo : 8;              // (more than eight such splits hold more than kRescoreCap candidates by themselves)
    for (int q = 0; q < n_redo; ++q) {
        const uint32_t split = (uint32_t)sh->redo[q], f0 = fwd[2 * split].idx & ~kThirdMark, f1 = fwd[2 * split + 1].idx;
        const uint32_t col0 = split * cols_per_split, col1 = dc - col0 < cols_per_split ? dc : col0 + cols_per_split;
        for (uint32_t col = col0 + threadIdx.x; col < col1; col += blockDim.x) {
            const ColKey key = column_key(seed_lo, seed_hi, col);
            double dot = 0.0, n2 = 0.0;
            for (int row = 0; row < k; row += 2) {
                const float2 z = half2_bits_to_float2(z_pair_from_word(key.ck + (uint32_t)(row >> 1) * key.mk));
                dot = fma((double)z.x, r[row], dot); n2 = fma((double)z.x, (double)z.x, n2);
                if (row + 1 < k) { dot = fma((double)z.y, r[row + 1], dot); n2 = fma((double)z.y, (double)z.y, n2); }
            }
            if (!(n2 > 0.0) || fabs(dot) < thr * sqrt(n2) || col == f0 || col == f1 || taken(col)) continue;
            const int slot = atomicAdd(&sh->n_c, 1);
            if (slot < kRescoreCap) sh->cidx[slot] = col;
        }
    }
    __syncthreads();
}

// SIMT route: the candidates are the columns that phase A left within 2e-3 (relative) of the best fp32 score.
// only != nullptr: a second chance for the recoveries that the tensor-core route marked unresolved; skipped unless *gate
// names this iteration.
__global__ void __launch_bounds__(kPickMaxThreads, 4) k_chunk_pick(ChunkArgs a, int iter, const int* gate, const unsigned char* only) {
    __shared__ PickSmem sh;
    const int res = blockIdx.x, m = res & 1, t = threadIdx.x, j = iter;
    const ChunkRef ref = a.table[res >> 1];
    // what earlier picks left is complete when this grid starts (phase A, the kernel before this one, has waited for the last
    // pick, and lets this one's blocks in only then), so it can be fetched before waiting for phase A itself
    if (gate == nullptr) pick_stage(a, ref, m, j);
    if (t == 0) sh.n_c = sh.n_redo = 0;
    after_previous_kernel(a.early);
    if (gate != nullptr && *gate != a.epoch0 + iter) return;
    if (only != nullptr && !only[res]) return;
    if (ref.cnt->stopped[m]) return;
    if (gate != nullptr) pick_stage(a, ref, m, j);
    const Cand* cc = a.cand + (size_t)res * a.splits * 2;
    const int n_entries = a.splits * 2;
    float mx = -1.0f;
    Cand first[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        first[u].score = -1.0f; first[u].idx = kNoColumn;
        const int e = t + u * (int)blockDim.x;
        if (e < n_entries) { const float2 f = __ldcg(reinterpret_cast<const float2*>(cc + e)); first[u].score = f.x; first[u].idx = __float_as_uint(f.y); }
        if (first[u].idx != kNoColumn) mx = fmaxf(mx, first[u].score);
    }
    for (int e = t + 2 * (int)blockDim.x; e < n_entries; e += blockDim.x) if (cc[e].idx != kNoColumn) mx = fmaxf(mx, cc[e].score);
    mx = pick_max(sh, mx);                                          // (its barriers also publish n_c = 0)
    const float thr = mx - 2e-3f * fabsf(mx);
    auto offer = [&](const Cand& c, int e) {
        if (c.idx != kNoColumn && c.score >= thr && c.score > 0.0f) {
            const int slot = atomicAdd(&sh.n_c, 1);
            if (slot < kRescoreCap) sh.cidx[slot] = c.idx & ~kThirdMark;
            if ((c.idx & kThirdMark) && c.score >= mx * (1.0f - kKeyWindow)) {
                const int q = atomicAdd(&sh.n_redo, 1);
                if (q < 8) sh.redo[q] = e >> 1;
            }
        }
    };
    offer(first[0], t); offer(first[1], t + (int)blockDim.x);
    for (int e = t + 2 * (int)blockDim.x; e < n_entries; e += blockDim.x) offer(cc[e], e);
    __syncthreads();
    if (sh.n_redo > 0 || mx == 0.0f)
        pick_rare(&sh, cc, a.seed_lo, a.seed_hi, a.k, (uint32_t)a.dc, (uint32_t)a.cols_per_split, a.lam + (size_t)res * a.s, j, (double)thr);
    int nc = sh.n_c;
    if (nc > kRescoreCap) {
        if (t == 0) atomicOr(&ref.cnt->status, (unsigned int)SGC_STATUS_CANDIDATE_OVERFLOW);
        nc = kRescoreCap;
    }
    pick_finish(a, ref, sh, res, j, nc);
}

// ---- tensor-core route of phase A (k_c > 32) --------------------------------------------------------------------
// The contraction Z^T R of an iteration (all columns of A against the residuals of all recoveries) is what the screening
// pass of sgc_pass.cu computes on the tensor cores: k_chunk_rt lays the residuals out as its binary16 rows (each scaled
// by a power of two, rows k_c.. of the padded height zero) with a report threshold of z_rep noise deviations, the pass
// reports every (column, recovery) pair above it, and k_chunk_pick_rep takes the candidates from the reports: every
// column within twice the pass's error bound of the best report.  Whatever that cannot settle (no report, too many, a
// window that reaches below the threshold, a zero residual) is marked unresolved and goes through the fp32 route.
__global__ void __launch_bounds__(64) k_chunk_rt(ChunkArgs a, int n_rows, int iter) {
    __shared__ double red[2];
    const int row = blockIdx.x, t = threadIdx.x;
    const float inf = __int_as_float(0x7f800000);
    bool live = row < 2 * a.c;
    const ChunkRef* ref = live ? &a.table[row >> 1] : nullptr;
    if (live && ref->cnt->stopped[row & 1]) live = false;
    if (!live) {
        if (t == 0) { a.tau[row] = inf; a.rep_count[row] = 0u; if (row < 2 * a.c) a.unresolved[row] = 0; }
        return;
    }
    const double* r = ref->r64 + (size_t)(row & 1) * a.k;
    double rn2 = 0.0;
    for (int q = t; q < a.k; q += 64) rn2 += r[q] * r[q];
    rn2 = warp_sum_d(rn2);
    if ((t & 31) == 0) red[t >> 5] = rn2;
    __syncthreads();
    const double rn = sqrt(red[0] + red[1]);
    if (!(rn > 0.0) || !isfinite(rn)) {                               // nothing to screen: the fp32 route decides
        if (t == 0) { a.tau[row] = inf; a.rep_count[row] = 0u; a.unresolved[row] = 1; a.flags[0] = a.epoch0 + iter; }   // every writer of an iteration stores the same value
        return;
    }
    const double sc = residual_scale(rn);
    uint16_t* dst = a.rt + (size_t)row * a.kp64;
    for (int q = t; q < a.kp64; q += 64) dst[q] = q < a.k ? half_rn_bits(r[q] * sc) : (uint16_t)0;
    if (t == 0) {
        a.tau[row] = (float)(a.z_rep * rn / sqrt((double)a.k) * sc);
        a.inv_scale[row] = (float)(1.0 / sc);
        a.rep_count[row] = 0u;
        a.rnv[row] = rn;
        a.unresolved[row] = 0;
    }
}

__global__ void __launch_bounds__(kPickMaxThreads) k_chunk_pick_rep(ChunkArgs a, int iter) {
    __shared__ PickSmem sh;
    const int res = blockIdx.x, m = res & 1, t = threadIdx.x, j = iter;
    const ChunkRef ref = a.table[res >> 1];
    if (ref.cnt->stopped[m] || a.unresolved[res]) return;
    pick_stage(a, ref, m, j);
    const unsigned int count = a.rep_count[res];
    const bool timed_out = a.flags[1] != 0;                          // a wait inside a pass of this step ran out: its reports are void
    bool give_up = timed_out || count == 0u || count > (unsigned int)kChunkRepCap;      // the same in every thread
    const uint2* rp = a.rep + (size_t)res * kChunkRepCap;
    const uint32_t* sup = ref.lam + (size_t)m * a.s;
    float smax = -1.0f;
    if (!give_up) {
        for (unsigned int e = t; e < count; e += blockDim.x) {
            const uint2 v = rp[e];
            bool taken = false;
            for (int q = 0; q < j; ++q) taken |= (sup[q] == v.x);
            if (!taken) smax = fmaxf(smax, __uint_as_float(v.y));
        }
        smax = pick_max(sh, smax);
        if (smax < 0.0f) give_up = true;
    }
    float lo = 0.0f;
    if (!give_up) {
        const double rn = a.rnv[res];
        lo = (float)((double)smax - 2.0 * screen_margin(rn, (double)smax, a.kp64));
        // the window must stay above the report threshold, or a column inside it may not have been reported
        if (!((double)lo > a.z_rep * rn / sqrt((double)a.k) * 1.001)) give_up = true;
    }
    if (!give_up) {
        if (t == 0) sh.n_c = 0;
        __syncthreads();
        for (unsigned int e = t; e < count; e += blockDim.x) {
            const uint2 v = rp[e];
            if (__uint_as_float(v.y) < lo) continue;
            bool taken = false;
            for (int q = 0; q < j; ++q) taken |= (sup[q] == v.x);
            if (taken) continue;
            const int slot = atomicAdd(&sh.n_c, 1);
            if (slot < kRescoreCap) sh.cidx[slot] = v.x;
        }
        __syncthreads();
        if (sh.n_c > kRescoreCap) give_up = true;
    }
    if (give_up) {
        if (t == 0) {
            a.unresolved[res] = 1; a.flags[0] = a.epoch0 + iter;
            if (timed_out) atomicOr(&ref.cnt->status, (unsigned int)SGC_STATUS_TIMEOUT);
        }
        return;
    }
    pick_finish(a, ref, sh, res, j, sh.n_c);
}

// ---- a5: coefficients and Eq. (8) on the common support of the two recoveries of a chunk, one block of two warps per chunk ----
__global__ void __launch_bounds__(64) k_chunk_scatter(ChunkArgs a, float* __restrict__ weight, double alpha, double eps, double lr) {
    __shared__ uint32_t vidx[kChunkMaxS], lam_s[2][kChunkMaxS];
    __shared__ double x_s[2][kChunkMaxS];
    extern __shared__ double rows_s[];                                // [2][s][s]
    after_previous_kernel(0);
    const int ch = blockIdx.x, lane = threadIdx.x & 31, m = threadIdx.x >> 5, s = a.s;
    const ChunkRef ref = chunk_ref(a, ch);
    float* W = weight + (size_t)ch * a.dc;
    const int done[2] = {ref.cnt->done[0], ref.cnt->done[1]}, n = done[m];
    // warp = recovery, lane = pick: x_l = gamma_l (a_l - sum_{j > l} c^(j)_l x_j), last pick first
    {
        double* rows = rows_s + (size_t)m * s * s;
        {
            const double* src = ref.crow + (size_t)m * s * s;
#pragma unroll 8
            for (int e = lane; e < n * s; e += 32) rows[e] = src[e];
        }
        const uint32_t col = lane < n ? ref.lam[(size_t)m * s + lane] : kNoColumn;
        double acc = lane < n ? ref.acoef[(size_t)m * s + lane] : 0.0, x = 0.0;
        const double gam = lane < n ? ref.gam[(size_t)m * s + lane] : 0.0;
        __syncwarp();
        for (int j = n - 1; j >= 0; --j) {
            const double xj = __shfl_sync(0xffffffffu, gam * acc, j);
            if (lane == j) x = xj;
            if (lane < j) acc = fma(-rows[(size_t)j * s + lane], xj, acc);
        }
        x_s[m][lane] = x; lam_s[m][lane] = col;
        if (lane < s) { ref.x[(size_t)m * s + lane] = x; if (lane >= n) ref.lam[(size_t)m * s + lane] = kNoColumn; }   // unpicked slots read as "none"
    }
    __syncthreads();
    if (m != 0) return;
    bool mis = false, neg = false, upd = false;
    double val = 0.0;
    const uint32_t mine = lam_s[0][lane];
    if (lane < done[0]) {
        int hit = -1;
        for (int b = 0; b < done[1]; ++b) if (lam_s[1][b] == mine) { hit = b; break; }
        if (hit < 0) mis = true;
        else {
            const double xv = x_s[1][hit];
            if (!(xv > 0.0)) neg = true;
            else { val = lr * (alpha * x_s[0][lane] / (sqrt(xv) + eps)); upd = true; }
        }
    }
    vidx[lane] = upd ? mine : kNoColumn;
    __syncwarp();
    const int n_mis = __popc(__ballot_sync(0xffffffffu, mis)), n_neg = __popc(__ballot_sync(0xffffffffu, neg));
    const int n_valid = __popc(__ballot_sync(0xffffffffu, upd));
    if (upd) {
        int rank = 0;
        for (int b = 0; b < done[0]; ++b) rank += vidx[b] < mine ? 1 : 0;
        ref.upd_idx[rank] = mine;
        ref.upd_val[rank] = val;
        W[mine] = (float)((double)W[mine] - val);
    }
    if (lane == 0) {
        ref.cnt->n_upd = n_valid; ref.cnt->mismatch = n_mis; ref.cnt->negv = n_neg;
        unsigned int bits = 0;
        if (n_mis > 0 || done[0] != done[1]) bits |= (unsigned int)SGC_STATUS_SUPPORT_MISMATCH;
        if (n_neg > 0) bits |= (unsigned int)SGC_STATUS_NEGATIVE_V;
        if (bits) atomicOr(&ref.cnt->status, bits);
    }
}

}  // namespace

// ---- host side ----------------------------------------------------------------------------------------------
namespace {

unsigned long long list_key(sgc_state* const* sts, int c) {
    unsigned long long h = 1469598103934665603ull;                   // FNV-1a
    for (int i = 0; i < c; ++i) {                                     // host object and its device allocation
        h ^= (unsigned long long)(uintptr_t)sts[i]; h *= 1099511628211ull;
        h ^= (unsigned long long)(uintptr_t)sts[i]->base; h *= 1099511628211ull;
    }
    h ^= sts[0]->seed; h *= 1099511628211ull;                        // the norm table belongs to one matrix
    return h ^ (unsigned long long)c;
}

template <int KP>
cudaError_t corr_setup(size_t* smem_out) {
    constexpr int TC = corr_tile(KP), KB = corr_kb(KP);
    const size_t smem = (size_t)(TC / 16) * KB * 512 + (size_t)(2 * TC + KB * TC) * sizeof(float);
    *smem_out = smem;
    return cudaFuncSetAttribute(k_chunk_corr<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// blocks of k_chunk_corr<KP> that one SM holds at a time (0 on an error)
template <int KP>
int corr_resident() {
    size_t smem = 0;
    int blocks = 0;
    if (corr_setup<KP>(&smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_chunk_corr<KP>, corr_threads(KP), smem) != cudaSuccess) return 0;
    return blocks;
}

int corr_resident(int kp) {
    switch (kp) {
        case 8: return corr_resident<8>();
        case 16: return corr_resident<16>();
        case 32: return corr_resident<32>();
        case 64: return corr_resident<64>();
        case 128: return corr_resident<128>();
        default: return corr_resident<256>();
    }
}

template <int KP>
cudaError_t corr_launch(const ChunkArgs& a, int iter, size_t smem, cudaStream_t stream, const int* gate) {
    dim3 grid((unsigned int)a.splits, (unsigned int)((2 * a.c + corr_group(KP) - 1) / corr_group(KP)));
    ChainedLaunch l(grid, dim3((unsigned int)corr_threads(KP)), smem, stream);
    return cudaLaunchKernelEx(&l.cfg, k_chunk_corr<KP>, a, iter, gate);
}

ChunkRef ref_of(const sgc_state* st) {
    ChunkRef r;
    r.M = st->M; r.V = st->V; r.p = st->p; r.q = st->q; r.y64 = st->y64; r.r64 = st->r64;
    r.sel_idx = st->sel_idx; r.sel_val = st->sel_val;
    r.qb = st->q_basis; r.lam = st->lam; r.crow = st->F; r.gam = st->gam; r.acoef = st->acoef; r.x = st->x; r.rnorm = st->rnorm;
    r.upd_idx = st->upd_idx; r.upd_val = st->upd_val; r.cnt = st->cnt; r.ctl = st->ctl;
    return r;
}

// Shape of the cluster form for c chunks like st0's (cl == 0: they take the launches of the general form, because a cluster has no
// room for A, or because so many recoveries share it that scoring, which all SMs do there, outweighs the launches).  us per step,
// general / cluster form:  64 chunks of 2048, k = 217, s = 31: 647 / 456 (with 140 of projection);  100 of 412, 119, 17: 254 / 132;
// 16 of 40520, 28, 4: 85 / 58;  300 of 2068, 200, 25: 783 / 550;  100 of 24712, 14, 2: 47 / 54;  300 of 3276, 21, 3: 53 / 56;
// 256 of 65536, 8, 1: 52 / 83;  one of 4096, 256, 16: 212 / 111 (the general form of a single vector is the lock-step recovery).
ChunkPlan plan_for(const sgc_state* st0, int c) {
    const double general = chunk_general_us(c, st0->d, st0->k, st0->s, st0->sm_count);
    auto better = [&](const ChunkPlan& p) { return cluster_form_taken(p, c, general); };
    // what a device of this size holds as a rule; it is asked (some ms, once per process) only where that form would be taken
    const int rule[kChunkShapes] = {st0->sm_count, st0->sm_count / 2, st0->sm_count * 2 / 9, st0->sm_count / 9, st0->sm_count / 18};
    if (!better(chunk_plan(c, st0->d, st0->k, st0->s, rule))) return ChunkPlan{};
    int resident[kChunkShapes];
    if (chunk_cluster_configure(st0->device, resident) != cudaSuccess) { cudaGetLastError(); return ChunkPlan{}; }
    const ChunkPlan p = chunk_plan(c, st0->d, st0->k, st0->s, resident);
    return better(p) ? p : ChunkPlan{};
}

// Shape of the whole-GPU form (blocks == 0: the launches of the general form, see grid_form_taken).
GridPlan grid_plan_for(const sgc_state* st0, int c) {
    const GridPlan p = grid_plan(c, st0->d, st0->k, st0->s, st0->sm_count);
    if (!grid_form_taken(p, st0->k, chunk_launches_us(c, st0->d, st0->k, st0->s, st0->sm_count))) return GridPlan{};
    bool fits = false;
    if (chunk_grid_configure(st0->device, p.kc, &fits) != cudaSuccess || !fits) { cudaGetLastError(); return GridPlan{}; }
    return p;
}

// builds (or reuses) the workspace for this chunk list; the first build synchronises (one allocation, one copy)
cudaError_t ensure_ws(sgc_state* const* sts, int c) {
    sgc_state* st0 = sts[0];
    const unsigned long long key = list_key(sts, c);
    if (st0->chunk_ws && st0->chunk_ws->key == key && st0->chunk_ws->c == c) return cudaSuccess;
    {
        std::vector<sgc_state*> sorted(sts, sts + c);                // a state may appear once only
        std::sort(sorted.begin(), sorted.end());
        for (int i = 1; i < c; ++i) if (sorted[i] == sorted[i - 1]) return cudaErrorInvalidValue;
    }
    free_chunk_ws(st0);
    ChunkWs* ws = new (std::nothrow) ChunkWs();
    if (!ws) return cudaErrorMemoryAllocation;
    ws->c = c; ws->key = key; ws->kp = chunk_padded_k(st0->k);
    ws->plan = plan_for(st0, c);
    if (ws->plan.cl == 0) ws->grid = grid_plan_for(st0, c);
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t b_table = up((size_t)c * sizeof(ChunkRef));
    std::vector<ChunkRef> host((size_t)c);
    for (int i = 0; i < c; ++i) host[i] = ref_of(sts[i]);
    if (ws->plan.cl > 0) {
        cudaError_t e = cudaMalloc(&ws->base, b_table);
        if (e != cudaSuccess) { delete ws; return e; }
        ws->table = static_cast<ChunkRef*>(ws->base);
        e = cudaMemcpy(ws->table, host.data(), (size_t)c * sizeof(ChunkRef), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();           // (a copy from pageable memory returns before it has arrived)
        if (e != cudaSuccess) { cudaFree(ws->base); delete ws; return e; }
        st0->chunk_ws = ws;
        return cudaSuccess;
    }
    if (ws->grid.blocks > 0) {
        const size_t rows = (size_t)ws->grid.mt * 128;
        ws->kp64 = ws->grid.kc * 64;
        const size_t b_rt = up(rows * ws->kp64 * sizeof(uint16_t)), b_row = up(rows * sizeof(float)), b_rep = up((size_t)2 * c * kChunkRepCap * sizeof(uint2));
        const size_t total = b_table + b_rt + 2 * b_row + b_rep + 256;
        cudaError_t e = cudaMalloc(&ws->base, total);
        if (e == cudaSuccess) {
            unsigned char* base = static_cast<unsigned char*>(ws->base);
            ws->table = reinterpret_cast<ChunkRef*>(base);
            ws->rt = reinterpret_cast<uint16_t*>(base + b_table);
            ws->tau = reinterpret_cast<float*>(base + b_table + b_rt);
            ws->rep_count = reinterpret_cast<unsigned int*>(base + b_table + b_rt + b_row);
            ws->rep = reinterpret_cast<uint2*>(base + b_table + b_rt + 2 * b_row);
            ws->flags = reinterpret_cast<int*>(base + b_table + b_rt + 2 * b_row + b_rep);
            // 20 noise columns per recovery above the threshold: none at all, which sends a recovery through all columns, once in 5e8 picks
            ws->z_rep = sphere_tail_threshold((double)st0->d, st0->k, 20.0);
            std::vector<float> never(rows, INFINITY);                // rows without a recovery screen nothing
            e = cudaMemset(ws->base, 0, total);
            if (e == cudaSuccess) e = cudaMemcpy(ws->tau, never.data(), rows * sizeof(float), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) e = cudaMemcpy(ws->table, host.data(), (size_t)c * sizeof(ChunkRef), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) e = cudaDeviceSynchronize();       // set-up done before the caller's stream runs on it
            if (e != cudaSuccess) { cudaFree(ws->base); delete ws; return e; }
            st0->chunk_ws = ws;
            return cudaSuccess;
        }
        cudaGetLastError();                                          // no room for the report lists: the general form does without them
        ws->base = nullptr; ws->grid = GridPlan{};
    }
    // column splits: as many blocks as the SMs hold at a time (one wave), at least one tile per split
    const int groups = (2 * c + corr_group(ws->kp) - 1) / corr_group(ws->kp);
    constexpr int tile = 16;                                         // columns that an operand of the correlation holds
    int resident = corr_resident(ws->kp);
    if (resident < 1) { delete ws; return cudaErrorLaunchOutOfResources; }
    // with few columns per SM one block each will do: the kernel that follows then finds room beside it (see `early`)
    if ((double)st0->d * groups <= 256.0 * st0->sm_count) resident = 1;
    int splits = resident * st0->sm_count / groups;
    const long long max_splits = (st0->d + tile - 1) / tile;
    if (splits > max_splits) splits = (int)max_splits;
    if (splits < 1) splits = 1;
    long long per = (st0->d + splits - 1) / splits;
    per = (per + tile - 1) / tile * tile;
    splits = (int)((st0->d + per - 1) / per);
    ws->splits = splits;
    const int kf = ws->kp < 16 ? 16 : ws->kp;
    const size_t b_frag = up((size_t)2 * c * 2 * kf * sizeof(uint16_t)), b_back = up((size_t)2 * c * sizeof(float));
    const size_t b_cand = up((size_t)2 * c * splits * 2 * sizeof(Cand));
    const size_t b_lam = up((size_t)2 * c * st0->s * sizeof(uint32_t));
    // tensor-core route: worth it from k_c = 33 on; bounded by its report lists (n_rows * 16 KB)
    // (a pass has some 40 us of fixed cost: below ~1e9 multiply-adds per iteration the fp32 kernel is quicker)
    ws->tensor = chunk_on_tensor_cores(c, st0->d, ws->kp);
    ws->kp64 = (st0->k + 63) / 64 * 64;
    ws->n_rows = (2 * c + 31) / 32 * 32;
    ws->passes = chunk_passes(c);
    size_t b_rt = 0, b_row = 0, b_rep = 0, b_norm = 0, b_rn = 0, b_un = 0, b_flags = 0;
    if (ws->tensor) {
        b_rt = up((size_t)ws->n_rows * ws->kp64 * sizeof(uint16_t));
        b_row = up((size_t)ws->n_rows * sizeof(float));
        b_rep = up((size_t)ws->n_rows * kChunkRepCap * sizeof(uint2));
        b_norm = up((size_t)st0->d * sizeof(uint16_t));
        b_rn = up((size_t)2 * c * sizeof(double));
        b_un = up((size_t)2 * c);
        b_flags = 256;
    }
    cudaError_t e = cudaMalloc(&ws->base, b_table + b_frag + b_back + b_cand + b_lam + b_rt + 3 * b_row + b_rep + b_norm + b_rn + b_un + b_flags);
    if (e != cudaSuccess) { delete ws; return e; }
    unsigned char* base = static_cast<unsigned char*>(ws->base);
    size_t off = 0;
    ws->table = reinterpret_cast<ChunkRef*>(base + off); off += b_table;
    ws->frag = reinterpret_cast<uint16_t*>(base + off); off += b_frag;
    ws->back = reinterpret_cast<float*>(base + off); off += b_back;
    ws->cand = reinterpret_cast<Cand*>(base + off); off += b_cand;
    ws->lam = reinterpret_cast<uint32_t*>(base + off); off += b_lam;
    if (ws->tensor) {
        ws->rt = reinterpret_cast<uint16_t*>(base + off); off += b_rt;
        ws->tau = reinterpret_cast<float*>(base + off); off += b_row;
        ws->inv_scale = reinterpret_cast<float*>(base + off); off += b_row;
        ws->rep_count = reinterpret_cast<unsigned int*>(base + off); off += b_row;
        ws->rep = reinterpret_cast<uint2*>(base + off); off += b_rep;
        ws->inv_norm = reinterpret_cast<uint16_t*>(base + off); off += b_norm;
        ws->rnv = reinterpret_cast<double*>(base + off); off += b_rn;
        ws->unresolved = base + off; off += b_un;
        ws->flags = reinterpret_cast<int*>(base + off); off += b_flags;
        ws->z_rep = normal_tail_threshold((double)st0->d, 32.0);    // ~32 noise columns per recovery above the threshold
        const int h_flags[3] = {0, 0, 1};
        e = pass_configure(kPassMaxN);
        if (e == cudaSuccess) e = cudaMemset(ws->rt, 0, b_rt);
        if (e == cudaSuccess) e = cudaMemset(ws->unresolved, 0, b_un);
        if (e == cudaSuccess) e = cudaMemcpy(ws->flags, h_flags, sizeof(h_flags), cudaMemcpyHostToDevice);
        for (int p = 0; p < ws->passes && e == cudaSuccess; ++p) {
            const int n_p = ws->n_rows - p * kPassMaxN < kPassMaxN ? ws->n_rows - p * kPassMaxN : kPassMaxN;
            e = pass_encode_map(ws->tmap[p], ws->rt + (size_t)p * kPassMaxN * ws->kp64, n_p, ws->kp64);
        }
        if (e == cudaSuccess) e = launch_inv_norms(st0->seed, (uint64_t)st0->d, st0->k, ws->inv_norm, 0);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();           // the table is ready before any stream uses it
        if (e != cudaSuccess) { cudaFree(ws->base); delete ws; return e; }
    }
    e = cudaMemcpy(ws->table, host.data(), (size_t)c * sizeof(ChunkRef), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(ws->frag, 0, b_frag);       // rows k..kf of every residual stay zero
    if (e == cudaSuccess) e = cudaDeviceSynchronize();               // set-up done before the caller's stream runs on it
    if (e != cudaSuccess) { cudaFree(ws->base); delete ws; return e; }
    st0->chunk_ws = ws;
    return cudaSuccess;
}

}  // namespace

void free_chunk_ws(sgc_state* st) {
    if (!st || !st->chunk_ws) return;
    cudaFree(st->chunk_ws->base);
    delete st->chunk_ws;
    st->chunk_ws = nullptr;
}

// The batched path serves chunk lists whose states are alike in everything but their moments: same shape, matrix, step
// count and hyper-parameters, Algorithm 2 as printed, small s and k, and no request for the speculative recovery.
bool chunk_sized(const sgc_state* st) { return st->s <= kChunkMaxS && st->k <= kChunkMaxK; }

bool chunked_batch_eligible(sgc_state* const* sts, int c) {
    const sgc_state* a = sts[0];
    if (!chunk_sized(a) || (a->d & 3) || a->d >= (1ll << 31) || c > (1 << 20)) return false;
    for (int i = 0; i < c; ++i) {
        const sgc_state* b = sts[i];
        if (b->mode == SGC_MODE_SPECULATIVE || b->shared_support || b->residual_tol > 0.0 || b->profile) return false;
        if (b->d != a->d || b->k != a->k || b->s != a->s || b->seed != a->seed || b->t != a->t || b->lr != a->lr ||
            b->beta1 != a->beta1 || b->beta2 != a->beta2 || b->eps != a->eps || b->alpha != a->alpha || b->device != a->device)
            return false;
    }
    return true;
}

// arguments that every form of the step needs
static ChunkArgs common_args(const sgc_state* st0, int c) {
    ChunkArgs a;
    memset(&a, 0, sizeof(a));
    a.c = c; a.k = st0->k; a.s = st0->s; a.kp = chunk_padded_k(st0->k); a.dc = st0->d;
    a.seed_lo = (uint32_t)(st0->seed & 0xFFFFFFFFu); a.seed_hi = (uint32_t)(st0->seed >> 32);
    a.sigma = (double)(float)(1.0 / sqrt((double)st0->k));
    a.wait_ns = st0->wait_limit_ns;
    return a;
}

static cudaError_t launch_front(const sgc_state* st0, ChunkArgs& a, bool cluster_next, const float* grad, cudaStream_t stream, int* launches) {
    const double b1 = (double)st0->beta1, b2 = (double)st0->beta2;
    const double c1 = 1.0 - pow(b1, (double)st0->t), c2 = 1.0 - pow(b2, (double)st0->t);
    // blocks per chunk: up to two blocks per SM, at least four vectors per thread (256 chunks of 65536 in 512 blocks: 22 -> 35 us)
    int split = 1;
    while (split < kFrontMaxSplit && 2 * split * a.c <= 2 * st0->sm_count && st0->d >= (int64_t)2 * split * kFrontThreads * 16) split *= 2;
    // (blocks of the next kernel that wait must not hold the places of this one's)
    a.early_front = cluster_next && a.c * split <= st0->sm_count ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)(a.c * split)); cfg.blockDim = dim3(kFrontThreads); cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_chunk_front, a, grad, b1, b2, c1, c2);
    if (e == cudaSuccess) *launches += 1;
    return e;
}

static cudaError_t launch_scatter(const sgc_state* st0, const ChunkArgs& a, float* weight, cudaStream_t stream, int* launches) {
    ChainedLaunch l(dim3((unsigned int)a.c), dim3(64), (size_t)2 * a.s * a.s * sizeof(double), stream);
    const cudaError_t e = cudaLaunchKernelEx(&l.cfg, k_chunk_scatter, a, weight, (double)st0->alpha, (double)st0->eps, (double)st0->lr);
    if (e != cudaSuccess) return e;
    *launches += 1;
    return cudaGetLastError();
}

static void set_form(sgc_state* st, int form, int batches, int warps, int q_shared) {
    st->form[0] = form; st->form[1] = batches; st->form[2] = warps; st->form[3] = q_shared;
}

// A single small state as a list of one chunk: selection, projection and moments in one launch, the recovery in one cluster.  It is what a
// state that recovers in lock-step does, faster (see k_chunk_cluster): a state that speculates, or has, keeps lists that this form does
// not know.
static bool small_step_plan(const sgc_state* st, ChunkPlan* plan) {
    if (!chunk_sized(st) || st->d >= (1ll << 31) || st->mode == SGC_MODE_SPECULATIVE || st->shared_support || st->residual_tol > 0.0 ||
        st->profile || st->spec_ready || will_speculate(st))
        return false;
    *plan = plan_for(st, 1);
    return plan->cl > 0;
}
bool takes_small_step(const sgc_state* st) { ChunkPlan p; return small_step_plan(st, &p); }
cudaError_t launch_small_step(sgc_state* st, const float* grad, float* weight, cudaStream_t stream, int* launches) {
    ChunkPlan plan;
    if (!small_step_plan(st, &plan)) return cudaErrorInvalidConfiguration;
    ChunkArgs a = common_args(st, 1);
    a.one = ref_of(st);
    cudaError_t e = launch_front(st, a, true, grad, stream, launches);
    if (e == cudaSuccess) e = launch_chunk_cluster(a, plan, true, stream);
    if (e != cudaSuccess) return e;
    *launches += 1;
    set_form(st, 3, plan.batches, plan.gw, plan.q_shared);
    return launch_scatter(st, a, weight, stream, launches);
}

// One step of all chunks (the caller has already advanced every state's step count).
cudaError_t launch_chunked_batch(sgc_state* const* sts, int c, const float* grad, float* weight, cudaStream_t stream,
                                 int* launches) {
    sgc_state* st0 = sts[0];
    cudaError_t e = ensure_ws(sts, c);
    if (e != cudaSuccess) return e;
    const ChunkWs* ws = st0->chunk_ws;
    ChunkArgs a = common_args(st0, c);
    a.table = ws->table;
    for (int i = 0; i < c; ++i)
        if (ws->plan.cl > 0) set_form(sts[i], 3, ws->plan.batches, ws->plan.gw, ws->plan.q_shared);
        else if (ws->grid.blocks > 0) set_form(sts[i], 4, 0, ws->grid.gw, 0);
        else set_form(sts[i], ws->tensor ? 2 : 1, 0, 0, 0);
    if (ws->plan.cl > 0) {
        e = launch_front(st0, a, true, grad, stream, launches);
        if (e != cudaSuccess) return e;                              // (nothing is counted: the caller takes the step count back)
        e = launch_chunk_cluster(a, ws->plan, true, stream);
        if (e != cudaSuccess) return e;
        *launches += 1;
        return launch_scatter(st0, a, weight, stream, launches);
    }
    if (ws->grid.blocks > 0) {
        a.kp64 = ws->kp64; a.rt = ws->rt; a.tau = ws->tau; a.rep_count = ws->rep_count; a.rep = ws->rep; a.flags = ws->flags; a.z_rep = ws->z_rep;
        e = launch_front(st0, a, false, grad, stream, launches);
        if (e != cudaSuccess) return e;
        e = launch_chunk_grid(a, ws->grid, stream);
        if (e != cudaSuccess) return e;
        *launches += 1;
        return launch_scatter(st0, a, weight, stream, launches);
    }
    a.frag = ws->frag; a.back = ws->back; a.kf = ws->kp < 16 ? 16 : ws->kp; a.cand = ws->cand; a.lam = ws->lam; a.splits = ws->splits;
    {
        const int groups = (2 * c + corr_group(ws->kp) - 1) / corr_group(ws->kp);
        a.early = (ws->splits * groups <= st0->sm_count && 2 * c <= st0->sm_count) ? 1 : 0;
    }
    a.cols_per_split = (int)((st0->d + ws->splits - 1) / ws->splits);
    a.cols_per_split = (a.cols_per_split + 15) / 16 * 16;
    a.kp64 = ws->kp64; a.rt = ws->rt; a.tau = ws->tau; a.inv_scale = ws->inv_scale; a.rep_count = ws->rep_count; a.rep = ws->rep;
    a.rnv = ws->rnv; a.unresolved = ws->unresolved; a.flags = ws->flags; a.z_rep = ws->z_rep;
    // names the iterations of this step in the gate word: 1 + (step count mod 2^20) * 64 + iteration, never 0
    a.epoch0 = 1 + (int)((st0->t & 0xFFFFF) * 64);
    if (ws->tensor) {
        e = cudaMemsetAsync(ws->flags + 1, 0, sizeof(int), stream);      // the time-out flag is per step
        if (e != cudaSuccess) return e;
    }
    const int s = st0->s;
    e = launch_front(st0, a, false, grad, stream, launches);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_chunk_pick, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pick_dyn_bytes(kChunkMaxS, kChunkMaxK));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_chunk_pick_rep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pick_dyn_bytes(kChunkMaxS, kChunkMaxK));
    if (e != cudaSuccess) return e;
    size_t smem = 0;
    switch (ws->kp) {
        case 8: e = corr_setup<8>(&smem); break;
        case 16: e = corr_setup<16>(&smem); break;
        case 32: e = corr_setup<32>(&smem); break;
        case 64: e = corr_setup<64>(&smem); break;
        case 128: e = corr_setup<128>(&smem); break;
        default: e = corr_setup<256>(&smem); break;
    }
    if (e != cudaSuccess) return e;
    for (int iter = 0; iter < s; ++iter) {
        const int* gate = nullptr;
        if (ws->tensor) {
            // phase A on the tensor cores; the fp32 kernels below then only run for what the reports left open
            k_chunk_rt<<<ws->n_rows, 64, 0, stream>>>(a, ws->n_rows, iter);
            const int* gates[kPassMaxBatch] = {ws->flags + 2};
            int* errors[kPassMaxBatch] = {ws->flags + 1};
            for (int p = 0; p < ws->passes && e == cudaSuccess; ++p) {
                const int n_p = ws->n_rows - p * kPassMaxN < kPassMaxN ? ws->n_rows - p * kPassMaxN : kPassMaxN;
                const size_t r0 = (size_t)p * kPassMaxN;
                e = launch_pass(ws->tmap[p], st0->seed, (uint64_t)st0->d, ws->kp64, n_p, ws->tau + r0, ws->inv_scale + r0,
                                ws->inv_norm, ws->rep_count + r0, ws->rep + r0 * kChunkRepCap, kChunkRepCap, gates, errors,
                                st0->sm_count, stream, nullptr, nullptr, 0, st0->wait_limit_ns);
            }
            if (e != cudaSuccess) return e;
            k_chunk_pick_rep<<<2 * c, pick_threads(st0->k), pick_dyn_bytes(s, st0->k), stream>>>(a, iter);
            *launches += 2 + ws->passes;
            gate = ws->flags;
        }
        switch (ws->kp) {
            case 8: e = corr_launch<8>(a, iter, smem, stream, gate); break;
            case 16: e = corr_launch<16>(a, iter, smem, stream, gate); break;
            case 32: e = corr_launch<32>(a, iter, smem, stream, gate); break;
            case 64: e = corr_launch<64>(a, iter, smem, stream, gate); break;
            case 128: e = corr_launch<128>(a, iter, smem, stream, gate); break;
            default: e = corr_launch<256>(a, iter, smem, stream, gate); break;
        }
        {
            ChainedLaunch l(dim3((unsigned int)(2 * c)), dim3(pick_threads(st0->k)), pick_dyn_bytes(s, st0->k), stream);
            const unsigned char* only = gate ? ws->unresolved : nullptr;
            if (e == cudaSuccess) e = cudaLaunchKernelEx(&l.cfg, k_chunk_pick, a, iter, gate, only);
        }
        if (e != cudaSuccess) return e;
        *launches += 2;
    }
    return launch_scatter(st0, a, weight, stream, launches);
}

}  // namespace sgc
