// Shape of the chunk recovery on thread-block clusters (sgc_chunk_cluster.cu): plain integer arithmetic, which a C++ compiler
// without CUDA takes as well, so that it can be checked over every size the library accepts.
#pragma once

#include <math.h>
#include <stddef.h>
#include <stdint.h>

namespace sgc {

constexpr int kChunkMaxS = 32;
constexpr int kChunkMaxK = 256;
constexpr int kClusterWarps = 16;                     // warps per block of the cluster form
constexpr int kClusterTiles = 63;                     // column tiles of 16 per warp: a key has room for 1023 columns
constexpr int kChunkShapes = 5;                       // clusters of 1, 2, 4, 8 and 16 blocks
constexpr size_t kClusterSmem = 224 * 1024;           // dynamic shared memory of a block, at most
constexpr size_t kClusterHead = 32;                   // barriers
constexpr size_t kClusterBook = 1296;                 // a recovery's small records (ChunkBook)

struct ChunkPlan {
    int cl;                            // blocks per cluster; 0: the recoveries do not fit
    int clusters, per_cluster;         // clusters of the launch, chunks that each serves ...
    int batch, batches;                // ... so many at a time
    int cols, tiles, kb;               // columns of a block, the same in tiles of 16; 16-row blocks of A
    int nt;                            // tiles of four recoveries
    int slots;                         // warps that share the block's tiles; kClusterWarps / slots share the recoveries
    int own, gw;                       // recoveries whose books a block keeps, warps that work on one of them
    int kq;                            // rows of a vector, a multiple of 64
    int rec_bytes;                     // a residual as an operand, with what keeps the banks apart
    int cl_log, slots_log, quads_log;  // logarithms: cl, slots, 16-byte pieces of a residual (rounded up)
    int q_shared;                      // the orthogonal vectors are in shared memory (else in the chunk's own records)
    size_t off_inv, off_frag, off_top, off_ent, off_book, off_r, off_x, off_q, bytes;
    double us;                         // estimate of the whole launch
};

// resident[i]: clusters of 1 << i blocks that the device holds at a time (0: that shape is not available)
inline ChunkPlan chunk_plan(int c, long long dc, int k, int s, const int (&resident)[kChunkShapes]) {
    ChunkPlan best = {};
    auto up16 = [](size_t b) { return (b + 15) / 16 * 16; };
    for (int shape = 0; shape < kChunkShapes; ++shape) {
        if (resident[shape] < 1) continue;
        ChunkPlan p = {};
        p.cl = 1 << shape;
        p.kb = (k + 15) / 16;
        p.kq = (k + 63) / 64 * 64;
        p.cl_log = shape;
        p.rec_bytes = (p.kb | 1) * 64;
        while ((1 << p.quads_log) < 4 * p.kb) ++p.quads_log;
        const long long cols = (dc + p.cl - 1) / p.cl;
        if (cols > 1 << 20) continue;
        p.cols = (int)((cols + 15) / 16 * 16);
        p.tiles = p.cols / 16;
        const size_t b_z = (size_t)p.tiles * p.kb * 512, b_inv = (size_t)p.cols * sizeof(float);
        if (kClusterHead + b_z + b_inv > kClusterSmem) continue;
        p.per_cluster = (c + resident[shape] - 1) / resident[shape];
        p.clusters = (c + p.per_cluster - 1) / p.per_cluster;
        for (p.batches = 1; p.batches <= p.per_cluster; ++p.batches) {
            p.batch = (p.per_cluster + p.batches - 1) / p.batches;
            if (p.batches > 1 && (p.per_cluster + p.batches - 2) / (p.batches - 1) == p.batch) continue;
            p.nt = (2 * p.batch + 3) / 4;
            p.own = (2 * p.batch + p.cl - 1) / p.cl;
            p.gw = kClusterWarps;
            while (p.gw > 1 && p.gw * p.own > kClusterWarps) p.gw >>= 1;
            // how the warps share (tiles, recoveries): the fewest rounds of a warp
            long long rounds = 0;
            p.slots = p.slots_log = 0;
            for (int slots = 1; slots <= kClusterWarps; slots <<= 1) {
                const int share = kClusterWarps / slots, per = (p.tiles + slots - 1) / slots;
                const int parts = (p.nt + share - 1) / share;
                if (per > kClusterTiles) continue;
                const long long r = (long long)per * parts;
                if (p.slots == 0 || r <= rounds) { rounds = r; p.slots = slots; }
            }
            if (p.slots == 0) break;
            while ((1 << p.slots_log) < p.slots) ++p.slots_log;
            p.off_inv = kClusterHead + b_z;
            p.off_frag = up16(p.off_inv + b_inv);
            p.off_top = p.off_frag + (size_t)4 * (p.nt + 3) * p.rec_bytes;                 // (tiles of recoveries are taken up to four at a time)
            p.off_ent = p.off_top + (size_t)2 * p.batch * p.slots * 16;
            p.off_book = p.off_ent + (size_t)p.own * p.cl * 16;
            p.off_r = p.off_book + (size_t)p.own * kClusterBook;
            p.off_x = p.off_r + (size_t)p.own * p.kq * sizeof(double);               // (a column per team)
            p.off_q = p.off_x + (size_t)(kClusterWarps / p.gw) * p.kq * sizeof(double);
            const size_t q = (size_t)p.own * s * p.kq * sizeof(double);
            p.q_shared = p.off_q + q <= kClusterSmem ? 1 : 0;
            p.bytes = p.off_q + (p.q_shared ? q : 0);
            if (p.bytes <= kClusterSmem) break;
        }
        if (p.slots == 0 || p.batches > p.per_cluster || p.bytes > kClusterSmem) continue;
        // Cycles, from timings of the phases: a warp generates a tile; per iteration, a tile of columns meets a tile of recoveries, the
        // warps' findings are joined, books are kept (a group of warps takes own / groups of them one after the other), and what is
        // sent arrives; 8 us for the launch and what comes before the first pick.  (Wider clusters wait longer for
        // one another: 64 chunks of 2048, k = 217: clusters of 16 / 8: 464 / 456 us per step;  32 of 1920, 140: 16 / 8 / 4: 220 / 216 / 213.)
        const int groups = kClusterWarps / p.gw, turns = (p.own + groups - 1) / groups, lone = (p.tiles + kClusterWarps - 1) / kClusterWarps;
        const double gen = lone * (700.0 + 530.0 * p.kb);
        const double corr = 900.0 + (double)p.tiles * p.nt * (7.9 + 3.8 * p.kb) + 700.0 * ((2 * p.batch + 31) / 32);
        const double fewer = p.gw >= 16 ? 1.0 : p.gw == 8 ? 1.1 : p.gw == 4 ? 1.4 : p.gw == 2 ? 2.3 : 3.0;
        const double book = turns * (3800.0 + 0.6 * s * k) * fewer;
        p.us = 8.0 + (gen + (double)p.batches * s * (corr + book + 1000.0 + 70.0 * p.cl)) / 1.9e3;
        if (best.cl == 0 || p.us < best.us) best = p;
    }
    return best;
}

// Share z of ||r|| / sqrt(k) that `target` of d columns score at least, when the columns' directions are uniform on the sphere of k
// dimensions: the normal law's tail is too heavy for that (k = 112, d = 65536: 32 columns expected, 20 found; k = 40: 12).
inline double sphere_tail_threshold(double d, int k, double target) {
    // P(|cos| > c): integral of (1 - x^2)^((k - 3) / 2) from c to 1 over that from 0 to 1, in x = sin(u)
    auto mass = [k](double c) {
        const double lo = asin(c), hi = 1.5707963267948966;
        const int n = 200;
        double sum = 0.0;
        for (int i = 0; i < n; ++i) sum += pow(cos(lo + (hi - lo) * (i + 0.5) / n), (double)(k - 2));
        return sum * (hi - lo) / n;
    };
    const double all = mass(0.0), share = target / d < 0.5 ? target / d : 0.5;
    double lo = 0.0, hi = 1.0;
    for (int i = 0; i < 30; ++i) { const double mid = 0.5 * (lo + hi); if (mass(mid) > share * all) lo = mid; else hi = mid; }
    return 0.5 * (lo + hi) * sqrt((double)k);
}

// Shape of the recoveries on the whole GPU (sgc_chunk_grid.cu): one block per SM keeps a share of the columns.
constexpr size_t kGridHead = 80;                      // barriers
constexpr int kGridQueue = 1024;                      // reports that a block collects before they join the lists
constexpr size_t kGridSmem = 226 * 1024;              // dynamic shared memory, at most (1 KB of it for alignment)
struct GridPlan {
    int blocks, cols, nb;              // 0 blocks: no room; columns of a block (multiple of 16), in blocks of up to 256
    int kc, ks, kq;                    // 64-row chunks, 16-row steps, rows of a vector (multiple of 64)
    int mt, row_bufs;                  // tiles of 128 residual rows; how many of them are in shared memory at a time
    int own, gw;                       // recoveries of a block, warps that work on one of them
    size_t off_rows, off_inv, off_queue, off_head, off_book, off_r, off_x, bytes;
    double us;                         // estimate of the launch, without what the general form needs as well
};
inline GridPlan grid_plan(int c, long long dc, int k, int s, int sms) {
    GridPlan p = {};
    const long long cols = ((dc + sms - 1) / sms + 15) / 16 * 16;
    if (cols > 1 << 16) return p;
    p.cols = (int)cols;
    p.nb = (p.cols + 255) / 256;
    const int blocks = (int)((dc + cols - 1) / cols);
    p.kc = (k + 63) / 64; p.ks = (k + 15) / 16; p.kq = p.kc * 64;
    p.mt = (2 * c + 127) / 128;
    p.own = (2 * c + blocks - 1) / blocks;
    p.gw = kClusterWarps;
    while (p.gw > 4 && p.gw * p.own > kClusterWarps) p.gw >>= 1;
    // Generating the columns; per pick, a tile of residuals meets a block of columns, and books are kept (a group of warps takes own / groups of
    // them one after the other).  Fitted to 236 lists of 2 to 5000 chunks, half of them random sizes (10 % off on average).
    {
        const int groups = kClusterWarps / p.gw, turns = (p.own + groups - 1) / groups, passes = (p.cols + 543) / 544;
        const double scores = p.mt * (0.40 * p.nb + p.cols * (2.6e-3 + 6.3e-5 * p.ks)), books = turns * (7.2 + (1.9e-3 * s * k + 0.011 * k) / p.gw);
        p.us = 1.0 + 2.85 * p.kc * passes + s * (4.6 + scores + books);
    }
    for (p.row_bufs = p.mt > 1 ? 2 : 1; p.row_bufs >= 1; --p.row_bufs) {
        p.off_rows = (size_t)p.cols * p.kc * 128;                     // (cols is a multiple of 8: the rows start on 1024 bytes)
        p.off_rows = (p.off_rows + 1023) / 1024 * 1024;
        p.off_inv = p.off_rows + (size_t)p.row_bufs * p.kc * 16384;
        p.off_queue = p.off_inv + (size_t)p.cols * 4;
        p.off_head = (p.off_queue + (size_t)kGridQueue * 12 + 15) / 16 * 16;
        p.off_book = p.off_head + kGridHead;
        p.off_r = p.off_book + (size_t)p.own * kClusterBook;
        p.off_x = p.off_r + (size_t)p.own * p.kq * 8;
        p.bytes = p.off_x + (size_t)(kClusterWarps / p.gw) * p.kq * 8;
        if (p.bytes + 1024 <= kGridSmem) { p.blocks = blocks; return p; }
    }
    return p;
}

// The same for the general form (a correlation and a decision per pick, each a launch; on the tensor cores three launches, of which
// the pass over 256 residuals takes most): us per step.
inline bool chunk_on_tensor_cores(int c, long long dc, int kp) { return kp >= 64 && 2 * c <= 2048 && (double)dc * kp * 2.0 * c >= 1.0e9; }
inline int chunk_passes(int c) { return ((2 * c + 31) / 32 * 32 + 255) / 256; }
inline int chunk_padded_k(int k) { return k <= 8 ? 8 : k <= 16 ? 16 : k <= 32 ? 32 : k <= 64 ? 64 : k <= 128 ? 128 : 256; }
inline double chunk_general_us(int c, long long dc, int k, int s, int sms) {
    const int kp = chunk_padded_k(k);
    if (chunk_on_tensor_cores(c, dc, kp)) return s * (22.0 + 16.0 * chunk_passes(c));
    const double units = (double)((dc + 15) / 16) * ((2 * c + 3) / 4) / sms;
    const double books = 1.2 * s * k * ((2 * c + sms - 1) / sms);      // (cycles, for the recoveries of one SM)
    return s * (11.0 + (books + units * (7.9 + 3.8 * ((k + 15) / 16))) / 1.9e3);
}
// The general form once more, where the other choice is the whole-GPU form: us of its iterations, fitted to the same lists as that one's (14 % off on
// average).  On the tensor cores a pass over 256 residuals reads and compares all columns; else a block generates its columns for every group of
// recoveries, of which it holds as many as its registers take, and books cost the SM of the recovery.
constexpr int chunk_corr_group(int kp) { return kp <= 64 ? 256 : kp <= 128 ? 128 : 64; }      // recoveries per block of the correlation
inline double chunk_launches_us(int c, long long dc, int k, int s, int sms) {
    const int kp = chunk_padded_k(k), passes = chunk_passes(c);
    const double per_sm = 2.0 * c / sms;
    if (chunk_on_tensor_cores(c, dc, kp)) return s * (18.4 + passes * (5.2 + 6.6e-7 * (double)dc * k) + 4.9 * per_sm);
    const int group = chunk_corr_group(kp), groups = (2 * c + group - 1) / group;
    const double tiles = (double)groups * (double)((dc + 15) / 16) / sms;
    return s * (10.6 + tiles * (0.82 + 0.0095 * (kp / 16)) + 1.6e-4 * per_sm * s * k);
}
// The whole-GPU form is taken from k_c = 33 on (with fewer rows the general form's correlation costs little more than its two launches: 256 chunks of
// 65536, k = 8, s = 1: 52 us, 55 here) where its estimate is below that by a twentieth.  us per step, general / whole-GPU form:  256 chunks of 65536, k = 112,
// s = 16: 884 / 423;  64 of 30000, 200, 25: 947 / 441;  1024 of 16384, 128, 16: 2390 / 964;  3 of 77688, 76, 2: 99 / 52;  but 1024 of 3416, 35, 5: 167 / 327;
// 1100 of 1024, 200, 2: 189 / 322;  2000 of 4000, 64, 8: 434 / 821;  21 of 2840, 177, 2: 34 / 48.  Over 236 lists the rule's choices take 0.1 % more
// than the better form of each, the whole-GPU form wherever it fits 16 %, the general form 36 %.
inline bool grid_form_taken(const GridPlan& p, int k, double launches_us) { return p.blocks > 0 && k > 32 && 1.05 * p.us < launches_us; }
// The cluster form is taken where its estimate beats that one by a tenth.  (The general form of a single vector is the lock-step recovery of
// a whole matrix: it is taken for one wherever it fits.)
inline bool cluster_form_taken(const ChunkPlan& p, int c, double general_us) { return p.cl > 0 && (c == 1 || 1.1 * p.us < general_us); }

}  // namespace sgc
