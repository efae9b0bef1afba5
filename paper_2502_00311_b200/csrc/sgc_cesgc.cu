// CESGC (Section 4.4, "Compute Efficient SGC"): SGC runs on the projected gradient B G (r x n) instead of G (m x n), and
// its update goes back through B^T:  W <- W - eta B^T SGC(B G).  B (r x m, the first r left-singular vectors of a
// gradient, refreshed by the caller every few hundred steps) is an input here; the two projections around the SGC core
// are the kernels of this file.
//   k_cesgc_project   P = B G in fp64, rounded to fp32 once, so that the top-s selection that follows decides on the exactly
//                     projected gradient.  64 fp64 multiply-adds per cycle and SM bound it (30 us for a 4096 x 4096 gradient at
//                     r = 32); conversions from fp32, a quarter as fast, are kept out of the way: a thread owns four columns and
//                     eight rows, converts each element of G once for its eight products and reads B as fp64 from a slab that
//                     the block has converted on the way in.  (An error-free two-float form took 276 us, fp64 with both operands
//                     converted per product 1.1 ms.)  The rows of G are split over the CTAs of a thread-block cluster; their
//                     partial sums meet through distributed shared memory, added in rank order.
//   k_cesgc_back      W += B^T U for the r x n matrix U that the SGC core left (U = -eta N has at most s non-zeros):
//                     block = one column of U; columns without a non-zero cost one read of r values.
#include "sgc_internal.cuh"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace sgc {
namespace {

constexpr int kCesgcMaxR = 64;
constexpr int kProjCols = 128;           // columns of G per block: 32 lanes of four
constexpr int kProjRows = 8;             // rows of B per thread
constexpr int kProjPer = 4;              // rows of a slab of G per thread
constexpr int kProjMaxSplit = 8;         // CTAs of a cluster (the portable limit), each with a range of G's rows
constexpr int kProjResident = 148;       // one wave

// groups of 8 rows of B (warps of a part), parts (each with every parts-th row of G) that make up 16 warps at most, rows of G per slab
__host__ __device__ constexpr int proj_groups(int r) { return (r + kProjRows - 1) / kProjRows; }
__host__ __device__ constexpr int proj_parts(int r) { return proj_groups(r) > 4 ? 2 : proj_groups(r) > 2 ? 4 : 8; }
__host__ __device__ constexpr int proj_slab(int r) { return kProjPer * proj_parts(r); }
// slabs of B (two, fp64) and, at the end, the partial sums of the parts
__host__ __device__ constexpr size_t proj_smem(int r) {
    const size_t slab = 2 * (size_t)proj_groups(r) * kProjRows * proj_slab(r) * sizeof(double);
    const size_t part = (size_t)proj_groups(r) * kProjRows * kProjCols * sizeof(double);
    return slab > part ? slab : part;
}
constexpr size_t proj_smem_max() {
    size_t v = 0;
    for (int r = 1; r <= kCesgcMaxR; ++r) if (proj_smem(r) > v) v = proj_smem(r);
    return v;
}

template <bool VEC>
__global__ void __launch_bounds__(512, 1)
k_cesgc_project(const float* __restrict__ B, const float* __restrict__ G, float* __restrict__ P, int r, int m, int n) {
    extern __shared__ double smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int groups = proj_groups(r), rows8 = groups * kProjRows, parts = proj_parts(r), slab_rows = proj_slab(r);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ig = warp % groups, part = warp / groups;
    const int j0 = blockIdx.x * kProjCols + 4 * lane;                 // this thread's four columns
    // this CTA's rows of G: whole slabs, the same number for every CTA of the cluster (the last ranges may be empty)
    const int slabs = (m + slab_rows - 1) / slab_rows;
    const int part_rows = (slabs + (int)gridDim.y - 1) / (int)gridDim.y * slab_rows;
    const int m_begin = (int)blockIdx.y * part_rows;
    const int m_end = m_begin + part_rows < m ? m_begin + part_rows : m;
    double acc[kProjRows][4];
#pragma unroll
    for (int u = 0; u < kProjRows; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[u][c] = 0.0;
    // slab of B as [row of G][row of B]: a thread reads its eight values of a row of G in four 16-byte broadcasts
    auto stage = [&](double* dst, int row0) {
        for (int e = threadIdx.x; e < rows8 * slab_rows; e += blockDim.x) {
            const int i = e / slab_rows, q = e % slab_rows;
            dst[q * rows8 + i] = (i < r && row0 + q < m_end) ? (double)B[(size_t)i * m + row0 + q] : 0.0;
        }
    };
    auto load = [&](int row) -> float4 {
        float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (row < m_end) {
            const float* src = G + (size_t)row * n + j0;
            if (VEC) { if (j0 < n) f = __ldcs(reinterpret_cast<const float4*>(src)); }        // n is a multiple of 4
            else {
                if (j0 < n) f.x = src[0];
                if (j0 + 1 < n) f.y = src[1];
                if (j0 + 2 < n) f.z = src[2];
                if (j0 + 3 < n) f.w = src[3];
            }
        }
        return f;
    };
    double* bufs[2] = {smem, smem + (size_t)rows8 * slab_rows};
    float4 next[kProjPer];
    if (m_begin < m_end) {
        stage(bufs[0], m_begin);
#pragma unroll
        for (int q = 0; q < kProjPer; ++q) next[q] = load(m_begin + q * parts + part);
    }
    int b = 0;
    for (int row0 = m_begin; row0 < m_end; row0 += slab_rows, b ^= 1) {
        __syncthreads();                                              // this slab is staged, the other one used up
        float4 g[kProjPer];
#pragma unroll
        for (int q = 0; q < kProjPer; ++q) g[q] = next[q];
        if (row0 + slab_rows < m_end) {
#pragma unroll
            for (int q = 0; q < kProjPer; ++q) next[q] = load(row0 + slab_rows + q * parts + part);
            stage(bufs[b ^ 1], row0 + slab_rows);
        }
        const double* slab = bufs[b] + ig * kProjRows;
#pragma unroll
        for (int q = 0; q < kProjPer; ++q) {
            const double2* bq = reinterpret_cast<const double2*>(slab + (size_t)(q * parts + part) * rows8);
            const double gx = (double)g[q].x, gy = (double)g[q].y, gz = (double)g[q].z, gw = (double)g[q].w;
#pragma unroll
            for (int u = 0; u < kProjRows / 2; ++u) {
                const double2 v = bq[u];
                acc[2 * u][0] = fma(v.x, gx, acc[2 * u][0]); acc[2 * u][1] = fma(v.x, gy, acc[2 * u][1]);
                acc[2 * u][2] = fma(v.x, gz, acc[2 * u][2]); acc[2 * u][3] = fma(v.x, gw, acc[2 * u][3]);
                acc[2 * u + 1][0] = fma(v.y, gx, acc[2 * u + 1][0]); acc[2 * u + 1][1] = fma(v.y, gy, acc[2 * u + 1][1]);
                acc[2 * u + 1][2] = fma(v.y, gz, acc[2 * u + 1][2]); acc[2 * u + 1][3] = fma(v.y, gw, acc[2 * u + 1][3]);
            }
        }
    }
    // the parts of this CTA, one after the other (a fixed order), into shared memory; then the CTAs of the cluster
    double* sums = smem;                                              // [rows8][kProjCols]
    for (int p = 0; p < parts; ++p) {
        __syncthreads();
        if (part != p) continue;
#pragma unroll
        for (int u = 0; u < kProjRows; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                double* d = sums + (size_t)(ig * kProjRows + u) * kProjCols + 32 * c + lane;      // (column 4 lane + c at 32 c + lane)
                *d = p == 0 ? acc[u][c] : *d + acc[u][c];
            }
    }
    cluster.sync();
    const unsigned split = cluster.num_blocks(), rank = cluster.block_rank();
    // the CTAs share the additions: rank order, whoever adds, so the result does not depend on the schedule
    for (int e = (int)(rank * blockDim.x + threadIdx.x); e < r * kProjCols; e += (int)(split * blockDim.x)) {
        const int i = e / kProjCols, x = e % kProjCols, col = blockIdx.x * kProjCols + 4 * (x & 31) + (x >> 5);
        double v = 0.0;
        for (unsigned y = 0; y < split; ++y) v += cluster.map_shared_rank(sums, y)[(size_t)i * kProjCols + x];
        if (col < n) P[(size_t)i * n + col] = (float)v;
    }
    cluster.sync();                                                   // nobody leaves while its sums may still be read
}

__global__ void __launch_bounds__(256)
k_cesgc_back(const float* __restrict__ B, const float* __restrict__ U, float* __restrict__ W, int r, int m, int n) {
    __shared__ float us[kCesgcMaxR];
    __shared__ int idx[kCesgcMaxR];
    __shared__ int n_nz;
    const int j = blockIdx.x;
    if (threadIdx.x == 0) n_nz = 0;
    __syncthreads();
    if ((int)threadIdx.x < r) {
        const float u = U[(size_t)threadIdx.x * n + j];
        if (u != 0.0f) { const int slot = atomicAdd(&n_nz, 1); us[slot] = u; idx[slot] = threadIdx.x; }
    }
    __syncthreads();
    const int nz = n_nz;
    if (nz == 0) return;
    // ascending row order of B, whatever order the atomics gave: the sum below does not depend on the schedule
    if (threadIdx.x == 0) {
        for (int a = 1; a < nz; ++a) {
            const int ia = idx[a]; const float ua = us[a];
            int b = a - 1;
            while (b >= 0 && idx[b] > ia) { idx[b + 1] = idx[b]; us[b + 1] = us[b]; --b; }
            idx[b + 1] = ia; us[b + 1] = ua;
        }
    }
    __syncthreads();
    for (int row = threadIdx.x; row < m; row += 256) {
        double acc = 0.0;
        for (int a = 0; a < nz; ++a) acc += (double)B[(size_t)idx[a] * m + row] * (double)us[a];
        float* w = W + (size_t)row * n + j;
        *w = (float)((double)*w + acc);
    }
}

}  // namespace

bool cesgc_shape_ok(int r, int m, int n) { return r >= 1 && r <= kCesgcMaxR && m >= 1 && n >= 1; }

cudaError_t launch_cesgc_project(const float* B, const float* G, float* P, int r, int m, int n, cudaStream_t stream) {
    const int col_blocks = (n + kProjCols - 1) / kProjCols;
    const int slabs = (m + proj_slab(r) - 1) / proj_slab(r);
    int split = kProjResident / col_blocks;                                         // one wave; a function of the shape alone
    if (split > kProjMaxSplit) split = kProjMaxSplit;
    if (split > slabs / 2) split = slabs / 2;                                       // at least two slabs per CTA
    if (split < 1) split = 1;
    const bool vec = n % 4 == 0 && ((uintptr_t)G & 15u) == 0;
    const void* fn = vec ? (const void*)k_cesgc_project<true> : (const void*)k_cesgc_project<false>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)proj_smem_max());
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)col_blocks, (unsigned)split, 1);
    cfg.blockDim = dim3((unsigned)(32 * proj_groups(r) * proj_parts(r)), 1, 1);
    cfg.dynamicSmemBytes = proj_smem(r);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = (unsigned)split; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return vec ? cudaLaunchKernelEx(&cfg, k_cesgc_project<true>, B, G, P, r, m, n)
               : cudaLaunchKernelEx(&cfg, k_cesgc_project<false>, B, G, P, r, m, n);
}

cudaError_t launch_cesgc_back(const float* B, const float* U, float* W, int r, int m, int n, cudaStream_t stream) {
    k_cesgc_back<<<n, 256, 0, stream>>>(B, U, W, r, m, n);
    return cudaGetLastError();
}

}  // namespace sgc
