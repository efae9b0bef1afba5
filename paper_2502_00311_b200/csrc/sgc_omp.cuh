// Arguments and small device helpers shared by the recovery kernels (sgc_omp.cu, sgc_recover.cu).  Not part of the C ABI.
#pragma once

#include "sgc_internal.cuh"

namespace sgc {

struct OmpArgs {
    uint32_t seed_lo, seed_hi;
    unsigned long long d;
    int k, s;
    int kp;                            // row stride of rt and zlist: k rounded up to a multiple of 64, the rows beyond k are zero
    double sigma;
    int half_n;                        // residuals per stream in one screening pass
    int rows_wide, rows_narrow;        // rows of the pass that serves both streams / the first stream alone
    double z_harvest, z_floor;         // screening thresholds in units of ||r|| / sqrt(k)
    float4* corr_cand;                 // [2][blocks] (score, column, best score not forwarded, -)
    const double* y64; float* r32;     // r32 viewed as float[2k] (interleaved pairs)
    uint32_t* lam;                     // [2][s]
    // Orthogonal form of Algorithm 3's recurrences, one record per pick j: q_j (unit vector, the new column made orthogonal
    // to the earlier ones), c^(j)_l = <q_l, a_new> for l < j, gamma_j = 1 / ||a_new - sum c_l q_l||, a_j = <q_j, r>
    double* q;                         // [2][s][k]
    double* crow; double* ccol;        // [2][s][s]  c^(j)_l at [j * s + l] and at [l * s + j]
    double* gam; double* acoef; double* rnorm;       // [2][s]
    Counters* cnt; SpecCtl* ctl;
    uint16_t* rt; float* tau; float* inv_scale; unsigned int* rep_count; double* pick_score;
    double* rhist;                     // fp64 copies of the screened residuals (row = m * half_n + position), for the resolve kernel
    // two-level screening
    float* wide_tau; double z_wide; int wide_every; unsigned int* wide_count; unsigned int* wide_bits;
    int mini;                          // 1: speculation ahead of a list pass (at most `depth` picks)
    int depth;
    const uint32_t* cand_list;
    uint16_t* zlist; double* gram; double* p0; double* wgram; double* pnorm;      // Gram path
    int q_cols;                        // columns of q that a bookkeeping block keeps in shared memory
    int book_correlates;               // lock-step: the bookkeeping blocks correlate, too
    int z_words;                       // 32-bit words of shared memory that the correlation may use to keep generated entries
};

__device__ __forceinline__ bool better(float sa, uint32_t ia, float sb, uint32_t ib) {
    return (sa > sb) || (sa == sb && ia < ib);
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// threshold of a wide list: every column scoring at least z_wide noise deviations against a screened residual (norm rn)
// in place c of its stream, in the scaled units of that row; +inf where the place feeds no list
__device__ __forceinline__ float wide_threshold(const OmpArgs& a, int c, double rn) {
    if (c % a.wide_every != 0) return __int_as_float(0x7f800000);
    return (float)(a.z_wide * rn / sqrt((double)a.k) * residual_scale(rn));
}

// threshold of a screened residual (norm rn) whose pick scored ps, in the caller's units: any column that could refute the
// pick must be reported, and z_harvest / z_floor bound how many others are
__device__ __forceinline__ double report_threshold(const OmpArgs& a, double rn, double ps) {
    const double unit = rn / sqrt((double)a.k);
    double t = ps - screen_margin(rn, ps, a.k);
    if (t > a.z_harvest * unit) t = a.z_harvest * unit;
    if (t < a.z_floor * unit) t = a.z_floor * unit;
    return t;
}

cudaError_t omp_configure(sgc_state* st);
cudaError_t launch_omp(sgc_state* st, const OmpArgs& a, int mode, cudaStream_t stream);

}  // namespace sgc
