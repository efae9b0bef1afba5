"""Shapes and shared-memory sizes of the recovery kernel, checked on the host over what sgc_create accepts.

csrc/sgc_omp_plan.h is plain integer arithmetic; g++ compiles it here together with the sweeps below.
"""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include "sgc_omp_plan.h"
using namespace sgc;

// do the buffers that k_omp carves for every role of a block end inside its shared memory?
static bool inside(int cl, int k, int s, const OmpBudget& b) {
    const int gs = group_blocks(cl);
    const long long pb = (long long)frag_bytes(k);
    const long long books = (long long)(book_doubles(k, s, gs, cl == 16) + (size_t)b.q_cols * slice_rows(k, gs)) * 8;
    const long long words = 4ll * b.z_words;
    if (b.q_cols < 0 || b.q_cols > s || words < 64 * 32 * 4) return false;          // (64 split tiles of partial sums)
    if (b.book_correlates) return ((pb + books + 15) & ~15ll) + words <= kOmpDynBytes;
    return books <= kOmpDynBytes && ((pb + 15) & ~15ll) + words <= kOmpDynBytes;
}

// first size whose launch would not fit, as (k, s, d); 0 when there is none
extern "C" int sweep_budget(int k0, int k1, long long* out) {
    static const int ss[] = {1, 2, 3, 4, 5, 7, 16, 31, 64, 73, 83, 100, 128, 200, 256, 333, 500, 512, 700, 900, 1000, 1023, 1024};
    for (int k = k0; k <= k1; ++k)
        for (int s : ss) {
            if (s > k) break;
            const long long limit = (long long)(1.2e6 / k);
            const long long ds[] = {s, s + 1, 64, 73, 83, limit, limit + 1, 999ll * s, 1000ll * s, 65536, 45088768, (1ll << 32) - 1};
            for (long long d : ds) {
                if (d < s || d < 1) continue;
                for (int mode = 0; mode < 2; ++mode)
                    for (int device = 0; device < 3; ++device) {      // a whole GPU, one without clusters of 16, one with few of 8
                        const int cl = omp_shape(d, k, s, mode, device == 0, device < 2);
                        const OmpBudget b = omp_budget(cl, k, s, mode);
                        if (b.fits && inside(cl, k, s, b) && (device < 2 || cl == 2)) continue;
                        out[0] = k; out[1] = s; out[2] = d;
                        return 1;
                    }
            }
        }
    return 0;
}
// are the blocks' shares of n columns whole, one after the other and inside their memory?
extern "C" int shares(unsigned n, int k, int nblk) {
    unsigned long long at = 0;
    for (int b = 0; b < nblk; ++b) {
        const CorrPlan c = corr_plan(n, k, 20000, b, nblk);
        if (c.cnt < 0 || (unsigned long long)c.tiles * 16 < (unsigned long long)c.cnt || (c.cnt > 0 && c.e0 != at)) return 0;
        at += (unsigned long long)c.cnt;
        if (c.norms && c.inv_off + (size_t)c.tiles * 32 > 20000) return 0;
        if (c.cached && c.z_off + (size_t)c.tiles * c.kblocks * 128 > 20000) return 0;
    }
    return at == n;
}
extern "C" int shape(long long d, int k, int s, int mode, int one) { return omp_shape(d, k, s, mode, one != 0, true); }
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("plan")
    src, so = str(tmp / "plan.cpp"), str(tmp / "plan.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2502_00311_b200", "csrc"), src, "-o", so])
    return C.CDLL(so)


def test_every_accepted_size_fits_the_shared_memory_of_its_form(plan):
    out = (C.c_longlong * 3)()
    assert plan.sweep_budget(1, 16384, out) == 0, list(out)


def test_many_rows_and_few_columns_leave_the_one_cluster_form(plan):
    # books and operands of the one cluster do not fit one block there
    assert [plan.shape(C.c_longlong(d), k, s, 1, 1) for d, k, s in [(73, 16384, 4), (83, 14369, 83), (64, 16384, 64)]] == [8, 8, 8]
    assert [plan.shape(C.c_longlong(d), k, s, 1, 1) for d, k, s in [(4096, 256, 16), (80, 14000, 16), (1171, 1024, 1024)]] == [16, 16, 16]


@pytest.mark.parametrize("nblk", [8, 16, 104, 120, 148, 160])
def test_shares_of_the_correlation_are_whole(plan, nblk):
    for n in [1, 7, nblk - 1, nblk, nblk + 1, 16 * nblk + 1, 24_576, 45_088_768, 2**31 - 1, 2**31, 2**31 + 12_345, 3 * 2**30 + 5,
              2**32 - nblk, 2**32 - nblk + 1, 2**32 - 2, 2**32 - 1]:
        for k in (1, 64, 300, 16384):
            assert plan.shares(C.c_uint(n), k, nblk), (n, k)
