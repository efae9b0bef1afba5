"""Shapes of the one-launch chunk recoveries, checked on the host over what the batched chunk path accepts.

csrc/sgc_chunk_plan.h is plain arithmetic; g++ compiles it here together with the sweeps below.
"""
import ctypes as C
import math
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# lists (chunks, columns of a chunk, rows of A, picks) whose chunks come in batches: more of them than the clusters have room for at a time.
# One pick, where a batch ends as soon as it has begun, and several; 4, 8 and 16 warps on a recovery
BATCHED = [(256, 8064, 164, 1), (400, 1684, 248, 8), (800, 856, 200, 8), (80, 6448, 212, 12)]

SHIM = r"""
#include "sgc_chunk_plan.h"
using namespace sgc;

// buffers of the cluster form that a block addresses, one behind the other and inside its shared memory
static bool whole(const ChunkPlan& p, int c, long long dc, int k, int s) {
    if (p.clusters < 1 || p.per_cluster * (long long)p.clusters < c || p.batch * p.batches < p.per_cluster || p.per_cluster > c) return false;
    if ((long long)p.cols * p.cl < dc || p.cols != 16 * p.tiles || p.kb * 16 < k || p.kq < k || p.kq < 16 * p.kb || p.kq % 64) return false;
    if ((1 << p.slots_log) != p.slots || (1 << p.cl_log) != p.cl || (1 << p.quads_log) < 4 * p.kb) return false;
    if ((p.tiles + p.slots - 1) / p.slots > kClusterTiles || p.slots > kClusterWarps) return false;              // a key's room
    if (4 * p.nt < 2 * p.batch || p.own * p.cl < 2 * p.batch || p.gw < 1 || kClusterWarps % p.gw) return false;
    if ((p.rec_bytes / 64) % 2 == 0 || p.rec_bytes < p.kb * 64) return false;                                  // every bank once
    if (p.off_inv < kClusterHead + (size_t)p.tiles * p.kb * 512 || p.off_frag < p.off_inv + (size_t)p.cols * 4) return false;
    if (p.off_top < p.off_frag + (size_t)4 * (p.nt + 3) * p.rec_bytes || p.off_ent < p.off_top + (size_t)2 * p.batch * p.slots * 16) return false;
    if (p.off_book < p.off_ent + (size_t)p.own * p.cl * 16 || p.off_r < p.off_book + (size_t)p.own * kClusterBook) return false;
    if (p.off_x < p.off_r + (size_t)p.own * p.kq * 8 || p.off_q < p.off_x + (size_t)(kClusterWarps / p.gw) * p.kq * 8) return false;
    if (p.bytes < p.off_q + (p.q_shared ? (size_t)p.own * s * p.kq * 8 : 0) || p.bytes > kClusterSmem) return false;
    return p.off_frag % 16 == 0 && p.off_top % 16 == 0 && p.off_ent % 16 == 0 && p.off_book % 16 == 0 && p.off_r % 16 == 0 && p.off_x % 16 == 0;
}
static bool whole(const GridPlan& p, int c, long long dc, int k, int sms) {
    if (p.blocks > sms || (long long)p.blocks * p.cols < dc || p.cols % 16 || p.nb * 256 < p.cols || (p.nb - 1) * 256 >= p.cols) return false;
    if (p.kc * 64 < k || p.kc > 4 || p.ks * 16 < k || p.ks > 4 * p.kc || p.kq != 64 * p.kc || p.mt * 128 < 2 * c || p.own * p.blocks < 2 * c) return false;
    if (p.gw < 4 || kClusterWarps % p.gw || p.row_bufs < 1 || p.row_bufs > 2) return false;
    if (p.off_rows % 1024 || p.off_rows < (size_t)p.cols * p.kc * 128 || p.off_inv < p.off_rows + (size_t)p.row_bufs * p.kc * 16384) return false;
    if (p.off_queue < p.off_inv + (size_t)p.cols * 4 || p.off_head < p.off_queue + (size_t)kGridQueue * 12 || p.off_head % 16) return false;
    if (p.off_book < p.off_head + kGridHead || p.off_r < p.off_book + (size_t)p.own * kClusterBook || p.off_r % 16) return false;
    if (p.off_x < p.off_r + (size_t)p.own * p.kq * 8 || p.bytes < p.off_x + (size_t)(kClusterWarps / p.gw) * p.kq * 8) return false;
    return p.bytes + 1024 <= kGridSmem;
}

// first size whose plan does not hold, as (c, dc, k, s, form); 0 when there is none.  taken: how many plans of each form there were.
extern "C" int sweep(int k, long long* out, long long* taken) {
    const int resident[4][kChunkShapes] = {{148, 74, 33, 15, 7}, {148, 74, 33, 15, 0}, {20, 10, 5, 2, 1}, {1, 0, 0, 0, 0}};
    const int cs[] = {1, 2, 3, 7, 16, 40, 64, 100, 256, 300, 1000, 1024, 5000};
    for (int c : cs)
        for (int e = 3; e <= 21; ++e)
            for (int odd = 0; odd < 3; ++odd) {
                const long long dc = (1ll << e) + (odd == 0 ? 0 : odd == 1 ? 4 : (1ll << e) / 3);
                for (int s = 1; s <= 32 && s <= k; s = s < 3 ? s + 1 : s < 30 ? s * 2 + 1 : s + 1) {
                    for (const auto& r : resident) {
                        const ChunkPlan p = chunk_plan(c, dc, k, s, r);
                        if (p.cl == 0) continue;
                        ++taken[0];
                        if (!whole(p, c, dc, k, s)) { out[0] = c; out[1] = dc; out[2] = k; out[3] = s; out[4] = 0; return 1; }
                    }
                    if (s > 1) continue;
                    for (int sms = 20; sms <= 148; sms += 128) {
                        const GridPlan g = grid_plan(c, dc, k, s, sms);
                        if (g.blocks == 0) continue;
                        ++taken[1];
                        if (!whole(g, c, dc, k, sms)) { out[0] = c; out[1] = dc; out[2] = k; out[3] = sms; out[4] = 1; return 1; }
                    }
                }
            }
    return 0;
}
// the cluster form of that list as the dispatch decides it on 148 SMs that hold `eight` / `sixteen` clusters of those widths: batches, warps per
// recovery, whether the q_l are in shared memory; all zero where the list takes another form
extern "C" void cluster_form(int c, long long dc, int k, int s, int eight, int sixteen, int* out) {
    const int resident[kChunkShapes] = {148, 74, 2 * eight, eight, sixteen};
    const ChunkPlan p = chunk_plan(c, dc, k, s, resident);
    const bool taken = cluster_form_taken(p, c, chunk_general_us(c, dc, k, s, 148));
    out[0] = taken ? p.batches : 0; out[1] = taken ? p.gw : 0; out[2] = taken ? p.q_shared : 0;
}
extern "C" int whole_gpu_form(int c, long long dc, int k, int s) { return grid_form_taken(grid_plan(c, dc, k, s, 148), k, chunk_launches_us(c, dc, k, s, 148)); }
extern "C" double tail(double d, int k, double target) { return sphere_tail_threshold(d, k, target); }
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    lib = str(d / "libplan.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2502_00311_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", lib])
    L = C.CDLL(lib)
    L.cluster_form.argtypes = [C.c_int, C.c_longlong, C.c_int, C.c_int, C.c_int, C.c_int, C.POINTER(C.c_int)]
    L.whole_gpu_form.argtypes = [C.c_int, C.c_longlong, C.c_int, C.c_int]
    L.tail.restype, L.tail.argtypes = C.c_double, [C.c_double, C.c_int, C.c_double]
    return L


def test_every_plan_holds_what_its_blocks_address(plan):
    taken = (C.c_longlong * 2)()
    for k in list(range(1, 34)) + [47, 48, 49, 63, 64, 65, 96, 112, 127, 128, 129, 192, 193, 217, 255, 256]:
        out = (C.c_longlong * 5)()
        assert plan.sweep(k, out, taken) == 0, list(out)
    assert taken[0] > 10_000 and taken[1] > 1_000                         # both forms are taken


@pytest.mark.parametrize("eight,sixteen", [(15, 7), (16, 8), (16, 7)])
@pytest.mark.parametrize("c,dc,k,s", BATCHED)
def test_lists_that_come_in_batches(plan, c, dc, k, s, eight, sixteen):
    # what test_gpu_variants runs as lists whose clusters take several batches, with several warps on a recovery
    out = (C.c_int * 3)()
    plan.cluster_form(c, dc, k, s, eight, sixteen, out)
    assert out[0] > 1 and out[1] > 1, list(out)


# lists whose step was timed in both forms (148 SMs; the clusters refuse them): chunks, columns of a chunk, rows of A, picks, us general / whole GPU
@pytest.mark.parametrize("c,dc,k,s,general,whole", [
    (1839, 1196, 96, 6, 439, 1047), (522, 616, 199, 2, 93, 204), (1024, 3416, 35, 5, 167, 327), (2000, 4000, 64, 8, 434, 821), (1100, 1024, 200, 2, 189, 322),
    (5000, 2048, 40, 2, 358, 599), (1024, 7096, 56, 8, 344, 448), (21, 2840, 177, 2, 34, 48), (27, 9008, 121, 1, 26, 31), (256, 65_536, 112, 16, 884, 423),
    (48, 22_456, 84, 12, 272, 184), (16, 100_000, 56, 8, 432, 146), (1024, 16_384, 128, 16, 2381, 964), (64, 30_000, 200, 25, 947, 441), (3, 77_688, 76, 2, 99, 52),
    (2, 51_712, 48, 6, 192, 93), (37, 39_428, 244, 2, 98, 60)])
def test_the_whole_gpu_form_is_taken_where_it_is_quicker(plan, c, dc, k, s, general, whole):
    assert plan.whole_gpu_form(c, dc, k, s) == (whole < general)


@pytest.mark.parametrize("d,k", [(65_536, 112), (20_000, 40), (30_000, 256)])
def test_report_threshold_follows_the_sphere(plan, d, k):
    # the share of uniform directions beyond it, by the beta law of the squared cosine
    from scipy.special import betainc
    z = plan.tail(d, k, 20.0)
    share = 1.0 - betainc(0.5, (k - 1) / 2, z * z / k)
    assert math.isclose(share * d, 20.0, rel_tol=1e-2)
