"""The variants the dispatch rules choose between, at the sizes where they change over or leave remainders.

Same bar as test_gpu_parity (index sets bit-exact, state 1e-5, update 1e-4): the comparisons are its own.
"""
import numpy as np
import pytest

import oracle
import test_gpu_parity as parity
from paper_2502_00311_b200 import inputs
from test_chunk_plan import BATCHED
from test_gpu_parity import cuda, run_both, sgc  # noqa: F401  (sgc is the module's fixture)

pytestmark = pytest.mark.gpu


# one block holds the whole gradient up to 32768 entries; above, maxima of units of vectors; remainders of four and of a unit
@pytest.mark.parametrize("d,s", [(3, 2), (1024, 1024), (4097, 1), (32767, 1024), (32768, 31), (32770, 1024), (65_537, 3),
                                 ((1 << 22) - 1, 200), ((1 << 22) + 5, 1024)])
def test_selection_without_a_threshold(sgc, d, s):  # noqa: F811
    import torch
    rng = np.random.default_rng(d + s)
    idx, val = torch.empty(s, dtype=torch.int32, device="cuda"), torch.empty(s, device="cuda")
    cases = [(rng.standard_t(3.0, size=d) * 1e-3).astype(np.float32), np.round(rng.standard_normal(d) * 2).astype(np.float32) / 2]
    cluster = cases[0].copy()
    cluster[max(0, d - 3 * s):] += 4.0                                    # all kept entries in the last units
    for g in cases + [cluster, np.full(d, -0.75, dtype=np.float32)]:
        sgc.sparsify_static(cuda(g), s, idx, val)
        widx, wval = oracle.sparsify(g, s)
        assert np.array_equal(idx.cpu().numpy().view(np.uint32), widx) and np.array_equal(val.cpu().numpy(), wval)


def test_selection_after_the_scale_of_the_gradient_jumps(sgc):  # noqa: F811
    # the threshold of the last step is far too high, far too low, then right again
    d, s = 300_001, 40
    st = sgc.Sgc(d, 64, s, 3, 1e-3, 0.9, 0.999, 1e-8)
    w = cuda(np.zeros(d, dtype=np.float32))
    for step, scale in enumerate([1.0, 1.0, 1e-4, 1e4, 1.0, 1.0]):
        g = (np.random.default_rng(step).standard_t(3.0, size=d) * scale).astype(np.float32)
        st.step(cuda(g), w)
        widx, wval = oracle.sparsify(g, s)
        assert np.array_equal(st.get("sel_idx"), widx) and np.array_equal(st.get("sel_val"), wval), step
    st.close()


# lock-step: one cluster up to k d = 1.2e6, groups of eight blocks, pairs from d = 1000 s on; fewer columns than blocks, odd k, many rows
@pytest.mark.parametrize("d,k,s", [(37, 5, 1), (4800, 250, 9), (4801, 250, 9), (700, 257, 130), (1001, 1199, 3), (66_000, 3100, 4),
                                   (1_000_003, 201, 6), (30_000, 7001, 3)])
def test_lockstep_cluster_shapes(sgc, d, k, s):  # noqa: F811
    run_both(sgc, d, k, s, 6, "student", 2, cfg_id=2, mode=1)


# the screening pass: rows of A in one or two chunks per slot, the long and the short sweep of the 128-row form, wide lists
@pytest.mark.parametrize("d,k,s,redraw", [(30_001, 64, 2, False), (40_000, 960, 64, False), (40_003, 1024, 64, False),
                                          (200_000, 1024, 60, True), (20_000, 1088, 120, False)])
def test_screening_pass_forms(sgc, d, k, s, redraw):  # noqa: F811
    run_both(sgc, d, k, s, 7, "student", 3, cfg_id=2, mode=2, redraw_support=redraw)


def test_a_state_chooses_between_speculation_and_lockstep(sgc):  # noqa: F811
    # k no multiple of 64 speculates on its own accord when k > 1.2 s ln d; below that size and below d = 65536 it does not
    for d, k, s, speculates in [(70_000, 333, 10, True), (65_535, 333, 10, False), (70_000, 70, 10, False)]:
        stats = []
        run_both(sgc, d, k, s, 5, "student", 2, cfg_id=2, stats=stats)
        assert all((rounds >= 1) == speculates for rounds, _, _ in stats), (d, k, s, stats)


# chunks: several blocks per chunk in the first kernel, one, equal magnitudes across the blocks of a chunk, as many picks as a
# chunk has rows but one
@pytest.mark.parametrize("c,dc,k,sc", [(2, 200_000, 217, 31), (3, 65_540, 7, 1), (12, 3000, 8, 7), (150, 4100, 16, 2)])
def test_chunk_variants(sgc, c, dc, k, sc):  # noqa: F811
    parity.test_mesgc_small_chunks_batched_path_matches_independent_oracles(sgc, c, dc, k, sc, "student")
    m = sgc.Mesgc(c * dc, c, k, sc, 8, *(inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")))
    g = np.full(c * dc, 0.25, dtype=np.float32)
    g[1::2] *= -1
    m.step(cuda(g), cuda(np.zeros(c * dc, dtype=np.float32)))
    for st in m.chunks:
        assert np.array_equal(st.get("sel_idx"), np.arange(sc, dtype=np.uint32))
    m.close()


# projection: columns that are no multiple of four (no 16-byte copies) or of a block's columns, r at its ends, ragged rows
@pytest.mark.parametrize("m,n,r,c,k,sc", [(333, 97, 8, 2, 28, 4), (70, 33, 12, 1, 40, 5), (130, 68, 64, 4, 56, 7),
                                          (257, 260, 1, 1, 40, 5), (4099, 130, 34, 5, 60, 6)])
def test_cesgc_remainders(sgc, m, n, r, c, k, sc):  # noqa: F811
    parity.test_cesgc_step_matches_its_oracle(sgc, m, n, r, c, k, sc)


# many rows and a handful of columns: the one-cluster form has no room for its books there, groups of eight serve
@pytest.mark.parametrize("d,k,s", [(73, 16384, 4), (83, 14369, 83), (40, 16384, 33), (80, 13999, 16)])
def test_lockstep_with_far_more_rows_than_columns(sgc, d, k, s):  # noqa: F811
    run_both(sgc, d, k, s, 6, "student", 2, cfg_id=2, mode=1)


# picks refuted while the list stays short: a round on the Gram matrix starts from a prescribed pick, of one recovery or of both
@pytest.mark.parametrize("d,k,s", [(200, 64, 10), (256, 128, 40), (250, 64, 3)])
def test_prescribed_picks_on_a_short_list(sgc, d, k, s):  # noqa: F811
    stats = []
    run_both(sgc, d, k, s, 7, "student", 12, cfg_id=2, mode=2, redraw_support=True, n_planted=2 * s, stats=stats)
    assert any(rounds > 1 and not fallback for rounds, fallback, _ in stats), stats
    assert all(n_cand <= 256 for _, _, n_cand in stats)


# several blocks per chunk with short shares: each writes its bound into the others' shared memory
@pytest.mark.parametrize("c,dc,sc", [(1, 16_384, 31), (20, 65_536, 5), (70, 16_388, 1), (9, 32_772, 17)])
def test_chunk_selection_over_a_cluster(sgc, c, dc, sc):  # noqa: F811
    m = sgc.Mesgc(c * dc, c, 8 * sc, sc, 8, *(inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")))
    w = cuda(np.zeros(c * dc, dtype=np.float32))
    for step in range(20):
        g = np.random.default_rng(100 * c + step).standard_t(3.0, size=c * dc).astype(np.float32)
        m.step(cuda(g), w)
        for i, st in enumerate(m.chunks):
            idx, val = oracle.sparsify(g[i * dc:(i + 1) * dc], sc)
            assert np.array_equal(st.get("sel_idx"), idx) and np.array_equal(st.get("sel_val"), val), (step, i)
    m.close()


# Columns of 16 neighbours, all in the share of one block of the chunk correlation, whose scores agree to 1e-5: closer than the keys
# resolve that pick what the block forwards (2^-13), far above the fp64 scores that decide.  More of them than it forwards.
@pytest.mark.parametrize("dc,k,c,tied", [(2048, 64, 1, 3), (2048, 24, 1, 3), (4096, 200, 2, 3), (512, 8, 3, 3), (2048, 100, 1, 5),
                                         (4096, 16, 40, 4)])
def test_chunk_picks_among_near_tied_columns(sgc, dc, k, c, tied):  # noqa: F811
    hp = [inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")]
    for trial in range(12):
        rng, seed = np.random.default_rng(trial), 100 + trial
        cols = 16 * int(rng.integers(0, dc // 16)) + np.sort(rng.choice(16, tied, replace=False))
        A = float(oracle.sigma(k)) * np.concatenate([oracle.z_block(seed, 0, k, int(q), 1) for q in cols], axis=1).astype(np.float64)
        G = (A.T @ A) / np.sqrt((A * A).sum(axis=0))[:, None]
        x = np.linalg.solve(G, 1.0 + 1e-5 * np.arange(tied))              # the last of the columns wins by 1e-5
        g = np.zeros(dc, dtype=np.float32)
        g[cols] = x.astype(np.float32)
        m = sgc.Mesgc(c * dc, c, k, tied, seed, *hp)
        ref = oracle.Oracle(dc, k, tied, seed, *hp)
        m.step(cuda(np.tile(g, c)), cuda(np.zeros(c * dc, dtype=np.float32)))
        ref.step(g, np.zeros(dc, dtype=np.float32))
        for st in (m.chunks[0], m.chunks[-1]):
            assert np.array_equal(st.get("lamM"), ref.get("lamM")), (trial, st.get("lamM"), ref.get("lamM"))
            assert np.array_equal(st.get("lamV"), ref.get("lamV")), trial
        m.close()
        ref.close()


# lists a little longer than the Gram path takes, many rows of A and kept entries of nearly equal size: two columns of one block's
# share come within the rescoring window, and more columns than 16 within the screening margin of a pick
@pytest.mark.parametrize("drift", [3, 30])
def test_near_equal_entries_on_a_list_of_some_hundred_columns(sgc, drift):  # noqa: F811
    d, k, s = 65_600, 16_384, 250
    hp = [inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")]
    supp, sign = inputs.planted_support(d, s, 30 + drift)
    supp, rng = supp.astype(np.int64), np.random.default_rng(drift)
    st, twin = sgc.Sgc(d, k, s, 5, *hp), sgc.Sgc(d, k, s, 5, *hp)
    twin.set_mode(sgc.MODE_LOCKSTEP)
    w, wt = cuda(np.zeros(d, dtype=np.float32)), cuda(np.zeros(d, dtype=np.float32))
    for step in range(10):
        if 0 < step <= 4:
            supp[rng.choice(s, drift, replace=False)] = np.setdiff1d(rng.integers(0, d, size=200), supp)[:drift]
        g = (rng.standard_t(3.0, size=d) * 1e-3).astype(np.float32)
        g[supp] = sign * (1.0 + 0.02 * rng.random(s)).astype(np.float32)
        st.step(cuda(g), w)
        twin.step(cuda(g), wt)
        assert int(st.get("fallback")) == 0 and int(st.get("rounds")) >= 2, step
        for name in ("lamM", "lamV"):
            assert np.array_equal(st.get(name), twin.get(name)), (step, name)
        assert np.array_equal(w.cpu().numpy(), wt.cpu().numpy())
    assert 256 < int(st.get("n_cand")) < 768
    st.close()
    twin.close()


# more picks than one pass has room for: two or three passes without a refuted pick are a confirmed step, and the state goes on
# speculating
@pytest.mark.parametrize("d,k,s,passes", [(131_072, 2048, 130, 2), (70_001, 4096, 260, 3)])
def test_a_state_confirmed_in_several_passes_keeps_speculating(sgc, d, k, s, passes):  # noqa: F811
    hp = [inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")]
    supp, sign = inputs.planted_support(d, s, 3)
    st, twin = sgc.Sgc(d, k, s, 5, *hp), sgc.Sgc(d, k, s, 5, *hp)
    twin.set_mode(sgc.MODE_LOCKSTEP)
    w, wt = cuda(np.zeros(d, dtype=np.float32)), cuda(np.zeros(d, dtype=np.float32))
    for step in range(6):
        g = cuda(inputs.gradient(d, "student", supp, sign, 100 + step))
        st.step(g, w)
        twin.step(g, wt)
        assert (int(st.get("rounds")), int(st.get("fallback"))) == (passes, 0), step
        assert np.array_equal(st.get("lamM"), twin.get("lamM")) and np.array_equal(st.get("lamV"), twin.get("lamV"))
    assert np.array_equal(w.cpu().numpy(), wt.cpu().numpy())
    st.close()
    twin.close()


# a zero gradient leaves zero residuals: all scores are equal and the lowest free column is picked every time
@pytest.mark.parametrize("d,k,s", [(4096, 256, 16), (16_384, 64, 16), (50_000, 16, 5), (300_000, 40, 6), (30_000, 128, 8)])
def test_lockstep_on_a_zero_gradient(sgc, d, k, s):  # noqa: F811
    st = sgc.Sgc(d, k, s, 5, *(inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")))
    st.set_mode(sgc.MODE_LOCKSTEP)
    g, w = cuda(np.zeros(d, dtype=np.float32)), cuda(np.ones(d, dtype=np.float32))
    for _ in range(40):
        st.step(g, w)
        assert np.array_equal(st.get("lamM"), np.arange(s)) and np.array_equal(st.get("lamV"), np.arange(s))
        assert int(st.get("doneM")) == s and int(st.get("n_upd")) == 0
    assert bool((w == 1).all())
    st.close()


# chunks without a gradient beside ordinary ones, and chunks with fewer non-zeros than are kept: the first zeros fill up, and a zero
# residual takes the lowest free columns
@pytest.mark.parametrize("c,dc,k,s", [(5, 4096, 16, 2), (3, 40_000, 112, 16), (40, 2048, 217, 31), (2, 1 << 17, 8, 1), (6, 32, 40, 31)])
def test_chunks_of_zeros(sgc, c, dc, k, s):  # noqa: F811
    hp = [inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")]
    m = sgc.Mesgc(c * dc, c, k, s, 8, *hp)
    refs = [oracle.Oracle(dc, k, s, 8, *hp) for _ in range(c)]
    w, wr = cuda(np.zeros(c * dc, dtype=np.float32)), np.zeros((c, dc), dtype=np.float32)
    rng = np.random.default_rng(c)
    for step in range(2):
        g = rng.standard_t(3.0, size=(c, dc)).astype(np.float32)
        g[0] = 0.0
        g[1] = 0.0
        g[1, rng.choice(dc, s // 2, replace=False)] = 1.0 + rng.random(s // 2).astype(np.float32)
        m.step(cuda(g.reshape(-1)), w)
        for i, (st, ref) in enumerate(zip(m.chunks, refs)):
            idx, val = oracle.sparsify(g[i], s)
            assert np.array_equal(st.get("sel_idx"), idx) and np.array_equal(st.get("sel_val"), val), (step, i)
            if i > 3:
                continue
            ref.step(g[i], wr[i])
            if i != 1:                                                    # (past the non-zeros its residual is rounding noise)
                for name in ("lamM", "lamV", "doneM", "doneV"):
                    assert np.array_equal(st.get(name), ref.get(name)), (step, i, name)
            assert not int(st.get("status")) & sgc.STATUS_CANDIDATE_OVERFLOW or i == 1
        got = w.cpu().numpy().reshape(c, dc)
        assert not got[0].any() and parity.rel(got[:min(c, 4)], wr[:min(c, 4)]) < 1e-4
    m.close()


def test_the_first_speculating_step_leaves_another_streams_capture_alone(sgc):  # noqa: F811
    # k no multiple of 64: the buffers of the speculation are allocated inside that step
    import torch
    d, k, s = 70_000, 333, 10
    hp = [inputs.ADAM[n] for n in ("lr", "beta1", "beta2", "eps")]
    supp, sign = inputs.planted_support(d, s, 3)
    g, w = cuda(inputs.gradient(d, "student", supp, sign, 1)), cuda(np.zeros(d, dtype=np.float32))
    warm = sgc.Sgc(d, k, s, 5, *hp)                                       # (a kernel's first launch loads it, which no capture survives)
    warm.step(g, w.clone())
    warm.close()
    st, x, side, graph = sgc.Sgc(d, k, s, 5, *hp), cuda(np.ones(4, dtype=np.float32)), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x.mul_(2.0)
        st.step(g, w, stream=side)
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 4
    assert int(st.get("rounds")) >= 1 and int(st.get("fallback")) == 0
    ref = oracle.Oracle(d, k, s, 5, *hp)
    ref.step(inputs.gradient(d, "student", supp, sign, 1), np.zeros(d, dtype=np.float32))
    assert np.array_equal(st.get("lamM"), ref.get("lamM")) and np.array_equal(st.get("lamV"), ref.get("lamV"))
    graph.reset()
    st.close()


def _chunk_parity(sgc, c, dc, k, sc, form):  # noqa: F811
    parity.test_mesgc_small_chunks_batched_path_matches_independent_oracles(sgc, c, dc, k, sc, "student", form=form)


# chunk recoveries inside clusters (form 3): fewer columns than blocks, ragged last block, odd k and the largest, one pick and the most, several
# recoveries per group of 4 warps, of 2, and per warp, orthogonal vectors in global memory
@pytest.mark.parametrize("c,dc,k,sc", [(3, 12, 9, 3), (1, 2052, 255, 32), (7, 1300, 256, 32), (200, 640, 33, 2), (33, 2064, 241, 12), (2, 60_000, 15, 4),
                                       (300, 64, 20, 3), (1000, 64, 20, 3), (150, 64, 212, 20), (300, 64, 68, 32)])
def test_chunk_recoveries_in_clusters(sgc, c, dc, k, sc):  # noqa: F811
    _chunk_parity(sgc, c, dc, k, sc, 3)


# the same with more chunks than the clusters have room for: a batch begins while the records of the one before are still being written
@pytest.mark.parametrize("c,dc,k,sc", BATCHED)
def test_chunk_recoveries_in_batches(sgc, c, dc, k, sc):  # noqa: F811
    _chunk_parity(sgc, c, dc, k, sc, 3)


def test_records_of_the_chunk_form_name_batches_and_teams(sgc):  # noqa: F811
    hp = [inputs.ADAM[q] for q in ("lr", "beta1", "beta2", "eps")]
    g = cuda(np.random.default_rng(0).standard_t(3.0, size=256 * 8064).astype(np.float32))
    seen = set()
    for c, dc, k, s in BATCHED + [(300, 64, 20, 3), (1000, 64, 20, 3), (150, 64, 212, 20)]:
        me = sgc.Mesgc(c * dc, c, k, s, 3, *hp)
        me.step(g, cuda(np.zeros(c * dc, dtype=np.float32)))
        form, batches, warps, shared = (int(v) for v in me.chunks[-1].get("chunk_form"))
        assert form == 3 and ((c, dc, k, s) not in BATCHED or (batches > 1 and warps > 1))
        seen |= {("warps", warps), ("shared", shared)}
        me.close()
    assert {("warps", 1), ("warps", 2), ("warps", 4), ("shared", 0), ("shared", 1)} <= seen


# the general form's side of the rules: a correlation and a decision per pick (form 1), the correlations on the tensor cores (form 2: more than
# 1e9 multiply-adds, too many columns for the whole GPU's shared memory; one pass over the residuals, and two)
@pytest.mark.parametrize("c,dc,k,sc,form", [(40, 508, 3, 1, 1), (700, 260, 17, 2, 1), (1000, 52, 250, 2, 1), (260, 20_000, 7, 1, 1), (522, 616, 199, 2, 1),
                                            (10, 200_000, 256, 2, 2), (130, 60_000, 250, 1, 2), (70, 65_540, 130, 2, 2)])
def test_chunk_lists_in_the_general_form(sgc, c, dc, k, sc, form):  # noqa: F811
    _chunk_parity(sgc, c, dc, k, sc, form)


# the first step of a list builds its table; a stream that does not wait for the default one finds it complete, whichever form the list takes
# (cluster, whole GPU, general)
@pytest.mark.parametrize("c,dc,k,sc,form", [(600, 64, 20, 4, 3), (3, 40_004, 130, 3, 4), (1000, 512, 8, 1, 1)])
def test_first_chunked_step_on_a_side_stream(sgc, c, dc, k, sc, form):  # noqa: F811
    import torch
    hp = [inputs.ADAM[q] for q in ("lr", "beta1", "beta2", "eps")]
    g = cuda(np.random.default_rng(c).standard_t(3.0, size=c * dc).astype(np.float32))
    side, want = torch.cuda.Stream(), None
    torch.cuda.synchronize()
    for turn in range(4):
        me, w = sgc.Mesgc(c * dc, c, k, sc, 3, *hp), torch.zeros(c * dc, device="cuda")
        torch.cuda.synchronize()
        me.step(g, w, stream=side if turn else None)
        side.synchronize()
        assert int(me.chunks[0].get("chunk_form")[0]) == form
        got = w.cpu().numpy()
        want = got if want is None else want
        assert np.array_equal(got, want) and (got != 0).any()
        me.close()


# chunk recoveries on the whole GPU (form 4; too many columns for a cluster): 64 to 256 rows of A, a ragged last block, tiles of residual rows
# that are full, nearly empty, and brought in one after the other where there is room for one only; books in several turns
@pytest.mark.parametrize("c,dc,k,sc", [(65, 60_000, 40, 2), (3, 40_004, 130, 3), (130, 22_004, 250, 1), (70, 30_000, 97, 2), (1, 70_016, 64, 5),
                                       (400, 14_000, 40, 2)])
def test_chunk_recoveries_on_the_whole_gpu(sgc, c, dc, k, sc):  # noqa: F811
    _chunk_parity(sgc, c, dc, k, sc, 4)


# single vectors small enough for one cluster: every remainder of four, several blocks in the first kernel, kept entries in the tail
@pytest.mark.parametrize("d,k,s,n", [(33, 32, 32, 1), (1026, 100, 7, 1), (4095, 256, 16, 2), (20_001, 64, 5, 3), (65_533, 16, 3, 1)])
def test_small_states_recover_in_one_cluster(sgc, d, k, s, n):  # noqa: F811
    hp = [inputs.ADAM[q] for q in ("lr", "beta1", "beta2", "eps")]
    sts, refs = [sgc.Sgc(d, k, s, 6, *hp) for _ in range(n)], [oracle.Oracle(d, k, s, 6, *hp) for _ in range(n)]
    ws, wr = [cuda(inputs.weights(d, i)) for i in range(n)], [inputs.weights(d, i) for i in range(n)]
    for step in range(3):
        gs = [np.random.default_rng(10 * step + i).standard_t(3.0, size=d).astype(np.float32) for i in range(n)]
        for g in gs:
            g[d - 1 - step] = 30.0
        if n == 1:
            sts[0].step(cuda(gs[0]), ws[0])
        else:
            sgc.step_group(sts, [cuda(g) for g in gs], ws)
        for st, ref, g, w in zip(sts, refs, gs, wr):
            ref.step(g, w)
            assert st.last_launches() == 3 and int(st.get("fallback")) == 1 and int(st.get("chunk_form")[0]) == 3
            for name in ("sel_idx", "sel_val", "lamM", "lamV", "doneM", "doneV", "upd_idx"):
                assert np.array_equal(st.get(name), ref.get(name)), (step, name)
    for w, r in zip(ws, wr):
        assert parity.rel(w.cpu().numpy(), r) < 1e-5
    for st in sts + refs:
        st.close()


def _near_tie(k, seed, supp, p, c, gap, rng):
    """A float32 vector of the columns `supp`, some 2e-7 of it left over once they are projected out, and column c ahead of column p there by `gap` of a
    score.  The lead is linear in the vector, so that units in the last place of its entries set it, to some 1e-10."""
    ext = np.longdouble                                                    # (a mantissa of 64 bits)
    z = np.stack([oracle.z_block(seed, 0, k, int(i), 1).reshape(-1) for i in [*supp, p, c]], 1).astype(ext)
    z /= np.sqrt((z * z).sum(0))
    q = np.zeros((k, len(supp)), ext)

    def rest(v, n=len(supp)):
        for _ in range(2):
            v = v - q[:, :n] @ (q[:, :n].T @ v)
        return v
    for j in range(len(supp)):
        v = rest(z[:, j], j)
        q[:, j] = v / np.sqrt(v @ v)
    hp, hc = rest(z[:, -2]), rest(z[:, -1])
    y = (z[:, :-2] @ (np.linspace(1.0, 0.6, len(supp)) * rng.choice([-1, 1], len(supp))).astype(ext) + ext(2e-7) * (z[:, -2] + z[:, -1])).astype(np.float32)
    unit = np.spacing(np.abs(y)).astype(ext)
    step, left, n = (hc - hp) * unit, ext(gap) * (hc @ y.astype(ext)) - (hc - hp) @ y.astype(ext), np.zeros(k, int)
    coarse = np.argsort(-np.abs(step))[::8]
    for i in coarse:
        n[i] = int(np.clip(np.rint(float(left / step[i])), -4, 4))
        left -= n[i] * step[i]
    fine = np.setdiff1d(np.arange(k), coarse)                              # one unit up here, one down there, and one more of a third entry
    a, b, sign = fine[:300], np.tile(fine[300:], 2), np.repeat([1, -1], fine.size - 300)
    pair = (step[a][:, None] - step[a][None, :]).astype(float).ravel()
    order, want = np.argsort(pair), (left - sign * step[b]).astype(float)
    at = np.clip(np.searchsorted(pair[order], want), 0, pair.size - 1)
    i = int(np.argmin(np.abs(pair[order][at] - want)))
    u, v = divmod(int(order[at[i]]), 300)
    n[b[i]] += sign[i]; n[a[u]] += 1; n[a[v]] -= 1
    y = (y.astype(ext) + n * unit).astype(np.float32)
    lead = float((hc - hp) @ y.astype(ext) / (hc @ y.astype(ext)))
    assert abs(lead - gap) < 0.25 * abs(gap)
    return y


# a pick of the candidate list against a column that only the screening pass has seen, 2e-9 of a score apart (some 2e-10 is what double precision
# leaves open at a residual of 1e-7): the confirmed order is that of the scores
@pytest.mark.parametrize("gap", [2e-9, -2e-9])
def test_a_pick_and_its_challenger_a_hair_apart(sgc, gap):  # noqa: F811
    import torch
    d, k, s, seed = 1 << 18, 1024, 18, 5
    rng = np.random.default_rng(3)
    for _ in range(4):
        cols = rng.choice(d, s + 1, replace=False)
        supp, p, c = cols[:16], cols[16], cols[18]                         # (p has been kept, c has not)
        y = _near_tie(k, seed, supp, p, c, gap, rng)
        st, w = sgc.Sgc(d, k, s, seed, 1e-3, 0.5, 0.999, 1e-8), torch.zeros(d, device="cuda")
        st.set_mode(sgc.MODE_SPECULATIVE)
        g = np.zeros(d, dtype=np.float32)
        g[cols[:18]] = rng.choice([-1, 1], 18) * (1 + rng.random(18))
        st.step(cuda(g), w)
        st.set_state(y, st.get("V"), 0)                                    # beta1 = 1/2 and t = 0: M^ is y to the last bit
        st.step(cuda(g * np.float32(1e-30)), w)
        lam = st.get("lamM")
        assert set(lam[:16]) == set(supp.astype(np.uint32)) and lam[16] == (c if gap > 0 else p) and lam[17] == (p if gap > 0 else c)
        assert int(st.get("fallback")) == 0
        st.close()
