"""The failure path of the tensor-core screening pass, exercised without breaking anything.

Every wait on a hardware barrier inside the pass is bounded.  With the bound set to one nanosecond (sgc_set_wait_limit)
ordinary waits run out: the kernel is intact, its warps merely give up early, flag the error, let what is in flight
finish, return their tensor memory and exit.  The caller must see the flag, the step must still produce Algorithm 3's
result (finished in lock-step) with SGC_STATUS_TIMEOUT set, and the next ordinary step must be an ordinary one again.
"""
import numpy as np
import pytest

import oracle
from paper_2502_00311_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sgc():
    import torch
    assert torch.cuda.is_available()
    from paper_2502_00311_b200 import binding
    binding.lib()
    return binding


def cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def screen_case(sgc, seed, d, k, n):
    import torch
    rng = np.random.default_rng(5)
    R = rng.standard_normal((n, k)).astype(np.float16)
    tau = np.full(n, 4.0 * np.sqrt(k) * 1.0, dtype=np.float32)           # ~4 noise deviations of a unit-variance residual
    return torch.from_numpy(R.view(np.int16)).cuda(), torch.from_numpy(tau).cuda()


def test_screen_reports_an_expired_wait_and_the_next_pass_is_clean(sgc):
    import torch
    seed, d, k, n = 4, 100_003, 256, 64
    rt, tau = screen_case(sgc, seed, d, k, n)
    ref_count, _, err = sgc.screen(seed, d, k, rt, tau, 256)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    try:
        sgc.set_screen_wait_limit(1)
        _, _, err = sgc.screen(seed, d, k, rt, tau, 256)
        torch.cuda.synchronize()                                        # the kernel returned: nothing hangs, nothing faults
        assert int(err.item()) == 1
    finally:
        sgc.set_screen_wait_limit(0)
    count, _, err = sgc.screen(seed, d, k, rt, tau, 256)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert np.array_equal(count.cpu().numpy(), ref_count.cpu().numpy())


def compare_step(st, ref, g, w_gpu, w_ref):
    st.step(cuda(g), w_gpu)
    ref.step(g, w_ref)
    for name in ("sel_idx", "lamM", "lamV"):
        assert np.array_equal(st.get(name), ref.get(name)), name
    n = int(ref.get("n_upd"))
    assert st.get("n_upd") == n and np.array_equal(st.get("upd_idx")[:n], ref.get("upd_idx")[:n])
    a, b = st.get("upd_val")[:n], ref.get("upd_val")[:n]
    assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max()


def test_step_survives_an_expired_wait_and_recovers(sgc):
    d, k, s, seed = 1 << 17, 512, 16, 2
    hp = inputs.ADAM
    st = sgc.Sgc(d, k, s, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    ref = oracle.Oracle(d, k, s, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    supp, sign = inputs.planted_support(d, s, 31)
    w0 = inputs.weights(d, 3)
    w_gpu, w_ref = cuda(w0.copy()), w0.copy()
    grads = [inputs.gradient(d, "student", supp, sign, 900 + i) for i in range(5)]
    for i in range(2):
        compare_step(st, ref, grads[i], w_gpu, w_ref)
    assert int(st.get("fallback")) == 0 and not st.status() & sgc.STATUS_TIMEOUT
    st.set_wait_limit(1)
    compare_step(st, ref, grads[2], w_gpu, w_ref)                       # the pass gives up; lock-step finishes the step
    assert st.status() & sgc.STATUS_TIMEOUT
    assert int(st.get("fallback")) == 1
    st.set_wait_limit(0)
    st.clear_status()
    compare_step(st, ref, grads[3], w_gpu, w_ref)
    compare_step(st, ref, grads[4], w_gpu, w_ref)
    assert int(st.get("fallback")) == 0 and int(st.get("rounds")) == 1   # one screening pass confirms every pick again
    assert not st.status() & sgc.STATUS_TIMEOUT
    st.close()
    ref.close()


# form 4: all picks in one launch on the whole GPU; form 2: a screening pass per pick
@pytest.mark.parametrize("c,dc,k,sc,form", [(64, 65_536, 112, 4, 4), (10, 200_000, 256, 2, 2)])
def test_chunked_tensor_route_survives_an_expired_wait(sgc, c, dc, k, sc, form):
    # MESGC chunks with k_c > 32 and many columns screen on the tensor cores (steps 0 and 2 check that route against the oracles); an expired
    # wait (step 1) sends every recovery of that step through all columns (4) or through the fp32 kernels (2), and is reported in the
    # chunks' status words
    seed = 9
    hp = inputs.ADAM
    me = sgc.Mesgc(c * dc, c, k, sc, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    refs = [oracle.Oracle(dc, k, sc, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"]) for _ in range(c)]
    supp, sign = inputs.planted_support(c * dc, c * sc, 77)
    w0 = inputs.weights(c * dc, 5)
    w_gpu, w_ref = cuda(w0.copy()), w0.copy()
    for step in range(3):
        g = inputs.gradient(c * dc, "student", supp, sign, 300 + step)
        me.chunks[0].set_wait_limit(1 if step == 1 else 0)               # the first state of the list owns the passes
        me.step(cuda(g), w_gpu)
        for i, ref in enumerate(refs):
            ref.step(g[i * dc:(i + 1) * dc], w_ref[i * dc:(i + 1) * dc])
            assert np.array_equal(me.chunks[i].get("lamM"), ref.get("lamM")), (step, i)
            assert np.array_equal(me.chunks[i].get("lamV"), ref.get("lamV")), (step, i)
        assert int(me.chunks[0].get("chunk_form")[0]) == form
        timed_out = any(ch.status() & sgc.STATUS_TIMEOUT for ch in me.chunks)
        assert timed_out == (step == 1)
        for ch in me.chunks:
            ch.clear_status()
        np.testing.assert_allclose(w_gpu.cpu().numpy(), w_ref, rtol=0, atol=1e-6)
    me.close()
    for ref in refs:
        ref.close()


# one batch of chunks per cluster; several batches, with the orthogonal vectors in shared memory and in global memory
@pytest.mark.parametrize("c,dc,k,sc", [(5, 4096, 100, 8), (256, 8064, 164, 2), (400, 1684, 248, 8)])
def test_cluster_recoveries_go_on_when_a_wait_expires(sgc, c, dc, k, sc):
    # the picks of small problems are made inside clusters whose blocks wait for one another's data; an expired wait (step 1) is
    # reported, every block makes the picks of its recoveries by itself, and the next step is an ordinary one
    seed = 9
    hp = inputs.ADAM
    me = sgc.Mesgc(c * dc, c, k, sc, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    refs = [oracle.Oracle(dc, k, sc, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"]) for _ in range(c)]
    supp, sign = inputs.planted_support(c * dc, c * sc, 77)
    w_gpu, w_ref = cuda(np.zeros(c * dc, dtype=np.float32)), np.zeros(c * dc, dtype=np.float32)
    for step in range(3):
        g = inputs.gradient(c * dc, "student", supp, sign, 300 + step)
        me.chunks[0].set_wait_limit(1 if step == 1 else 0)
        me.step(cuda(g), w_gpu)
        for i, ref in enumerate(refs):
            ref.step(g[i * dc:(i + 1) * dc], w_ref[i * dc:(i + 1) * dc])
            for name in ("doneM", "doneV", "lamM", "lamV", "upd_idx"):
                assert np.array_equal(me.chunks[i].get(name), ref.get(name)), (step, i, name)
        assert any(ch.status() & sgc.STATUS_TIMEOUT for ch in me.chunks) == (step == 1)
        for ch in me.chunks:
            ch.clear_status()
        np.testing.assert_allclose(w_gpu.cpu().numpy(), w_ref, rtol=0, atol=1e-6)
    me.close()
    for ref in refs:
        ref.close()


def test_small_state_goes_on_when_a_wait_expires(sgc):
    d, k, s, seed = 4096, 256, 16, 4
    hp = inputs.ADAM
    st = sgc.Sgc(d, k, s, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    ref = oracle.Oracle(d, k, s, seed, hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    supp, sign = inputs.planted_support(d, s, 31)
    w_gpu, w_ref = cuda(inputs.weights(d, 3)), inputs.weights(d, 3)
    for step in range(3):
        st.set_wait_limit(1 if step == 1 else 0)
        compare_step(st, ref, inputs.gradient(d, "student", supp, sign, 900 + step), w_gpu, w_ref)
        assert bool(st.status() & sgc.STATUS_TIMEOUT) == (step == 1)
        st.clear_status()
    st.close()
    ref.close()


# a list in clusters, on the whole GPU and in the general form; a single small state and one that is not small
@pytest.mark.parametrize("c,dc,k,s,form", [(6, 512, 100, 8, 3), (3, 40_004, 130, 3, 4), (1000, 512, 8, 1, 1), (0, 4096, 256, 16, 3), (0, 40_000, 300, 4, 0)])
def test_a_step_whose_first_launch_fails_does_not_count(sgc, c, dc, k, s, form):
    # launches into a stream whose capture has become invalid are refused by the runtime: M, V and t stay what they were
    import ctypes
    import torch
    rt = ctypes.CDLL("libcudart.so.12")
    hp = [inputs.ADAM[q] for q in ("lr", "beta1", "beta2", "eps")]
    grads = [cuda(np.random.default_rng(i).standard_t(3.0, size=max(c, 1) * dc).astype(np.float32)) for i in range(2)]
    side, outs = torch.cuda.Stream(), []
    torch.cuda.synchronize()
    for refused in (False, True):
        opt = sgc.Mesgc(c * dc, c, k, s, 3, *hp) if c else sgc.Sgc(dc, k, s, 3, *hp)
        st, w = opt.chunks[-1] if c else opt, torch.zeros(max(c, 1) * dc, device="cuda")
        torch.cuda.synchronize()
        opt.step(grads[0], w, stream=side)
        assert int(st.get("chunk_form")[0]) == form
        if refused:
            before = st.get("M"), st.get("V"), w.cpu().numpy()
            cs = ctypes.c_void_p(side.cuda_stream)
            assert rt.cudaStreamBeginCapture(cs, 2) == 0
            assert rt.cudaStreamSynchronize(cs) != 0                       # not allowed while capturing, which ends the capture's validity
            with pytest.raises(sgc.SgcError):
                opt.step(grads[1], w, stream=side)
            graph = ctypes.c_void_p()
            assert rt.cudaStreamEndCapture(cs, ctypes.byref(graph)) != 0 and not graph.value
            rt.cudaGetLastError()
            assert int(st.get("t")) == 1
            for a, b in zip(before, (st.get("M"), st.get("V"), w.cpu().numpy())):
                assert np.array_equal(a, b)
        opt.step(grads[1], w, stream=side)
        side.synchronize()
        assert int(st.get("t")) == 2
        outs.append((st.get("M"), w.cpu().numpy()))
        opt.close()
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


def test_a_chunk_list_without_room_for_reports_takes_the_general_form(sgc):
    # the recoveries on the whole GPU keep report lists of 16 KB each; when they cannot be allocated the step is made in launches that need none
    import ctypes
    import torch
    rt = ctypes.CDLL("libcudart.so.12")
    hp = [inputs.ADAM[q] for q in ("lr", "beta1", "beta2", "eps")]
    c, dc, k, s = 200, 19_000, 100, 2
    g = cuda(np.random.default_rng(0).standard_t(3.0, size=c * dc).astype(np.float32))
    small, forms, outs = sgc.Mesgc(27 * 9008, 27, 121, 1, 3, *hp), [], []
    small.step(g, torch.zeros(27 * 9008, device="cuda"))                   # (its kernels are those of the general form below: they are loaded now)
    assert int(small.chunks[0].get("chunk_form")[0]) == 1
    for full in (False, True):
        me, w, held = sgc.Mesgc(c * dc, c, k, s, 3, *hp), torch.zeros(c * dc, device="cuda"), []
        torch.cuda.synchronize()
        try:
            for size in (1 << 30, 1 << 26, 1 << 22) if full else ():
                p = ctypes.c_void_p()
                while rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0:
                    held.append(p)
                    p = ctypes.c_void_p()
            if full:
                rt.cudaGetLastError()
                assert rt.cudaFree(held.pop()) == 0                        # 4 MB, and less than 4 more, for lists of 6.5
            me.step(g, w)
            torch.cuda.synchronize()
        finally:
            for p in held:
                rt.cudaFree(p)
        forms.append(int(me.chunks[0].get("chunk_form")[0]))
        outs.append(w.cpu().numpy())
        me.close()
    small.close()
    assert forms == [4, 1] and np.array_equal(outs[0] != 0, outs[1] != 0)
    assert np.abs(outs[0] - outs[1]).max() <= 1e-6 * np.abs(outs[0]).max()


def test_states_of_very_different_k_live_side_by_side(sgc):
    # the lock-step kernel's shared-memory opt-in belongs to the kernel, not to a state: creating a small-k state must
    # not take away what a large-k state needs
    hp = inputs.ADAM
    big = dict(d=1 << 16, k=16384, s=2, seed=5)
    small = dict(d=1 << 16, k=256, s=4, seed=6)
    sts, refs, ws, wr = [], [], [], []
    for cfg in (big, small):                                             # the small state is created second
        st = sgc.Sgc(cfg["d"], cfg["k"], cfg["s"], cfg["seed"], hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
        st.set_mode(sgc.MODE_LOCKSTEP)
        sts.append(st)
        refs.append(oracle.Oracle(cfg["d"], cfg["k"], cfg["s"], cfg["seed"], hp["lr"], hp["beta1"], hp["beta2"], hp["eps"]))
        w0 = inputs.weights(cfg["d"], 11)
        ws.append(cuda(w0.copy()))
        wr.append(w0.copy())
    for step in range(2):
        for cfg, st, ref, w_gpu, w_ref in zip((big, small), sts, refs, ws, wr):
            supp, sign = inputs.planted_support(cfg["d"], cfg["s"], 40 + cfg["k"])
            g = inputs.gradient(cfg["d"], "student", supp, sign, 700 + step)
            compare_step(st, ref, g, w_gpu, w_ref)
    for st, ref in zip(sts, refs):
        st.close()
        ref.close()
