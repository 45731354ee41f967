"""Calls of different sizes from two host threads at once, each on a stream and a
workspace of its own (what the header asks of concurrent calls): every call
succeeds, and the last one gave the oracle's result (SEQUENTIAL dispatch, which
changes its inputs, is checked by its status).  The sizes differ in the shared memory
that the same kernel is launched with."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_2609_15359_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2609_15359_gb300 import maps
    return maps


def dev(x, dt=np.int32):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=dt)).cuda()


# Each form: the call's arguments up to its workspace, and what it gives.  The
# library is called with plain addresses, so that little else lies between two
# calls of a thread.

def sequential(M, oracle, big):
    D, H, J = (32, 16384, 6) if big else (2, 100, 3)
    rng = np.random.default_rng(D)
    K = rng.integers(0, 50, (D, H)).astype(np.int32)
    cap, Q = np.full(D, 2**30, np.int32), np.zeros(D, np.int32)
    cp, cb = np.zeros(J, np.int32), np.ones(J, np.int32)  # K at one step grows by one a candidate
    t = [dev(x) for x in (K, cap, Q, cp, cb)]
    out, head = dev(np.zeros(J)), dev(np.zeros(J), np.int64)
    Kd, capd, Qd, cpd, cbd = (x.data_ptr() for x in t)
    args = (1, D, H, 1, Kd, None, capd, Qd, None, 0, None, None, None, J, cpd, cbd, out.data_ptr(),
            head.data_ptr())
    return M.lib.maps_dispatch, args, [], (t, out, head)


def snapshot(M, oracle, big):
    D, H, J = (512, 4096, 700) if big else (400, 4096, 700)  # one tile width, past the direct form
    rng = np.random.default_rng(D)
    K = rng.integers(0, 5000, (D, H)).astype(np.int32)
    cap, Q = rng.integers(5000, 9000, D).astype(np.int32), rng.integers(0, 4, D).astype(np.int32)
    cp, cb = rng.integers(0, 500, J).astype(np.int32), rng.integers(1, H, J).astype(np.int32)
    _, ch, hr, _, _ = oracle.dispatch(0, D, H, 1, K, cap, Q, cp, cb)
    t = [dev(x) for x in (K, cap, Q, cp, cb)]
    out, head = dev(np.zeros(J)), dev(np.zeros(J), np.int64)
    Kd, capd, Qd, cpd, cbd = (x.data_ptr() for x in t)
    args = (0, D, H, 1, Kd, None, capd, Qd, None, 0, None, None, None, J, cpd, cbd, out.data_ptr(),
            head.data_ptr())
    return M.lib.maps_dispatch, args, [(out, ch), (head, hr)], t


def order(M, oracle, big):
    N, D = (20000, 1024) if big else (120000, 8)  # both bucketed by the same kernel
    rng = np.random.default_rng(D)
    x = [rng.integers(0, hi, N).astype(np.int32) for hi in (D, 3000, 20, N)]
    _, po, so = oracle.order_local(D, *x, 10)
    t = [dev(v) for v in x]
    perm, seg = dev(np.zeros(N)), dev(np.zeros(D + 1), np.int64)
    args = (N, D, *(v.data_ptr() for v in t), 10, perm.data_ptr(), seg.data_ptr())
    return M.lib.maps_order_local, args, [(perm, po), (seg, so)], t


def stream(M, oracle, big):
    # a window past the one-block loop's: every batch is launched from the host
    N, D, B = (300, 40, 60) if big else (60, 3, 12)
    cfg = (N, D, 1024, 20000, B, 5000, 500000, 100)
    w = W.make_stream(n_requests=N)
    w["arrival_ms"] = w["arrival_ms"] * 40  # completions between the batches
    _, co, qo, so = oracle.stream(*cfg, w["arrival_ms"], w["prompt"], w["true"], w["pred"])
    nb = len(qo)
    assert (qo >= 0).any()
    t = [dev(w["arrival_ms"], np.int64)] + [dev(w[k]) for k in ("prompt", "true", "pred")]
    ch, q, st = dev(np.zeros(N)), dev(np.zeros(nb)), dev(np.zeros((nb, 4)), np.int64)
    c = M.stream_cfg(*cfg)
    args = (ctypes.byref(c), *(v.data_ptr() for v in t), None, ch.data_ptr(), q.data_ptr(), st.data_ptr(), None)
    return M.lib.maps_stream_run, args, [(ch, co), (q, qo), (st, so)], (t, c)


@pytest.mark.parametrize("make,calls", [(sequential, 4000), (snapshot, 8000), (order, 2000), (stream, 20)])
def test_two_threads_of_different_sizes(M, oracle, make, calls):
    sides = [make(M, oracle, big) for big in (True, False)]
    spaces = [M.Workspace(64 << 20) for _ in sides]
    streams = [torch.cuda.Stream() for _ in sides]
    torch.cuda.synchronize()
    failed, done = [], threading.Event()

    def run(i):  # the larger calls, and the smaller ones for as long
        call, args = sides[i][0], (*sides[i][1], spaces[i].buf.data_ptr(), spaces[i].nbytes,
                                   streams[i].cuda_stream)
        n = 0
        while not failed and (n < calls if i == 0 else not done.is_set()):
            status = call(*args)
            n += 1
            if status != 0:
                failed.append((i, n, status, M.lib.maps_last_cuda_error()))
            if n % 50 == 0:
                streams[i].synchronize()
        if i == 0:
            done.set()

    threads = [threading.Thread(target=run, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for (_, _, outs, _), ws in zip(sides, spaces):
        assert M.maps_check(ws) == 0
        for got, want in outs:
            assert np.array_equal(got.cpu().numpy().reshape(want.shape), want)
