"""GPU parity: the CUDA path through the C ABI against the CPU oracle.

Integer work throughout, so every comparison is bit-exact (tolerance 0).
Sizes: the hand-derived goldens, seeded random instances with ragged shapes
that span several tiles, and the benchmark workloads at full size (whole
outputs where the oracle finishes in seconds, sampled candidates otherwise).
"""
import numpy as np
import pytest
import torch

from paper_2609_15359_gb300 import workloads as W

pytestmark = pytest.mark.gpu

I32_MAX = 2**31 - 1


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2609_15359_gb300 import maps
    return maps


@pytest.fixture(scope="module")
def ws(M):
    return M.Workspace()


def dev(x, dtype=None):
    a = np.ascontiguousarray(x if dtype is None else np.asarray(x, dtype=dtype))
    return torch.from_numpy(a).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


# ---------------------------------------------------------------------------
# helpers running one op on the GPU and returning (status, outputs)
# ---------------------------------------------------------------------------

def gpu_calibrate(M, ws, L, P, a, query=None):
    m = 0 if query is None else len(query)
    U = torch.empty(max(m, 1), dtype=torch.int32, device="cuda")
    qd = torch.zeros(1, dtype=torch.int32, device="cuda")
    st, q = M.maps_calibrate(dev(L, np.int32), dev(P, np.int32), a,
                             None if query is None else dev(query, np.int32),
                             U[:m] if m else None, qd, q_host=True, ws=ws)
    return st, q, int(host(qd)[0]), host(U[:m])


def gpu_occupancy(M, ws, D, H, off, p, g, u, with_kmax=False):
    K = torch.full((D, H), -7, dtype=torch.int32, device="cuda")
    km = torch.full(M.kmax_shape(D, H), -7, dtype=torch.int32, device="cuda") if with_kmax else None
    st = M.maps_project_occupancy(D, H, dev(off, np.int64), dev(p, np.int32), dev(g, np.int32),
                                  dev(u, np.int32), K, km, ws=ws)
    assert st == 0
    if with_kmax:
        return M.maps_check(ws), host(K), host(km).view(np.uint32)
    return M.maps_check(ws), host(K)


def kmax_of(K):
    """16-step block maxima of K + t (the summary's definition, in numpy)."""
    D, H = K.shape
    x = K.astype(np.int64) + np.arange(H)
    nb = (H + 15) // 16
    pad = np.full((D, nb * 16), -1, np.int64)
    pad[:, :H] = x
    return pad.reshape(D, nb, 16).max(axis=2).astype(np.uint32)


def gpu_dispatch(M, ws, mode, D, H, S, K, cap, Q, cp, cb, res=None, kmax=None):
    J = len(cp)
    Kd = None if K is None else dev(K, np.int32)
    kmd = None if kmax is None else dev(np.ascontiguousarray(kmax).view(np.int32))
    Qd = dev(Q, np.int32)
    ch = torch.full((max(J, 1),), -9, dtype=torch.int32, device="cuda")
    hr = torch.full((max(J, 1),), -9, dtype=torch.int64, device="cuda")
    kw = {}
    if res is not None:
        kw = dict(res_off=dev(res[0], np.int64), prompt=dev(res[1], np.int32),
                  gen=dev(res[2], np.int32), bound=dev(res[3], np.int32))
    st = M.maps_dispatch(mode, D, H, S, Kd, dev(cap, np.int32), Qd, dev(cp, np.int32),
                         dev(cb, np.int32), ch[:J], hr[:J], kmax=kmd, ws=ws, **kw)
    assert st == 0, st
    st = M.maps_check(ws)
    return st, host(ch[:J]), host(hr[:J]), (None if Kd is None else host(Kd)), host(Qd)


def gpu_order(M, ws, D, dec, U, wait, arr, mw):
    N = len(dec)
    perm = torch.full((max(N, 1),), -1, dtype=torch.int32, device="cuda")
    seg = torch.full((D + 1,), -1, dtype=torch.int64, device="cuda")
    st = M.maps_order_local(D, dev(dec, np.int32), dev(U, np.int32), dev(wait, np.int32),
                            dev(arr, np.int32), mw, perm[:N], seg, ws=ws)
    assert st == 0
    return M.maps_check(ws), host(perm[:N]), host(seg)


# ---------------------------------------------------------------------------
# golden worked examples
# ---------------------------------------------------------------------------

def test_golden_worked_example(M, ws, golden):
    c = golden["calibration"]
    for case in c["cases"]:
        st, q, qd, _ = gpu_calibrate(M, ws, c["true_len"], c["pred_len"], case["alpha_ppm"])
        assert st == case["status"]
        if st == 0:
            assert q == qd == case["q"]
    m = c["misround_case"]
    assert gpu_calibrate(M, ws, m["true_len"], m["pred_len"], m["alpha_ppm"])[1] == m["q"]
    b = c["bound"]
    st, q, _, U = gpu_calibrate(M, ws, [9, 9, 9, 9, 9, 9, 9, 9, 13], [9] * 9, 100000, b["pred"])
    assert st == 0 and q == 4 and U.tolist() == b["U"]

    d, cd = golden["decoders"], golden["candidates"]
    st, K = gpu_occupancy(M, ws, 2, 8, d["res_off"], d["res_prompt"], d["res_gen"], d["res_bound"])
    assert st == 0 and K.tolist() == d["K"]
    res = (d["res_off"], d["res_prompt"], d["res_gen"], d["res_bound"])
    st, ch, hr, _, _ = gpu_dispatch(M, ws, 0, 2, 8, 1, d["K"], d["cap"], d["Q"], cd["prompt"], cd["bound"])
    assert st == 0 and ch.tolist() == golden["snapshot"]["choice"]
    assert hr.tolist() == golden["snapshot"]["headroom"]
    s = golden["sequential"]
    st, ch, hr, Ka, Qa = gpu_dispatch(M, ws, 1, 2, 8, 1, d["K"], d["cap"], d["Q"], cd["prompt"], cd["bound"])
    assert st == 0 and ch.tolist() == s["choice"] and hr.tolist() == s["headroom"]
    assert Ka.tolist() == s["K_after"] and Qa.tolist() == s["Q_after"]
    a = golden["alg1"]
    st, ch, hr, _, _ = gpu_dispatch(M, ws, 2, 2, 8, 1, None, d["cap"], d["Q"], cd["prompt"], cd["bound"], res)
    assert st == 0 and ch.tolist() == a["choice"] and hr.tolist() == a["headroom"]
    st, ch, hr, _, Qa = gpu_dispatch(M, ws, 3, 2, 8, 1, None, d["cap"], d["Q"], cd["prompt"], cd["bound"], res)
    assert st == 0 and ch.tolist() == a["sequential_choice"]
    assert hr.tolist() == a["sequential_headroom"] and Qa.tolist() == a["sequential_Q_after"]
    o = golden["order"]
    st, perm, seg = gpu_order(M, ws, 1, o["dec"], o["bound"], o["wait"], o["arrival"], o["max_wait"])
    assert st == 0 and perm.tolist() == o["perm"] and seg.tolist() == o["seg_off"]


# ---------------------------------------------------------------------------
# calibration
# ---------------------------------------------------------------------------

# one-block sizes: ranked by counting up to 128 scores, then the histogram select
# with 1, 4, 8 and 16 scores a thread; past 16,384 the cooperative kernel
@pytest.mark.parametrize("n", [1, 2, 3, 9, 10, 127, 128, 129, 1000, 1024, 1025, 2048, 2049, 4096, 4097,
                               8192, 8193, 16384, 16385, 65537, 1000003])
def test_calibrate_random(M, ws, oracle, n):
    rng = np.random.default_rng(n)
    L = rng.integers(-(2**31), 2**31, n, dtype=np.int64).astype(np.int32) if n % 2 else \
        rng.integers(0, 3000, n).astype(np.int32)
    P = rng.integers(-(2**31), 2**31, n, dtype=np.int64).astype(np.int32) if n % 3 == 0 else \
        rng.integers(0, 3000, n).astype(np.int32)
    if n > 10:
        P[: n // 4] = L[: n // 4]  # exact zeros
    query = rng.integers(0, 5000, 4099).astype(np.int32)
    for a in (1, 50000, 100000, 200000, 900000, 999999):
        sto, qo = oracle.calibrate(L, P, a)
        if sto == 0:  # the call also bounds the queries, which may overflow
            sto, Uo = oracle.bound(query, qo)
        st, q, qd, U = gpu_calibrate(M, ws, L, P, a, query)
        assert st == sto, (n, a)
        if st == 0:
            assert q == qd == qo
            assert np.array_equal(U, Uo)


def test_calibrate_unaligned_and_ranges(M, ws, oracle):
    rng = np.random.default_rng(3)
    L = rng.integers(0, 10**6, 10001).astype(np.int32)
    P = rng.integers(0, 10**6, 10001).astype(np.int32)
    Ld, Pd = dev(L), dev(P)
    qd = torch.zeros(1, dtype=torch.int32, device="cuda")
    st, q = M.maps_calibrate(Ld[1:], Pd[1:], 100000, q_dev_out=qd, q_host=True, ws=ws)
    assert st == 0 and q == oracle.calibrate(L[1:], P[1:], 100000)[1]
    # score above INT32_MAX -> range error
    st, _ = M.maps_calibrate(dev([I32_MAX] * 3, np.int32), dev([-5] * 3, np.int32), 500000,
                             q_host=True, ws=ws)
    assert st == M.MAPS_E_RANGE
    # bound above INT32_MAX -> range error
    U = torch.empty(1, dtype=torch.int32, device="cuda")
    st, _ = M.maps_calibrate(dev([10] * 3, np.int32), dev([0] * 3, np.int32), 500000,
                             dev([I32_MAX - 3], np.int32), U, q_host=True, ws=ws)
    assert st == M.MAPS_E_RANGE
    # rank above n: unbounded, returned at once
    assert gpu_calibrate(M, ws, [1] * 8, [0] * 8, 100000)[0] == M.MAPS_E_UNBOUNDED
    assert gpu_calibrate(M, ws, [], [], 100000)[0] == M.MAPS_E_UNBOUNDED
    assert M.maps_calibrate(Ld, Pd, 0, ws=ws)[0] == M.MAPS_E_INVALID


@pytest.mark.parametrize("seed,n", [(0, 20011), (1, 20011), (2, 20011), (0, 16384), (1, 9001), (2, 5003),
                                    (0, 4096), (1, 1024), (2, 1000), (0, 128)])
def test_calibrate_grid_bucket_edges(M, ws, oracle, seed, n):
    """Grid form (n above the one-block limit) and the one-block forms: scores
    on the first pass's bin edges (the last exact bin, each leading-bit boundary,
    each 7-bit step) and up to 2^32 - 1, so that quantiles resolve after one, two
    or three passes and some lie above INT32_MAX (range error)."""
    rng = np.random.default_rng(seed)
    edges = {0, 1, 1022, 1023, 1024, 1025, 2**32 - 1}
    for e in range(10, 32):
        step = 1 << (e - 7)
        edges |= {(1 << e) - 1, 1 << e, (1 << e) + 1, (1 << e) + step - 1, (1 << e) + step}
    edges = np.array(sorted(edges), dtype=np.int64)
    s = rng.choice(edges, n)
    s[: n // 3] = rng.integers(0, 2**32, n // 3, dtype=np.int64)  # full range
    P = np.full(n, -(2**31), dtype=np.int64)
    small = s < 2**31 - 5000
    P[small] = rng.integers(-2000, 2000, int(small.sum()))
    L, P = (P + s).astype(np.int32), P.astype(np.int32)
    assert np.array_equal(np.maximum(L.astype(np.int64) - P, 0), s)
    seen = set()
    for a in (1, 30, 1000, 100000, 333333, 500000, 700000, 900000, 999000, 999999):
        sto, qo = oracle.calibrate(L, P, a)
        st, q, qd, _ = gpu_calibrate(M, ws, L, P, a)
        assert st == sto, (seed, a)
        seen.add(st)
        if st == 0:
            assert q == qd == qo, (seed, a)
    assert {0, M.MAPS_E_RANGE} <= seen


@pytest.mark.parametrize("n,m,shift", [
    # more scores than the grid keeps in registers: every pass reads them again
    (1300007, 4099, 0),
    # more predictions than the grid keeps in registers, at an unaligned address
    (20011, 1300003, 1),
    # no queries; then a ragged, unaligned few
    (8193, 0, 0), (10001, 777, 1), (4096, 16384, 0),
    # the one-block form at 16,384 residuals and queries, and past each limit;
    # a thread's last items, and queries past those loaded before the select
    (16384, 16384, 0), (16384, 16385, 1), (16385, 0, 0), (16385, 777, 1), (1024, 8193, 1),
    (1025, 1, 0), (15361, 9000, 0)])
def test_calibrate_fused_register_limits(M, ws, oracle, n, m, shift):
    """Calibration sets above 16,384 scores take one cooperative kernel; its
    scores and predictions live in registers up to eight per thread, else they
    are read from memory, as the one-block form's queries past its eight are: q,
    the bounds and the status match the oracle either way."""
    rng = np.random.default_rng(n + m)
    L = rng.integers(0, 40000, n).astype(np.int32)
    P = rng.integers(0, 40000, n).astype(np.int32)
    P[: n // 5] = L[: n // 5]
    query = rng.integers(0, 70000, m + shift).astype(np.int32)
    Ld, Pd, Qd = dev(L), dev(P), dev(query)
    U = torch.full((m + shift + 1,), -9, dtype=torch.int32, device="cuda")
    qd = torch.zeros(1, dtype=torch.int32, device="cuda")
    for a in (1000, 100000, 999999):  # ranks within n at every size here
        sto, qo = oracle.calibrate(L, P, a)
        st, q = M.maps_calibrate(Ld, Pd, a, Qd[shift:] if m else None, U[shift:shift + m] if m else None,
                                 qd, q_host=True, ws=ws)
        assert st == sto == 0 and q == qo == int(host(qd)[0]), (n, m, a)
        if m:
            Uh = host(U)
            assert np.array_equal(Uh[shift:shift + m], oracle.bound(query[shift:], qo)[1])
            assert Uh[:shift].tolist() == [-9] * shift and Uh[shift + m] == -9
    # a bound above INT32_MAX: the range error, the others still bounded
    big = query[shift:].copy() if m else np.zeros(1, np.int32)
    big[-1] = I32_MAX - 3
    Ub = torch.empty(len(big), dtype=torch.int32, device="cuda")
    st, q = M.maps_calibrate(Ld, Pd, 100000, dev(big), Ub, q_host=True, ws=ws)
    assert st == M.MAPS_E_RANGE
    assert np.array_equal(host(Ub)[:-1], oracle.bound(big[:-1], oracle.calibrate(L, P, 100000)[1])[1])


@pytest.mark.parametrize("n", [3, 16384, 16385])
@pytest.mark.parametrize("m", [5, 16384, 16385])
def test_calibrate_range_error_keeps_no_earlier_quantile(M, oracle, n, m):
    """A quantile above INT32_MAX, in every form: the range error, and what is
    written beside it (the host's quantile, the bounds) does not depend on the
    call that used the workspace before."""
    query = np.arange(m, dtype=np.int32)
    U = torch.empty(m, dtype=torch.int32, device="cuda")
    L, P = dev(np.full(n, I32_MAX, np.int32)), dev(np.full(n, -5, np.int32))
    seen = []
    for earlier in (77, 123456):
        ws = M.Workspace()
        st, q = M.maps_calibrate(dev(np.full(9, earlier, np.int32)), dev(np.zeros(9, np.int32)),
                                 500000, q_host=True, ws=ws)
        assert st == 0 and q == earlier
        U.fill_(-9)
        st, q = M.maps_calibrate(L, P, 500000, dev(query), U, q_host=True, ws=ws)
        assert st == M.MAPS_E_RANGE
        seen.append((q, host(U).tolist()))
    assert seen[0] == seen[1]
    assert seen[0] == (0, query.tolist())


@pytest.mark.parametrize("name", ["tiny", "d16", "d64", "large"])
def test_calibrate_workloads(M, ws, oracle, name):
    w = W.make(name)
    query = np.concatenate([w["res_pred"], w["cand_pred"]])
    for a in w["alphas_ppm"]:
        sto, qo = oracle.calibrate(w["cal_true"], w["cal_pred"], a)
        st, q, qd, U = gpu_calibrate(M, ws, w["cal_true"], w["cal_pred"], a, query)
        assert st == sto == 0 and q == qd == qo
        assert np.array_equal(U, oracle.bound(query, qo)[1])


# ---------------------------------------------------------------------------
# occupancy
# ---------------------------------------------------------------------------

def random_residents(rng, D, H, per_max, with_empty=True):
    R_per = rng.integers(0 if with_empty else 1, per_max + 1, D)
    off = np.concatenate([[0], np.cumsum(R_per)]).astype(np.int64)
    R = int(off[-1])
    p = rng.integers(0, 3000, R).astype(np.int32)
    g = rng.integers(0, 2 * H + 3, R).astype(np.int32)
    U = rng.integers(0, 3 * H + 5, R).astype(np.int32)
    return off, p, g, U


@pytest.mark.parametrize("D,H", [(1, 1), (3, 3), (2, 8), (5, 511), (4, 512), (3, 513), (7, 4095),
                                 (2, 4097), (9, 4100), (3, 12289), (2, 65536),
                                 # 128 horizon tiles (the most the bucketed form takes), then
                                 # more, which stream every resident per tile instead; grids
                                 # past 640 tiles at those, and with few steps a tile
                                 (2, 524288), (2, 524292), (1, 600001), (6, 524288), (6, 524292),
                                 (170, 16384), (700, 1000)])
def test_occupancy_random(M, ws, oracle, D, H):
    rng = np.random.default_rng(D * 100003 + H)
    off, p, g, U = random_residents(rng, D, H, 700)
    sto, Ko = oracle.occupancy(D, H, off, p, g, U)
    st, K, km = gpu_occupancy(M, ws, D, H, off, p, g, U, with_kmax=True)
    assert st == sto == 0
    assert np.array_equal(K, Ko)
    assert np.array_equal(km, kmax_of(Ko))


@pytest.mark.parametrize("name", ["tiny", "d16", "d64", "large"])
def test_occupancy_workloads(M, ws, oracle, name):
    w = W.make(name)
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    sto, Ko = oracle.occupancy(w["D"], w["H"], w["res_off"], w["res_prompt"], w["res_gen"], U)
    st, K, km = gpu_occupancy(M, ws, w["D"], w["H"], w["res_off"], w["res_prompt"], w["res_gen"],
                              U, with_kmax=True)
    assert st == sto == 0
    assert np.array_equal(K, Ko)
    assert np.array_equal(km, kmax_of(Ko))


@pytest.mark.parametrize("D,H,per", [(2, 20000, 9000), (3, 3000, 4097),
                                     (16, 65536, 4096), (16, 65536, 4097), (2, 60001, 40000),
                                     (3, 400000, 4097),
                                     # 640 tiles, and past them and three a decoder, bucketed;
                                     # 768 tiles of three a decoder, one launch
                                     (40, 65536, 2049), (41, 65535, 4097), (129, 20001, 2500),
                                     (7, 400000, 9000), (161, 12289, 1500), (256, 12288, 700)])
def test_occupancy_many_residents_per_decoder(M, ws, oracle, D, H, per):
    """More residents on one decoder than a block stages at once."""
    rng = np.random.default_rng(H + per)
    off = np.arange(D + 1, dtype=np.int64) * per
    R = D * per
    p = rng.integers(0, 300, R).astype(np.int32)
    g = rng.integers(0, H, R).astype(np.int32)
    U = rng.integers(0, 2 * H, R).astype(np.int32)
    sto, Ko = oracle.occupancy(D, H, off, p, g, U)
    st, K, km = gpu_occupancy(M, ws, D, H, off, p, g, U, with_kmax=True)
    assert st == sto == 0
    assert np.array_equal(K, Ko)
    assert np.array_equal(km, kmax_of(Ko))


def test_occupancy_errors(M, ws, oracle):
    # K above INT32_MAX
    big = I32_MAX // 2
    st, _ = gpu_occupancy(M, ws, 1, 4, [0, 2], [big, big], [0, 0], [4, 4])
    assert st == M.MAPS_E_RANGE == oracle.occupancy(1, 4, [0, 2], [big, big], [0, 0], [4, 4])[0]
    st, K = gpu_occupancy(M, ws, 1, 4, [0, 1], [I32_MAX - 4], [0], [4])
    assert st == 0 and K[0].tolist() == [I32_MAX - 3, I32_MAX - 2, I32_MAX - 1, I32_MAX]
    st, _ = gpu_occupancy(M, ws, 1, 8, [0, 1], [-1], [0], [3])
    assert st == M.MAPS_E_RANGE
    st, _ = gpu_occupancy(M, ws, 2, 8, [0, 2, 1], [1, 1], [0, 0], [3, 3])
    assert st == M.MAPS_E_RANGE
    st, _ = gpu_occupancy(M, ws, 1, 8, [0, 5], [1, 1], [0, 0], [3, 3])  # beyond R
    assert st == M.MAPS_E_RANGE
    K = torch.empty((1, 8), dtype=torch.int32, device="cuda")
    assert M.maps_project_occupancy(0, 8, dev([0], np.int64), dev([1], np.int32), dev([0], np.int32),
                                    dev([1], np.int32), K, ws=ws) == M.MAPS_E_INVALID


# ---------------------------------------------------------------------------
# dispatch
# ---------------------------------------------------------------------------

def diverse_caps(rng, K, spread):
    """Capacities straddling each decoder's occupancy so that the feasible set
    changes from candidate to candidate (test input built from the oracle)."""
    base = K[:, 0].astype(np.int64)
    off = rng.integers(-spread, spread // 2, K.shape[0])
    off[rng.integers(K.shape[0])] = spread // 2 - 1  # at least one roomy decoder
    return np.clip(base + off, 0, I32_MAX).astype(np.int32)


def check_dispatch(M, ws, oracle, mode, D, H, K, cap, Q, cp, cb, S=1, res=None):
    sto, co, ho, Ko, Qo = oracle.dispatch(mode, D, H, S, K, cap, Q, cp, cb,
                                          *(res if res is not None else ()))
    runs = [None, kmax_of(np.asarray(K))] if mode == 0 else [None]
    for km in runs:  # SNAPSHOT: summary derived inside, and passed in
        st, ch, hr, Ka, Qa = gpu_dispatch(M, ws, mode, D, H, S, K, cap, Q, cp, cb, res, km)
        assert st == sto
        if st == 0:
            assert np.array_equal(ch, co)
            assert np.array_equal(hr, ho)
            if mode == 1:
                assert np.array_equal(Ka, Ko)
            assert np.array_equal(Qa, Qo)
    return co, ho


@pytest.mark.parametrize("D,H,J", [(1, 1, 1), (1, 9, 33), (2, 8, 40), (3, 100, 700), (5, 511, 1000),
                                   (17, 4100, 3000), (64, 4096, 5000), (255, 1000, 3000),
                                   (256, 8192, 6000), (257, 2048, 2000), (300, 777, 1500),
                                   (1024, 1024, 2000),
                                   # 32-column tiles (129..256 decoders), copied by TMA and,
                                   # with H not a multiple of 4, by plain loads
                                   (129, 3000, 2000), (200, 1001, 2000)])
def test_dispatch_snapshot_random(M, ws, oracle, D, H, J):
    rng = np.random.default_rng(D * 7919 + H)
    off, p, g, U = random_residents(rng, D, H, 40)
    _, K = oracle.occupancy(D, H, off, p, g, U)
    cap = diverse_caps(rng, K, 4000)
    # tied queue lengths for even D, all distinct for odd D
    Q = (rng.integers(0, 4, D) if D % 2 == 0 else rng.permutation(D)).astype(np.int32)
    cp = rng.integers(0, 3000, J).astype(np.int32)
    cb = rng.integers(0, 2 * H + 2, J).astype(np.int32)
    co, ho = check_dispatch(M, ws, oracle, 0, D, H, K, cap, Q, cp, cb)
    if J >= 100:
        assert (ho >= 0).any() and (ho < 0).any()  # both branches exercised
        if D >= 8:
            assert len(set(co.tolist())) > 1


@pytest.mark.parametrize("D,H,J,unaligned", [
    # the one-launch form at its limits and the bucketed form just past them:
    # scores, scores times spans of the horizon, cells of K
    (16, 2048, 8192, False), (16, 2048, 8193, False), (32, 9001, 2048, False),
    (32, 9001, 2049, False), (1000, 1048, 60, False), (1000, 1049, 60, False),
    (7, 32768, 300, False), (7, 32769, 300, False),
    # summary rows of whole 16-byte words and not, at an aligned address and
    # not; 32-decoder groups at their edges; one candidate
    (31, 640, 100, True), (33, 1000, 1, False), (64, 64, 65, False), (1024, 100, 9, True),
    # rows read word by word, around 128 blocks of the summary and past twice as many;
    # the most candidates of the one-launch form, of few decoders and of 18 in four groups
    (330, 2047, 20, False), (330, 2081, 20, False), (9, 4400, 70, True), (3, 30001, 33, False),
    (2, 300, 16384, False), (2, 300, 16385, False), (18, 104, 4096, False), (18, 104, 4097, False),
    # wide tiles of the bucketed form (few decoders, many candidates)
    (5, 4099, 60000, False), (40, 4096, 9000, True)])
def test_dispatch_snapshot_forms(M, ws, oracle, D, H, J, unaligned):
    rng = np.random.default_rng(D * 37 + H + J)
    off, p, g, U = random_residents(rng, D, H, 12)
    _, K = oracle.p_occupancy(D, H, off, p, g, U)
    cap = diverse_caps(rng, K, 4000)
    Q = rng.integers(0, 4, D).astype(np.int32)
    cp = rng.integers(0, 3000, J).astype(np.int32)
    cb = rng.integers(0, H + 2, J).astype(np.int32)
    cb[: min(J, 5)] = [0, 15, 16, 17, H][: min(J, 5)]
    _, co, ho = oracle.p_dispatch_snapshot(D, H, K, cap, Q, cp, cb)
    km = kmax_of(K)
    shift = 1 if unaligned else 0
    kd = torch.empty(km.size + shift, dtype=torch.int32, device="cuda")[shift:].view(*km.shape)
    kd.copy_(torch.from_numpy(km.view(np.int32)))
    Kd = torch.empty(K.size + shift, dtype=torch.int32, device="cuda")[shift:].view(*K.shape)
    Kd.copy_(torch.from_numpy(K))
    ch = torch.empty(J, dtype=torch.int32, device="cuda")
    hr = torch.empty(J, dtype=torch.int64, device="cuda")
    for summary in (kd, None):
        assert M.maps_dispatch(0, D, H, 1, Kd, dev(cap), dev(Q), dev(cp), dev(cb), ch, hr,
                               kmax=summary, ws=ws) == 0
        assert M.maps_check(ws) == 0
        assert np.array_equal(host(ch), co) and np.array_equal(host(hr), ho)
    # a negative cell is reported: without a summary, and with one too in the
    # one-launch form (the bucketed form reads only the candidates' tiles then)
    rows = next(8 * s for s in (1, 2, 4, 8) if 8 * s >= D or s == 8)  # whole groups of 8 a warp
    one_launch = (J * (-(-D // rows) * rows) <= 2**17 and J * D * max(1, H // 2048) <= 2**18
                  and H <= 32768 and D * H <= 2**20)
    Kd[D - 1, H // 2] = -5
    for summary in (kd, None) if one_launch else (None,):
        M.maps_dispatch(0, D, H, 1, Kd, dev(cap), dev(Q), dev(cp), dev(cb), ch, hr, kmax=summary, ws=ws)
        assert M.maps_check(ws) in (M.MAPS_E_RANGE, M.MAPS_E_INVALID)


@pytest.mark.parametrize("name", ["tiny", "d16", "d64"])
@pytest.mark.parametrize("variant", ["given", "feasible", "diverse"])
def test_dispatch_snapshot_workloads(M, ws, oracle, name, variant):
    w = W.make(name, feasible=(variant == "feasible"))
    rng = np.random.default_rng(11)
    for a in w["alphas_ppm"]:
        q = oracle.calibrate(w["cal_true"], w["cal_pred"], a)[1]
        U = oracle.bound(w["res_pred"], q)[1]
        cb = oracle.bound(w["cand_pred"], q)[1]
        _, K = oracle.occupancy(w["D"], w["H"], w["res_off"], w["res_prompt"], w["res_gen"], U)
        cap, Q = w["cap"], w["Q"]
        if variant == "diverse":
            cap = diverse_caps(rng, K, 3000)
            Q = rng.integers(0, 3, w["D"]).astype(np.int32)
        check_dispatch(M, ws, oracle, 0, w["D"], w["H"], K, cap, Q, w["cand_prompt"], cb)


@pytest.mark.parametrize("variant", ["given", "feasible", "diverse"])
def test_dispatch_snapshot_large_full(M, ws, oracle, variant):
    """Full size, in the benchmark's launch configuration: every one of the
    65,536 candidates against the plain oracle (pinned to the by-definition
    one in test_oracle_tier_p.py), and a sample of them against the
    by-definition oracle itself."""
    w = W.make("large", feasible=(variant == "feasible"))
    D, H, J = w["D"], w["H"], w["J"]
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1]
    _, K = oracle.p_occupancy(D, H, w["res_off"], w["res_prompt"], w["res_gen"], U)
    cap, Q = w["cap"], w["Q"]
    rng = np.random.default_rng(5)
    if variant == "diverse":
        cap = diverse_caps(rng, K, 6000)
        Q = rng.integers(0, 3, D).astype(np.int32)
    st, ch, hr, _, _ = gpu_dispatch(M, ws, 0, D, H, 1, K, cap, Q, w["cand_prompt"], cb,
                                    kmax=kmax_of(K))
    stp, cp_, hp_ = oracle.p_dispatch_snapshot(D, H, K, cap, Q, w["cand_prompt"], cb)
    assert st == stp == 0
    assert np.array_equal(ch, cp_)
    assert np.array_equal(hr, hp_)
    st2, ch2, hr2, _, _ = gpu_dispatch(M, ws, 0, D, H, 1, K, cap, Q, w["cand_prompt"], cb)
    assert st2 == 0 and np.array_equal(ch, ch2) and np.array_equal(hr, hr2)
    idx = np.concatenate([np.argsort(cb)[-32:], rng.choice(J, 300, replace=False)])
    sto, co, ho, _, _ = oracle.dispatch(0, D, H, 1, K, cap, Q, w["cand_prompt"][idx], cb[idx])
    assert sto == 0
    assert np.array_equal(ch[idx], co)
    assert np.array_equal(hr[idx], ho)


@pytest.mark.parametrize("D,H,J", [(1, 5, 20), (2, 8, 50), (3, 100, 300), (7, 513, 400),
                                   (32, 2048, 256), (100, 1000, 300), (1024, 64, 100)])
def test_dispatch_sequential_random(M, ws, oracle, D, H, J):
    rng = np.random.default_rng(D * 31 + H)
    off, p, g, U = random_residents(rng, D, H, 30)
    _, K = oracle.occupancy(D, H, off, p, g, U)
    cap = diverse_caps(rng, K, 3000)
    Q = rng.integers(0, 3, D).astype(np.int32)
    cp = rng.integers(0, 500, J).astype(np.int32)
    cb = rng.integers(0, H + 5, J).astype(np.int32)
    check_dispatch(M, ws, oracle, 1, D, H, K, cap, Q, cp, cb)


@pytest.mark.parametrize("name", ["tiny", "d16", "d64"])
def test_dispatch_sequential_workloads(M, ws, oracle, name):
    w = W.make(name, feasible=True)
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1]
    _, K = oracle.occupancy(w["D"], w["H"], w["res_off"], w["res_prompt"], w["res_gen"], U)
    check_dispatch(M, ws, oracle, 1, w["D"], w["H"], K, w["cap"], w["Q"], w["cand_prompt"], cb)


@pytest.mark.parametrize("D,H,J,spread", [
    # one column warp and many, and several decoders a lane; horizons around a
    # 128-step chunk and a 16-step block; rows past what shared memory holds; a
    # last refill of candidates that is not full
    (1, 127, 33, 3000), (8, 129, 65, 3000), (9, 1000, 64, 3000), (16, 16384, 200, 6000),
    (17, 2049, 100, 3000), (32, 4111, 150, 3000), (33, 4096, 100, 3000), (64, 9001, 130, 6000),
    (100, 5000, 60, 3000), (300, 700, 50, 3000), (1, 300000, 40, 100000),
    # one and two candidates (no row in shared memory), and three; candidates that end
    # in either of the two global chunks in flight
    (1, 5, 1, 3000), (3, 130, 2, 3000), (24, 16509, 2, 6000), (8, 32768, 3, 6000), (200, 4801, 1, 3000),
    (64, 9001, 4, 6000), (1, 300001, 2, 100000), (40, 20003, 30, 6000), (12, 30004, 25, 6000),
    # headrooms further apart than the 32-bit keys hold
    (5, 600, 60, 2**30), (40, 600, 60, 2**30)])
def test_dispatch_sequential_edges(M, ws, oracle, D, H, J, spread):
    rng = np.random.default_rng(D * 131 + H)
    off, p, g, U = random_residents(rng, D, H, 20)
    _, K = oracle.occupancy(D, H, off, p, g, U)
    cap = diverse_caps(rng, K, spread)
    Q = rng.integers(0, 3, D).astype(np.int32)
    cp = rng.integers(0, 500, J).astype(np.int32)
    cb = np.where(rng.random(J) < 0.5, rng.integers(0, H + 5, J), rng.integers(0, 40, J)).astype(np.int32)
    cb[: min(J, 4)] = ([H] if J < 3 else [0, 16, 128, H])[: min(J, 4)] * (2 if J == 2 else 1)
    check_dispatch(M, ws, oracle, 1, D, H, K, cap, Q, cp, cb)
    cp[J // 2] = -1  # skipped and reported
    check_dispatch(M, ws, oracle, 1, D, H, K, cap, Q, cp, cb)


def test_dispatch_sequential_ranges(M, ws, oracle):
    """Queue lengths far apart (past the 32-bit keys), one that passes int32,
    and a reservation that takes K past int32."""
    K = np.zeros((40, 50), np.int32)
    cap = np.full(40, 10**6, np.int32)
    cp, cb = np.full(30, 7, np.int32), np.full(30, 20, np.int32)
    Q = (np.arange(40)[::-1] * 50_000_000).astype(np.int32)
    check_dispatch(M, ws, oracle, 1, 40, 50, K, cap, Q, cp, cb)
    check_dispatch(M, ws, oracle, 1, 40, 50, K, cap, np.full(40, I32_MAX, np.int32), cp, cb)
    check_dispatch(M, ws, oracle, 1, 3, 50, np.full((3, 50), I32_MAX - 60, np.int32), cap[:3],
                   Q[:3], cp, cb)


@pytest.mark.parametrize("S", [1, 16])
@pytest.mark.parametrize("name", ["tiny", "d16", "d64", "large"])
def test_dispatch_alg1_workloads(M, ws, oracle, name, S):
    w = W.make(name, feasible=True)
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1]
    res = (w["res_off"], w["res_prompt"], w["res_gen"], U)
    rng = np.random.default_rng(S)
    cap = (w["cap"].astype(np.int64) // 2 + rng.integers(0, w["cap"].max() // 8, w["D"])).astype(np.int32)
    Q = rng.integers(0, 3, w["D"]).astype(np.int32)
    co, ho = check_dispatch(M, ws, oracle, 2, w["D"], w["H"], None, cap, Q, w["cand_prompt"], cb, S, res)
    # SEQUENTIAL over every candidate (65,536 reservations in order at Large)
    check_dispatch(M, ws, oracle, 3, w["D"], w["H"], None, cap, Q, w["cand_prompt"], cb, S, res)


@pytest.mark.parametrize("D,J,S,spread", [
    # decoders at the edges of the registers-per-lane variants; a last chunk of
    # candidates that is not full, and one candidate
    (1, 33, 1, 2000), (31, 65, 16, 3000), (32, 1, 16, 3000), (33, 700, 1, 3000),
    (64, 1000, 16, 5000), (65, 500, 32, 5000), (200, 500, 16, 5000), (257, 300, 1, 4000),
    (600, 400, 16, 4000), (1024, 300, 16, 4000),
    # up to eight candidates on more than 256 decoders, a thread a decoder; and beside it
    (257, 1, 16, 4000), (512, 2, 1, 4000), (1024, 8, 16, 4000), (1000, 7, 1, 2**24), (256, 8, 16, 4000),
    (257, 9, 16, 4000),
    # budgets further apart than a 32-bit key holds (the wide comparison), from
    # the start and after some reservations
    (5, 400, 1, 2**30), (1000, 300, 1, 2**24), (2, 3000, 1, 2**29)])
def test_dispatch_alg1_sequential_edges(M, ws, oracle, D, J, S, spread):
    rng = np.random.default_rng(D * 31 + J)
    per = 3
    off = np.arange(D + 1, dtype=np.int64) * per
    p = rng.integers(0, 400, D * per).astype(np.int32)
    g = rng.integers(0, 300, D * per).astype(np.int32)
    U = rng.integers(0, 600, D * per).astype(np.int32)
    cap = rng.integers(0, spread, D).astype(np.int32)
    Q = rng.integers(0, 4, D).astype(np.int32)
    big = 600 if spread < 2**20 else 500000
    cp = rng.integers(0, big, J).astype(np.int32)
    cb = rng.integers(0, big, J).astype(np.int32)
    check_dispatch(M, ws, oracle, 3, D, 1, None, cap, Q, cp, cb, S, (off, p, g, U))
    # invalid candidates are skipped and reported; a queue length that passes
    # int32 is reported
    cp[J // 2] = -1
    check_dispatch(M, ws, oracle, 3, D, 1, None, cap, Q, cp, cb, S, (off, p, g, U))
    cp[J // 2] = 1
    full = np.full(D, I32_MAX, np.int32)
    check_dispatch(M, ws, oracle, 3, D, 1, None, cap, full, cp, cb, S, (off, p, g, U))


def test_dispatch_errors(M, ws, oracle):
    K = np.zeros((2, 8), np.int32)
    st, ch, _, _, _ = gpu_dispatch(M, ws, 0, 2, 8, 1, K, [5, 5], [0, 0], [1, -1], [2, 2])
    assert st == M.MAPS_E_RANGE and ch[1] == -1
    K[1, 3] = -1
    assert gpu_dispatch(M, ws, 0, 2, 8, 1, K, [5, 5], [0, 0], [1], [2])[0] == M.MAPS_E_RANGE
    assert gpu_dispatch(M, ws, 1, 2, 8, 1, K, [5, 5], [0, 0], [1], [2])[0] == M.MAPS_E_RANGE
    assert gpu_dispatch(M, ws, 0, 2, 8, 1, np.zeros((2, 8), np.int32), [5, -5], [0, 0], [1], [2])[0] \
        == M.MAPS_E_RANGE
    ch = torch.empty(1, dtype=torch.int32, device="cuda")
    z = dev([0, 0], np.int32)
    Kd = dev(np.zeros((2, 8), np.int32))
    assert M.maps_dispatch(7, 2, 8, 1, Kd, z, z, dev([1], np.int32), dev([1], np.int32), ch,
                           ws=ws) == M.MAPS_E_INVALID
    assert M.maps_dispatch(0, 1025, 8, 1, Kd, z, z, dev([1], np.int32), dev([1], np.int32), ch,
                           ws=ws) == M.MAPS_E_INVALID
    small = M.Workspace(256)
    assert M.lib.maps_dispatch(0, 2, 8, 1, M._ptr(Kd), None, M._ptr(z), M._ptr(z), None, 0, None, None,
                               None, 1, M._ptr(dev([1], np.int32)), M._ptr(dev([1], np.int32)),
                               M._ptr(ch), None, small.ptr, 256, M._stream(None)) == M.MAPS_E_WORKSPACE


# ---------------------------------------------------------------------------
# local order
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("N,D,sorted_arrival", [(0, 3, True), (1, 1, True), (2, 2, False),
                                                (100, 3, False), (4096, 8, True), (4097, 8, False),
                                                (50000, 64, True), (50001, 300, False),
                                                (300000, 256, False), (1000, 70000, True),
                                                # one-block calls: bitonic up to 1,024
                                                # entries, then stable passes
                                                (700, 5, True), (1024, 16, False),
                                                (1025, 16, True), (3000, 40, False),
                                                # the one-block form at its decoder limit,
                                                # then past it
                                                (2000, 4096, True), (2000, 4097, True),
                                                # one decoder's queue at, and past, the most a
                                                # block sorts in shared memory
                                                (4608, 1, True), (4609, 1, True),
                                                (5632, 1, True), (5633, 1, True),
                                                (20000, 2, True), (300000, 256, True),
                                                # a queue of 22 chunks: five merge levels
                                                (100000, 1, True),
                                                # more decoders than the stable scatter takes
                                                (60000, 1500, True),
                                                # the bucketing pass at its decoder limit, and
                                                # with a count not a multiple of four
                                                (200000, 1024, True), (200000, 1023, False),
                                                # bucketing by two entries a thread: its last
                                                # range full and of one entry, the most of them
                                                # and one more, and counts past their room
                                                (5120, 6, True), (5121, 900, False),
                                                (102400, 333, False), (102401, 333, True),
                                                (50001, 1023, True),
                                                # past 304 x 4,096 entries the bucketing blocks
                                                # take several rounds (loads issued twice);
                                                # arrival out of order: the global key pass
                                                (1500000, 256, True), (1500000, 1024, False)])
def test_order_random(M, ws, oracle, N, D, sorted_arrival):
    rng = np.random.default_rng(N + D)
    dec = rng.integers(0, D, N).astype(np.int32)
    U = rng.integers(0, 60 if N < 5000 else 2**31 - 1, N, dtype=np.int64).astype(np.int32)
    wait = rng.integers(-10, 3000, N).astype(np.int32)
    if sorted_arrival:
        arr = np.sort(rng.integers(0, max(N // 2, 1), N)).astype(np.int32)
    else:
        arr = rng.integers(0, 2**31 - 1, N, dtype=np.int64).astype(np.int32)
        arr[: N // 3] = rng.integers(0, 50, N // 3)  # ties on arrival too
    sto, po, so = oracle.order_local(D, dec, U, wait, arr, 1000)
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 1000)
    assert st == sto == 0
    assert np.array_equal(perm, po)
    assert np.array_equal(seg, so)


@pytest.mark.parametrize("N,D,ubits,abits", [
    # one-block calls with arrival out of index order: when (decoder, not
    # promoted, bound, arrival, index) fits 64 bits one sort on it gives the
    # order (bitonic, then stable passes), otherwise two sorts do
    (700, 5, 15, 20), (3000, 40, 15, 20), (1000, 1, 31, 31), (4000, 300, 31, 31),
    # exactly 64 bits, and one bit more
    (1024, 16, 18, 31), (1024, 16, 19, 31)])
def test_order_small_unsorted_key_widths(M, ws, oracle, N, D, ubits, abits):
    rng = np.random.default_rng(N + D + ubits)
    dec = rng.integers(0, D, N).astype(np.int32)
    U = rng.integers(0, 2**ubits, N, dtype=np.int64).astype(np.int32)
    wait = rng.integers(-10, 3000, N).astype(np.int32)
    i = rng.integers(0, N)
    U[i], wait[i] = 2**ubits - 1, 0  # the full width, on an entry that is not promoted
    arr = rng.integers(0, 2**abits, N, dtype=np.int64).astype(np.int32)
    arr[rng.integers(0, N)] = 2**abits - 1
    arr[: N // 4] = arr[N // 4]  # ties on arrival
    sto, po, so = oracle.order_local(D, dec, U, wait, arr, 1000)
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 1000)
    assert st == sto == 0
    assert np.array_equal(perm, po)
    assert np.array_equal(seg, so)


def test_order_bucketing_rounds_range_error(M, ws, oracle):
    """An entry outside the decoder domain in a call whose bucketing blocks
    take several rounds: counted and placed at decoder 0 in both of its
    passes, reported as MAPS_E_RANGE, every write inside the outputs."""
    rng = np.random.default_rng(5)
    N, D = 1300000, 64
    dec = rng.integers(0, D, N).astype(np.int32)
    dec[777777] = -3
    dec[1299999] = D + 5
    U = rng.integers(0, 5000, N).astype(np.int32)
    wait = rng.integers(0, 3000, N).astype(np.int32)
    arr = np.arange(N, dtype=np.int32)
    assert oracle.order_local(D, dec, U, wait, arr, 1000)[0] == -2
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 1000)
    assert st == M.MAPS_E_RANGE
    assert perm.min() >= -1 and perm.max() < N


# blocks of 1,024 entries (64 a warp) and of 4,096 (256 a warp), one round each
@pytest.mark.parametrize("N,D,per_warp", [(20500, 8, 64), (200003, 60, 256)])
@pytest.mark.parametrize("ordered", [True, False])
def test_order_bucketing_largest_in_each_warp(M, ws, oracle, N, D, per_warp, ordered):
    """The widths of the key's fields come from the largest bound and the
    largest arrival of all entries: each in turn held by one entry of one warp
    of a block, far above the rest (a width too small runs the fields into
    each other)."""
    rng = np.random.default_rng(N)
    dec = rng.integers(0, D, N).astype(np.int32)
    wait = rng.integers(0, 5, N).astype(np.int32)
    for warp in range(16):
        U = rng.integers(0, 200, N).astype(np.int32)
        arr = np.sort(rng.integers(0, 500, N)).astype(np.int32)
        if not ordered:
            arr = rng.permutation(arr)
        block = int(rng.integers(0, N // (16 * per_warp)))
        at = (block * 16 + warp) * per_warp
        U[at + int(rng.integers(0, per_warp))] = 2**20 + 7
        if ordered:
            arr[at:] += 2**18  # non-decreasing still
        else:
            arr[at + int(rng.integers(0, per_warp))] = 2**18 + 3
        sto, po, so = oracle.order_local(D, dec, U, wait, arr, 5)
        st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 5)
        assert st == sto == 0
        assert np.array_equal(perm, po) and np.array_equal(seg, so), warp


@pytest.mark.parametrize("N,D,blo,bhi,skew", [
    # one queue far past a block (16 chunks), bounds of 17 bits
    (70000, 256, 0, 70000, 0.95),
    # several long queues with ragged last chunks, 31-bit bounds
    (60001, 8, 0, 2**31 - 1, 0.0),
    # bounds in [2^20, 2^20 + 200): keys share their high bits
    (30000, 3, 2**20, 2**20 + 200, 0.5),
    # more decoders than the stable scatter takes, one long queue
    (40000, 1100, 0, 2**31 - 1, 0.9),
    # every entry in one queue of 15 runs (ranked pairwise: 210 pairs)
    (65536, 256, 0, 70000, 1.0),
    # sixteen queues of about 16 runs each: the first to reserve their pairs within
    # the budget are ranked pairwise, the others merged level by level
    (1120000, 16, 0, 2**31 - 1, 0.0)])
def test_order_long_queues(M, ws, oracle, N, D, blo, bhi, skew):
    rng = np.random.default_rng(N + D)
    dec = rng.integers(0, D, N).astype(np.int32)
    dec[rng.random(N) < skew] = D // 2
    U = rng.integers(blo, bhi, N, dtype=np.int64).astype(np.int32)
    wait = rng.integers(-10, 3000, N).astype(np.int32)
    arr = np.sort(rng.integers(0, N, N)).astype(np.int32)
    sto, po, so = oracle.order_local(D, dec, U, wait, arr, 1000)
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 1000)
    assert st == sto == 0
    assert np.array_equal(perm, po)
    assert np.array_equal(seg, so)


@pytest.mark.parametrize("N,D,ubits,abits,skew", [
    # arrival out of index order past one block: (not promoted, bound, arrival,
    # index) in exactly 63 bits, sorted per decoder, and in 64, sorted globally
    (16384, 5, 17, 31, 0.0), (16384, 5, 18, 31, 0.0),
    # one decoder; ragged last chunks ranked pairwise; a queue past the pairwise
    # ranks merged level by level; many queues of two runs; the most decoders
    (4609, 1, 14, 20, 0.0), (60001, 3, 14, 20, 0.5), (90000, 2, 14, 24, 0.9),
    (300000, 60, 14, 22, 0.0), (50000, 1024, 14, 20, 0.0),
    # one entry past a bucketing round, and ranges of several rounds
    (4097, 9, 10, 10, 0.0), (1300000, 300, 14, 25, 0.0),
    # seven merge levels
    (400000, 1, 14, 22, 0.0)])
def test_order_shuffled_arrival_forms(M, ws, oracle, N, D, ubits, abits, skew):
    rng = np.random.default_rng(N + D + ubits)
    dec = rng.integers(0, D, N).astype(np.int32)
    dec[rng.random(N) < skew] = D // 2
    U = rng.integers(0, 2**ubits, N, dtype=np.int64).astype(np.int32)
    wait = rng.integers(-10, 3000, N).astype(np.int32)
    U[7], wait[7] = 2**ubits - 1, 0  # the full widths
    arr = rng.integers(0, 2**abits, N, dtype=np.int64).astype(np.int32)
    arr[N // 2] = 2**abits - 1
    arr[: N // 4] = arr[N // 4]  # ties on arrival: by index
    sto, po, so = oracle.order_local(D, dec, U, wait, arr, 1000)
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 1000)
    assert st == sto == 0
    assert np.array_equal(perm, po)
    assert np.array_equal(seg, so)


@pytest.mark.parametrize("sizes,D", [
    # runs of 4,608 ranked pairwise: one entry past a run, whole runs, the most
    # runs (16), and a queue past them merged by levels beside ranked ones
    ([4609], 1), ([9216], 1), ([9217, 0, 4608, 1, 13823], 5), ([73728], 2), ([73729, 5000, 9000], 4),
    # merges at the most entries of one and of three outputs a thread, and past them
    ([77824], 1), ([77825], 1), ([390000, 76944], 2), ([390000, 76945], 2),
    # the last run within, and at, one and two outputs a thread
    ([4608 + 511, 4608 + 512, 4608 + 513, 4608 * 2 + 256], 9),
    # listed by size (at most 511 decoders) and not; items around half a run
    ([5000, 2304, 2305, 1, 4608, 6912, 6913, 0, 12000] * 3, 511), ([5000, 2304, 2305, 9, 7000], 512)])
@pytest.mark.parametrize("ordered", [True, False])
def test_order_queue_sizes(M, ws, oracle, sizes, D, ordered):
    """Queues of given lengths, keys with ties in every field."""
    rng = np.random.default_rng(sum(sizes) + D)
    dec = rng.permutation(np.repeat(np.arange(len(sizes)) * D // len(sizes), sizes)).astype(np.int32)
    N = len(dec)
    U = rng.integers(0, 300, N).astype(np.int32)
    wait = rng.integers(0, 1200, N).astype(np.int32)
    arr = rng.integers(0, 4000, N).astype(np.int32)
    if ordered:
        arr.sort()
    sto, po, so = oracle.order_local(D, dec, U, wait, arr, 1000)
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, 1000)
    assert st == sto == 0
    assert np.array_equal(perm, po)
    assert np.array_equal(seg, so)


def test_order_degenerate_keys(M, ws, oracle):
    # every key identical: all digit passes trivial -> identity order
    N = 9000
    z = np.zeros(N, np.int32)
    st, perm, seg = gpu_order(M, ws, 1, z, z, z, z, 5)
    assert st == 0 and np.array_equal(perm, np.arange(N)) and seg.tolist() == [0, N]
    st, perm, _ = gpu_order(M, ws, 2, [3], [1], [0], [0], 5)
    assert st == M.MAPS_E_RANGE


@pytest.mark.parametrize("name,one_queue", [("d64", False), ("large", False), ("large", True)])
def test_order_workload_pipeline(M, ws, oracle, name, one_queue):
    """The benchmark's order step: residents plus dispatched candidates (spread over the
    decoders, or all on one decoder as when every candidate falls back to the same one)."""
    w = W.make(name)
    R, J, D = w["R"], w["J"], w["D"]
    rng = np.random.default_rng(1)
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(np.concatenate([w["res_pred"], w["cand_pred"]]), q)[1]
    cand_dec = np.full(J, 37, np.int32) if one_queue else rng.integers(0, D, J).astype(np.int32)
    dec = np.concatenate([w["res_dec"], cand_dec])
    wait = np.concatenate([w["res_wait"], np.zeros(J, np.int32)])
    arr = np.arange(R + J, dtype=np.int32)
    sto, po, so = oracle.order_local(D, dec, U, wait, arr, w["max_wait"])
    st, perm, seg = gpu_order(M, ws, D, dec, U, wait, arr, w["max_wait"])
    assert st == sto == 0
    assert np.array_equal(perm, po) and np.array_equal(seg, so)


def test_dispatch_snapshot_invalid_candidates(M, ws, oracle):
    """Candidates with a negative prompt or bound get choice -1 and headroom 0
    and record MAPS_E_RANGE; the others are still decided."""
    w = W.make("tiny", feasible=True)
    D, H = w["D"], w["H"]
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1].copy()
    cp = w["cand_prompt"].copy()
    cp[3], cb[7] = -1, -5
    _, K = oracle.occupancy(D, H, w["res_off"], w["res_prompt"], w["res_gen"], U)
    st, ch, hr, _, _ = gpu_dispatch(M, ws, M.MODE_SNAPSHOT, D, H, 1, K, w["cap"], w["Q"], cp, cb)
    sto, cho, hro, _, _ = oracle.dispatch(0, D, H, 1, K, w["cap"], w["Q"], cp, cb)
    assert st == sto == M.MAPS_E_RANGE
    assert np.array_equal(ch, cho) and np.array_equal(hr, hro)


def test_dispatch_kmax_checked_against_K(M, ws, oracle):
    """A caller's 16-step summary is compared with K at four blocks of every
    row: the summary of K itself passes, one that disagrees with K in the first
    block of a row is MAPS_E_INVALID."""
    w = W.make("d16", feasible=True)
    D, H = w["D"], w["H"]
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1]
    _, K = oracle.occupancy(D, H, w["res_off"], w["res_prompt"], w["res_gen"], U)
    km = kmax_of(K)
    st, ch, hr, _, _ = gpu_dispatch(M, ws, M.MODE_SNAPSHOT, D, H, 1, K, w["cap"], w["Q"],
                                    w["cand_prompt"], cb, kmax=km)
    _, cho, hro, _, _ = oracle.dispatch(0, D, H, 1, K, w["cap"], w["Q"], w["cand_prompt"], cb)
    assert st == 0 and np.array_equal(ch, cho) and np.array_equal(hr, hro)
    bad = km.copy()
    bad[5, 0] += 1
    st, _, _, _, _ = gpu_dispatch(M, ws, M.MODE_SNAPSHOT, D, H, 1, K, w["cap"], w["Q"],
                                  w["cand_prompt"], cb, kmax=bad)
    assert st == M.MAPS_E_INVALID


def test_dispatch_scoring_events(M, ws, oracle):
    """The benchmarking hook records its events around the scoring kernel and
    leaves the decisions unchanged."""
    w = W.make("tiny", feasible=True)
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], w["alphas_ppm"][0])[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1]
    _, K = oracle.occupancy(w["D"], w["H"], w["res_off"], w["res_prompt"], w["res_gen"], U)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    e1.record()
    assert M.maps_set_dispatch_events(e0, e1) == 0
    try:
        st, ch, hr, _, _ = gpu_dispatch(M, ws, 0, w["D"], w["H"], 1, K, w["cap"], w["Q"],
                                        w["cand_prompt"], cb)
    finally:
        M.maps_set_dispatch_events(None, None)
    torch.cuda.synchronize()
    _, cho, hro, _, _ = oracle.dispatch(0, w["D"], w["H"], 1, K, w["cap"], w["Q"],
                                        w["cand_prompt"], cb)
    assert st == 0 and np.array_equal(ch, cho) and np.array_equal(hr, hro)
    assert e0.elapsed_time(e1) > 0.0


# ---------------------------------------------------------------------------
# CUDA graph capture of the whole pass
# ---------------------------------------------------------------------------

def test_graph_capture_replay(M, oracle):
    """The four calls (calibrate + bound, occupancy, SNAPSHOT dispatch, local
    order) captured once in a CUDA graph: every replay reads the inputs as they
    are then and matches the oracle, including after the inputs change."""
    w0, w1 = W.make("tiny", feasible=True), W.make("tiny", seed=11)
    D, H, R, J = w0["D"], w0["H"], w0["R"], w0["J"]
    assert (D, H, R, J) == (w1["D"], w1["H"], w1["R"], w1["J"])
    a = w0["alphas_ppm"][0]
    n = len(w0["cal_true"])
    z = lambda k, dt=torch.int32: torch.zeros(k, dtype=dt, device="cuda")  # noqa: E731
    x = dict(cal_true=z(n), cal_pred=z(n), pred=z(R + J), off=z(D + 1, torch.int64), prompt=z(R),
             gen=z(R), cap=z(D), Q=z(D), cprompt=z(J), dec=z(R + J), wait=z(R + J),
             arr=torch.arange(R + J, dtype=torch.int32, device="cuda"))
    U, q = z(R + J), z(1)
    K = z(D * H).view(D, H)
    km = torch.zeros(M.kmax_shape(D, H), dtype=torch.int32, device="cuda")
    hr, perm, seg = z(J, torch.int64), z(R + J), z(D + 1, torch.int64)
    need = max(M.lib.maps_calibrate_workspace_size(n, R + J),
               M.lib.maps_project_occupancy_workspace_size(D, H, R),
               M.lib.maps_dispatch_workspace_size(M.MODE_SNAPSHOT, D, H, J),
               M.lib.maps_order_local_workspace_size(R + J, D))
    gws = M.Workspace(need, torch.device("cuda"))

    def load(w):
        for k, v in dict(cal_true=w["cal_true"], cal_pred=w["cal_pred"],
                         pred=np.concatenate([w["res_pred"], w["cand_pred"]]), off=w["res_off"],
                         prompt=w["res_prompt"], gen=w["res_gen"], cap=w["cap"], Q=w["Q"],
                         cprompt=w["cand_prompt"], wait=np.concatenate([w["res_wait"], np.zeros(J)]),
                         dec=np.concatenate([w["res_dec"], np.zeros(J)])).items():
            x[k].copy_(torch.from_numpy(np.ascontiguousarray(v).astype(x[k].cpu().numpy().dtype)))

    def run():
        assert M.maps_calibrate(x["cal_true"], x["cal_pred"], a, x["pred"], U, q, ws=gws)[0] == 0
        assert M.maps_project_occupancy(D, H, x["off"], x["prompt"], x["gen"], U[:R], K, km,
                                        ws=gws) == 0
        assert M.maps_dispatch(M.MODE_SNAPSHOT, D, H, 1, K, x["cap"], x["Q"], x["cprompt"],
                               U[R:], x["dec"][R:], hr, kmax=km, ws=gws) == 0
        assert M.maps_order_local(D, x["dec"], U, x["wait"], x["arr"], w0["max_wait"], perm, seg,
                                  ws=gws) == 0

    load(w0)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        run()  # warm-up outside the capture
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side, capture_error_mode="relaxed"):
        run()
    for w in (w0, w1, w0):
        load(w)
        g.replay()
        torch.cuda.synchronize()
        assert M.maps_check(gws) == 0
        sto, qo = oracle.calibrate(w["cal_true"], w["cal_pred"], a)
        Uo = oracle.bound(np.concatenate([w["res_pred"], w["cand_pred"]]), qo)[1]
        _, Ko = oracle.occupancy(D, H, w["res_off"], w["res_prompt"], w["res_gen"], Uo[:R])
        _, cho, hro, _, _ = oracle.dispatch(0, D, H, 1, Ko, w["cap"], w["Q"], w["cand_prompt"],
                                            Uo[R:])
        deco = np.concatenate([w["res_dec"], cho]).astype(np.int32)
        _, po, so = oracle.order_local(D, deco, Uo, np.concatenate([w["res_wait"], np.zeros(J, np.int32)]),
                                       np.arange(R + J, dtype=np.int32), w0["max_wait"])
        assert int(host(q)[0]) == qo and np.array_equal(host(U), Uo)
        assert np.array_equal(host(K), Ko)
        assert np.array_equal(host(x["dec"])[R:], cho) and np.array_equal(host(hr), hro)
        assert np.array_equal(host(perm), po) and np.array_equal(host(seg), so)


# ---------------------------------------------------------------------------
# determinism
# ---------------------------------------------------------------------------

def test_repeat_runs_identical(M, ws, oracle):
    w = W.make("d64")
    q = oracle.calibrate(w["cal_true"], w["cal_pred"], 100000)[1]
    U = oracle.bound(w["res_pred"], q)[1]
    cb = oracle.bound(w["cand_pred"], q)[1]
    outs = []
    for _ in range(3):
        _, K = gpu_occupancy(M, ws, w["D"], w["H"], w["res_off"], w["res_prompt"], w["res_gen"], U)
        _, ch, hr, _, _ = gpu_dispatch(M, ws, 0, w["D"], w["H"], 1, K, w["cap"], w["Q"],
                                       w["cand_prompt"], cb)
        outs.append((K, ch, hr))
    for o in outs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(o, outs[0]))


# ---------------------------------------------------------------------------
# streaming loop
# ---------------------------------------------------------------------------

def gpu_stream(M, ws, N, D, H, cap, B, Wn, a, mw, arrival, prompt, true, pred):
    nb = (N + B - 1) // B
    ch = torch.full((N,), -9, dtype=torch.int32, device="cuda")
    q = torch.full((nb,), -9, dtype=torch.int32, device="cuda")
    stats = torch.full((nb, 4), -9, dtype=torch.int64, device="cuda")
    cfg = M.stream_cfg(N, D, H, cap, B, Wn, a, mw)
    st = M.maps_stream_run(cfg, dev(arrival[:N], np.int64), dev(prompt[:N], np.int32),
                           dev(true[:N], np.int32), dev(pred[:N], np.int32), ch, q, stats, ws=ws)
    return st, host(ch), host(q), host(stats)


def check_stream(M, ws, oracle, N, D, H, cap, B, Wn, a, mw, w):
    args = (N, D, H, cap, B, Wn, a, mw, w["arrival_ms"], w["prompt"], w["true"], w["pred"])
    sto, cho, qo, so = oracle.stream(*args)
    st, ch, q, s = gpu_stream(M, ws, *args)
    assert st == sto
    if st == 0:
        assert np.array_equal(q, qo)
        assert np.array_equal(s, so)
        assert np.array_equal(ch, cho)
    return qo, so


def test_stream_golden(M, ws, stream_golden):
    c, r = stream_golden["config"], stream_golden["requests"]
    st, ch, q, s = gpu_stream(M, ws, c["N"], c["D"], c["H"], c["cap"], c["batch"], c["window"],
                              c["alpha_ppm"], c["max_wait"], np.array(r["arrival_ms"]),
                              np.array(r["prompt"]), np.array(r["true_len"]), np.array(r["pred"]))
    assert st == 0
    assert ch.tolist() == stream_golden["choice"]
    assert q.tolist() == stream_golden["q"]
    assert s.tolist() == stream_golden["stats"]


@pytest.mark.parametrize("N,D,H,cap,B,Wn,a,mw", [
    (1, 32, 16384, 262144, 256, 500, 100000, 1000),       # one request, round robin
    (300, 32, 16384, 262144, 256, 500, 100000, 1000),     # ragged last batch
    (20000, 32, 16384, 262144, 256, 500, 100000, 1000),   # the streaming workload's prefix
    (20000, 4, 4096, 12000, 256, 500, 100000, 1000),      # queues back up and block
    (20000, 3, 2048, 9000, 100, 37, 300000, 50),          # promotions, small window
    (5000, 5, 1000, 20000, 33, 7, 500000, 0),             # horizon below many bounds
    # capacity far below demand: waiting queues push M, and the deficits,
    # past 2^21 (the dispatch's 64-bit key comparison)
    (3000, 8, 16384, 3000, 256, 500, 100000, 1000),
    # 200 decoders x batches of 256: the end-step tables would need about 800 KB of
    # shared memory, so the loop dispatches through the dense projection instead
    (3000, 200, 2048, 60000, 256, 300, 100000, 1000),
    # 48 decoders: the shared-memory walk past one warp's decoders, with queues
    (4000, 48, 4096, 30000, 64, 200, 100000, 1000),
    # a window of 10,000 completions, more than the one-block loop holds: batch by
    # batch from the host, the quantile by the one-block calibration
    (30000, 8, 16384, 262144, 512, 10000, 100000, 1000),
    # and one of 17,000, past that: by the cooperative kernel
    (40000, 8, 16384, 262144, 512, 17000, 100000, 1000),
])
def test_stream_prefix(M, ws, oracle, N, D, H, cap, B, Wn, a, mw):
    w = W.make_stream(n_requests=N)
    qo, so = check_stream(M, ws, oracle, N, D, H, cap, B, Wn, a, mw, w)
    assert (qo >= 0).any() or N < 1000


@pytest.mark.parametrize("N,D,cap,B", [
    # lists around 32, 64 and 128 pairs a decoder, some outgrowing the variant
    # they start on within a batch; one decoder, and as many as a warp's lanes
    (1500, 1, 30000, 16), (2000, 1, 9000, 40), (2000, 2, 50000, 90), (3000, 3, 40000, 200),
    (4000, 31, 9000, 256), (4000, 32, 14000, 300), (4000, 32, 60, 100)])
def test_stream_walk_list_sizes(M, ws, oracle, N, D, cap, B):
    w = W.make_stream(n_requests=N)
    check_stream(M, ws, oracle, N, D, 16384, cap, B, 300, 100000, 1000, w)


@pytest.mark.parametrize("N,D,cap,B,Wn", [
    # more batches than one launch of the one-block loop runs
    (700, 4, 30000, 2, 50), (257, 3, 30000, 1, 20),
    # the window at what the loop holds, and past it
    (9000, 8, 262144, 512, 4096), (9000, 8, 262144, 512, 4097),
    # queues past the ranked groups (512), and a system that outgrows the loop
    # and comes back into it; batches and systems around 2,048 requests
    (3000, 2, 40000, 100, 300), (9000, 2, 60000, 300, 500), (5000, 16, 262144, 2000, 500),
    (5000, 16, 262144, 2048, 500), (5000, 64, 20000, 2049, 500),
    # one decoder, and as many as a warp's lanes, with more picks than threads
    (4000, 1, 262144, 1500, 300), (6000, 32, 262144, 1100, 300),
    # many completions in one batch: sorted by the network
    (9000, 40, 262144, 900, 700),
    # sorted lists past 128 pairs a decoder: walked in the loop (short), left to the
    # host at the dispatch (long), both in turn, on one decoder and on as many as a
    # warp's lanes; no room for them with 16 decoders and more
    (3000, 4, 229000, 40, 300), (2453, 5, 87144, 458, 980), (4501, 5, 97355, 348, 262),
    (1983, 1, 57103, 47, 50), (3000, 15, 30000, 300, 200), (3000, 16, 30000, 300, 200),
    (6000, 32, 15000, 400, 300), (3000, 33, 20000, 300, 200)])
def test_stream_one_block_loop_limits(M, ws, oracle, N, D, cap, B, Wn):
    w = W.make_stream(n_requests=N)
    check_stream(M, ws, oracle, N, D, 16384, cap, B, Wn, 100000, 1000, w)


@pytest.mark.parametrize("seed,a", [(0, 100000), (1, 300000), (2, 20000), (3, 700000)])
def test_stream_quantile_bin_edges(M, ws, oracle, seed, a):
    """The loop's own quantile, of a window of scores on the bin edges of its
    passes (each batch completes the one before, whose true lengths are those
    scores over predictions of zero)."""
    rng = np.random.default_rng(seed)
    edges = {1, 1022, 1023, 1024, 1025, 2**30 + 2**24}
    for e in range(10, 31):
        step = 1 << (e - 7)
        edges |= {(1 << e) - 1, 1 << e, (1 << e) + 1, (1 << e) + step - 1, (1 << e) + step}
    N, B = 1200, 15
    spread = rng.choice(np.array(sorted(edges)), N)
    true = np.where(np.arange(N) // 300 % 2 == 0, spread, rng.integers(1, 2**30, N))
    zeros = np.zeros(N, np.int32)
    w = dict(arrival_ms=np.arange(N) // B * 2**32, prompt=zeros, pred=zeros, true=true.astype(np.int32))
    qo, so = check_stream(M, ws, oracle, N, 8, 64, I32_MAX, B, 250, a, 1000, w)
    assert (so[1:, 0] == B).all() and (qo[-60:] > 0).all() and len(set(qo.tolist())) >= 10


def test_stream_full_workload(M, ws, oracle):
    """All 1,000,000 requests of the streaming workload, bit for bit."""
    w = W.make_stream()
    c = W.WORKLOADS["stream"]
    qo, so = check_stream(M, ws, oracle, w["N"], w["D"], w["H"], w["cap"], w["batch"],
                          w["window"], w["alpha_ppm"], w["max_wait"], w)
    assert len(qo) == (w["N"] + c["batch"] - 1) // c["batch"]
