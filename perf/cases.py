"""The scheduler's measured work: whole passes through its public entry points.

A pass is what a program that embeds the scheduler does between receiving its
state and acting on the answers, from a scheduler of four decoders to one of
256 with a million residents:

* ``step``        calibrate, project the occupancy, dispatch every candidate
                  against the same state, put every queue in local order;
* ``sequential``  project the occupancy, then dispatch candidates one after
                  another, each reserving its footprint (K and Q are updated);
* ``alg1``        Algorithm 1 on block budgets, one request after another or
                  all against the same state;
* ``order``       the local order alone, entries in slots that are reused, so
                  that arrival does not follow the entry index, or in order;
* ``stream``      the whole streaming loop over a trace of arrivals;
* ``rr``          the round-robin KV-pressure simulation of a load sweep.

Every result is a whole number (lengths, choices, orders, times in integer
steps or microseconds), so any correct implementation gives the same ones.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_15359_gb300 import maps as M
from paper_2609_15359_gb300 import workloads as W

MAX_WAIT = W.MAX_WAIT_STEPS

# output-length distributions of the workloads: (kind, parameters, clip, noise)
LENGTHS = {
    "lognormal": ((5.5, 1.0), 16384, 0.4),
    "pareto": ((1.5, 16.0), 32768, 0.6),
    "bimodal": ((0.7, 4.5, 0.8, 7.5, 0.7), 65536, 0.5),
}


def listed():
    return [
        # a small cluster's scheduler asked for one step: four decoders, 32
        # candidates; launches and latency are all there is
        dict(name="step_tiny", kind="step", D=4, per=64, H=4096, J=32, n=1000, alpha=100000,
             load=1.0, lengths="lognormal", pmax=2048),
        # sixteen decoders near their capacity, uneven queues and odd sizes (a
        # horizon that is no multiple of four): some decoders have room, some none
        dict(name="step_d16_odd", kind="step", D=16, per=509, H=16381, J=1021, n=10007,
             alpha=100000, load=1.05, lengths="lognormal", pmax=2048),
        # 64 decoders with room: candidates take the shortest queue that fits
        dict(name="step_d64_feasible", kind="step", D=64, per=2048, H=32768, J=8192, n=100000,
             alpha=50000, load=0.6, lengths="pareto", pmax=2048),
        # the largest: 256 decoders, a million residents, far over capacity
        dict(name="step_large", kind="step", D=256, per=4096, H=65536, J=65536, n=1000000,
             alpha=100000, load=32.0, lengths="bimodal", pmax=8192),
        # one request after another with reservation, near capacity
        dict(name="sequential_d16", kind="sequential", D=16, per=512, H=16384, J=1024, load=0.97,
             lengths="lognormal", pmax=2048),
        # the same over 64 decoders, odd sizes, most of them with room
        dict(name="sequential_d64_odd", kind="sequential", D=64, per=2039, H=32763, J=2003,
             load=0.7, lengths="pareto", pmax=2048),
        # Algorithm 1 on block budgets, reserving after each choice
        dict(name="alg1_d64", kind="alg1", D=64, per=2048, J=8192, S=16, reserve=True, load=0.7,
             lengths="pareto", pmax=2048),
        # local order of entries kept in reused slots, many queues
        dict(name="order_shuffled", kind="order", N=200003, D=64, arrival="shuffled",
             lengths="lognormal"),
        # the streaming loop at its workload's capacity: no queue forms
        dict(name="stream_roomy", kind="stream", N=30000, D=32, cap=262144, H=16384, batch=256,
             window=500, alpha=100000, dispatch=0, local=0, accounting=0, per_step=0, beta=-1),
        # the same loop where capacity binds and queues form
        dict(name="stream_tight", kind="stream", N=20011, D=32, cap=16000, H=16384, batch=256,
             window=500, alpha=100000, dispatch=0, local=0, accounting=0, per_step=0, beta=-1),
        # admission on every step with preemption, predictions that come late
        dict(name="stream_per_step", kind="stream", N=20011, D=32, cap=16000, H=16384, batch=256,
             window=500, alpha=100000, dispatch=0, local=0, accounting=0, per_step=1, beta=1000),
        # the load sweep of App. A: six utilisations of several drawn workloads
        dict(name="rr_sweep", kind="rr", seeds=64, n_req=10000, N=4, C=50000),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "sequential", "alg1", "order", "order", "stream",
                       "stream", "rr"])
    lengths = rng.choice(sorted(LENGTHS))
    pmax = rng.choice([512, 2048, 8192])
    load = rng.choice([0.6, 0.9, 1.0, 1.3, 8.0])
    alpha = rng.choice([50000, 100000, 200000])
    if kind == "step":
        return dict(kind=kind, D=_log(rng, 1, 256), per=_log(rng, 16, 4096), H=_log(rng, 500, 65536),
                    J=_log(rng, 1, 65536), n=_log(rng, 100, 1000000), alpha=alpha, load=load,
                    lengths=lengths, pmax=pmax)
    if kind == "sequential":
        return dict(kind=kind, D=_log(rng, 2, 100), per=_log(rng, 16, 2048), H=_log(rng, 500, 32768),
                    J=_log(rng, 16, 2048), load=load, lengths=lengths, pmax=pmax)
    if kind == "alg1":
        return dict(kind=kind, D=_log(rng, 2, 1024), per=_log(rng, 16, 1024), J=_log(rng, 16, 8192),
                    S=rng.choice([1, 16, 32]), reserve=rng.random() < 0.7, load=load,
                    lengths=lengths, pmax=pmax)
    if kind == "order":
        return dict(kind=kind, N=_log(rng, 100, 1000000), D=_log(rng, 1, 1024),
                    arrival=rng.choice(["shuffled", "sorted"]), lengths=lengths)
    if kind == "stream":
        batch, D = _log(rng, 32, 512), _log(rng, 4, 48)
        return dict(kind=kind, N=_log(rng, 1000, min(30000, 117 * batch)), D=D,
                    cap=_log(rng, max(16000, 300000 // D), 262144),
                    H=rng.choice([4096, 10007, 16384]),
                    batch=batch, window=_log(rng, 50, 2000), alpha=alpha,
                    dispatch=rng.choice([0, 0, 0, 1, 2, 3]), local=rng.choice([0, 0, 1]),
                    accounting=0, per_step=rng.choice([0, 0, 1]), beta=rng.choice([-1, -1, 1000]))
    return dict(kind=kind, seeds=_log(rng, 1, 64), n_req=_log(rng, 200, 10000),
                N=rng.choice([2, 4, 4, 7, 16]), C=rng.choice([20000, 50000, 200000]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _lengths(rng, name, size):
    params, clip, _ = LENGTHS[name]
    if name == "lognormal":
        x = rng.lognormal(*params, size)
    elif name == "pareto":
        x = params[1] * (1.0 + rng.pareto(params[0], size))
    else:
        w, m1, s1, m2, s2 = params
        x = np.where(rng.random(size) < w, rng.lognormal(m1, s1, size), rng.lognormal(m2, s2, size))
    return np.clip(np.rint(x), 1, clip).astype(np.int32)


def _predictions(rng, name, true):
    _, clip, sigma = LENGTHS[name]
    x = true * np.exp(rng.normal(0.0, sigma, true.shape[0]))
    return np.clip(np.rint(x), 1, clip).astype(np.int32)


def _prompts(rng, pmax, size):
    return rng.integers(32, pmax + 1, size, dtype=np.int32)


def _cluster(c, rng):
    """Decoders with residents (uneven queues), capacities at the stated load
    (tokens held over capacity, 15% apart) and waiting-queue lengths."""
    D, R = c["D"], c["D"] * c["per"]
    share = rng.uniform(0.5, 1.5, D)
    off = np.zeros(D + 1, np.int64)
    off[1:] = np.floor(np.cumsum(share) / share.sum() * R + 0.5)
    true = _lengths(rng, c["lengths"], R)
    w = dict(off=off, prompt=_prompts(rng, c["pmax"], R),
             gen=np.floor(rng.random(R) * true).astype(np.int32),
             pred=_predictions(rng, c["lengths"], true),
             Q=rng.integers(0, c["per"] // 4 + 1, D, dtype=np.int32))
    held = np.zeros(D + 1, np.int64)
    held[1:] = np.cumsum(w["prompt"].astype(np.int64) + w["gen"] + 1)[off[1:] - 1]
    held = np.diff(held)
    w["cap"] = np.maximum(held / c["load"] * rng.uniform(0.85, 1.15, D), 1000).astype(np.int32)
    return w


def _inputs(c, seed):
    """Numpy arrays of one case, from the seed alone."""
    kind = c["kind"]
    rng = np.random.default_rng([seed, 2609])
    if kind in ("step", "sequential", "alg1"):
        w = _cluster(c, rng)
        true = _lengths(rng, c["lengths"], c["J"])
        w["cprompt"] = _prompts(rng, c["pmax"], c["J"])
        w["cpred"] = _predictions(rng, c["lengths"], true)
        if kind == "step":
            R = len(w["prompt"])
            w["cal_true"] = _lengths(rng, c["lengths"], c["n"])
            w["cal_pred"] = _predictions(rng, c["lengths"], w["cal_true"])
            w["dec"] = np.repeat(np.arange(c["D"], dtype=np.int32), np.diff(w["off"]))
            w["wait"] = rng.integers(0, 2 * MAX_WAIT + 1, R, dtype=np.int32)
        else:
            margin = int(rng.integers(50, 400))  # a calibrated quantile
            w["bound"], w["cbound"] = w["pred"] + margin, w["cpred"] + margin
        return w
    if kind == "order":
        N = c["N"]
        w = dict(dec=rng.integers(0, c["D"], N, dtype=np.int32),
                 bound=_lengths(rng, c["lengths"], N) + np.int32(200),
                 wait=rng.integers(0, 2 * MAX_WAIT + 1, N, dtype=np.int32),
                 arrival=np.sort(rng.integers(0, 10 * N, N)).astype(np.int32))
        if c["arrival"] == "shuffled":
            w["arrival"] = w["arrival"][rng.permutation(N)]
        return w
    if kind == "stream":
        return W.make_stream(seed=seed, n_requests=c["N"])
    return W.make_rr(c["seeds"], n_req=c["n_req"], seed0=1000 * seed)


def _dev(x, dtype=None):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=dtype)).cuda()


def _empty(*shape, dtype=torch.int32):
    return torch.empty(shape, dtype=dtype, device="cuda")


def prepare(case, seed):
    """The device tensors a scheduler holds before the call: its inputs, the
    outputs it reuses and one workspace, sized once for the calls of a pass."""
    c, w = case, _inputs(case, seed)
    s = dict(c=c, ws=M.Workspace())
    kind, lib = c["kind"], M.lib
    if kind in ("step", "sequential", "alg1"):
        D, J, R = c["D"], c["J"], len(w["prompt"])
        H = c.get("H", 1)
        for k in ("off", "prompt", "gen", "cap", "cprompt"):
            s[k] = _dev(w[k])
        s["Q0"] = _dev(w["Q"])
        s["headroom"] = _empty(J, dtype=torch.int64)
        if kind != "alg1":
            s["K"] = _empty(D, H)
            s["ws"].ensure(lib.maps_project_occupancy_workspace_size(D, H, R))
        if kind == "step":
            s["cal_true"], s["cal_pred"] = _dev(w["cal_true"]), _dev(w["cal_pred"])
            s["pred"] = _dev(np.concatenate([w["pred"], w["cpred"]]))
            s["U"], s["q"] = _empty(R + J), _empty(1)
            s["kmax"] = _empty(*M.kmax_shape(D, H))
            s["dec"] = _dev(np.concatenate([w["dec"], np.zeros(J, np.int32)]))
            s["wait"] = _dev(np.concatenate([w["wait"], np.zeros(J, np.int32)]))
            s["arrival"] = _dev(np.arange(R + J), np.int32)
            s["perm"], s["seg"] = _empty(R + J), _empty(D + 1, dtype=torch.int64)
            s["ws"].ensure(max(lib.maps_calibrate_workspace_size(c["n"], R + J),
                               lib.maps_dispatch_workspace_size(M.MODE_SNAPSHOT, D, H, J),
                               lib.maps_order_local_workspace_size(R + J, D)))
        else:
            s["bound"], s["cbound"] = _dev(w["bound"]), _dev(w["cbound"])
            s["Q"], s["choice"] = s["Q0"].clone(), _empty(J)
            s["ws"].ensure(lib.maps_dispatch_workspace_size(_mode(c), D, H, J))
    elif kind == "order":
        for k in ("dec", "bound", "wait", "arrival"):
            s[k] = _dev(w[k])
        s["perm"], s["seg"] = _empty(c["N"]), _empty(c["D"] + 1, dtype=torch.int64)
        s["ws"].ensure(lib.maps_order_local_workspace_size(c["N"], c["D"]))
    elif kind == "stream":
        nb = -(-c["N"] // c["batch"])
        s["cfg"] = M.stream_cfg(c["N"], c["D"], c["H"], c["cap"], c["batch"], c["window"],
                                c["alpha"], MAX_WAIT, c["dispatch"], c["local"], c["accounting"],
                                c["per_step"], c["beta"])
        for k in ("arrival_ms", "prompt", "true", "pred"):
            s[k] = _dev(w[k])
        s["delay"] = _dev(w["pred_delay_ms"]) if c["beta"] >= 0 else None
        s["choice"], s["q"] = _empty(c["N"]), _empty(nb)
        s["stats"] = _empty(nb, 4, dtype=torch.int64)
        s["dec_stats"] = _empty(c["D"], 4, dtype=torch.int64)
        s["ws"].ensure(lib.maps_stream_workspace_size(s["cfg"]))
    else:
        for k in ("arrival_us", "prompt", "out_len"):
            s[k] = _dev(w[k])
        n_real, n_req = w["arrival_us"].shape
        s["t_tok_us"], s["theta_ppm"] = w["t_tok_us"], w["theta_ppm"]
        s["admit"] = _empty(n_real, n_req, dtype=torch.int64)
        s["done"] = _empty(n_real, n_req, dtype=torch.int64)
        s["stats"] = _empty(n_real, c["N"], 6, dtype=torch.int64)
        s["t_sim"] = _empty(n_real, dtype=torch.int64)
        s["ws"].ensure(lib.maps_rr_pressure_workspace_size(
            M.RRCfg(n_req, c["N"], c["C"], w["t_tok_us"], w["theta_ppm"]), n_real))
    return s


def _mode(c):
    if c["kind"] == "sequential":
        return M.MODE_SEQUENTIAL
    return M.MODE_ALG1_SEQUENTIAL if c["reserve"] else M.MODE_ALG1_SNAPSHOT


def _ok(status):
    if status != M.MAPS_OK:
        raise M.MapsError(status)


def run(state):
    s, c = state, state["c"]
    kind, ws = c["kind"], s["ws"]
    if kind == "step":
        D, H, R = c["D"], c["H"], s["prompt"].numel()
        st, _ = M.maps_calibrate(s["cal_true"], s["cal_pred"], c["alpha"], s["pred"], s["U"],
                                 s["q"], ws=ws)
        _ok(st)
        _ok(M.maps_project_occupancy(D, H, s["off"], s["prompt"], s["gen"], s["U"][:R], s["K"],
                                     s["kmax"], ws=ws))
        _ok(M.maps_dispatch(M.MODE_SNAPSHOT, D, H, 1, s["K"], s["cap"], s["Q0"], s["cprompt"],
                            s["U"][R:], s["dec"][R:], s["headroom"], kmax=s["kmax"], ws=ws))
        _ok(M.maps_order_local(D, s["dec"], s["U"], s["wait"], s["arrival"], MAX_WAIT, s["perm"],
                               s["seg"], ws=ws))
        return {k: s[k] for k in ("q", "U", "K", "kmax", "headroom", "perm", "seg")} | {
            "choice": s["dec"][R:]}
    if kind == "sequential":
        D, H = c["D"], c["H"]
        s["Q"].copy_(s["Q0"])
        _ok(M.maps_project_occupancy(D, H, s["off"], s["prompt"], s["gen"], s["bound"], s["K"],
                                     ws=ws))
        _ok(M.maps_dispatch(M.MODE_SEQUENTIAL, D, H, 1, s["K"], s["cap"], s["Q"], s["cprompt"],
                            s["cbound"], s["choice"], s["headroom"], ws=ws))
        return {k: s[k] for k in ("choice", "headroom", "K", "Q")}
    if kind == "alg1":
        s["Q"].copy_(s["Q0"])
        _ok(M.maps_dispatch(_mode(c), c["D"], 1, c["S"], None, s["cap"], s["Q"], s["cprompt"],
                            s["cbound"], s["choice"], s["headroom"], s["off"], s["prompt"],
                            s["gen"], s["bound"], ws=ws))
        return {k: s[k] for k in ("choice", "headroom", "Q")}
    if kind == "order":
        _ok(M.maps_order_local(c["D"], s["dec"], s["bound"], s["wait"], s["arrival"], MAX_WAIT,
                               s["perm"], s["seg"], ws=ws))
        return {k: s[k] for k in ("perm", "seg")}
    if kind == "stream":
        _ok(M.maps_stream_run(s["cfg"], s["arrival_ms"], s["prompt"], s["true"], s["pred"],
                              s["choice"], s["q"], s["stats"], s["dec_stats"], ws=ws,
                              pred_delay=s["delay"]))
        return {k: s[k] for k in ("choice", "q", "stats", "dec_stats")}
    _ok(M.maps_rr_pressure(c["N"], c["C"], s["t_tok_us"], s["theta_ppm"], s["arrival_us"],
                           s["prompt"], s["out_len"], s["admit"], s["done"], s["stats"],
                           s["t_sim"], ws=ws))
    return {k: s[k] for k in ("admit", "done", "stats", "t_sim")}


def work(case):
    """Bytes of the inputs read once and the outputs written once.  The path
    is integer compares and sums: no floating-point operations are counted."""
    c, kind = case, case["kind"]
    if kind in ("step", "sequential", "alg1"):
        D, J, R = c["D"], c["J"], c["D"] * c["per"]
        b = 8 * (D + 1) + 12 * R + 8 * D + 8 * J + 12 * J  # residents, decoders, candidates
        if kind == "step":
            nb = -(-c["H"] // 16)
            b += 8 * c["n"] + 8 * (R + J)             # residuals; predictions and bounds
            b += 4 * D * c["H"] + 4 * D * nb          # K and its summary
            b += 16 * (R + J) + 8 * (D + 1)           # wait, arrival, decoder; the order
        elif kind == "sequential":
            b += 4 * D * c["H"] + 4 * D
        else:
            b += 4 * D
    elif kind == "order":
        b = 20 * c["N"] + 8 * (c["D"] + 1)
    elif kind == "stream":
        nb = -(-c["N"] // c["batch"])
        b = (24 + (4 if c["beta"] >= 0 else 0)) * c["N"] + 36 * nb + 32 * c["D"]
    else:
        n_real = c["seeds"] * len(W.WORKLOADS["rr"]["rhos"])
        b = n_real * (32 * c["n_req"] + 48 * c["N"] + 8)
    return {"bytes": b, "flops": 0}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------------------
# the same results from the definitions, in 64-bit numpy
# ---------------------------------------------------------------------------

def _occupancy(D, H, off, p, g, U):
    """K[k][t] = sum over the residents of k with t < e of (b + t)."""
    b = p.astype(np.int64) + g + 1
    e = np.minimum(np.maximum(U.astype(np.int64) - g, 1), H)
    K = np.empty((D, H), np.int64)
    t = np.arange(H)
    for k in range(D):
        r = slice(off[k], off[k + 1])
        gone_n = np.bincount(e[r], minlength=H + 1)[:H].cumsum()
        gone_b = np.zeros(H + 1, np.int64)
        np.add.at(gone_b, e[r], b[r])
        K[k] = b[r].sum() - gone_b[:H].cumsum() + (off[k + 1] - off[k] - gone_n) * t
    return K


def _order(D, dec, bound, wait, arrival):
    promoted = wait > MAX_WAIT
    perm = np.lexsort((np.arange(len(dec)), arrival, np.where(promoted, 0, bound), ~promoted, dec))
    seg = np.zeros(D + 1, np.int64)
    seg[1:] = np.bincount(dec, minlength=D).cumsum()
    return perm.astype(np.int32), seg


def _pick(h, Q):
    """Smallest queue among the decoders that fit, else the most headroom."""
    fit = h >= 0
    return int(np.argmin(np.where(fit, Q, np.iinfo(np.int64).max)) if fit.any() else np.argmax(h))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("stream", "rr"):
        return None  # step-by-step simulations: minutes in plain numpy
    w = _inputs(c, seed)
    if kind == "order":
        perm, seg = _order(c["D"], w["dec"], w["bound"], w["wait"], w["arrival"])
        return dict(perm=perm, seg=seg)
    D, J = c["D"], c["J"]
    cap, Q, cp = w["cap"].astype(np.int64), w["Q"].astype(np.int64), w["cprompt"].astype(np.int64)
    choice, head = np.empty(J, np.int32), np.empty(J, np.int64)
    if kind == "step":
        n, H, R = c["n"], c["H"], len(w["prompt"])
        k = -(-(1000000 - c["alpha"]) * (n + 1) // 1000000)
        s = np.maximum(w["cal_true"].astype(np.int64) - w["cal_pred"], 0)
        q = int(np.partition(s, k - 1)[k - 1])
        U = np.concatenate([w["pred"], w["cpred"]]).astype(np.int64) + q
        K = _occupancy(D, H, w["off"], w["prompt"], w["gen"], U[:R])
        t = np.arange(H)
        Kt = np.pad(K + t, ((0, 0), (0, -H % 16)))
        kmax = Kt.reshape(D, -1, 16).max(2)
        peak = np.maximum.accumulate(K + t, axis=1)
        by_queue = np.lexsort((np.arange(D), Q))
        u = np.minimum(np.maximum(U[R:], 1), H)
        for a in range(0, J, 4096):
            z = slice(a, min(a + 4096, J))
            h = cap[:, None] - (peak[:, u[z] - 1] + cp[z] + 1)
            fit = h[by_queue] >= 0
            ch = np.where(fit.any(0), by_queue[fit.argmax(0)], h.argmax(0))
            choice[z], head[z] = ch, h[ch, np.arange(h.shape[1])]
        dec = np.concatenate([w["dec"], choice])
        perm, seg = _order(D, dec, U, np.concatenate([w["wait"], np.zeros(J, np.int32)]),
                           np.arange(R + J))
        return dict(q=np.array([q], np.int32), U=U.astype(np.int32), K=K.astype(np.int32),
                    kmax=kmax.astype(np.int32), headroom=head, perm=perm, seg=seg, choice=choice)
    if kind == "sequential":
        H = c["H"]
        K = _occupancy(D, H, w["off"], w["prompt"], w["gen"], w["bound"])
        t = np.arange(H)
        peak = np.maximum.accumulate(K + t, axis=1)
        u = np.minimum(np.maximum(w["cbound"].astype(np.int64), 1), H)
        for j in range(J):
            h = cap - (peak[:, u[j] - 1] + cp[j] + 1)
            k = _pick(h, Q)
            choice[j], head[j] = k, h[k]
            K[k, :u[j]] += cp[j] + 1 + t[:u[j]]
            peak[k] = np.maximum.accumulate(K[k] + t)
            Q[k] += 1
        return dict(choice=choice, headroom=head, K=K.astype(np.int32), Q=Q.astype(np.int32))
    S = c["S"]
    held = w["prompt"].astype(np.int64) + np.maximum(w["bound"], w["gen"] + 1)
    blocks = np.concatenate([[0], np.cumsum(-(-held // S))])
    B = cap // S - np.diff(blocks[w["off"]])
    need = -(-(cp + w["cbound"]) // S)
    for j in range(J):
        h = B - need[j]
        k = _pick(h, Q)
        choice[j], head[j] = k, h[k]
        if c["reserve"]:
            B[k] -= need[j]
            Q[k] += 1
    return dict(choice=choice, headroom=head, Q=Q.astype(np.int32))
