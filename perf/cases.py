"""The measured cases: what users of this framework have it do, through its public entry points.

Sizes and options come from the workloads of gen.py, the tests and bench.py: single Tabu
searches from 10 to 400 missions (penalty and hard caps, one and two vehicle types,
arrive-by times, helicopter-only missions), a search called on host data, mixed batches,
a backlog of requests drained by the serving kernels, the paper's own sweeps with and
without random loop orders, and travel matrices from coordinates.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

from paper_2002_11710_gb300 import _lib, api, gen, serve

MODES = {"penalty": api.PENALTY, "hard": api.HARD}


def listed():
    return [
        # the smallest search: a handful of missions planned at a desk, 200 iterations
        dict(name="solve-tiny", kind="solve", fleet="uniform", M=10, V=3, iterations=200, tenure=7),
        # one paper-sized scenario (Section 5 of the paper): planes and helicopters, helicopter-only
        # missions, arrive-by times, the duty cap as a constraint
        dict(name="solve-paper-fleet", kind="solve", fleet="paper", M=24, V=12, iterations=1000, tenure=7),
        # the paper-shaped search: 100 missions, 20 vehicles, 5,000 iterations
        dict(name="solve-paper-shaped", kind="solve", fleet="clustered", M=100, V=20, iterations=5000, tenure=10),
        # the large search of the headline benchmark: 400 missions, 50 vehicles, 10,000 iterations
        dict(name="solve-large", kind="solve", fleet="zipf", M=400, V=50, iterations=10000, tenure=15),
        # one re-planning request handled by itself, host arrays in and host arrays out
        dict(name="solve-host", kind="host", fleet="clustered", M=61, V=13, iterations=1000, tenure=10),
        # the batch of uneven instances (3-30 vehicles, 10-200 missions) of the batched benchmark
        dict(name="batch-mixed", kind="batch", B=1024, M_lo=10, M_hi=200, V_lo=3, V_hi=30, iterations=2000,
             tenure=10),
        # many paper-sized scenarios (12-33 missions) under the hard cap with arrive-by times
        dict(name="batch-paper-fleet", kind="batch-paper", B=300, M_lo=12, M_hi=33, iterations=1000, tenure=7),
        # a backlog of re-planning requests (10-400 missions) drained by both serving lanes
        dict(name="serve-backlog", kind="serve", B=128, iterations=1000, tenure=10),
        # the paper's Algorithm 2 on a large set of paper-sized scenarios (each drawn scenario
        # planned several times, so that the set stays quick to draw)
        dict(name="sweep-neighbourhood", kind="sweep", algorithm="neighbourhood", B=16384, distinct=2048,
             M_lo=12, M_hi=33, orders=False, sweeps=100, tenure=0),
        # the paper's Algorithm 3, 10 runs per scenario in random loop orders
        dict(name="sweep-tabu-orders", kind="sweep", algorithm="tabu", B=5120, distinct=512,
             M_lo=12, M_hi=33, orders=True, sweeps=100, tenure=7),
        # travel matrices of paper-sized scenarios (52 locations, two vehicle types) from kilometres
        dict(name="travel-euclidean", kind="travel", metric="euclidean", B=16384, L_lo=52, L_hi=52, types=2),
        # travel matrices of uneven regions (40-1,000 locations) from latitudes and longitudes
        dict(name="travel-haversine-ragged", kind="travel", metric="haversine", B=96, L_lo=40, L_hi=1000, types=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "host", "batch", "batch-paper", "serve", "sweep", "travel"])
    if kind in ("solve", "host"):
        fleet = rng.choice(["uniform", "clustered", "zipf", "paper"] if kind == "solve" else ["clustered", "paper"])
        if fleet == "paper":
            M, V = rng.randint(12, 33), 12
        else:
            M = _log_int(rng, 10, 400)
            V = min(50, max(3, int(round(M / rng.uniform(3.0, 9.0)))))
        return dict(kind=kind, fleet=fleet, M=M, V=V, iterations=_log_int(rng, 200, 10000), tenure=rng.randint(5, 20))
    if kind == "batch":
        lo = _log_int(rng, 10, 60)
        vlo = rng.randint(3, 8)
        return dict(kind=kind, B=_log_int(rng, 16, 512), M_lo=lo, M_hi=min(200, _log_int(rng, lo, 200)), V_lo=vlo,
                    V_hi=rng.randint(vlo, 30), iterations=_log_int(rng, 200, 2000), tenure=rng.randint(5, 20))
    if kind == "batch-paper":
        lo = rng.randint(12, 33)
        return dict(kind=kind, B=_log_int(rng, 16, 1024), M_lo=lo, M_hi=rng.randint(lo, 33),
                    iterations=_log_int(rng, 200, 2000), tenure=rng.randint(5, 15))
    if kind == "serve":
        return dict(kind=kind, B=_log_int(rng, 8, 128), iterations=_log_int(rng, 200, 1000), tenure=rng.randint(5, 15))
    if kind == "sweep":
        tabu = rng.random() < 0.5
        lo = rng.randint(12, 33)
        distinct = _log_int(rng, 64, 1024)
        return dict(kind=kind, algorithm="tabu" if tabu else "neighbourhood", B=distinct * rng.randint(1, 10),
                    distinct=distinct, M_lo=lo, M_hi=rng.randint(lo, 33), orders=rng.random() < 0.5, sweeps=100,
                    tenure=rng.randint(3, 12) if tabu else 0)
    lo = _log_int(rng, 10, 1000)
    hi = min(1000, _log_int(rng, lo, 1000))
    types = rng.randint(1, 2)
    cells = 16384 * 52 * 52  # at most half the cells of the largest listed case
    most = max(8, min(16384, int(cells / (types * hi * hi))))
    return dict(kind="travel", metric=rng.choice(["euclidean", "haversine"]), B=_log_int(rng, 8, most), L_lo=lo,
                L_hi=hi, types=types)


# ------------------------------------------------------------------ inputs

def _instance(case, seed):
    fleet, M, V = case["fleet"], case["M"], case["V"]
    if fleet == "uniform":
        return gen.make_instance(seed, n_bases=min(V, 12), n_vehicles=V, n_facilities=max(6, min(60, M)), n_missions=M,
                                 box_km=1000.0, duty_cap=720)
    if fleet == "clustered":
        return gen.make_instance(seed, n_bases=12, n_vehicles=V, n_facilities=60, n_missions=M, box_km=1500.0,
                                 geography="clustered", duty_cap=720)
    if fleet == "zipf":
        return gen.make_instance(seed, n_bases=40, n_vehicles=V, n_facilities=200, n_missions=M, box_km=3000.0,
                                 geography="clustered", pairs="zipf", duty_cap=960)
    # the paper's fleet: the first drawn scenario whose greedy start is feasible, as the paper
    # kept only valid scenarios
    params = api.make_params(case["tenure"], 0, api.HARD)
    for k in range(200):
        inst = gen.paper_fleet(1000 * seed + k, M)
        info = api.greedy_init(api.DeviceProblem(inst), params)[2]
        if int(info[api.INFO_STATUS]) == api.OK:
            break
    return inst


# The sizes of a case's instances are the same for every seed; a seed draws what they hold.

def _batch_instances(case, seed):
    rng = random.Random(case["B"])
    out = []
    for i in range(case["B"]):
        V = rng.randint(case["V_lo"], case["V_hi"])
        M = rng.randint(case["M_lo"], case["M_hi"])
        out.append(gen.make_instance(100000 * seed + i, n_bases=12, n_vehicles=V, n_facilities=60, n_missions=M,
                                     box_km=1500.0, geography="clustered", duty_cap=720))
    return out


def _paper_instances(case, seed, n):
    rng = random.Random(n)
    return [gen.paper_fleet(100000 * seed + i, rng.randint(case["M_lo"], case["M_hi"])) for i in range(n)]


def _travel_sizes(case):
    rng = random.Random(case["B"])
    return [_log_int(rng, case["L_lo"], case["L_hi"]) for _ in range(case["B"])]


def _travel_coords(case, seed):
    sizes = _travel_sizes(case)
    rng = np.random.default_rng(seed)
    n = sum(sizes)
    if case["metric"] == "euclidean":
        xy = rng.uniform(0.0, 1000.0, size=(n, 2))
    else:  # New South Wales and around: latitude, longitude
        xy = np.stack([rng.uniform(-37.0, -28.0, n), rng.uniform(141.0, 154.0, n)], axis=1)
    return sizes, np.ascontiguousarray(xy)


SPEEDS = [300.0, 500.0]


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("solve", "host"):
        inst = _instance(case, seed)
        mode = api.HARD if case["fleet"] == "paper" else api.PENALTY
        st["params"] = api.make_params(case["tenure"], case["iterations"], mode, 1000)
        st["problem"] = api.DeviceProblem(inst) if kind == "solve" else api.pin_instance(inst)
    elif kind in ("batch", "batch-paper"):
        if kind == "batch":
            insts, mode = _batch_instances(case, seed), api.PENALTY
        else:
            insts, mode = _paper_instances(case, seed, case["B"]), api.HARD
        st["params"] = api.make_params(case["tenure"], case["iterations"], mode, 1000)
        st["problem"] = api.BatchProblem(insts)
    elif kind == "serve":
        # Requests already published when the launches start, and the stop flag raised, so that
        # both lanes end once every request is taken: small ones on one-CTA workers, from 60
        # missions on clusters of 8 CTAs (the split of the serving benchmark).
        srv = serve.Server(max_loc=72, max_vehicles=80, max_missions=400, n_slots=case["B"], big_missions=60,
                           big_cluster=8, big_clusters=8)
        for i in range(case["B"]):
            srv.submit(gen.serving_request(100000 * seed + i), i)
        srv.copy_stream.synchronize()
        st["server"] = srv
        for name, control, published in (("control", srv.control, srv.next_ticket),
                                         ("control_big", srv.control_big, srv.next_ticket_big)):
            control.zero_()
            control[_lib.CTRL_PUBLISHED] = published
            control[_lib.CTRL_STOP] = 1
            st[name] = control.clone()
        st["params"] = api.make_params(case["tenure"], case["iterations"], api.PENALTY, 1000)
        st["params_big"] = api.make_params(case["tenure"], case["iterations"], api.PENALTY, 1000, cluster_size=8)
    elif kind == "sweep":
        insts = _paper_instances(case, seed, case["distinct"])
        copies = case["B"] // case["distinct"]
        bp = api.BatchProblem([i for i in insts for _ in range(copies)])
        st["problem"] = bp
        st["params"] = api.sweep_params(case["sweeps"], api.HARD, tenure=case["tenure"], repair=True)
        st["orders"] = None
        if case["orders"]:
            st["orders"] = api.sweep_orders_tensors(bp, [gen.sweep_orders(100000 * seed + b, 12, insts[b // copies].n_missions)
                                                         for b in range(case["distinct"] * copies)])
    else:
        sizes, xy = _travel_coords(case, seed)
        st["coords"] = torch.from_numpy(xy).cuda()
        st["problem"] = _travel_batch(sizes, case["types"])
    torch.cuda.synchronize()
    return st


def _travel_batch(sizes, types):
    """A batch whose travel matrices are still to be built: a mission and a vehicle per region."""
    one = np.zeros(1, np.int32)
    return api.BatchProblem([gen.Instance(travel=np.zeros((types, L, L), np.int32), veh_base=one, veh_type=one,
                                          pickup=one, delivery=one + 1, heli_only=None, deadline=None, duty_cap=600)
                             for L in sizes])


# ------------------------------------------------------------------ one pass

def _solve_outputs(out):
    return [out.route_off, out.route, out.flight, out.overflow, out.info]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        out = api.solve(state["problem"], state["params"], trajectory=True)
        return _solve_outputs(out) + [out.traj_move, out.traj_z]
    if kind == "host":
        res = api.solve_host(state["problem"], state["params"], trajectory=True)
        return [res[k] for k in ("route_off", "route", "flight", "overflow", "info", "traj_z")]
    if kind in ("batch", "batch-paper"):
        return _solve_outputs(api.solve_batch(state["problem"], state["params"]))
    if kind == "serve":
        return _drain(state)
    if kind == "sweep":
        algorithm = api.SWEEP_TABU if case["algorithm"] == "tabu" else api.SWEEP_NEIGHBOURHOOD
        out, _ = api.sweep_batch(state["problem"], algorithm, state["params"], orders=state["orders"])
        return _solve_outputs(out)
    metric = api.METRIC_HAVERSINE if case["metric"] == "haversine" else api.METRIC_EUCLIDEAN
    status = api.travel_into_batch(state["problem"], state["coords"], SPEEDS[:case["types"]], metric)
    return [state["problem"].travel, status]


def _drain(state):
    """Both serving lanes over the published requests, as Server.start launches them."""
    srv = state["server"]
    cur = torch.cuda.current_stream()
    srv.control.copy_(state["control"])
    srv.control_big.copy_(state["control_big"])
    srv.done.fill_(-1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lanes = ((srv.struct_big, state["params_big"], 64, srv.big_stream),
             (srv.struct, state["params"], sms - 64, srv.serve_stream))
    for struct, params, ctas, stream in lanes:
        stream.wait_stream(cur)
        _lib.check(_lib.load().asched_serve(ctypes.byref(struct), ctypes.byref(params), int(10e9), ctas,
                                            ctypes.c_void_p(stream.cuda_stream)), "asched_serve")
    for _, _, _, stream in lanes:
        cur.wait_stream(stream)
    return [srv.slot_out, srv.done]


# ------------------------------------------------------------------ work

# int32 operations of one evaluated move: a relocation about 20, a swap about 30.
def _search_work(M, V, iterations, words):
    return 4.0 * words, iterations * (20.0 * M * (M + V - 2) + 30.0 * M * (M - 1) / 2)


def work(case):
    """Inputs read once, outputs written once; int32 operations counted as flops (every move of
    every iteration considered once)."""
    kind = case["kind"]
    if kind in ("solve", "host"):
        M, V = case["M"], case["V"]
        L = {"uniform": min(V, 12) + max(6, min(60, M)), "clustered": 72, "zipf": 240, "paper": 52}[case["fleet"]]
        nt = 2 if case["fleet"] == "paper" else 1
        b, f = _search_work(M, V, case["iterations"], nt * L * L + 6 * V + 5 * M + 2 * case["iterations"])
        return {"bytes": b, "flops": f}
    if kind in ("batch", "batch-paper", "serve", "sweep"):
        if kind == "serve":
            ms, V, words = [math.exp(math.log(60.0) + 0.5 * z) for z in (-1.5, -0.7, 0.0, 0.7, 1.5)], None, 72 * 72
        else:
            lo, hi = case["M_lo"], case["M_hi"]
            ms = [lo + (hi - lo) * k / 4.0 for k in range(5)]
            V = (case["V_lo"] + case["V_hi"]) / 2.0 if kind == "batch" else 12
            words = 72 * 72 if kind == "batch" else 2 * 52 * 52
        bts = fl = 0.0
        for m in ms:
            v = V if V is not None else math.ceil(m / 5)
            if kind == "sweep":  # about two sweeps, each mission against every insertion point
                b, f = 4.0 * (words + 6 * v + 5 * m), 2.0 * 20.0 * m * (m + v)
            else:
                b, f = _search_work(m, v, case["iterations"], words + 6 * v + 5 * m)
            bts += b / len(ms)
            fl += f / len(ms)
        return {"bytes": bts * case["B"], "flops": fl * case["B"]}
    lo, hi = case["L_lo"], case["L_hi"]
    r = math.log(hi / lo) if hi > lo else 0.0
    mean_sq = (hi * hi - lo * lo) / (2.0 * r) if r > 0 else float(lo * lo)
    cells = case["B"] * mean_sq
    per = 8.0 if case["metric"] == "euclidean" else 30.0  # float operations per pair
    return {"bytes": 4.0 * case["types"] * cells + 16.0 * case["B"] * math.sqrt(mean_sq), "flops": per * cells}


# ------------------------------------------------------------------ the values in 64 bits

def exact(case, seed):
    """Travel matrices in plain float64 numpy; the searches are integer trajectories with no
    short restatement."""
    if case["kind"] != "travel":
        return None
    sizes, xy = _travel_coords(case, seed)
    parts, off = [], 0
    for L in sizes:
        c = xy[off:off + L]
        off += L
        if case["metric"] == "euclidean":
            d = np.sqrt((c[:, None, 0] - c[None, :, 0]) ** 2 + (c[:, None, 1] - c[None, :, 1]) ** 2)
        else:
            ang = c * (math.pi / 180.0)
            s1 = np.sin((ang[:, None, 0] - ang[None, :, 0]) * 0.5)
            s2 = np.sin((ang[:, None, 1] - ang[None, :, 1]) * 0.5)
            cs = np.cos(ang[:, 0])
            a = s1 * s1 + (cs[:, None] * cs[None, :]) * (s2 * s2)
            d = 2.0 * 6371.0 * np.arcsin(np.minimum(np.sqrt(a), 1.0))
        for v in SPEEDS[:case["types"]]:
            parts.append(np.rint(d / v * 60.0).reshape(-1))
    return [np.concatenate(parts), None]
