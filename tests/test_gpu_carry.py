"""The search with carried move values (batches, requests, wide searches on one cluster)
against the oracle, at the sizes where its pieces change: blocks of 32 missions and one or
several of them, lane groups of short slices, words of 32 vehicles in a vehicle set, the ring
of tabu stamps and its limit, travel times too long for the shifted detour key."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_11710_gb300 import api, gen

pytestmark = pytest.mark.gpu
HARD, PENALTY = gen.HARD, gen.PENALTY

# (missions, vehicles): block and lane-group edges, then vehicle-set edges
SIZES = [(1, 1), (2, 3), (5, 2), (16, 4), (17, 1), (31, 5), (32, 3), (33, 4), (64, 2), (65, 7), (9, 31), (12, 32),
         (20, 33), (33, 65)]


def _check_batch(insts, mode, tenure, iters, **kw):
    bp = api.BatchProblem(insts)
    out = api.solve_batch(bp, api.make_params(tenure, iters, mode, 1000, **kw))
    torch.cuda.synchronize()
    started = 0
    for b, inst in enumerate(insts):
        got = bp.unpack(out, b)
        r = oracle.tabu_search(oracle.Problem(inst, mode, 1000), tenure, iters)
        assert int(got["info"][api.INFO_STATUS]) == r["status"], b
        if r["status"] != 0:
            continue
        started += 1
        assert int(got["info"][api.INFO_Z_BEST]) == r["z_best"] and int(got["info"][api.INFO_BEST_IT]) == r["best_it"], b
        assert int(got["info"][api.INFO_Z_FINAL]) == (int(r["traj_z"][-1]) if iters else r["z_best"]), b
        np.testing.assert_array_equal(got["route_off"], r["route_off"])
        np.testing.assert_array_equal(got["route"], r["route"])
    return started


@pytest.mark.parametrize("cluster,threads", [(1, 256), (1, 64), (2, 128), (8, 512), (16, 64)])
@pytest.mark.parametrize("tenure", [0, 1, 7, 60])
def test_batch_sizes_match_oracle(cluster, threads, tenure):
    insts = [gen.random_instance(300 + 7 * k, n_loc=10 + k, n_vehicles=v, n_missions=m, n_types=2, heli_only_frac=0.2,
                                 duty_cap=500, max_minutes=90) for k, (m, v) in enumerate(SIZES)]
    assert _check_batch(insts, PENALTY, tenure, 70, cluster_size=cluster, block_threads=threads) >= 13  # (17, 1) may have no helicopter


@pytest.mark.parametrize("mode,deadlines", [(HARD, False), (HARD, True), (PENALTY, True)])
@pytest.mark.parametrize("compact", [False, True])
def test_batch_constraints_match_oracle(mode, deadlines, compact):
    insts = [gen.random_instance(500 + k, n_loc=14, n_vehicles=v, n_missions=m, n_types=2, heli_only_frac=0.2,
                                 deadlines=deadlines, deadline_lo=1000, duty_cap=400, max_minutes=25)
             for k, (m, v) in enumerate([(6, 4), (23, 6), (31, 9), (33, 12), (40, 34), (65, 30)])]
    assert _check_batch(insts, mode, 6, 90, compact=compact) >= 4


def test_long_times_take_the_multiplied_detour_key():
    """Under the hard cap the overflow guard lets times grow to where 4 maxT times the next
    power of two above M + V no longer fits 32 bits, though 4 maxT (M + V) does."""
    base = gen.random_instance(71, n_loc=12, n_vehicles=12, n_missions=24, max_minutes=1000)
    scale = (2 ** 31 - 1) // (2 * (2 * 24 + 12 + 2)) // int(base.travel.max())
    inst = gen.Instance(**{**base.__dict__, "travel": base.travel * scale, "duty_cap": 10 ** 9})
    assert 4 * int(inst.travel.max()) * 64 >= 2 ** 32 > 4 * int(inst.travel.max()) * 36
    assert _check_batch([inst], HARD, 5, 60) == 1


@pytest.mark.parametrize("tenure", [512, 513])
def test_longest_carried_tenure(tenure):
    inst = gen.random_instance(81, n_loc=9, n_vehicles=4, n_missions=14, duty_cap=700)
    assert _check_batch([inst], PENALTY, tenure, 80) == 1


@pytest.mark.parametrize("threads", [0, 64, 256])
def test_wide_search_on_one_cluster(threads):
    """asched_solve on a neighbourhood the plan spreads over clusters: carried on one cluster,
    the trajectory of the full evaluation on several."""
    inst = gen.random_instance(91, n_loc=20, n_vehicles=20, n_missions=360, n_types=2, heli_only_frac=0.1,
                               duty_cap=900, max_minutes=90)
    dp = api.DeviceProblem(inst)
    a = api.solve_one_cluster(dp, api.make_params(9, 150, PENALTY, 100, block_threads=threads), trajectory=True)
    params = api.make_params(9, 150, PENALTY, 100)
    assert api.plan(dp, params).grid_clusters > 1
    b = api.solve(dp, params, trajectory=True)
    torch.cuda.synchronize()
    assert int(a.info[api.INFO_STATUS]) == 0
    for k in ("route_off", "route", "flight", "overflow", "info", "traj_move", "traj_z"):
        assert torch.equal(getattr(a, k), getattr(b, k)), k
