"""The one-warp sweep kernel (at most 64 missions and vehicles together) against the oracle at
the edges of its registers: 31 to 33 and 63 to 64 nodes, no missions, routes that cross
position 32, times beyond 16 bits, and runs without a trace (needs a GB300)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_11710_gb300 import api, gen

pytestmark = pytest.mark.gpu

# (locations, vehicles, missions)
SIZES = [(6, 1, 0), (5, 64, 0), (6, 40, 1), (9, 1, 31), (9, 1, 32), (12, 2, 29), (12, 3, 29), (12, 3, 30), (14, 31, 2),
         (14, 32, 31), (20, 16, 16), (20, 12, 22), (20, 5, 40), (25, 2, 61), (25, 1, 63), (25, 24, 40), (30, 20, 44)]


def _instances(nt, deadlines, scale=1):
    out = []
    for s, (L, V, M) in enumerate(SIZES):
        inst = gen.random_instance(40 + s, n_loc=L, n_vehicles=V, n_missions=M, n_types=nt, heli_only_frac=0.2 * (nt - 1),
                                   deadlines=deadlines, deadline_lo=200, duty_cap=1500 * scale, max_minutes=60)
        if deadlines:
            inst.deadline = np.minimum(inst.deadline, inst.horizon - 120).astype(np.int32)
        if scale > 1:
            inst.travel = inst.travel * scale
        out.append(inst)
    return out


@pytest.mark.parametrize("algorithm,tenure,worse", [(api.SWEEP_NEIGHBOURHOOD, 0, False), (api.SWEEP_TABU, 7, False),
                                                    (api.SWEEP_TABU, 0, False), (api.SWEEP_TABU, 3, True)])
@pytest.mark.parametrize("mode", [api.HARD, api.PENALTY])
@pytest.mark.parametrize("nt,deadlines,scale", [(2, False, 1), (1, True, 1), (2, False, 600)])
def test_register_edges_match_oracle(algorithm, tenure, worse, mode, nt, deadlines, scale):
    insts = _instances(nt, deadlines, scale)
    rng = np.random.default_rng(3)
    for orders in (None, [(rng.permutation(i.n_vehicles).astype(np.int32), rng.permutation(i.n_missions).astype(np.int32))
                          for i in insts]):
        bp = api.BatchProblem(insts)
        p = api.sweep_params(12, mode, 7, tenure, worse, repair=True)
        out, trace = api.sweep_batch(bp, algorithm, p, trace_capacity=1024, orders=orders)
        plain, _ = api.sweep_batch(bp, algorithm, p, orders=orders)
        torch.cuda.synchronize()
        solved = 0
        for b, inst in enumerate(insts):
            vo, mr = orders[b] if orders else (None, None)
            pb = oracle.Problem(inst, mode, 7)
            if algorithm == api.SWEEP_NEIGHBOURHOOD:
                r = oracle.neighbourhood_search(pb, 12, repair=True, vorder=vo, mrank=mr)
            else:
                r = oracle.tabu_sweep(pb, tenure, 12, accept_worse=worse, repair=True, vorder=vo, mrank=mr)
            for o in (out, plain):
                got = bp.unpack(o, b)
                info = got["info"]
                assert info[api.INFO_STATUS] == r["status"]
                if r["status"] != 0:
                    continue
                for k, name in ((api.INFO_Z_BEST, "z_best"), (api.INFO_Z_INIT, "z_init"), (api.INFO_Z_FINAL, "z_final"),
                                (api.INFO_BEST_IT, "best_step"), (api.INFO_ITERS, "sweeps"), (api.INFO_MOVES, "n_moves"),
                                (api.INFO_STEPS, "steps")):
                    assert info[k] == r[name], (b, name)
                np.testing.assert_array_equal(got["route_off"], r["route_off"])
                np.testing.assert_array_equal(got["route"], r["route"])
                z, fl, ov = oracle.cost(pb, got["route_off"], got["route"])
                np.testing.assert_array_equal(got["flight"], fl)
                np.testing.assert_array_equal(got["overflow"], ov)
                solved += 1
            if r["status"] == 0:
                n = min(r["steps"], 1024)
                mv = trace.move[b * 1024:b * 1024 + n].cpu().numpy().view(np.uint32)
                np.testing.assert_array_equal(mv, r["trace_move"][:n])
                np.testing.assert_array_equal(trace.z[b * 1024:b * 1024 + n].cpu().numpy(), r["trace_z"][:n])
        assert solved > 0
