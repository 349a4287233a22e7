"""Searches of one or two items a thread (relocations singly or in pairs, sides of swaps)
against the oracle, on both sides of the sizes where the items' form changes (needs a GB300)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_11710_gb300 import api, gen

pytestmark = pytest.mark.gpu
HARD, PENALTY = gen.HARD, gen.PENALTY


def _chunks(m, v, pairs):
    return -(-(m + v) * ((m + 1) // 2 if pairs else m) // 32) - (-m * (m - 1) // 32)


def _form(m, v, warps):
    single, paired = _chunks(m, v, False), _chunks(m, v, True)
    if single <= warps:
        return "single"
    if single > 2 * warps:
        return "wide"
    return "pairs" if paired <= warps else "two rounds"


# (missions, vehicles, CTAs, threads a CTA) and the form of the items there
CASES = [(1, 1, 1, 64, "single"), (2, 5, 1, 64, "single"), (5, 3, 1, 64, "pairs"), (6, 4, 1, 64, "pairs"),
         (7, 4, 1, 96, "two rounds"), (9, 3, 1, 128, "two rounds"), (10, 3, 1, 192, "pairs"), (10, 3, 1, 256, "single"),
         (11, 8, 1, 192, "two rounds"), (12, 4, 1, 192, "two rounds"), (14, 4, 1, 192, "wide"), (15, 6, 2, 192, "two rounds"), (24, 12, 16, 128, "single"),
         (31, 9, 16, 128, "pairs"), (33, 12, 16, 128, "pairs"), (40, 12, 16, 128, "two rounds"),
         (41, 20, 16, 128, "wide"), (61, 13, 16, 384, "pairs"), (80, 16, 16, 512, "two rounds")]


@pytest.mark.parametrize("mode,deadlines,heli", [(PENALTY, False, 0.0), (HARD, False, 0.25), (HARD, True, 0.25),
                                                 (PENALTY, True, 0.25)])
@pytest.mark.parametrize("m,v,cluster,threads,form", CASES)
def test_item_forms_match_oracle(m, v, cluster, threads, form, mode, deadlines, heli):
    assert _form(m, v, cluster * threads // 32) == form
    iters, checked = 60, 0
    for seed in range(40):  # the first instances with a feasible greedy start
        inst = gen.random_instance(1000 * m + seed, n_loc=12, n_vehicles=v, n_missions=m, n_types=2, heli_only_frac=heli,
                                   deadlines=deadlines, deadline_lo=1000, duty_cap=120 * (m // v + 1), max_minutes=25)
        r = oracle.tabu_search(oracle.Problem(inst, mode, 1000), 7, iters)
        if r["status"] != 0:
            continue
        for compact in (False, True):
            out = api.solve(api.DeviceProblem(inst), api.make_params(7, iters, mode, 1000, cluster_size=cluster,
                                                                     block_threads=threads, compact=compact), trajectory=True)
            torch.cuda.synchronize()
            assert int(out.info[api.INFO_STATUS]) == 0
            np.testing.assert_array_equal(out.traj_move.cpu().numpy().view(np.uint32)[:iters], r["traj_move"])
            np.testing.assert_array_equal(out.traj_z.cpu().numpy()[:iters], r["traj_z"])
            np.testing.assert_array_equal(out.route.cpu().numpy()[:m], r["route"])
        checked += 1
        if checked == 2:
            break
    assert checked > 0
