"""Batches whose instances choose their form with several CTAs on an SM: the same results at
every block size, the oracle's for the largest, whose tables leave no room for a second CTA
(needs a GB300)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_11710_gb300 import api, gen

pytestmark = pytest.mark.gpu
PENALTY = gen.PENALTY


def _batch(n_small, n_large):
    rng = np.random.default_rng(9)
    insts = [gen.random_instance(900 + k, n_loc=72, n_vehicles=int(rng.choice([2, 3, 12])), n_missions=200,
                                 duty_cap=2000, max_minutes=90) for k in range(n_large)]
    for k in range(n_small):
        insts.append(gen.random_instance(1000 + k, n_loc=int(rng.integers(8, 30)), n_vehicles=int(rng.integers(1, 9)),
                                         n_missions=int(rng.integers(5, 40)), duty_cap=500, max_minutes=90))
    order = rng.permutation(len(insts))
    return [insts[i] for i in order]


@pytest.mark.parametrize("n_small,n_large", [(20, 4), (180, 20), (700, 12)])
def test_results_do_not_depend_on_the_block(n_small, n_large):
    insts = _batch(n_small, n_large)
    bp = api.BatchProblem(insts)
    outs = []
    for threads in (0, 64, 128, 256, 512):
        out = api.solve_batch(bp, api.make_params(7, 25, PENALTY, 1000, block_threads=threads))
        torch.cuda.synchronize()
        outs.append(out)
    for out in outs[1:]:
        for k in ("route_off", "route", "flight", "overflow", "info"):
            assert torch.equal(getattr(out, k), getattr(outs[0], k)), k
    large = [b for b, i in enumerate(insts) if i.n_missions == 200][:4]
    for b in large + [0, len(insts) - 1]:
        got = bp.unpack(outs[0], b)
        r = oracle.tabu_search(oracle.Problem(insts[b], PENALTY, 1000), 7, 25)
        assert r["status"] == 0 == int(got["info"][api.INFO_STATUS])
        assert int(got["info"][api.INFO_Z_BEST]) == r["z_best"] and int(got["info"][api.INFO_BEST_IT]) == r["best_it"]
        np.testing.assert_array_equal(got["route"], r["route"])
