"""Batches by the full evaluation, either side of the size from which its item lists take
relocations of four missions and neighbours in a pass of their own (6 chunks of 32 items a
warp), at every mission count mod 4, against the oracle (needs a GB300)."""
import pytest

from paper_2002_11710_gb300 import gen
from test_gpu_carry import _check_batch

pytestmark = pytest.mark.gpu
HARD, PENALTY = gen.HARD, gen.PENALTY

# 64 threads: pairs up to 384 items, (19, 2) with 381 and (19, 3) with 391 on either side
SIZES = [(13, 2), (15, 2), (18, 3), (19, 2), (19, 3), (20, 1), (21, 2), (23, 2), (40, 2), (65, 1), (66, 2), (67, 1)]


@pytest.mark.parametrize("mode", [HARD, PENALTY])
@pytest.mark.parametrize("compact", [False, True])
def test_lists_match_oracle(mode, compact):
    insts = [gen.random_instance(700 + 3 * k, n_loc=9 + k, n_vehicles=v, n_missions=m, n_types=2,
                                 heli_only_frac=0.2 if v > 1 else 0.0, duty_cap=60 * m if mode == HARD else 500,
                                 max_minutes=90) for k, (m, v) in enumerate(SIZES)]
    assert _check_batch(insts, mode, 6, 60, block_threads=64, compact=compact) >= 9


@pytest.mark.parametrize("mode", [HARD, PENALTY])
@pytest.mark.parametrize("cluster", [1, 2])
def test_lists_with_deadlines_match_oracle(mode, cluster):
    insts = []
    for k, (m, v) in enumerate(SIZES):
        i = gen.random_instance(800 + 3 * k, n_loc=9 + k, n_vehicles=v, n_missions=m, deadlines=True, duty_cap=30 * m + 300,
                                max_minutes=20)
        insts.append(gen.Instance(**{**i.__dict__, "deadline": 100 + 60 * i.deadline, "horizon": 100000}))
    assert _check_batch(insts, mode, 6, 60, block_threads=64, cluster_size=cluster) >= 9
