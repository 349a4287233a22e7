"""The search with carried move values on one cluster against the oracle: slices of every size,
empty ones among them, both matrix types, and a key that never arrives; over several clusters
and with few vehicles the full evaluation runs (needs a GB300)."""
import pytest
import torch

from paper_2002_11710_gb300 import api, gen
from test_gpu_carry import _check_batch
from test_gpu_parity import _check_solve_vs_oracle

pytestmark = pytest.mark.gpu
HARD, PENALTY = gen.HARD, gen.PENALTY


def _instance(M, V, **kw):
    return gen.random_instance(131, n_loc=18, n_vehicles=V, n_missions=M, n_types=2, heli_only_frac=0.2, **kw)


def _carried(inst, mode=PENALTY, **kw):
    """Only the carried form keeps a ring of moves, two words per iteration of tenure."""
    dp = api.DeviceProblem(inst)
    smem = [api.plan(dp, api.make_params(t, 50, mode, 1000, block_threads=64, **kw)).smem_bytes for t in (8, 108)]
    assert smem[1] - smem[0] in (0, 800)
    return smem[1] > smem[0]


# missions, vehicles, CTAs: slices of 75 missions, 75 (the last shorter), 19, 10 and 10 (the last
# CTA without missions)
@pytest.mark.parametrize("M,V,cluster", [(150, 30, 2), (149, 33, 2), (151, 40, 8), (151, 60, 16), (150, 60, 16)])
@pytest.mark.parametrize("compact", [False, True])
def test_trajectory_on_one_cluster(M, V, cluster, compact):
    inst = _instance(M, V, duty_cap=900, max_minutes=90)
    kw = dict(cluster_size=cluster, grid_clusters=1, compact=compact)
    assert _carried(inst, **kw)
    _check_solve_vs_oracle(inst, PENALTY, 8, 90, block_threads=64, **kw)


@pytest.mark.parametrize("mode", [HARD, PENALTY])
@pytest.mark.parametrize("cluster", [1, 2, 8])
def test_trajectory_on_one_cluster_with_deadlines(mode, cluster):
    inst = _instance(120, 40, duty_cap=400, max_minutes=20, deadlines=True, deadline_lo=1100)
    kw = dict(cluster_size=cluster, grid_clusters=1)
    assert _carried(inst, mode, **kw)
    _check_solve_vs_oracle(inst, mode, 6, 90, block_threads=64, **kw)


@pytest.mark.parametrize("cluster", [2, 8])
def test_withheld_key_times_out(cluster):
    """A CTA that never publishes its first key ends every other wait of the carried loop."""
    inst = _instance(150, 50, duty_cap=900, max_minutes=90)
    kw = dict(cluster_size=cluster, grid_clusters=1)
    assert _carried(inst, **kw)
    params = api.make_params(8, 50, PENALTY, 1000, block_threads=64, timeout_ns=50_000_000, **kw)
    params.flags |= api._lib.TEST_WITHHOLD_KEY
    out = api.solve(api.DeviceProblem(inst), params)
    torch.cuda.synchronize()
    assert int(out.info[api.INFO_STATUS]) == api.E_TIMEOUT
    assert int(out.info[api.INFO_ITERS]) == 0
    _check_solve_vs_oracle(inst, PENALTY, 8, 50, block_threads=64, **kw)


@pytest.mark.parametrize("cluster,grid", [(1, 2), (4, 4)])
def test_full_evaluation_over_several_clusters(cluster, grid):
    inst = _instance(150, 50, duty_cap=900, max_minutes=90)
    kw = dict(cluster_size=cluster, grid_clusters=grid)
    assert not _carried(inst, **kw)
    _check_solve_vs_oracle(inst, PENALTY, 8, 60, block_threads=64, **kw)


# lane groups of short slices, blocks of 32 missions, words of 32 vehicles
EDGES = [(8, 250), (9, 260), (16, 150), (17, 150), (31, 65), (32, 64), (33, 63), (63, 32), (64, 31), (65, 33), (96, 12),
         (97, 30), (150, 5)]


@pytest.mark.parametrize("tenure", [0, 1, 7, 60, 512])
@pytest.mark.parametrize("compact", [False, True])
def test_sizes_on_one_cta(tenure, compact):
    insts = [gen.random_instance(300 + 7 * k, n_loc=10 + k, n_vehicles=v, n_missions=m, n_types=2, heli_only_frac=0.2,
                                 duty_cap=500, max_minutes=90) for k, (m, v) in enumerate(EDGES)]
    for i in insts:
        assert _carried(i, cluster_size=1, grid_clusters=1, compact=compact), (i.n_missions, i.n_vehicles)
    assert _check_batch(insts, PENALTY, tenure, 70, block_threads=64, compact=compact) == len(EDGES)


def test_long_times_take_the_multiplied_detour_key():
    """Under the hard cap times may grow to where 4 maxT times the next power of two above M + V
    no longer fits 32 bits, though 4 maxT (M + V) does."""
    base = gen.random_instance(71, n_loc=12, n_vehicles=70, n_missions=24, max_minutes=1000)
    scale = (2 ** 31 - 1) // (2 * (2 * 24 + 70 + 2)) // int(base.travel.max())
    inst = gen.Instance(**{**base.__dict__, "travel": base.travel * scale, "duty_cap": 10 ** 9})
    assert 4 * int(inst.travel.max()) * 128 >= 2 ** 32 > 4 * int(inst.travel.max()) * 94
    assert _carried(inst, HARD, cluster_size=1, grid_clusters=1)
    assert _check_batch([inst], HARD, 5, 60, block_threads=64) == 1


@pytest.mark.parametrize("M,V,cluster,carried", [(100, 1, 1, False), (100, 2, 1, False), (40, 4, 1, False), (100, 8, 1, True),
                                                 (200, 2, 8, False), (100, 12, 8, False), (200, 40, 8, True)])
def test_the_form_follows_the_vehicles(M, V, cluster, carried):
    inst = gen.random_instance(133, n_loc=18, n_vehicles=V, n_missions=M, duty_cap=900, max_minutes=90)
    kw = dict(cluster_size=cluster, grid_clusters=1)
    assert _carried(inst, **kw) == carried
    _check_solve_vs_oracle(inst, PENALTY, 8, 60, block_threads=64, **kw)
