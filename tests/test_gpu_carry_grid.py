"""The search with carried move values over several clusters, and its bounded waits, against
the oracle: slices of every size, empty ones among them, both matrix types, and a key that
never arrives (needs a GB300)."""
import pytest
import torch

from paper_2002_11710_gb300 import api, gen
from test_gpu_parity import _check_solve_vs_oracle

pytestmark = pytest.mark.gpu
HARD, PENALTY = gen.HARD, gen.PENALTY
WARPS = 2  # per CTA, at 64 threads


def _instance(M, V, **kw):
    return gen.random_instance(131, n_loc=18, n_vehicles=V, n_missions=M, n_types=2, heli_only_frac=0.2, **kw)


def _carried(inst, ctas):
    """More than 6 chunks of 32 items (pairs of relocations, swaps) a warp."""
    M, V = inst.n_missions, inst.n_vehicles
    return (M + V) * ((M + 1) // 2) + M * (M - 1) // 2 > 32 * 6 * ctas * WARPS


# missions, vehicles, CTAs of a cluster, clusters; slices 41, 27, 14, 6 (two CTAs without
# missions), 4 (two without) and 5 missions
SHAPES = [(81, 10, 1, 2), (81, 10, 1, 3), (83, 33, 2, 3), (81, 10, 4, 4), (120, 9, 16, 2), (120, 1, 8, 3)]


@pytest.mark.parametrize("M,V,cluster,grid", SHAPES)
@pytest.mark.parametrize("compact", [False, True])
def test_trajectory_over_clusters(M, V, cluster, grid, compact):
    inst = _instance(M, V, duty_cap=900, max_minutes=90)
    if V == 1:  # the one vehicle may be a plane
        inst = gen.Instance(**{**inst.__dict__, "heli_only": None})
    assert _carried(inst, cluster * grid)
    _check_solve_vs_oracle(inst, PENALTY, 8, 90, cluster_size=cluster, grid_clusters=grid, block_threads=32 * WARPS,
                           compact=compact)


@pytest.mark.parametrize("mode", [HARD, PENALTY])
@pytest.mark.parametrize("cluster,grid", [(1, 3), (2, 2), (4, 4)])
def test_trajectory_over_clusters_with_deadlines(mode, cluster, grid):
    inst = _instance(81, 34, duty_cap=400, max_minutes=25, deadlines=True, deadline_lo=1000)
    assert _carried(inst, cluster * grid)
    _check_solve_vs_oracle(inst, mode, 6, 90, cluster_size=cluster, grid_clusters=grid, block_threads=32 * WARPS)


@pytest.mark.parametrize("cluster,grid", [(2, 1), (8, 1), (1, 3), (2, 3), (4, 4)])
def test_withheld_key_times_out(cluster, grid):
    """A CTA (one cluster) or a cluster (several) that never publishes its first key."""
    inst = _instance(81, 10, duty_cap=900, max_minutes=90)
    assert _carried(inst, cluster * grid)
    params = api.make_params(8, 50, PENALTY, 1000, cluster_size=cluster, grid_clusters=grid, block_threads=32 * WARPS,
                             timeout_ns=50_000_000)
    params.flags |= api._lib.TEST_WITHHOLD_KEY
    out = api.solve(api.DeviceProblem(inst), params)
    torch.cuda.synchronize()
    assert int(out.info[api.INFO_STATUS]) == api.E_TIMEOUT
    assert int(out.info[api.INFO_ITERS]) == 0
    _check_solve_vs_oracle(inst, PENALTY, 8, 50, cluster_size=cluster, grid_clusters=grid, block_threads=32 * WARPS)
