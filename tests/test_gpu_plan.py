"""asched_plan tells the shared memory of the form of the search that a call then launches
(needs a GB300)."""
import pytest

from paper_2002_11710_gb300 import api, gen

pytestmark = pytest.mark.gpu


def _smem(inst, tenure, **kw):
    return api.plan(api.DeviceProblem(inst), api.make_params(tenure, 20, gen.PENALTY, 1000, **kw)).smem_bytes


@pytest.mark.parametrize("cluster,threads,compact", [(1, 64, False), (1, 256, False), (1, 128, True), (2, 64, False)])
def test_plan_follows_the_form_of_the_search(cluster, threads, compact):
    """Carried move values keep a ring of two words per iteration of tenure; past 512 the full
    evaluation runs, whose layout holds no ring."""
    inst = gen.random_instance(141, n_loc=20, n_vehicles=20, n_missions=120, duty_cap=900, max_minutes=90)
    kw = dict(cluster_size=cluster, block_threads=threads, grid_clusters=1, compact=compact)
    assert _smem(inst, 500, **kw) - _smem(inst, 10, **kw) == 4 * 2 * 490
    assert _smem(inst, 513, **kw) == _smem(inst, 600, **kw) != _smem(inst, 10, **kw)


def test_plan_of_a_small_search_holds_no_ring():
    inst = gen.tiny(0)
    assert _smem(inst, 10) == _smem(inst, 500)
