"""Travel matrices of small instances around the date line and the globe, where longitudes lie
more than half a turn apart: the shared-memory build and the tiles give the same integers, the
oracle's wherever the time is not within 1e-6 of a half minute (needs a GB300)."""
import numpy as np
import pytest

from paper_2002_11710_gb300 import api
from test_gpu_travel_tiles import _build, _check, _points

pytestmark = pytest.mark.gpu


def _coords(region, n, lo, hi):
    rng = np.random.default_rng(17)
    out = []
    for _ in range(n):
        L = int(rng.integers(lo, hi + 1))
        if region == "strip":  # a few degrees either side of the date line, as -180..180
            lon = rng.uniform(176.0, 184.0, L)
            out.append(np.stack([rng.uniform(-20.0, -14.0, L), np.where(lon > 180.0, lon - 360.0, lon)], axis=1))
        elif region == "turns":  # the same places, given as any number of turns
            lon = rng.uniform(176.0, 184.0, L) + 360.0 * rng.integers(-2, 3, L)
            out.append(np.stack([rng.uniform(-20.0, -14.0, L), lon], axis=1))
        else:
            out.append(_points(rng, L, region))
    return out


@pytest.mark.parametrize("region", ["strip", "turns", "dateline", "turn"])
@pytest.mark.parametrize("speeds", [[10.0], [300.0, 500.0]])
def test_small_instances_across_the_date_line(region, speeds):
    """640 instances fill the chip and take the shared-memory build; slow speeds make long
    times, whose absolute error is the larger."""
    _check(_coords(region, 640, 30, 55), speeds, region)


@pytest.mark.parametrize("region", ["strip", "turn"])
def test_both_builds_agree(region):
    coords = _coords(region, 640, 30, 55)
    many = _build(coords, [10.0], api.METRIC_HAVERSINE)
    large = _coords(region, 1, 90, 90)
    for k in range(0, 640, 64):  # 64 instances beside a larger one join its tiles
        for a, b in zip(_build(coords[k:k + 64] + large, [10.0], api.METRIC_HAVERSINE), many[k:k + 64]):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("lo,hi,n", [(1, 20, 9), (30, 64, 64), (65, 78, 64), (65, 78, 200)])
def test_few_small_instances_alone(lo, hi, n):
    """Batches of small instances only, too few to fill the chip: by their own kernel up to a
    tile's side or above one per SM, else by tiles."""
    _check(_coords("dateline", n, lo, hi), [300.0], "dateline")
    rng = np.random.default_rng(5)
    _check([_points(rng, int(rng.integers(lo, hi + 1)), "plane") for _ in range(n)], [300.0], "plane")
