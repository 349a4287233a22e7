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


@pytest.mark.parametrize("region", ["region", "dateline", "strip", "poles", "close"])
def test_tiles_at_slow_speeds(region):
    """At 2 and 10 km/h times run to 10^5 minutes and more, where a float32 error above its screen
    would show as a wrong integer: half a million pairs each, around the poles and a few hundred
    metres apart among them."""
    rng = np.random.default_rng(23)
    n = 1000
    if region == "poles":
        c = np.stack([np.where(rng.random(n) < 0.5, 90.0, -90.0) * (1.0 - 10.0 ** rng.uniform(-9.0, -1.2, n)),
                      rng.uniform(-180.0, 180.0, n)], axis=1)
        c[:, 0] = np.abs(c[:, 0])  # one pole: no pair nearly half a turn apart
    elif region == "close":
        c = np.stack([rng.uniform(47.0, 47.01, n), rng.uniform(8.0, 8.01, n)], axis=1)
    elif region == "strip":
        lon = rng.uniform(176.0, 184.0, n)
        c = np.stack([rng.uniform(-20.0, -14.0, n), np.where(lon > 180.0, lon - 360.0, lon)], axis=1)
    else:
        c = _points(rng, n, region)
    _check([c, c[:333]], [2.0, 10.0], region)
