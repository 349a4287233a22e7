"""Travel matrices by tiles: tile edges, runs of tiles that cross instances, small instances
that join the tiles or keep their own kernel, and longitudes either side of the date line
(needs a GB300)."""
import numpy as np
import pytest
import torch

from oracle import travel
from paper_2002_11710_gb300 import api, gen

pytestmark = pytest.mark.gpu

EDGES = [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 193, 256]


def _build(coords, speeds, metric):
    one = np.zeros(1, np.int32)
    nt = len(speeds)
    bp = api.BatchProblem([gen.Instance(travel=np.zeros((nt, len(c), len(c)), np.int32), veh_base=one, veh_type=one,
                                        pickup=one, delivery=one + 1, heli_only=None, deadline=None, duty_cap=600)
                           for c in coords])
    bp.travel.fill_(-7)
    xy = torch.from_numpy(np.concatenate(coords)).to("cuda", torch.float64)
    status = api.travel_into_batch(bp, xy, speeds, metric)
    torch.cuda.synchronize()
    assert int(status.item()) == api.OK
    return [bp.travel[int(bp.h_travel_off[b]):int(bp.h_travel_off[b]) + nt * len(c) ** 2].cpu().numpy()
            .reshape(nt, len(c), len(c)) for b, c in enumerate(coords)]


def _points(rng, n, region):
    if region == "plane":
        return rng.uniform(-800.0, 1800.0, size=(n, 2))
    if region == "dateline":  # 160 E to 160 W, as -180..180
        lon = rng.uniform(160.0, 200.0, n)
        return np.stack([rng.uniform(-50.0, 70.0, n), np.where(lon > 180.0, lon - 360.0, lon)], axis=1)
    if region == "turn":  # the globe, as 0..360
        return np.stack([rng.uniform(-90.0, 90.0, n), rng.uniform(0.0, 360.0, n)], axis=1)
    return np.stack([rng.uniform(-37.0, -28.0, n), rng.uniform(141.0, 154.0, n)], axis=1)


def _check(coords, speeds, region):
    hav = region != "plane"
    got = _build(coords, speeds, api.METRIC_HAVERSINE if hav else api.METRIC_EUCLIDEAN)
    metric = travel.HAVERSINE if hav else travel.EUCLIDEAN
    for g, c in zip(got, coords):
        want = travel.travel_minutes(c, speeds, metric)
        if hav:  # device and host trigonometry differ in the last bits: exact away from half minutes
            raw = travel.minutes_unrounded(c, speeds, metric)
            sure = np.abs(np.abs(raw - np.floor(raw)) - 0.5) >= 1e-6
            assert np.array_equal(g[sure], want[sure])
            assert np.abs(g.astype(np.int64) - want).max() <= 1
        else:
            np.testing.assert_array_equal(g, want)
        assert (g == np.transpose(g, (0, 2, 1))).all()


@pytest.mark.parametrize("region", ["plane", "region", "dateline", "turn"])
@pytest.mark.parametrize("speeds", [[300.0], [300.0, 500.0]])
def test_tile_edges(speeds, region):
    rng = np.random.default_rng(len(speeds))
    _check([_points(rng, n, region) for n in EDGES + [1000]], speeds, region)


@pytest.mark.parametrize("region", ["plane", "region"])
def test_small_instances_with_and_without_their_own_kernel(region):
    """640 small instances take the shared-memory build, with the larger ones in tiles beside
    them; 200 join the tiles."""
    rng = np.random.default_rng(3)
    for n_small in (200, 640):
        sizes = [int(x) for x in rng.integers(1, 20, n_small)] + [int(x) for x in rng.integers(79, 200, 70)]
        rng.shuffle(sizes)
        _check([_points(rng, n, region) for n in sizes], [300.0], region)


def test_every_entry_uncertain_overflows_the_queue():
    """Half the times of a 200-point line are exact ties, more than the queue of deferred
    entries holds."""
    line = np.stack([0.5 * np.arange(200) + 1000.0, np.zeros(200)], axis=1)
    _check([line, line[:65]], [60.0, 120.0], "plane")
