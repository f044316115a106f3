"""Batches whose events have more than 10,000 tracks on average, for which the
vertex finder sorts, scans and joins in kernels of their own over every SM:
several events, uneven and empty ones, tracks that take no part, and one
event beyond the limit beside others; against the oracle."""
import numpy as np
import pytest

from oracle import postfit
from paper_2008_13461_gb300 import _lib as L

from test_gpu_vertices import CUTS, KEYS, _compare, _gpu

pytestmark = pytest.mark.gpu

MOST = 512


def event(n: int, e: int, seed: int, idle: int = 0) -> dict:
    """n tracks of event e around n / 25 vertices, and idle ones that no cut lets in."""
    rng = np.random.default_rng(seed)
    centres = rng.uniform(-15.0, 15.0, max(1, n // 25))
    k = n + idle
    z = centres[rng.integers(0, len(centres), k)] + 0.003 * rng.standard_normal(k)
    take = np.zeros(k, bool)
    take[rng.permutation(k)[:n]] = True
    return dict(ev=np.full(k, e, np.int32), z0=z.astype(np.float32),
                ez0=(0.003 * rng.uniform(0.5, 2.0, k)).astype(np.float32),
                pt=np.where(take, rng.uniform(0.6, 5.0, k), 0.3).astype(np.float32),
                nhits=np.full(k, 4, np.uint8), keep=np.ones(k, np.uint8))


def batch(sizes, idle, seed, shuffled):
    d = [event(n, e, seed + e, i) for e, (n, i) in enumerate(zip(sizes, idle)) if n + i]
    d = {k: np.concatenate([v[k] for v in d]) for k in KEYS}
    if shuffled:
        order = np.random.default_rng(seed).permutation(len(d["ev"]))
        d = {k: v[order] for k, v in d.items()}
    assert len(d["ev"]) // len(sizes) > 10000           # the rule of the split path
    return d


@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("sizes,idle", [
    ((10003, 10001), (0, 9)),
    ((0, 11111, 0, 0, 9001, 1, 0), (7, 30001, 3, 0, 29989, 2, 8)),      # empty, single, first and last
    ((33, 4097, 31, 2, 12345), (20011, 1, 0, 20000, 0)),
    ((1, 1, 1, 1), (20000, 1, 20001, 10001)),
])
def test_events_of_a_large_batch_match_the_oracle(sizes, idle, shuffled):
    d = batch(sizes, idle, sum(sizes), shuffled)
    want, vidx = postfit.find_vertices(*(d[k] for k in KEYS), len(sizes), CUTS)
    assert sum(len(w) for w in want) > 0 or max(sizes) == 1
    assert max(len(w) for w in want) <= MOST
    _compare(_gpu(d, len(sizes), max_vertices=MOST), want, vidx, len(sizes), MOST)


@pytest.mark.parametrize("big", [0, 1, 2])
def test_an_event_beyond_the_limit_beside_others_of_a_large_batch(big):
    n = [4099, 5003, 33]
    n[big] = L.PT_VTX_MAX_TRACKS + 1
    d = batch(n, (12000, 5, 9000), 3, True)
    g = _gpu(d, 3, max_vertices=MOST)
    assert int(g["status"][0]) == L.PT_VTX_EVENT_TOO_LARGE
    assert int(g["n"][big]) == 0 and np.all(g["track_vertex"][d["ev"] == big] == -1)
    rest = {k: v[d["ev"] != big] for k, v in d.items()}
    want, vidx = postfit.find_vertices(*(rest[k] for k in KEYS), 3, CUTS)
    assert sum(len(w) for w in want) > 0
    g["track_vertex"] = g["track_vertex"][d["ev"] != big]
    g["status"][0] = 0
    _compare(g, want, vidx, 3, MOST)


@pytest.mark.parametrize("n", [L.PT_VTX_MAX_TRACKS - 1, L.PT_VTX_MAX_TRACKS])
def test_events_at_the_limit(n):
    d = batch((n, 17), (0, 20000), 5, False)
    want, vidx = postfit.find_vertices(*(d[k] for k in KEYS), 2, CUTS)
    g = _gpu(d, 2, max_vertices=MOST)
    if len(want[0]) <= MOST:
        _compare(g, want, vidx, 2, MOST)
    else:
        assert int(g["status"][0]) == L.PT_VTX_TOO_MANY
