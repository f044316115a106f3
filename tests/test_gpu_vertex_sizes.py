"""The vertex finder at the sizes where its work changes hands: crowded z0
tiles, candidates beyond the members held in registers, tracks beyond the
tiles' range, and events large enough for windows in kernels of their own;
against the oracle, as in test_gpu_vertices."""
import numpy as np
import pytest

from oracle import postfit

from test_gpu_vertices import CUTS, _compare, _gpu

pytestmark = pytest.mark.gpu


def tracks(z0, ez0, seed):
    rng = np.random.default_rng(seed)
    n = len(z0)
    order = rng.permutation(n)
    return dict(ev=np.zeros(n, np.int32), z0=np.asarray(z0, np.float32)[order],
                ez0=np.full(n, ez0, np.float32) * rng.uniform(0.5, 2.0, n).astype(np.float32),
                pt=rng.uniform(0.6, 5.0, n).astype(np.float32), nhits=np.full(n, 4, np.uint8), keep=np.ones(n, np.uint8))


def check(d):
    want, vidx = postfit.find_vertices(*(d[k] for k in ("ev", "z0", "ez0", "pt", "nhits", "keep")), 1, CUTS)
    assert len(want[0]) > 0
    _compare(_gpu(d, 1), want, vidx, 1)


@pytest.mark.parametrize("m", [31, 32, 33, 255, 256, 257, 300])
@pytest.mark.parametrize("spread", [0.0, 0.004, 0.05])
def test_crowded_tiles_and_large_candidates(m, spread):
    """m tracks in one z0 tile (ties, or all distinct), and some far away."""
    rng = np.random.default_rng(m)
    z = np.concatenate([0.005 + spread * rng.random(m), rng.uniform(-6.0, 6.0, 90), [30.0, 30.001, -41.0, -41.002, 1e6]])
    check(tracks(z, 0.004, m))


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 9999, 10000, 10011])
def test_event_sizes(n):
    rng = np.random.default_rng(n)
    z = rng.uniform(-20.0, 20.0, max(1, n // 20))[rng.integers(0, max(1, n // 20), n)] + 0.003 * rng.standard_normal(n)
    d = tracks(z, 0.003, n)
    if n == 1:
        assert int(_gpu(d, 1)["n"][0]) == 0
    else:
        want, vidx = postfit.find_vertices(*(d[k] for k in ("ev", "z0", "ez0", "pt", "nhits", "keep")), 1, CUTS)
        most = 512
        assert n < 100 or 0 < len(want[0]) <= most
        _compare(_gpu(d, 1, max_vertices=most), want, vidx, 1)
