"""The search's writing of n-tuplets by the warp: events in which one walk
finds more n-tuplets than a warp holds, and capacities that end inside a
warp's block of them."""
import numpy as np
import pytest
import torch

from synth import cuts as CU
from synth import events as E
from synth import geometry as G

from parity import compare_sets, gpu_run, make_pipeline, oracle_run, to_dev

pytestmark = pytest.mark.gpu


def straight_bundle(m: int, seed: int) -> dict:
    """m hits on each barrel layer, all within a pencil of straight lines so
    narrow that every hit connects to every hit: ~m^4 maximal paths."""
    rng = np.random.default_rng(seed)
    pts, layer = [], []
    for L, r in enumerate(G.BARREL_R):
        phi, z = rng.uniform(-2e-4, 2e-4, m), 0.3 * r + rng.uniform(-1e-3, 1e-3, m)
        pts.append(np.stack([r * np.cos(phi), r * np.sin(phi), z], 1))
        layer.append(np.full(m, L))
    p, layer = np.concatenate(pts), np.concatenate(layer)
    order = rng.permutation(len(p))
    p, layer = E.snap(p[order]), layer[order]
    base = np.array([np.nonzero(G.module_layer_table() == k)[0][0] for k in range(4)])
    f = lambda v: v.astype(np.float32)
    return dict(x=f(p[:, 0]), y=f(p[:, 1]), z=f(p[:, 2]), r=f(E.snap(np.hypot(p[:, 0], p[:, 1]))),
                module=base[layer].astype(np.int32), ev_off=np.array([0, len(p)], np.int32))


def loose_cuts():
    return dict(CU.make_cuts(pt_min=0.3, barrel_only=True), fishbone_eps2=float(np.float32(2.0 ** -30)))


@pytest.mark.parametrize("m", [1, 2, 3, 5, 9])
def test_more_paths_than_a_warp_holds(m):
    batch = straight_bundle(m, m)
    want = oracle_run(batch, loose_cuts(), stage=3)
    assert len(want["tuple_n"]) >= m ** 3
    compare_sets(gpu_run(batch, loose_cuts()), want)


@pytest.mark.parametrize("capacity", [1, 31, 32, 33, 63, 64, 100])
def test_capacity_ends_inside_a_block(capacity):
    from paper_2008_13461_gb300 import _lib as L
    batch = straight_bundle(4, 4)
    want = oracle_run(batch, loose_cuts(), stage=3)
    n = len(want["tuple_n"])
    assert n > 100
    pipe = make_pipeline(loose_cuts())
    t = to_dev(batch)
    args = [t[k] for k in ("x", "y", "z", "r", "module", "ev_off")]
    bufs = pipe.allocate(16, 1, dict(cells=4096, edges=4096, tuples=capacity, tracks=4096))
    guard = torch.full((capacity + 64,), 77, dtype=torch.uint8, device="cuda:0")
    bufs.tup_alive = guard[:capacity]
    pipe.launch(bufs, *args)
    st, c = pipe.counts(bufs, *args)
    assert st == L.PT_ERR_CAPACITY and c.flags & L.FLAG_TUPLES and c.n_tuples == n
    assert bool((guard[capacity:] == 77).all())
