"""The connection's writing of edges by the warp: cells with more incoming
edges than a warp remembers or may keep, several of them in turn, and
capacities that end inside a warp's edges."""
import numpy as np
import pytest

from synth import cuts as CU
from synth import events as E
from synth import geometry as G

from parity import compare_sets, gpu_run, make_pipeline, oracle_run, to_dev

pytestmark = pytest.mark.gpu


def straight_bundle(m, seed: int) -> dict:
    """m[L] hits on barrel layer L, all within a pencil of straight lines so
    narrow that every hit connects to every hit."""
    rng = np.random.default_rng(seed)
    pts = []
    for L, k in enumerate(m):
        r = G.BARREL_R[L]
        phi, z = rng.uniform(-1e-3, 1e-3, k), 0.3 * r + rng.uniform(-3e-3, 3e-3, k)
        pts.append(np.stack([r * np.cos(phi), r * np.sin(phi), z], 1))
    p = np.unique(E.snap(np.concatenate(pts)), axis=0)
    layer = np.argmin(np.abs(np.hypot(p[:, 0], p[:, 1])[:, None] - np.asarray(G.BARREL_R[:len(m)])), 1)
    order = rng.permutation(len(p))
    p, layer = p[order], layer[order]
    base = np.array([np.nonzero(G.module_layer_table() == k)[0][0] for k in range(4)])
    f = lambda v: v.astype(np.float32)
    return dict(x=f(p[:, 0]), y=f(p[:, 1]), z=f(p[:, 2]), r=f(E.snap(np.hypot(p[:, 0], p[:, 1]))),
                module=base[layer].astype(np.int32), ev_off=np.array([0, len(p)], np.int32))


def loose_cuts():
    return dict(CU.make_cuts(pt_min=0.3, barrel_only=True), fishbone_eps2=float(np.float32(2.0 ** -30)))


@pytest.mark.parametrize("m", [(1, 1, 1), (31, 2, 3), (33, 3, 1), (97, 2, 2), (120, 2, 2), (127, 1, 2), (128, 1, 2),
                               (129, 2, 1), (140, 2, 2), (150, 1, 2), (170, 2, 3), (400, 1, 2), (1100, 1, 2)])
def test_cells_with_many_edges(m):
    batch = straight_bundle(m, sum(m))
    want = oracle_run(batch, loose_cuts(), stage=3)
    assert len(want["edges"]) >= 0.4 * np.prod(m)
    compare_sets(gpu_run(batch, loose_cuts()), want)


@pytest.mark.parametrize("capacity", [1, 31, 32, 33, 127, 160, 161])
def test_capacity_ends_inside_the_edges(capacity):
    import torch
    from paper_2008_13461_gb300 import _lib as L
    batch = straight_bundle((50, 2, 2), 7)
    want = oracle_run(batch, loose_cuts(), stage=3)
    n = len(want["edges"])
    assert n > 161
    pipe = make_pipeline(loose_cuts())
    t = to_dev(batch)
    args = [t[k] for k in ("x", "y", "z", "r", "module", "ev_off")]
    bufs = pipe.allocate(len(batch["x"]), 1, dict(cells=4096, edges=capacity, tuples=4096, tracks=4096))
    pipe.launch(bufs, *args)
    st, c = pipe.counts(bufs, *args)
    assert st == L.PT_ERR_CAPACITY and c.flags & L.FLAG_EDGES and c.n_edges == n
