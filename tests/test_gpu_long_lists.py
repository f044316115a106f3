"""Outer hits with many cells: the Fishbone and the connection at the list
lengths where the work passes from one kernel or loop to the next, compared
with the oracle cell by cell and edge by edge."""
import numpy as np
import pytest

from synth import cuts as CU
from synth import events as E
from synth import geometry as G

from parity import compare_sets, gpu_run, oracle_run


def crowded_event(n: int, seed: int) -> dict:
    """n hits on the first barrel layer, all within the window of 3 hits on
    the second; half of them come as a pair on the line to the first of
    those, so that the Fishbone has aligned cells; 2 hits on the third."""
    rng = np.random.default_rng(seed)
    outer = np.array([(6.65, 0.0, 0.5), (6.95 * np.cos(0.01), 6.95 * np.sin(0.01), -0.3),
                      (6.65 * np.cos(-0.012), 6.65 * np.sin(-0.012), 0.1)])
    third = np.array([(10.75 * np.cos(0.004), 10.75 * np.sin(0.004), 1.0), (11.05, 0.02, -0.6)])
    m = n // 2
    phi, z = rng.uniform(-0.03, 0.03, n - m), rng.uniform(-6.0, 6.0, n - m)
    first = np.stack([2.75 * np.cos(phi), 2.75 * np.sin(phi), z], 1)
    t = np.full((m, 1), 0.3 / (6.65 - 2.75))
    pairs = first[:m] + t * (outer[0] - first[:m])
    p = np.concatenate([first, pairs, outer, third])
    layer = np.concatenate([np.zeros(n, int), np.ones(3, int), np.full(2, 2)])
    order = rng.permutation(len(p))
    p, layer = E.snap(p[order]), layer[order]
    base = np.array([np.nonzero(G.module_layer_table() == k)[0][0] for k in range(3)])
    f = lambda v: v.astype(np.float32)
    return dict(x=f(p[:, 0]), y=f(p[:, 1]), z=f(p[:, 2]), r=f(E.snap(np.hypot(p[:, 0], p[:, 1]))),
                module=base[layer].astype(np.int32), ev_off=np.array([0, len(p)], np.int32))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 12, 13, 31, 33, 63, 65, 128, 129, 192, 193, 224, 225, 256, 257, 288, 289, 320, 321, 512, 513, 1024, 1025])
def test_lists_of_any_length(n):
    batch, cuts = crowded_event(n, n), CU.make_cuts(pt_min=0.3)
    want = oracle_run(batch, cuts, stage=3)
    cells = np.asarray(want["cells"])
    assert np.bincount(cells[cells[:, 2] == 0, 1]).max() == n
    res = gpu_run(batch, cuts)
    compare_sets(res, want)
