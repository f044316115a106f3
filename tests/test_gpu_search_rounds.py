"""The n-tuplets that a warp of the search holds, over several rounds: each
lane has to see the same number of them before the warp meets to write them,
whatever the lanes that are ahead have found since."""
import os
import re

import numpy as np
import pytest

from parity import make_pipeline, oracle_run, to_dev
from test_gpu_many_tuplets import loose_cuts, straight_bundle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_number_held_is_read_between_two_meetings_of_the_warp():
    """Its only readers are the atomic additions and dfs_held, which no lane
    leaves before all have read (CPU: the source)."""
    src = open(os.path.join(ROOT, "paper_2008_13461_gb300", "csrc", "pt_ntuplets.cu")).read()
    code = re.sub(r"//[^\n]*", "", src)
    uses = [u for u in re.findall(r"[^;{}]*hold\.count\[[^;]*;", code)]
    reads = [u for u in uses if "atomicAdd(&hold.count" not in u and not re.search(r"hold\.count\[\w+\] = 0;", u)]
    assert len(reads) == 1
    assert re.search(r"__syncwarp\(\);\s*const int n = hold\.count\[threadIdx\.x >> 5\];\s*__syncwarp\(\);\s*return n;",
                     code)


@pytest.mark.gpu
@pytest.mark.parametrize("m,rounds", [(1, 4), (1, 5), (2, 3), (3, 3), (5, 3)])
def test_rounds_that_end_around_what_a_warp_writes(m, rounds):
    """Copies of a small bundle as events, enough for every warp to take
    several rounds of 32 edges: a round finds about 24 n-tuplets for m = 1
    (a warp writes from 32 on, so in every other one), 51 for m = 2, 40 for
    m = 3 and 54 for m = 5, where it holds 64."""
    import torch
    one = straight_bundle(m, m)
    want = oracle_run(one, loose_cuts(), stage=3)
    edges, paths = len(want["edges"]), len(want["tuple_n"])
    assert paths >= m ** 3
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = rounds * sms * 256 // edges + 1
    k = len(one["x"])
    off = np.arange(n, dtype=np.int64) * k
    batch = {q: np.tile(one[q], n) for q in ("x", "y", "z", "r", "module")}
    batch["ev_off"] = np.append(off, n * k).astype(np.int32)
    pipe = make_pipeline(loose_cuts(), dict(n_phi_bins=16, n_t_bins=1, blocks_per_sm=1))
    t = to_dev(batch)
    bufs = pipe.allocate(n * k, n, dict(cells=n * len(want["cells"]) + 64, edges=n * edges + 64, tuples=n * paths + 64,
                                        tracks=n * paths + 64))
    res, _ = pipe.run(*(t[q] for q in ("x", "y", "z", "r", "module", "ev_off")), bufs=bufs)
    assert res.counts.n_edges == n * edges and res.counts.n_tuples == n * paths
    got = res.tuples["hits"].cpu().numpy().astype(np.int64)
    length = res.tuples["n"].cpu().numpy()
    used = np.arange(got.shape[1]) < length[:, None]
    got = np.where(used, got, -1)
    ref = np.asarray(want["tuple_hits"], np.int64)
    ref = np.where(np.arange(ref.shape[1]) < np.asarray(want["tuple_n"])[:, None], ref, -1)
    ref = np.where(ref[None] >= 0, ref[None] + off[:, None, None], -1).reshape(n * paths, -1)
    rows = lambda a: a[np.lexsort(a.T[::-1])]
    assert np.array_equal(rows(got), rows(ref))
