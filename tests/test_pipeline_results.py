"""What Pipeline.result makes of the buffers (host logic, no GPU)."""
import torch

from paper_2008_13461_gb300 import _lib as L
from paper_2008_13461_gb300.pipeline import Pipeline
from synth import cuts as CU
from synth import geometry as G


def _pipe():
    return Pipeline(G.layers(), G.module_layer_table(), CU.cuts_for("pu50-ttbar-like"), CU.FIT_PARAMS, device="cpu")


def _counts(n):
    c = L.Counts()
    c.n_cells = c.n_edges = c.n_tuples = c.n_tracks = n
    return c


def test_counts_beyond_the_capacities_give_what_the_buffers_hold():
    """After an overflow the counters say what was found; the result holds
    the rows there are, and nothing beyond a buffer that is part of a larger
    tensor."""
    pipe, cap = _pipe(), 10
    hits = [torch.zeros(16) for _ in range(4)] + [torch.zeros(16, dtype=torch.int32),
                                                  torch.tensor([0, 16], dtype=torch.int32)]
    bufs = pipe.allocate(16, 1, dict.fromkeys(("cells", "edges", "tuples", "tracks"), cap))
    big = dict(tup_hits=L.NMAX, tup_cells=L.NMAX, trk_params=5, trk_cov=15)
    for name, w in big.items():
        whole = torch.zeros((cap + 20) * w, dtype=getattr(bufs, name).dtype)
        whole[cap * w:] = 77
        setattr(bufs, name, whole[:cap * w])
    for n in (0, 1, cap, cap + 1, cap + 15, 10 ** 6):
        r = pipe.result(bufs, _counts(n), *hits)
        tables = (r.tuples["hits"], r.tuples["cells"], r.tracks["params"], r.tracks["cov"])
        assert [t.shape for t in tables] == [(min(n, cap), w) for w in big.values()]
        assert not any(bool((t == 77).any()) for t in tables)
        for t in (*r.cells.values(), *r.edges.values(), r.tuples["n"], r.tracks["chi2"], r.tracks["tuple"]):
            assert t.shape[0] == min(n, cap)
