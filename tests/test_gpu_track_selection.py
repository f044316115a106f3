"""The fit's track list: every live n-tuplet of at least min_hits hits,
grouped by hit count and in n-tuplet order within a count, whatever the
number of n-tuplets per slice of the selection."""
import numpy as np
import pytest
import torch

from synth import cuts as CU
from synth import events as E
from synth import geometry as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["barrel-50-helices", "pu50-ttbar-like"])
def finished(request):
    from paper_2008_13461_gb300.pipeline import Pipeline
    batch = E.make_batch(request.param)
    dev = torch.device("cuda:0")
    hits = [torch.as_tensor(batch[k]).to(dev) for k in ("x", "y", "z", "r", "module", "ev_off")]
    pipe = Pipeline(G.layers(), G.module_layer_table(), CU.cuts_for(request.param), CU.FIT_PARAMS, device=dev)
    res, bufs = pipe.run(*hits)
    return pipe, bufs, hits, res.counts.n_tuples, bufs.tup_alive.clone()


@pytest.mark.parametrize("live", [0.0, 0.03, 0.6, 1.0])
def test_selected_tracks(finished, live):
    from paper_2008_13461_gb300.autograd import DifferentiableFit
    pipe, bufs, hits, nt, alive0 = finished
    rng = np.random.default_rng(5)
    alive = (rng.random(nt) < live).astype(np.uint8)
    bufs.tup_alive[:nt] = torch.as_tensor(alive).to(bufs.tup_alive.device)
    try:
        fit = DifferentiableFit(pipe, bufs, *hits[3:])
        params, chi2 = fit.fit(*hits[:3])
        got = fit.tuple[:params.shape[0]].cpu().numpy()
    finally:
        bufs.tup_alive.copy_(alive0)
    n = bufs.tup_n[:nt].cpu().numpy().astype(int)
    sel = np.nonzero(alive)[0]
    want = sel[np.argsort(np.minimum(n[sel], 6), kind="stable")]
    assert np.array_equal(got, want)
    assert bool(torch.isfinite(params).all()) and bool(torch.isfinite(chi2).all())
