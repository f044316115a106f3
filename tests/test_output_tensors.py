"""The tensors that the host path returns are each the caller's own (host
logic, no GPU; the library's calls are stand-ins): one can be changed in
place, also by a factor that is being learned, and another saved by autograd
meanwhile, although several share an allocation."""
import types

import pytest
import torch

from paper_2008_13461_gb300 import _lib as L
from paper_2008_13461_gb300 import pipeline as P
from paper_2008_13461_gb300.autograd import DifferentiableFit
from synth import cuts as CU
from synth import geometry as G

N_HITS, N_TRACKS, N_MODULES = 7, 5, 3


@pytest.fixture
def pipe(monkeypatch):
    for name in ("fit_tracks", "fit_tracks_grad", "align_hits", "align_hits_grad", "track_summary", "find_vertices"):
        monkeypatch.setattr(L, name, lambda *a: None)
    c = L.Counts()
    c.n_tracks = N_TRACKS
    monkeypatch.setattr(L, "read_counts", lambda *a: (L.PT_OK, c))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=0))
    return P.Pipeline(G.layers(), G.module_layer_table(), CU.cuts_for("pu50-ttbar-like"), CU.FIT_PARAMS, device="cpu")


def _refit(pipe):
    bufs = pipe.allocate(N_HITS, 1, dict.fromkeys(("cells", "edges", "tuples", "tracks"), 16))
    module = torch.zeros(N_HITS, dtype=torch.int32)
    return DifferentiableFit(pipe, bufs, torch.zeros(N_HITS), module, torch.tensor([0, N_HITS], dtype=torch.int32),
                             torch.zeros(N_MODULES, 3))


def _leaves(*shapes):
    return [torch.zeros(s, requires_grad=True) for s in shapes]


def _outputs(pipe, what):
    if what == "gradients of the refit":
        x, y, z = _leaves(*(N_HITS,) * 3)
        params, chi2 = _refit(pipe).fit(x, y, z)
        return torch.autograd.grad(params.sum() + chi2.sum(), (x, y, z))
    if what == "gradients of the alignment":
        x, y, z, shift, rot = _leaves(*(N_HITS,) * 3, (N_MODULES, 3), (N_MODULES, 3))
        moved = _refit(pipe).align(x, y, z, shift, rot)
        return torch.autograd.grad(sum(m.sum() for m in moved), (x, y, z, shift, rot))
    if what == "track summary":
        fit = _refit(pipe)
        c = L.Counts()
        c.n_tracks = N_TRACKS
        x = torch.zeros(N_HITS)
        return list(pipe.track_summary(fit.bufs, c, x, x, x, x, fit.module, fit.ev_off).values())
    i, f, u = (torch.zeros(N_TRACKS, dtype=d) for d in (torch.int32, torch.float32, torch.uint8))
    v = P.find_vertices(i, f, f, f, u, None, 2, max_vertices=4)
    return [t for n, t in v.items() if n != "scratch"]


@pytest.mark.parametrize("what", ["gradients of the refit", "gradients of the alignment", "track summary", "vertices"])
def test_each_output_stands_alone(pipe, what):
    out = _outputs(pipe, what)
    spans = sorted((t.data_ptr(), t.numel() * t.element_size()) for t in out)
    assert all(a + n <= b for (a, n), (b, _) in zip(spans, spans[1:]))          # no element in two of them
    versions = [t._version for t in out]
    out[0].add_(1)
    assert [t._version - v for t, v in zip(out, versions)] == [1] + [0] * (len(out) - 1)
    floats = [t for t in out if t.is_floating_point()]
    assert len(floats) >= 3
    for k in range(len(floats)):                          # in place, with a gradient
        floats = [t for t in _outputs(pipe, what) if t.is_floating_point()]
        scale = torch.ones((), requires_grad=True)
        floats[k].mul_(scale)
        assert [t.requires_grad for t in floats] == [j == k for j in range(len(floats))]
        saved = (floats[k - 1].zero_() * scale).sum()
        floats[k].sum().backward()
        saved.backward()
