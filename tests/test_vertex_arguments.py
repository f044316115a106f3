"""Sizes that the vertex finder refuses, it refuses with the library's status
(host logic: the library looks at them before any CUDA call)."""
import types

import pytest
import torch

from paper_2008_13461_gb300 import _lib as L
from paper_2008_13461_gb300.pipeline import find_vertices


@pytest.mark.parametrize("tracks", [0, 8])
@pytest.mark.parametrize("n_events,max_vertices", [(-1, 256), (-5, 3), (1, 0), (2, -1), (-1, -1)])
def test_refused_sizes_raise_the_status(monkeypatch, tracks, n_events, max_vertices):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=0))
    i, f, u = (torch.zeros(tracks, dtype=d) for d in (torch.int32, torch.float32, torch.uint8))
    with pytest.raises(L.PtError) as e:
        find_vertices(i, f, f, f, u, None, n_events, max_vertices=max_vertices)
    assert e.value.status == L.PT_ERR_INVALID_ARG
