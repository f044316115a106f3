"""tuning.blocks_per_sm limits what every persistent kernel puts on the
device: no more threads per SM than that many blocks of 256 (the adjoint: of
128), and as many as it did where the kernel's blocks are smaller.  The grids
are read from a captured graph; nothing of it runs."""
import ctypes as C

import numpy as np
import pytest
import torch

from synth import cuts as CU
from synth import events as E

from parity import make_pipeline, to_dev

pytestmark = pytest.mark.gpu

# kernels whose grid follows the problem's size or is fixed
SIZED = ("k_scan_small", "k_scan_reduce", "k_scan_partials", "k_scan_apply", "k_count_tracks", "k_select_tracks")


class NodeParams(C.Structure):
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def captured(stream, enqueue):
    """{kernel name: (blocks, threads per block)} of what enqueue() puts on the stream."""
    cu = C.CDLL("libcuda.so.1")

    def call(name, *args):
        assert getattr(cu, name)(*args) == 0, name

    s, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t()
    call("cuStreamBeginCapture_v2", s, 1)
    try:
        enqueue()
    finally:
        call("cuStreamEndCapture", s, C.byref(graph))
    call("cuGraphGetNodes", graph, None, C.byref(n))
    nodes = (C.c_void_p * n.value)()
    call("cuGraphGetNodes", graph, nodes, C.byref(n))
    out = {}
    for node in nodes:
        kind = C.c_int()
        call("cuGraphNodeGetType", C.c_void_p(node), C.byref(kind))
        if kind.value != 0:
            continue
        q, name = NodeParams(), C.c_char_p()
        call("cuGraphKernelNodeGetParams_v2", C.c_void_p(node), C.byref(q))
        if q.func:
            call("cuFuncGetName", C.byref(name), C.c_void_p(q.func))
        else:
            call("cuKernelGetName", C.byref(name), C.c_void_p(q.kern))
        out[name.value.decode()] = (q.grid[0] * q.grid[1] * q.grid[2], q.block[0] * q.block[1] * q.block[2])
    call("cuGraphDestroy", graph)
    return out


def grids(factor):
    b = E.make_batch("barrel-50-helices", n_events=1)
    pipe = make_pipeline(CU.cuts_for("barrel-50-helices"), dict(blocks_per_sm=factor))
    t = to_dev(b)
    args = [t[k] for k in ("x", "y", "z", "r", "module", "ev_off")]
    from paper_2008_13461_gb300 import _lib as L
    bufs = pipe.allocate(args[0].numel(), 1)
    g = torch.zeros(len(b["x"]), device="cuda:0")
    gp = torch.zeros(bufs.trk_params.numel(), device="cuda:0")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def enqueue():
        pipe.launch(bufs, *args, stream=stream)
        _, _, tuples, tracks = bufs.structs()
        L.fit_tracks_grad(bufs.ws.data_ptr(), bufs.ws.numel(), pipe._hits(*args), pipe._cfg(bufs.capacity), tuples,
                          tracks, gp.data_ptr(), None, g.data_ptr(), g.data_ptr(), g.data_ptr(), stream.cuda_stream)

    return captured(stream, enqueue)


def test_no_kernel_puts_more_on_an_sm_than_the_factor_allows():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    full = grids(32)
    names = {k for k in full if not any(q in k for q in SIZED)}
    assert len(names) == 4 + 4 + 14                       # fits, adjoints, the others
    for factor in (1, 2, 3, 5, 8, 14):
        got = grids(factor)
        for k in names:
            blocks, threads = got[k]
            unit = 128 if "k_fit_grad" in k else 256
            assert blocks * threads <= sms * factor * unit, (k, factor, blocks, threads)
            assert blocks <= full[k][0] and threads == full[k][1]
            # a kernel that the limit does not reach is not held back by counting small blocks
            if "k_connect" in k and "exact" not in k:
                assert blocks == min(2 * factor, 12) * sms
            if "k_fit<" in k or "k_fitILi" in k:
                assert blocks == min(4 * factor * sms, full[k][0])


def test_the_default_and_the_largest_factor_launch_the_same():
    assert grids(24) == grids(32)


def test_the_tuner_tries_no_two_factors_that_launch_the_same():
    from paper_2008_13461_gb300.autotune import SPACE
    tried = [grids(f) for f in dict(SPACE)["blocks_per_sm"]]
    assert all(tried[i] != tried[j] for i in range(len(tried)) for j in range(i))


def test_results_do_not_depend_on_the_factor():
    from parity import compare_sets, compare_tracks, gpu_run, oracle_run
    b = E.make_batch("barrel-50-helices", n_events=1)
    cuts = CU.cuts_for("barrel-50-helices")
    want = oracle_run(b, cuts)
    for factor in (1, 3, 32):
        res = gpu_run(b, cuts, dict(blocks_per_sm=factor))
        compare_sets(res, want)
        compare_tracks(res, want)
    assert np.all(res.tracks["chi2"].cpu().numpy() >= 0)
