"""The doublets' shared-memory buffers: outer hits whose cells fill the buffer
that two of them share, to the last entry and beyond it, for every number of
lanes per outer hit, compared with the oracle cell by cell."""
import numpy as np
import pytest

from synth import cuts as CU

from parity import compare_sets, gpu_run, oracle_run
from test_gpu_long_lists import crowded_event


def batch_of(sizes, least: int) -> dict:
    """Crowded events of the given sizes, over and over until they have least hits."""
    events, total = [], 0
    while total < least or len(events) < len(sizes):
        e = crowded_event(sizes[len(events) % len(sizes)], len(events))
        events.append(e)
        total += len(e["x"])
    off = np.concatenate([[0], np.cumsum([len(e["x"]) for e in events])]).astype(np.int32)
    return dict({k: np.concatenate([e[k] for e in events]) for k in ("x", "y", "z", "r", "module")}, ev_off=off)


@pytest.mark.gpu
@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
def test_buffers_full_and_beyond(lanes):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # with fewer hits than this the kernel would take more lanes
    least = 4 * 256 * sms // lanes if lanes < 32 else 0
    full = 40 * lanes
    sizes = [full - 1, full, full + 1, 10, full + full // 2, 1, 2 * full - 1, 2 * full, 2 * full + 1]
    batch, cuts = batch_of(sizes, least + 1), CU.make_cuts(pt_min=0.3)
    res = gpu_run(batch, cuts, tuning=dict(doublet_lanes=lanes, blocks_per_sm=1))
    compare_sets(res, oracle_run(batch, cuts, stage=3))
