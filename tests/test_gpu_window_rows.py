"""The rows of tiles that the doublet search looks through are those of the
float32 azimuth of the outer hit, with no error beyond float32 rounding: outer
hits whose window ends close to a tile's edge, 3 to 9 microradians inside
it or short of it, and inner hits one to a tile, so that the number of
candidates is the number of rows."""
import numpy as np
import pytest

from synth import cuts as CU
from synth import geometry as G

N_PHI = 1024
GRID = 2.0 ** -14
# float32 rounding moves an end of the window by less than 2.5e-6 rad: the
# azimuth by 3 ulp (7e-7, atan2f), the two sums by half an ulp each (1.2e-7,
# 2.4e-7), the scale by two roundings of up to 2 pi (7.5e-7)
SAFE = 2.5e-6


def _cuts():
    cuts = CU.make_cuts(pt_min=0.5, barrel_only=True)
    for pc in cuts["pairs"]:
        pc["tan2_dphi"], pc["k_pt"] = float(np.float32(0.09)), 2.0 ** -20        # PhiW's window, not narrowed
    return cuts


def _ends(phi):
    """Both ends of the window in rows, float64 from the float32 constants."""
    dphi = np.float64(np.float32(np.arctan(np.sqrt(np.float64(np.float32(0.09)))) + 1e-4))
    scale = np.float64(np.float32(N_PHI) * np.float32(0.159154943))
    pi = np.float64(np.float32(np.pi))
    return (phi - dphi + pi) * scale, (phi + dphi + pi) * scale


def _outer(inside: bool, lower: bool, n: int):
    """x, y of outer hits of which one end lies just inside a row (or just
    short of it) and the other nowhere near an edge."""
    rng = np.random.default_rng(7 + 2 * inside + lower)
    x, y, per_rad = [], [], N_PHI / (2 * np.pi)
    while len(x) < n:
        phi = rng.uniform(-np.pi, np.pi, 400000)
        xs, ys = np.round(6.8 * np.cos(phi) / GRID) * GRID, np.round(6.8 * np.sin(phi) / GRID) * GRID
        a, b = _ends(np.arctan2(ys, xs))
        if not lower:
            a, b = b, a
        d = (a - np.floor(a)) if inside else (np.ceil(a) - a)
        far = np.minimum(b - np.floor(b), np.ceil(b) - b)
        k = (d > SAFE * per_rad) & (d < 9e-6 * per_rad) & (far > 4e-5 * per_rad)
        x += list(xs[k])
        y += list(ys[k])
    return np.array(x[:n]), np.array(y[:n])


@pytest.mark.gpu
@pytest.mark.parametrize("inside", [True, False])
@pytest.mark.parametrize("lower", [True, False])
def test_candidates_are_the_rows_of_the_float32_window(inside, lower):
    from parity import make_pipeline, to_dev
    x, y = _outer(inside, lower, 400)
    lo, hi = _ends(np.arctan2(y, x))
    rows = np.floor(hi).astype(np.int64) - np.floor(lo).astype(np.int64) + 1
    mid = (np.arange(N_PHI) + 0.5) * 2 * np.pi / N_PHI - np.pi
    r = np.concatenate([np.full(N_PHI, 2.9), np.full(len(x), 6.8)])
    x = np.concatenate([np.round(2.9 * np.cos(mid) / GRID) * GRID, x])
    y = np.concatenate([np.round(2.9 * np.sin(mid) / GRID) * GRID, y])
    module = [int(np.nonzero(G.module_layer_table() == k)[0][0]) for k in (0, 1)]
    f = lambda v: v.astype(np.float32)
    batch = dict(x=f(x), y=f(y), z=f(0 * x), r=f(np.round(np.hypot(x, y) / GRID) * GRID),
                 module=np.repeat(np.array(module, np.int32), [N_PHI, len(x) - N_PHI]),
                 ev_off=np.array([0, len(x)], np.int32))
    pipe = make_pipeline(_cuts(), dict(n_phi_bins=N_PHI, n_t_bins=1))
    t = to_dev(batch)
    res, _ = pipe.run(*(t[k] for k in ("x", "y", "z", "r", "module", "ev_off")))
    assert res.counts.n_doublet_candidates == int(rows.sum())
