"""Decisions within rounding of the doublet cuts, and hits whose r is not the
hypotenuse of x and y.  The contract ties r to its layer's envelope only, and
every predicate reads r or (x, y), so the cells are exact whatever the two
say of each other: pairs next to the azimuth and curvature cuts where x and y
are far larger than r, next to the intercept cut over whole envelopes, and
pairs beyond the azimuth window that r alone would suggest."""
import numpy as np
import pytest

from synth import cuts as CU
from synth import geometry as G

from parity import gpu_run, gpu_sets, oracle_run, oracle_sets

LAYERS = {ly.index: ly for ly in G.layers()}
MODULE = {k: int(np.nonzero(G.module_layer_table() == k)[0][0]) for k in range(G.N_LAYERS)}
GRID = 2.0 ** -14


def _batch(pairs):
    """One event per pair ((x, y, z, r, layer) inner, the same outer)."""
    h = np.array([row for p in pairs for row in p], np.float64)
    f = lambda v: np.ascontiguousarray(v, np.float32)
    assert np.array_equal(f(h[:, :4]).astype(np.float64), h[:, :4]) and np.all(np.abs(h[:, :4]) < 64)
    return dict(x=f(h[:, 0]), y=f(h[:, 1]), z=f(h[:, 2]), r=f(h[:, 3]),
                module=np.array([MODULE[int(k)] for k in h[:, 4]], np.int32),
                ev_off=np.arange(0, len(h) + 1, 2).astype(np.int32))


def _cuts(tan2_dphi=None, k_pt=None):
    cuts = CU.make_cuts(pt_min=0.5, barrel_only=True)
    for pc in cuts["pairs"]:
        if tan2_dphi is not None:
            pc["tan2_dphi"] = float(np.float32(tan2_dphi))
        if k_pt is not None:
            pc["k_pt"] = float(np.float32(k_pt))
    return cuts


def _compare(pairs, cuts):
    batch = _batch(pairs)
    got, want = gpu_sets(gpu_run(batch, cuts))[0], oracle_sets(oracle_run(batch, cuts, stage=1))[0]
    assert set(got) == set(want), (len(set(got) - set(want)), len(set(want) - set(got)))
    return len(want)


def _snap(v):
    return np.round(np.asarray(v) / GRID) * GRID


def _near_the_cut(cut: str, far, seed: int, n: int):
    """Pairs within 2e-7 of the cut (relative to its terms), half on either side
    on average, with |(x, y)| = far (inner, outer) and r in the layers' envelopes."""
    rng = np.random.default_rng(seed)
    tan2, k_pt = (0.09, 2.0 ** -20) if cut == "phi" else (16.0, 2500.0)
    out = []
    while len(out) < n:
        m = 200000
        phi = rng.uniform(-np.pi, np.pi, m)
        if cut == "phi":
            dphi = np.full(m, np.arctan(np.sqrt(tan2)))
        else:                                   # chords of a circle of diameter sqrt(k_pt) through the beam line
            dphi = np.arcsin(far[1] / np.sqrt(k_pt)) - np.arcsin(far[0] / np.sqrt(k_pt))
        xi, yi = _snap(far[0] * np.cos(phi)), _snap(far[0] * np.sin(phi))
        xo, yo = _snap(far[1] * np.cos(phi + dphi)), _snap(far[1] * np.sin(phi + dphi))
        c2, d = (xi * yo - yi * xo) ** 2, xi * xo + yi * yo
        if cut == "phi":
            a, b = tan2 * d * d, c2
        else:
            a, b = ((xo - xi) ** 2 + (yo - yi) ** 2) * (xi * xi + yi * yi) * (xo * xo + yo * yo), k_pt * c2
        for k in np.nonzero(np.abs(a - b) <= 2e-7 * (a + b))[0]:
            out.append(((xi[k], yi[k], 0.0, 3.0, 0), (xo[k], yo[k], 0.0, 7.0, 1)))
    return out[:n], _cuts(tan2, k_pt)


@pytest.mark.gpu
@pytest.mark.parametrize("cut", ["phi", "pt"])
@pytest.mark.parametrize("far", [(3.0, 7.0), (20.0, 30.0), (40.0, 45.0)])
def test_pairs_within_rounding_of_a_cut(cut, far):
    pairs, cuts = _near_the_cut(cut, far, 3, 4000)
    kept = _compare(pairs, cuts)
    assert 0.1 * len(pairs) < kept < 0.9 * len(pairs)


def _near_the_intercept(inner: int, outer: int, seed: int, n: int):
    """Pairs on one azimuth within 2e-7 of the ZIP cut (relative to its
    terms), over the whole of both layers' envelopes."""
    rng = np.random.default_rng(seed)
    li, lo, zmax = LAYERS[inner], LAYERS[outer], 12.0
    out = []
    while len(out) < n:
        m = 200000
        ri, zi, zo = (_snap(rng.uniform(a + 0.01, b - 0.01, m))
                      for a, b in ((li.rmin, li.rmax), (li.zmin, li.zmax), (lo.zmin, lo.zmax)))
        side = rng.choice([-zmax, zmax], m)
        ro = _snap(ri * (zo - side) / np.where(zi == side, np.nan, zi - side))
        left, right = np.abs(zi * ro - zo * ri), zmax * (ro - ri)
        near = (ro > lo.rmin) & (ro < lo.rmax) & (ro > ri) & (np.abs(left - right) <= 2e-7 * (left + right))
        phi = rng.uniform(-np.pi, np.pi, m)
        for k in np.nonzero(near)[0]:
            xy = [(float(_snap(r * np.cos(phi[k]))), float(_snap(r * np.sin(phi[k])))) for r in (ri[k], ro[k])]
            out.append(((*xy[0], zi[k], ri[k], inner), (*xy[1], zo[k], ro[k], outer)))
    cuts = CU.make_cuts(pt_min=0.5)
    for pc in cuts["pairs"]:
        pc["zmax"], pc["zlo"], pc["zhi"] = zmax, -60.0, 60.0
    return out[:n], cuts


@pytest.mark.gpu
@pytest.mark.parametrize("inner,outer", [(0, 1), (2, 3), (0, 4), (1, 7), (4, 6), (8, 9)])
def test_pairs_within_rounding_of_the_intercept(inner, outer):
    pairs, cuts = _near_the_intercept(inner, outer, 8, 2000)
    kept = _compare(pairs, cuts)
    assert 0.1 * len(pairs) < kept < 0.9 * len(pairs)


@pytest.mark.gpu
@pytest.mark.parametrize("consistent", [True, False])
def test_pairs_beyond_the_window_that_r_suggests(consistent):
    """Azimuth differences up to the PhiW cut; with r = 3 and 7 cm the
    narrowed window ends far below what chords of 30 and 45 cm bend."""
    rng = np.random.default_rng(9)
    pairs = []
    for _ in range(600):
        far = (3.0, 7.0) if consistent else (rng.uniform(3, 40), rng.uniform(7, 60))
        phi, d = rng.uniform(-np.pi, np.pi), rng.uniform(-0.5, 0.5)
        pairs.append(((_snap(far[0] * np.cos(phi)), _snap(far[0] * np.sin(phi)), 0.0, 3.0, 0),
                      (_snap(far[1] * np.cos(phi + d)), _snap(far[1] * np.sin(phi + d)), 0.0, 7.0, 1)))
    assert _compare(pairs, _cuts(tan2_dphi=0.5)) > 20


@pytest.mark.gpu
@pytest.mark.parametrize("others", [1, 500])
def test_such_hits_beside_ordinary_ones(others):
    """Pairs off their radius among events of ordinary ones."""
    pairs, cuts = _near_the_cut("pt", (40.0, 45.0), 5, 300)
    plain, _ = _near_the_cut("pt", (3.0, 7.0), 6, others)
    _compare(plain + pairs + plain, cuts)


def test_the_pairs_do_what_the_tests_say():
    """CPU: the near pairs are contested in float32 and decided by the oracle
    on either side of the cut."""
    for cut in ("phi", "pt"):
        pairs, cuts = _near_the_cut(cut, (40.0, 45.0), 3, 500)
        kept = len(oracle_run(_batch(pairs), cuts, stage=1)["cells"])
        assert 0.1 * len(pairs) < kept < 0.9 * len(pairs)
