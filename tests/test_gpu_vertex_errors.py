"""The error of a vertex is the float32 nearest to the float64 1 / sqrt(sum of
weights): two-track vertices whose error lies within 1e-14 (relative) above
the midpoint between two float32, so that any shortfall of the float64 value
by more rounds the other way."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

# float32 bits of the z0 errors of the two tracks
PAIRS = (
    (0x3d0c2486, 0x3cbef98d), (0x3d20a835, 0x3d11d31b), (0x3d03683a, 0x3d0dc263), (0x3d21e09e, 0x3ceee470),
    (0x3bb387a8, 0x3cc452f0), (0x3c23f86b, 0x3c43738b), (0x3ca61dee, 0x3d086ace), (0x3bc05628, 0x3beaacf5),
    (0x3d314577, 0x3c301dd9), (0x3be469d2, 0x3bcbd478), (0x3cecd7a2, 0x3bde7462), (0x3cf3f9ef, 0x3c7c24da),
    (0x3d02cac3, 0x3be59923), (0x3cefa242, 0x3d157687), (0x3cad778a, 0x3cf7237e), (0x3c9aabec, 0x3cb647d0),
    (0x3d1a8162, 0x3d18b2e1), (0x3c9315a7, 0x3d31412e), (0x3d369816, 0x3cc479ca), (0x3cee0538, 0x3d23b1e5),
    (0x3c1d2cff, 0x3cbe5883), (0x3c78638d, 0x3c8b84b8), (0x3d23ad29, 0x3c9e2b04), (0x3d2ce3b4, 0x3d08956b),
    (0x3d0f2596, 0x3d02aa55), (0x3cbbce99, 0x3bf30045), (0x3d203dbf, 0x3ccd4550), (0x3c029aa6, 0x3d1bc8e9),
    (0x3d05ea1b, 0x3d15522a), (0x3ba14cbb, 0x3d016c5d), (0x3d31f5a8, 0x3c6f079e), (0x3c88030e, 0x3c9d9a5a),
    (0x3c95d5cf, 0x3cf34fae), (0x3cb2c90f, 0x3cc254f0), (0x3cac17c6, 0x3c6e92b0), (0x3bbf45f5, 0x3d0d7c80),
    (0x3b9a3a60, 0x3c0be8b2), (0x3d0a845d, 0x3ce3c080), (0x3d087cab, 0x3c88075f), (0x3d29ca78, 0x3c88d178),
    (0x3d34dc9f, 0x3c75cf9f), (0x3ba3b715, 0x3ce27bb8), (0x3c8406ca, 0x3cf9d3c7), (0x3cccb7dc, 0x3d1e45fd),
    (0x3cb292ee, 0x3c58bffa), (0x3cd2f10e, 0x3cc9a21c), (0x3cec1422, 0x3c647a62), (0x3d2ee578, 0x3d3283f8),
)


def exact(a, b):
    """1 / sqrt(1 / a^2 + 1 / b^2) to 40 digits."""
    getcontext().prec = 40
    return 1 / (1 / Decimal(float(a)) ** 2 + 1 / Decimal(float(b)) ** 2).sqrt()


def nearest(v):
    f = np.float32(float(v))
    around = [np.nextafter(f, np.float32(0)), f, np.nextafter(f, np.float32(1))]
    return min(around, key=lambda c: abs(Decimal(float(c)) - v))


def errors():
    return np.array(PAIRS, np.uint32).view(np.float32)


def test_the_pairs_lie_just_above_a_midpoint():
    for a, b in errors():
        v, up = exact(a, b), nearest(exact(a, b))
        mid = (Decimal(float(up)) + Decimal(float(np.nextafter(up, np.float32(0))))) / 2
        assert Decimal("1e-15") < (v - mid) / v < Decimal("1e-14")
        # what float64 makes of it is well inside that
        f64 = 1.0 / np.sqrt(1.0 / float(a) ** 2 + 1.0 / float(b) ** 2)
        assert abs(Decimal(float(f64)) - v) < v * Decimal("6e-16") and np.float32(f64) == up


@pytest.mark.gpu
def test_vertex_errors_round_from_float64():
    import torch
    from paper_2008_13461_gb300.pipeline import find_vertices
    from test_gpu_vertices import CUTS
    e = errors()
    n = len(e)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to("cuda:0")
    ev = dev(np.repeat(np.arange(n, dtype=np.int32), 2))
    one = torch.ones(2 * n, device="cuda:0")
    four = torch.full((2 * n,), 4, dtype=torch.uint8, device="cuda:0")
    v = find_vertices(ev, 0 * one, dev(e.reshape(-1)), one, four, None, n, dict(CUTS), 4)
    assert v["n"].tolist() == [1] * n and v["status"].tolist() == [0]
    got = v["ez"][:, 0].cpu().numpy()
    want = np.array([nearest(exact(a, b)) for a, b in e], np.float32)
    assert np.array_equal(got, want), int((got != want).sum())
