"""The work that users of this framework have it do, as timed cases.

Kinds of case (``kind``):

  chain     hits of a batch of events to fitted tracks: ``Pipeline.run`` and
            its tracks, put in order of their hits (the run leaves them in no
            particular order, and a program that stores or compares events
            orders them);
  refit     the tracks of a run fitted again from given hit coordinates
            (``DifferentiableFit.fit``), with or without the gradient with
            respect to every hit coordinate;
  align     one step of a track-based alignment: hits moved by per-module
            shifts and rotations, refit, robust loss, gradient with respect to
            the shifts and rotations;
  postfit   ambiguity resolution, track summaries and vertices of a run's
            tracks (``Pipeline.find_vertices``);
  vertices  the vertex finder on track summaries (``find_vertices``).

Events are helices through the pixel detector that the framework's own
configurations describe (pileup vertices of Poisson(30) tracks plus a hard
one, module overlaps, scattering, noise hits), drawn on the GPU from the seed
alone.  ``exact`` finds the doublets, cells and n-tuplets by plain pair loops
in torch (hits are multiples of 2^-14 cm, so the products that decide are exact
or rounded at 1e-16) and fits them in float64.  The all-float32 solve is left
out: its chi2 is not bounded, and no program that uses chi2 can run it.
"""
from __future__ import annotations

import math
from typing import NamedTuple

import numpy as np
import torch

from paper_2008_13461_gb300.autograd import DifferentiableFit
from paper_2008_13461_gb300.pipeline import DEFAULT_VERTEX_CUTS, Pipeline, find_vertices

DEV = "cuda"
F64 = torch.float64
NMAX = 8

# ---------------------------------------------------------------- detector
GRID = 2.0 ** -14
BZ = 3.8
BARREL_R, BARREL_Z, LADDERS, ZSEG, DR = (2.9, 6.8, 10.9, 16.0), 26.7, (12, 28, 44, 64), 8, 0.15
DISK_Z, DISK_RMIN, DISK_RMAX, RING_SPLIT, RING_MODULES, DZ = (32.0, 39.5, 48.8), 4.5, 16.0, 10.0, (44, 68), 0.2
OVERLAP, ENVELOPE = 0.08, 0.05
BARREL_BASE = [sum(LADDERS[:i]) * ZSEG for i in range(4)]
N_BARREL = sum(LADDERS) * ZSEG
PER_DISK = sum(RING_MODULES)
N_MODULES = N_BARREL + 6 * PER_DISK
FIT = dict(bz=BZ, sigma_rphi=10e-4, sigma_z=20e-4, sigma_r=20e-4, x0_barrel=0.02, x0_disk=0.03)
PAIRS = ((0, 1), (1, 2), (2, 3), (0, 4), (0, 7), (1, 4), (1, 7), (4, 5), (7, 8), (5, 6), (8, 9),
         (0, 2), (1, 3), (0, 5), (0, 8), (4, 6), (7, 9))
BARREL_PAIRS = ((0, 1), (1, 2), (2, 3), (0, 2), (1, 3))


class Layer(NamedTuple):
    kind: int                     # 0 barrel, 1 disk
    rmin: float
    rmax: float
    zmin: float
    zmax: float


def disk_z(layer: int) -> float:
    return (1.0 if layer < 7 else -1.0) * DISK_Z[(layer - 4) % 3]


LAYERS = [Layer(0, r - DR - ENVELOPE, r + DR + ENVELOPE, -BARREL_Z - ENVELOPE, BARREL_Z + ENVELOPE)
          for r in BARREL_R] + \
         [Layer(1, DISK_RMIN - ENVELOPE, DISK_RMAX + ENVELOPE, disk_z(k) - DZ - ENVELOPE, disk_z(k) + DZ + ENVELOPE)
          for k in range(4, 10)]


def module_layers() -> np.ndarray:
    return np.concatenate([np.repeat(np.arange(4), [n * ZSEG for n in LADDERS]),
                           np.repeat(np.arange(4, 10), PER_DISK)]).astype(np.int32)


def module_centres() -> np.ndarray:
    """float64[N_MODULES, 3], the points about which the modules turn."""
    c = []
    for r, n in zip(BARREL_R, LADDERS):
        for k in range(n):
            phi, rr = (k + 0.5) * 2 * math.pi / n, r + (DR if k % 2 else -DR)
            c += [(rr * math.cos(phi), rr * math.sin(phi), -BARREL_Z + (j + 0.5) * 2 * BARREL_Z / ZSEG)
                  for j in range(ZSEG)]
    for layer in range(4, 10):
        side, zd = math.copysign(1.0, disk_z(layer)), abs(disk_z(layer))
        for rr, n in zip(((DISK_RMIN + RING_SPLIT) / 2, (RING_SPLIT + DISK_RMAX) / 2), RING_MODULES):
            for k in range(n):
                phi = (k + 0.5) * 2 * math.pi / n
                c.append((rr * math.cos(phi), rr * math.sin(phi), side * (zd + (DZ if k % 2 else -DZ))))
    return np.array(c)


def radius_of_pt(pt):
    return pt / (0.299792458 * BZ) * 100.0


def make_cuts(pt_min: float, barrel_only: bool) -> dict:
    """The framework's cut table for tracks above pt_min (GeV): azimuth and z
    windows of the layer pairs, curvature, alignment and impact cuts."""
    rho, zmax, impact, f32 = radius_of_pt(pt_min), 12.0, 0.01, lambda v: float(np.float32(v))
    soft = max(1.0, 0.5 / pt_min)
    turn = lambda r: math.asin(min(1.0, r / (1.8 * rho)))
    pairs = []
    for i, o in (BARREL_PAIRS if barrel_only else PAIRS):
        Li, Lo = LAYERS[i], LAYERS[o]
        dphi = turn(Lo.rmax) - turn(Li.rmin) + math.asin(impact / Li.rmin) + math.asin(impact / max(Lo.rmin, Li.rmin)) + 0.005
        zlo, zhi = Li.zmin, Li.zmax
        if Li.kind == 0 and Lo.kind == 1:
            if disk_z(o) > 0:
                zlo = max(zlo, -zmax + (Lo.zmin + zmax) * Li.rmin / Lo.rmax - 0.5)
            else:
                zhi = min(zhi, zmax + (Lo.zmax - zmax) * Li.rmin / Lo.rmax + 0.5)
        pairs.append(dict(inner=i, outer=o, tan2_dphi=f32(math.tan(min(dphi, 1.2)) ** 2), zlo=f32(zlo), zhi=f32(zhi),
                          zmax=f32(zmax), k_pt=f32(4.0 * (0.9 * rho) ** 2)))
    region = [dict(tol_rz2=f32((tol * soft) ** 2), k_curv=f32(4.0 * (0.8 * rho) ** 2), rmax2=f32((rmax * soft) ** 2),
                   zmax=f32(zmax)) for tol, rmax in ((0.02, 0.05), (0.03, 0.1))]
    return dict(pairs=pairs, region=region, fishbone_eps2=f32(math.tan(2e-3) ** 2), min_hits=3)


# ------------------------------------------------------------------- cases
def event_case(kind: str, events: int, pileup: float, **more) -> dict:
    return dict(dict(kind=kind, events=events, pileup=pileup, pt_min=0.5, noise=0.02, inefficiency=0.0, ragged=False,
                     helices=0, grad=False), **more)


def listed() -> list[dict]:
    ev = event_case
    return [
        # the smallest call: 50 noiseless helices in the barrel, the event a new user or a monitoring probe runs
        dict(ev("chain", 1, 0.0, helices=50, pt_min=0.9, noise=0.0), name="chain-barrel-50-helices"),
        # an online trigger that takes one event at a time, at the paper's pileup and at that of the upgrade
        dict(ev("chain", 1, 50.0), name="chain-pu50"),
        dict(ev("chain", 1, 200.0), name="chain-pu200"),
        # offline throughput: batches of the paper's events, and the benchmark's batch
        dict(ev("chain", 32, 50.0), name="chain-pu50-batch32"),
        dict(ev("chain", 64, 200.0), name="chain-pu200-batch64"),
        # low-momentum tracking with dead channels and noise: the densest graph, the longest lists per hit
        dict(ev("chain", 24, 200.0, pt_min=0.3, noise=0.05, inefficiency=0.1), name="chain-stress-batch24"),
        # a real run's mix: every event another size, empty ones among them
        dict(ev("chain", 37, 90.0, ragged=True, noise=0.03), name="chain-ragged-batch37"),
        # refit of a batch after new hit positions
        dict(ev("refit", 24, 200.0), name="refit-pu200-batch24"),
        # gradient of a loss of the track parameters with respect to every hit
        dict(ev("refit", 24, 200.0, grad=True), name="refit-grad-pu200-batch24"),
        # one step of the alignment of a misaligned detector
        dict(ev("align", 32, 50.0), name="align-pu50-batch32"),
        # from fitted tracks to vertices, for a batch
        dict(ev("postfit", 24, 200.0), name="postfit-pu200-batch24"),
        # the vertex finder alone on one event's track summaries
        dict(ev("vertices", 1, 50.0), name="vertices-pu50"),
    ]


def draw(rng) -> dict:
    """Batches of 1 to 64 events at pileup 8 to 200, momentum thresholds 0.3
    to 0.9 GeV; fewer events where the threshold is low."""
    kind = rng.choice(["chain"] * 5 + ["refit"] * 2 + ["align", "postfit", "vertices"])
    pileup = round(math.exp(rng.uniform(math.log(8.0), math.log(200.0))), 1)
    pt_min = rng.choice([0.3, 0.5, 0.5, 0.5, 0.9])
    most = 24 if pt_min < 0.5 or kind != "chain" else 64
    events = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    case = event_case(kind, events, pileup, pt_min=pt_min, noise=round(rng.uniform(0.0, 0.05), 3),
                      inefficiency=round(rng.choice([0.0, rng.uniform(0.0, 0.1)]), 3), ragged=rng.random() < 0.3)
    if kind == "refit":
        case["grad"] = rng.random() < 0.5
    return case


def numbers(case: dict, pileup: float) -> tuple[float, float, float, float]:
    """Usual numbers of hits, doublets, n-tuplets and tracks of an event."""
    H = pileup * 134.0 + 270.0 if not case["helices"] else 4.0 * case["helices"]
    soft = 1.0 if case["pt_min"] >= 0.5 else 1.4
    D = 2.8e-3 * H * H * soft if not case["helices"] else 237.0
    if case["ragged"]:                       # mean of the squared relative size of the events
        D *= 1.5
    T = 0.7 * H + 0.022 * D * soft
    return H, D, T, 0.8 * T


def work(case: dict) -> dict:
    """Bytes and operations of one pass, from the case's usual numbers: 60
    operations for each doublet's cuts, 400 for each track's fit."""
    ev = case["events"]
    H, D, T, K = numbers(case, case["pileup"])
    if case["kind"] == "chain":
        return dict(bytes=ev * (20 * H + 10 * D + 8 * 0.03 * D + 66 * T + 89 * K), flops=ev * (60 * D + 400 * K))
    if case["kind"] == "vertices":
        n = 33.0 * case["pileup"] + 70.0
        return dict(bytes=ev * 22 * n, flops=ev * 400 * n)
    if case["kind"] == "postfit":
        return dict(bytes=ev * (44 + 32 + 22) * K, flops=ev * 60 * K)
    back = 2 if case["grad"] or case["kind"] == "align" else 1
    return dict(bytes=ev * (20 * H * back + (36 + 16 * 3.2 + 84) * K * back), flops=ev * 400 * K * (1 if back == 1 else 4))


# ------------------------------------------------------------------ events
def generator(seed: int) -> torch.Generator:
    return torch.Generator(device=DEV).manual_seed(int(seed))


def covering(phi, n, parity):
    """(covered, module): the module k of n, of the given parity, that spans
    phi; neighbours overlap by OVERLAP of their width."""
    u = torch.remainder(phi, 2 * math.pi) * (n / (2 * math.pi))
    k0, frac = u.floor().long() % n, u - u.floor()
    here, low, high = k0 % 2 == parity, frac <= OVERLAP / 2, frac >= 1 - OVERLAP / 2
    k = torch.where(here, k0, torch.where(low, (k0 - 1) % n, (k0 + 1) % n))
    return here | low | high, k


def module_of(layer, k, ring, z):
    if layer < 4:
        seg = ((z + BARREL_Z) * (ZSEG / (2 * BARREL_Z))).floor().clamp(0, ZSEG - 1).long()
        return BARREL_BASE[layer] + k * ZSEG + seg
    return N_BARREL + (layer - 4) * PER_DISK + torch.where(ring, RING_MODULES[0] + k, k)


def circle_point(x, y, phi, k, s):
    h = 0.5 * k * s
    f = s * torch.where(h.abs() > 1e-8, torch.sin(h) / h, 1.0)
    return x + f * torch.cos(phi + h), y + f * torch.sin(phi + h)


def make_events(case: dict, seed: int) -> dict:
    """Hits of a batch: x, y, z, r, module, ev_off, shuffled within each event."""
    g, E = generator(seed), case["events"]
    uni = lambda n, lo=0.0, hi=1.0: lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=F64)
    gauss = lambda n: torch.randn(n, generator=g, device=DEV, dtype=F64)
    poisson = lambda mean: torch.poisson(mean, generator=g).long()
    plain = case["helices"] > 0              # no overlaps, no scattering, one vertex at the origin
    if plain:
        vev, ntrk, hard = torch.arange(E, device=DEV), torch.full((E,), case["helices"], device=DEV), torch.zeros(E, dtype=torch.bool, device=DEV)
        vtx = torch.zeros(E, 3, device=DEV, dtype=F64)
    else:
        mean = torch.full((E,), float(case["pileup"]), device=DEV, dtype=F64)
        filled = torch.ones(E, dtype=torch.long, device=DEV)
        if case["ragged"]:
            mean = (2.0 * mean * uni(E)).clamp(max=200.0)
            filled[3::7] = 0
        nv = poisson(mean) * filled
        vev = torch.cat([torch.arange(E, device=DEV).repeat_interleave(nv), torch.arange(E, device=DEV)[filled > 0]])
        hard = torch.arange(vev.numel(), device=DEV) >= int(nv.sum())
        ntrk = poisson(torch.where(hard, 60.0, 30.0).to(F64))
        vtx = torch.stack([15e-4 * gauss(vev.numel()), 15e-4 * gauss(vev.numel()), 3.5 * gauss(vev.numel())], 1)
    vid = torch.arange(vev.numel(), device=DEV).repeat_interleave(ntrk)
    n = vid.numel()
    ev, u = vev[vid], uni(n)
    pmin = 1.0 if plain else torch.where(hard[vid], max(1.0, case["pt_min"]), case["pt_min"])
    pt = torch.exp(u * math.log(10.0)) if plain else pmin / (1.0 - u * (1.0 - pmin / 100.0))
    eta = uni(n, -2.0, 2.0) if plain else uni(n, -2.5, 2.5)
    phi, q = uni(n, -math.pi, math.pi), torch.where(uni(n) < 0.5, -1.0, 1.0)
    x, y, z = vtx[vid].unbind(1)
    tanl, p, k = torch.sinh(eta), pt * torch.cosh(eta), -q / radius_of_pt(pt)
    side = torch.where(tanl > 0, 1.0, -1.0).to(F64)
    if plain:
        surfaces = [(L, r, -1) for L, r in enumerate(BARREL_R)]
    else:
        surfaces = [(L, r + d, par) for L, r in enumerate(BARREL_R) for par, d in ((0, -DR), (1, DR))]
        surfaces += [(4 + d, zd + dz, par) for d, zd in enumerate(DISK_Z) for par, dz in ((0, -DZ), (1, DZ))]
    out = []
    for layer, val, par in surfaces:
        if layer < 4:
            arc = lambda r: 2.0 / k.abs() * torch.asin((0.5 * r * k.abs()).clamp(max=1.0))
            s = arc(torch.full_like(x, val)) - arc(torch.hypot(x, y))
            for _ in range(5):
                xs, ys = circle_point(x, y, phi, k, s)
                a = phi + k * s
                s = s - (xs * xs + ys * ys - val * val) / (2.0 * (xs * torch.cos(a) + ys * torch.sin(a)))
        else:
            s = (side * val - z) / tanl
        ok = torch.isfinite(s) & (s > 1e-7) & (k.abs() * s < math.pi)
        s = torch.where(ok, s, 0.0)
        xs, ys = circle_point(x, y, phi, k, s)
        zs, a, rr = z + s * tanl, phi + k * s, torch.hypot(xs, ys)
        where = torch.atan2(ys, xs)
        cosl = torch.rsqrt(1.0 + tanl * tanl)
        if layer < 4:
            if par < 0:
                kk = (torch.remainder(where, 2 * math.pi) * (LADDERS[layer] / (2 * math.pi))).long() % LADDERS[layer]
            else:
                cov, kk = covering(where, LADDERS[layer], par)
                ok = ok & cov
            ok = ok & (zs.abs() < BARREL_Z) & ((rr - val).abs() < 1e-6)
            module = module_of(layer, kk, None, zs)
            lay = torch.full_like(kk, layer)
            x0 = 0.02 / (cosl * (torch.cos(a) * xs + torch.sin(a) * ys) / rr).abs().clamp(min=1e-3)
        else:
            ring = rr >= RING_SPLIT
            (c0, k0), (c1, k1) = covering(where, RING_MODULES[0], par), covering(where, RING_MODULES[1], par)
            ok = ok & torch.where(ring, c1, c0) & (rr >= DISK_RMIN) & (rr <= DISK_RMAX)
            kk = torch.where(ring, k1, k0)
            lay = torch.where(side > 0, layer, layer + 3)
            module = torch.where(side > 0, module_of(layer, kk, ring, None), module_of(layer + 3, kk, ring, None))
            x0 = 0.03 / (tanl.abs() * cosl).clamp(min=1e-3)
        x, y, z, phi = torch.where(ok, xs, x), torch.where(ok, ys, y), torch.where(ok, zs, z), torch.where(ok, a, phi)
        kept = ok & (uni(n) >= case["inefficiency"])
        out.append([v[kept] for v in (xs, ys, zs, lay, module, ev)])
        if not plain:                        # scattering in the module just crossed
            th = torch.where(ok, 0.0136 / p * torch.sqrt(x0) * (1.0 + 0.038 * torch.log(x0)), 0.0)
            lam = torch.atan(tanl) + gauss(n) * th
            phi, tanl = phi + gauss(n) * th / cosl, torch.tan(lam)
            k = -q / radius_of_pt(p * torch.cos(lam))
    hx, hy, hz, lay, module, hev = (torch.cat(v) for v in zip(*out))
    m = hx.numel()
    disk, rr = lay >= 4, torch.hypot(hx, hy)
    ph = torch.atan2(hy, hx) + 10e-4 * gauss(m) / rr
    rr = rr + torch.where(disk, 20e-4 * gauss(m), 0.0)
    hx, hy, hz = rr * torch.cos(ph), rr * torch.sin(ph), hz + torch.where(disk, 0.0, 20e-4 * gauss(m))
    nn = int(poisson(torch.tensor([case["noise"] * m], device=DEV, dtype=F64))) if case["noise"] > 0 and m else 0
    if nn:                                   # noise: like the signal over events and layers, uniform on each
        at = (uni(nn) * m).long()
        ph, nl = uni(nn, -math.pi, math.pi), lay[at]
        rd, zb = torch.sqrt(uni(nn, DISK_RMIN ** 2 + 0.01, DISK_RMAX ** 2 - 0.01)), uni(nn, -BARREL_Z + 0.01, BARREL_Z - 0.01)
        ring = rd >= RING_SPLIT
        nx, nz, nm = torch.zeros_like(ph), torch.zeros_like(ph), torch.zeros_like(nl)
        for layer in range(10):
            if layer < 4:
                (c0, k0), (_, k1) = covering(ph, LADDERS[layer], 0), covering(ph, LADDERS[layer], 1)
                r_, z_, mod = torch.where(c0, BARREL_R[layer] - DR, BARREL_R[layer] + DR), zb, module_of(layer, torch.where(c0, k0, k1), None, zb)
            else:
                zd, sg = abs(disk_z(layer)), math.copysign(1.0, disk_z(layer))
                even = [covering(ph, c, 0) for c in RING_MODULES]
                c0 = torch.where(ring, even[1][0], even[0][0])
                ko = torch.where(ring, covering(ph, RING_MODULES[1], 1)[1], covering(ph, RING_MODULES[0], 1)[1])
                kk = torch.where(c0, torch.where(ring, even[1][1], even[0][1]), ko)
                r_, z_, mod = rd, sg * torch.where(c0, zd - DZ, zd + DZ), module_of(layer, kk, ring, None)
            here = nl == layer
            nx, nz, nm = torch.where(here, r_, nx), torch.where(here, z_, nz), torch.where(here, mod, nm)
        hx, hy, hz = torch.cat([hx, nx * torch.cos(ph)]), torch.cat([hy, nx * torch.sin(ph)]), torch.cat([hz, nz])
        module, hev = torch.cat([module, nm]), torch.cat([hev, hev[at]])
    order = torch.argsort(hev.to(F64) + uni(hev.numel()), stable=True)
    snap = lambda v: torch.round(v / GRID) * GRID
    x, y, z = (snap(v[order]) for v in (hx, hy, hz))
    off = torch.zeros(E + 1, dtype=torch.int32, device=DEV)
    off[1:] = torch.bincount(hev, minlength=E).cumsum(0).to(torch.int32)
    f = lambda v: v.to(torch.float32).contiguous()
    return dict(x=f(x), y=f(y), z=f(z), r=f(snap(torch.hypot(x, y))), module=module[order].to(torch.int32), ev_off=off)


def make_summaries(case: dict, seed: int) -> dict:
    """Track summaries of a batch, for the vertex finder: true tracks around
    their vertices, a tenth of fakes, in random order."""
    g, E = generator(seed), case["events"]
    uni = lambda n, lo=0.0, hi=1.0: lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=F64)
    nv = torch.poisson(torch.full((E,), float(case["pileup"]), device=DEV, dtype=F64), generator=g).long().clamp(min=1)
    if case["ragged"]:
        nv = (nv * uni(E) * 2.0).long()
    vev = torch.arange(E, device=DEV).repeat_interleave(nv)
    vz = 3.5 * torch.randn(vev.numel(), generator=g, device=DEV, dtype=F64)
    vid = torch.arange(vev.numel(), device=DEV).repeat_interleave(
        torch.poisson(torch.full((vev.numel(),), 30.0, device=DEV, dtype=F64), generator=g).long())
    nf = vid.numel() // 10
    n = vid.numel() + nf
    fake = torch.arange(n, device=DEV) >= vid.numel()
    ev = torch.cat([vev[vid], (uni(nf) * E).long()])
    pt, eta = 0.3 / (1.0 - uni(n) * (1.0 - 0.003)), uni(n, -2.5, 2.5)
    ez = 0.002 * (1.0 + eta.abs()) * torch.sqrt(1.0 + 1.0 / (pt * pt)) * torch.where(fake, 5.0, 1.0)
    z0 = torch.cat([vz[vid], uni(nf, -15.0, 15.0)]) + torch.where(fake, 0.0, ez) * torch.randn(n, generator=g, device=DEV, dtype=F64)
    u, order = uni(n), torch.argsort(uni(n))
    nh = torch.where(u < 0.35, 3, torch.where(u < 0.9, 4, 5))
    keep = uni(n) < 0.9
    f, b = lambda v: v[order].to(torch.float32), lambda v: v[order].to(torch.uint8)
    return dict(ev=ev[order].to(torch.int32), z0=f(z0), ez0=f(ez), pt=f(pt), nhits=b(nh), keep=b(keep))


# --------------------------------------------------------- a user's program
def make_record(case: dict) -> dict:
    """The program's own output arrays, of a fixed size that no batch of the
    case exceeds; the places after the last entry stay zero."""
    most = min(case["pileup"] * (2.0 if case["ragged"] else 1.0), 200.0)
    most += 5.0 * math.sqrt(most) + 5.0
    E = case["events"]
    H, K = (int(E * 1.5 * numbers(case, most)[0]) + 1000, int(E * 1.5 * numbers(case, most)[3]) + 1000)
    f32, sizes = torch.float32, {}
    track = dict(params=((K, 5), f32), chi2=((K,), f32))
    hit = {k: ((H,), f32) for k in ("gx", "gy", "gz")}
    if case["kind"] == "chain":
        sizes = dict(track, cov=((K, 15), f32), ndf=((K,), torch.int8), hits=((K, NMAX), torch.int32))
    elif case["kind"] == "vertices":
        sizes = dict(track_vertex=((int(E * 50.0 * most) + 1000,), torch.int32))
    elif case["kind"] == "postfit":
        sizes = dict(track_vertex=((K,), torch.int32), ev=((K,), torch.int32), z0=((K,), f32), ez0=((K,), f32),
                     pt=((K,), f32), nhits=((K,), torch.uint8), keep=((K,), torch.uint8))
    elif case["kind"] == "refit":
        sizes = dict(track, **hit) if case["grad"] else track
    else:
        sizes = track
    return {k: torch.zeros(shape, dtype=dtype, device=DEV) for k, (shape, dtype) in sizes.items()}


def fill(record: dict, values: dict) -> dict:
    """The record with the first entries of its arrays set; other values as
    they are."""
    for k in record:
        if values[k] is not None:
            record[k][:values[k].shape[0]] = values[k]
    return {**values, **{k: v if values[k] is not None else None for k, v in record.items()}}


def places():
    """The places of an n-tuplet, and a factor for each."""
    return torch.arange(NMAX, device=DEV), torch.tensor(
        [0x1E3779B97F4A7C15, 0x3F58476D1CE4E5B9, 0x14D049BB133111EB, 0x2545F4914F6CDD1D,
         0x369DEA0F31A53F85, 0x1B03738712FAD5C9, 0x2545F3C65D2C8A4F, 0x1CE4E5B9BF58476D], device=DEV)


def tuple_keys(hits, n, places):
    """The hits with unused places -1, and a 64-bit number made of each
    n-tuplet's hits: the program's n-tuplets are in the order of it."""
    hits = torch.where(places[0] < n[:, None], hits, -1)
    return hits, (hits * places[1]).sum(1)


def fix_order(bufs, counts) -> None:
    """Put the n-tuplets of a run in a fixed order, as a program does that
    refits the same tracks many times and compares them one by one."""
    nt = counts.n_tuples
    hits = bufs.tup_hits[:nt * NMAX].view(-1, NMAX)
    order = torch.argsort(tuple_keys(hits, bufs.tup_n[:nt], places())[1])
    cells = bufs.tup_cells[:nt * NMAX].view(-1, NMAX)
    for t in (hits, cells, bufs.tup_n[:nt], bufs.tup_alive[:nt]):
        t.copy_(t[order])


def fitted_order(n, alive, min_hits=3):
    """Indices of the n-tuplets that are fitted, in the fit's track order."""
    sel = torch.nonzero((alive != 0) & (n >= min_hits)).flatten()
    return sel[torch.argsort(n[sel].clamp(max=6).long(), stable=True)]


def pipeline_for(case: dict) -> Pipeline:
    return Pipeline(LAYERS, module_layers(), make_cuts(case["pt_min"], case["helices"] > 0), FIT, device=DEV)


def alignment(seed: int) -> list[torch.Tensor]:
    """Shifts of 50 um and rotations of 0.1 mrad per module and axis."""
    g = generator(seed + 1)
    return [scale * torch.randn(N_MODULES, 3, generator=g, device=DEV) for scale in (50e-4, 1e-4)]


def cotangents(seed: int, k: int):
    """Gradient of a loss with respect to k tracks' parameters and chi2: each
    parameter in units of its usual spread."""
    g = generator(seed + 2)
    scale = torch.tensor([100.0, 10.0, 10.0, 30.0, 1.0], device=DEV)
    return torch.randn(k, 5, generator=g, device=DEV) * scale, torch.rand(k, generator=g, device=DEV)


def prepare(case: dict, seed: int) -> dict:
    if case["kind"] == "vertices":
        return dict(case=case, summaries=make_summaries(case, seed), record=make_record(case))
    b = make_events(case, seed)
    hits = [b[k] for k in ("x", "y", "z", "r", "module", "ev_off")]
    pipe = pipeline_for(case)
    if case["kind"] == "chain":
        bufs = pipe.allocate(b["x"].numel(), case["events"])
        return dict(case=case, pipe=pipe, hits=hits, bufs=bufs, record=make_record(case), places=places())
    res, bufs = pipe.run(*hits)
    fix_order(bufs, res.counts)
    state = dict(case=case, pipe=pipe, hits=hits, bufs=bufs, counts=res.counts, record=make_record(case))
    if case["kind"] == "postfit":
        # the tracks to resolve are fitted here, in float64, so that no last
        # bit of the fit under way decides which tracks make a vertex
        nt = res.counts.n_tuples
        n, sel = bufs.tup_n[:nt], fitted_order(bufs.tup_n[:nt], bufs.tup_alive[:nt])
        par, cov, chi2 = fit_all(b, bufs.tup_hits[:nt * NMAX].view(-1, NMAX)[sel].long(), n[sel].long())
        K = sel.numel()
        bufs.trk_tuple[:K], bufs.trk_chi2[:K], bufs.trk_ndf[:K] = sel.to(torch.int32), chi2.float(), (2 * n[sel].long() - 5).to(torch.int8)
        bufs.trk_params[:K * 5], bufs.trk_cov[:K * 15] = par.float().flatten(), cov.float().flatten()
        return state
    centres = torch.as_tensor(module_centres())
    state["fit"] = DifferentiableFit(pipe, bufs, b["r"], b["module"], b["ev_off"], centres)
    if case["kind"] == "align":
        state["shift"], state["rot"] = alignment(seed)
    elif case["grad"]:
        state["cotangents"] = cotangents(seed, res.counts.n_tracks)
    return state


def ordered_tracks(res, record: dict, places) -> dict:
    t, which = res.tracks, res.tracks["tuple"]
    hits, key = tuple_keys(res.tuples["hits"], res.tuples["n"], places)
    order = torch.argsort(key[which])
    for k in ("params", "cov", "chi2", "ndf"):
        torch.index_select(t[k], 0, order, out=record[k][:order.numel()])
    torch.take(hits, torch.add(places[0], which[order][:, None], alpha=NMAX), out=record["hits"][:order.numel()])
    c = res.counts
    return dict(record, counts=[c.n_cells, c.n_alive_cells, c.n_edges, c.n_tuples, c.n_alive_tuples, c.n_tracks])


def used_rows(v: dict) -> dict:
    """The vertices without the unused rows of their table (zeros there)."""
    used = torch.arange(v["z"].shape[1], device=v["z"].device) < v["n"][:, None]
    f = torch.where(used, torch.stack([v["z"], v["ez"], v["chi2"], v["sumpt2"]]), 0.0)
    i = torch.where(used, torch.stack([v["ndf"], v["ntracks"]]), 0)
    return dict(n=v["n"], vertices=f, members=i, track_vertex=v["track_vertex"], status=v["status"])


def run(state: dict):
    case, record = state["case"], state["record"]
    if case["kind"] == "chain":
        res, state["bufs"] = state["pipe"].run(*state["hits"], bufs=state["bufs"])
        return ordered_tracks(res, record, state["places"])
    if case["kind"] == "vertices":
        s = state["summaries"]
        return fill(record, used_rows(find_vertices(s["ev"], s["z0"], s["ez0"], s["pt"], s["nhits"], s["keep"],
                                                    case["events"])))
    if case["kind"] == "postfit":
        v, s = state["pipe"].find_vertices(state["bufs"], state["counts"], *state["hits"])
        return fill(record, dict(used_rows(v), **s))
    fit, xyz = state["fit"], state["hits"][:3]
    if case["kind"] == "align":
        shift, rot = (state[k].detach().requires_grad_() for k in ("shift", "rot"))
        params, chi2 = fit.fit(*fit.align(*xyz, shift, rot))
        gshift, grot = torch.autograd.grad(torch.log1p(chi2).sum(), (shift, rot))
        return fill(record, dict(params=params.detach(), chi2=chi2.detach(), gshift=gshift, grot=grot))
    if not case["grad"]:
        params, chi2 = fit.fit(*xyz)
        return fill(record, dict(params=params, chi2=chi2))
    xyz = [t.detach().requires_grad_() for t in xyz]
    params, chi2 = fit.fit(*xyz)
    gx, gy, gz = torch.autograd.grad((params, chi2), xyz, state["cotangents"])
    return fill(record, dict(params=params.detach(), chi2=chi2.detach(), gx=gx, gy=gy, gz=gz))


# --------------------------------------- the same in 64 bits, in plain torch
def join(count, start):
    """For rows with count[i] partners from start[i] on: all (row, partner)."""
    row = torch.arange(count.numel(), device=count.device).repeat_interleave(count)
    first = count.cumsum(0) - count
    return row, torch.arange(row.numel(), device=count.device) - first[row] + start[row]


def ranges(sorted_keys, n):
    count = torch.bincount(sorted_keys, minlength=n)
    return count, count.cumsum(0) - count


def find_tuples(x, y, z, r, layer, cuts):
    """(hits [T, NMAX] with -1 in unused places, n, alive) of one event:
    doublets, Fishbone, connection, maximal paths, cleaning, by their definitions."""
    H, dev = x.numel(), x.device
    inner, outer, live = [], [], []
    for c in cuts["pairs"]:
        I, O = torch.nonzero(layer == c["inner"]).flatten(), torch.nonzero(layer == c["outer"]).flatten()
        I = I[(z[I] >= c["zlo"]) & (z[I] <= c["zhi"])]
        xi, yi, zi, ri = (v[I][None, :] for v in (x, y, z, r))
        xo, yo, zo, ro = (v[O][:, None] for v in (x, y, z, r))
        ok = (ro > ri) & ((zi * ro - zo * ri).abs() <= c["zmax"] * (ro - ri))
        C, D = xi * yo - yi * xo, xi * xo + yi * yo
        ok &= (D > 0) & (C * C <= c["tan2_dphi"] * D * D)
        ok &= c["k_pt"] * C * C <= ((xo - xi) ** 2 + (yo - yi) ** 2) * (xi * xi + yi * yi) * (xo * xo + yo * yo)
        o, i = torch.nonzero(ok).unbind(1)
        # Fishbone among the cells of one outer hit (in the order of nonzero, so sorted by it)
        cnt, start = ranges(o, O.numel())
        a, b = join(cnt[o], start[o])
        i, o = I[i], O[o]
        ux, uy, uz = x[i] - x[o], y[i] - y[o], z[i] - z[o]
        l2 = ux * ux + uy * uy + uz * uz
        cr = (uy[a] * uz[b] - uz[a] * uy[b]) ** 2 + (uz[a] * ux[b] - ux[a] * uz[b]) ** 2 + (ux[a] * uy[b] - uy[a] * ux[b]) ** 2
        dead = (ux[a] * ux[b] + uy[a] * uy[b] + uz[a] * uz[b] > 0) & (cr <= cuts["fishbone_eps2"] * l2[a] * l2[b])
        dead &= (l2[b] < l2[a]) | ((l2[b] == l2[a]) & (i[b] < i[a]))
        alive = torch.ones_like(i, dtype=torch.bool)
        alive[a[dead]] = False
        inner.append(i), outer.append(o), live.append(alive)
    inner, outer, live = torch.cat(inner), torch.cat(outer), torch.cat(live)
    cells = torch.nonzero(live).flatten()
    cells = cells[torch.argsort(outer[cells], stable=True)]
    inner, outer = inner[cells], outer[cells]
    cnt, start = ranges(outer, H)
    src, dst = [], []
    for c0 in range(0, inner.numel(), 200_000):
        cell = torch.arange(c0, min(c0 + 200_000, inner.numel()), device=dev)
        row, cand = join(cnt[inner[cell]], start[inner[cell]])
        row = cell[row]
        A, B, C = inner[cand], inner[row], outer[row]
        rg = (layer[B] >= 4).long()
        cut = {k: torch.tensor([q[k] for q in cuts["region"]], dtype=F64, device=dev) for k in cuts["region"][0]}
        X = (r[B] - r[A]) * (z[C] - z[B]) - (z[B] - z[A]) * (r[C] - r[B])
        ok = X * X <= cut["tol_rz2"][rg] * ((r[C] - r[A]) ** 2 + (z[C] - z[A]) ** 2)
        row, cand, A, B, C, rg = (v[ok] for v in (row, cand, A, B, C, rg))
        ok = (z[A] * r[C] - z[C] * r[A]).abs() <= cut["zmax"][rg] * (r[C] - r[A])
        bx, by, cx, cy, dx, dy = x[B] - x[A], y[B] - y[A], x[C] - x[A], y[C] - y[A], -x[A], -y[A]
        b2, c2, d2 = bx * bx + by * by, cx * cx + cy * cy, dx * dx + dy * dy
        P = b2 * ((x[C] - x[B]) ** 2 + (y[C] - y[B]) ** 2) * c2
        ok &= P >= cut["k_curv"][rg] * (bx * cy - by * cx) ** 2
        ok &= (bx * (cy * d2 - c2 * dy) - by * (cx * d2 - c2 * dx) + b2 * (cx * dy - cy * dx)) ** 2 <= cut["rmax2"][rg] * P
        src.append(cand[ok]), dst.append(row[ok])
    src, dst = torch.cat(src), torch.cat(dst)          # dst ascending
    n_in, first_in = ranges(dst, inner.numel())
    has_out = torch.zeros(inner.numel(), dtype=torch.bool, device=dev)
    has_out[src] = True
    first = torch.tensor([True, True, False, False, True, False, False, True, False, False], device=dev)
    path = torch.nonzero(~has_out & (n_in > 0)).flatten()[:, None]          # cells, outermost first
    found = []
    while path.numel():
        head = path[:, -1]
        if path.shape[1] >= 2:
            found.append(path[(n_in[head] == 0) & first[layer[inner[head]]]])
        row, e = join(n_in[head], first_in[head])
        path = torch.cat([path[row], src[e][:, None]], 1)
    rows, lens, longest = [], [], torch.zeros(inner.numel(), dtype=torch.long, device=dev)
    for f in found:
        hits = torch.cat([inner[f.flip(1)], outer[f[:, :1]]], 1)
        rows.append(torch.nn.functional.pad(hits, (0, NMAX - hits.shape[1]), value=-1))
        lens.append(torch.full((f.shape[0],), hits.shape[1], device=dev))
        longest[f.flatten()] = torch.maximum(longest[f.flatten()], torch.tensor(hits.shape[1], device=dev))
    if not rows:
        return torch.zeros(0, NMAX, dtype=torch.long, device=dev), *(torch.zeros(0, dtype=torch.long, device=dev),) * 2
    alive = torch.cat([(longest[f] <= f.shape[1] + 1).all(1) for f in found])
    return torch.cat(rows), torch.cat(lens), alive


def find_all(b, cuts):
    """The n-tuplets of a batch, in the fixed order: (hits, n, alive)."""
    layer = torch.as_tensor(module_layers(), device=DEV)[b["module"].long()].long()
    xyzr, off = [b[k].to(F64) for k in "xyzr"], b["ev_off"].tolist()
    parts = []
    for lo, hi in zip(off[:-1], off[1:]):
        if hi > lo:
            h, n, a = find_tuples(*(v[lo:hi] for v in xyzr), layer[lo:hi], cuts)
            parts.append((torch.where(h >= 0, h + lo, -1), n, a))
    hits, n, alive = (torch.cat(v) for v in zip(*parts))
    hits, key = tuple_keys(hits, n, places())
    order = torch.argsort(key)
    return hits[order], n[order], alive[order]


def asinc(q):
    q = q.clamp(-1.0, 1.0)
    small = q.abs() < 1e-4
    safe = torch.where(small, 1.0, q)
    return torch.where(small, 1.0 + q * q / 6.0, torch.asin(safe) / safe)


def fit64(x, y, z, disk):
    """Broken-line fit of K tracks of N hits (x, y, z, disk: [K, N]) in
    float64: (params [K, 5], cov [K, 15], chi2 [K]), differentiable."""
    K, N = x.shape
    m = N // 2
    abx, aby, acx, acy = x[:, m] - x[:, 0], y[:, m] - y[:, 0], x[:, -1] - x[:, 0], y[:, -1] - y[:, 0]
    dab = torch.hypot(abx, aby)
    k0 = 2.0 * (abx * acy - aby * acx) / (dab * torch.hypot(x[:, -1] - x[:, m], y[:, -1] - y[:, m]) * torch.hypot(acx, acy))
    psi0 = torch.atan2(aby, abx) - torch.asin((0.5 * k0 * dab).clamp(-1.0, 1.0))
    cs, sn, k = torch.cos(psi0), torch.sin(psi0), k0[:, None]
    dx, dy = x[:, 1:] - x[:, :1], y[:, 1:] - y[:, :1]
    dist = torch.hypot(dx, dy)
    zero = torch.zeros(K, 1, dtype=F64, device=x.device)
    s = torch.cat([zero, dist * asinc(0.5 * k * dist)], 1)
    X, Y = dx * cs[:, None] + dy * sn[:, None], dy * cs[:, None] - dx * sn[:, None]
    U = k * (X * X + Y * Y) - 2.0 * Y
    off = torch.cat([zero, -U / (1.0 + torch.sqrt((1.0 + k * U).clamp(min=0.0)))], 1)
    ds = (s[:, 1:] - s[:, :-1]).clamp(min=1e-4)
    tan0 = (z[:, -1] - z[:, 0]) / s[:, -1].clamp(min=1e-4)
    sec2, atl = 1.0 + tan0 * tan0, tan0.abs().clamp(min=1e-3)
    sec = torch.sqrt(sec2)
    f = {key: float(np.float32(v)) for key, v in FIT.items()}
    mom = 0.00299792458 * f["bz"] / k0.abs().clamp(min=1e-7) * sec
    x0 = torch.where(disk, (f["x0_disk"] * sec / atl)[:, None], (f["x0_barrel"] * sec)[:, None])[:, 1:-1]
    th2 = (0.0136 / mom[:, None] * torch.sqrt(x0) * (1.0 + 0.038 * torch.log(x0))) ** 2
    vt, vl = (th2 * sec2[:, None]).clamp(min=1e-20), (th2 * (sec2 * sec2)[:, None]).clamp(min=1e-20)
    i1 = 1.0 / ds
    G = torch.zeros(K, N - 2, N + 1, dtype=F64, device=x.device)            # kinks of u_0 .. u_{N-1}, dk
    at = torch.arange(N - 2, device=x.device)
    G[:, at, at], G[:, at, at + 1], G[:, at, at + 2] = i1[:, :-1], -(i1[:, :-1] + i1[:, 1:]), i1[:, 1:]
    G[:, at, -1] = -0.5 * (ds[:, :-1] + ds[:, 1:])
    wz = torch.where(disk, (1.0 / (f["sigma_r"] * atl) ** 2)[:, None], torch.tensor(1.0 / f["sigma_z"] ** 2, dtype=F64, device=x.device))
    wu = torch.full_like(off, 1.0 / f["sigma_rphi"] ** 2)
    A = torch.diag_embed(wz) + G[:, :, :N].mT @ (G[:, :, :N] / vl[:, :, None])
    B = torch.diag_embed(torch.cat([wu, zero], 1)) + G.mT @ (G / vt[:, :, None])
    v = torch.linalg.solve(A, (wz * z)[:, :, None])[:, :, 0]
    u = torch.linalg.solve(B, torch.cat([wu * off, zero], 1)[:, :, None])[:, :, 0]
    kl, kt = (G[:, :, :N] @ v[:, :, None])[:, :, 0], (G @ u[:, :, None])[:, :, 0]
    chi2 = (wz * (v - z) ** 2).sum(1) + (kl * kl / vl).sum(1) + (wu * (u[:, :N] - off) ** 2).sum(1) + (kt * kt / vt).sum(1)
    u0, u1, dk, d1 = u[:, 0], u[:, 1], u[:, -1], ds[:, 0]
    px, py, psi, kf = x[:, 0] - u0 * sn, y[:, 0] + u0 * cs, psi0 + (u1 - u0) / d1 - 0.5 * dk * d1, k0 + dk
    cp, sp = torch.cos(psi), torch.sin(psi)
    Xo, Yo = -(px * cp + py * sp), px * sp - py * cp
    R2 = Xo * Xo + Yo * Yo
    U = kf * R2 - 2.0 * Yo
    S = torch.sqrt((1.0 + kf * U).clamp(min=0.0))
    a, b = kf * Xo, 1.0 - kf * Yo
    dpsi = torch.atan2(a, b)
    phi0 = psi + dpsi
    arc = torch.where(kf != 0, dpsi / torch.where(kf != 0, kf, 1.0), Xo)
    tanl = (v[:, 1] - v[:, 0]) / d1
    par = torch.stack([-kf, phi0 - 2 * math.pi * torch.round(phi0 / (2 * math.pi)), tanl, -U / (1.0 + S), v[:, 0] + tanl * arc], 1)
    with torch.no_grad():                     # covariance: solved blocks through the perigee's Jacobian
        one, nil = torch.ones_like(d1), torch.zeros_like(d1)
        J = []
        for dpx, dpy, dps, dkk in ((-sn, cs, -1.0 / d1, nil), (nil, nil, 1.0 / d1, nil), (nil, nil, -0.5 * d1, one)):
            dX, dY = -(dpx * cp + dpy * sp) + Yo * dps, dpx * sp - dpy * cp - Xo * dps
            dU = R2 * dkk + 2.0 * kf * Xo * dX + (2.0 * kf * Yo - 2.0) * dY
            dS = 0.5 / S * (U * dkk + kf * dU)
            dpsi_ = (b * (Xo * dkk + kf * dX) + a * (Yo * dkk + kf * dY)) / (a * a + b * b)
            J.append(torch.stack([-dkk, dps + dpsi_, -dU / (1.0 + S) + U / (1.0 + S) ** 2 * dS], 1))
        J = torch.stack(J, 2)
        sel = torch.tensor([0, 1, N], device=x.device)
        Cc = J @ torch.linalg.inv(B)[:, sel][:, :, sel] @ J.mT
        Jl = torch.stack([torch.stack([-1.0 / d1, 1.0 / d1], 1), torch.stack([1.0 - arc / d1, arc / d1], 1)], 1)
        Cl = Jl @ torch.linalg.inv(A)[:, :2, :2] @ Jl.mT
        cov = torch.zeros(K, 15, dtype=F64, device=x.device)
        for (i, j), c in {(0, 0): Cc[:, 0, 0], (1, 0): Cc[:, 1, 0], (1, 1): Cc[:, 1, 1], (2, 2): Cl[:, 0, 0], (3, 0): Cc[:, 2, 0],
                          (3, 1): Cc[:, 2, 1], (3, 3): Cc[:, 2, 2], (4, 2): Cl[:, 1, 0], (4, 4): Cl[:, 1, 1]}.items():
            cov[:, i * (i + 1) // 2 + j] = c
    return par, cov, chi2


def fit_all(b, hits, n, xyz=None):
    """fit64 of n-tuplets of any lengths (hits [T, NMAX], n [T]), a million
    at a time, in their order."""
    xyz = xyz or [b[k].to(F64) for k in "xyz"]
    is_disk = torch.as_tensor(module_layers(), device=DEV)[b["module"].long()] >= 4
    where, outs = [], []
    for N in range(3, NMAX + 1):
        of = torch.nonzero(n == N).flatten()
        for sel in of.split(1_000_000) if of.numel() else ():
            h = hits[sel, :N]
            where.append(sel)
            outs.append(fit64(*(v[h] for v in xyz), is_disk[h]))
    if not outs:
        return tuple(torch.zeros(s, dtype=F64, device=DEV) for s in ((0, 5), (0, 15), (0,)))
    back = torch.argsort(torch.cat(where))
    return tuple(torch.cat(v)[back] for v in zip(*outs))


def resolve(hits, n, chi2, d0):
    """keep: cells keep the tracks of smallest chi2, then hits the triplets of
    smallest |d0| (float32 values; equal ones are all kept)."""
    K, inf = n.numel(), float("inf")
    cell = hits[:, :-1] * (1 << 31) + hits[:, 1:]
    is_cell = torch.arange(NMAX - 1, device=hits.device) < n[:, None] - 1
    _, cid = torch.unique(torch.where(is_cell, cell, -1), return_inverse=True)
    least = lambda idx, val, size: torch.full((size,), inf, device=hits.device).scatter_reduce(0, idx.flatten(), val.flatten(), "amin")
    c2 = chi2[:, None].expand(K, NMAX - 1)
    keep = ((c2 <= least(cid, torch.where(is_cell, c2, inf), int(cid.max()) + 1)[cid]) | ~is_cell).all(1)
    tri = keep & (n == 3)
    h3, tip = hits[tri, :3], d0[tri].abs()[:, None].expand(-1, 3)
    keep[tri] = (tip <= least(h3, tip, int(hits.max()) + 1)[h3]).all(1)
    return keep


def cluster(z0, ez, pt):
    """Vertices of one event's eligible tracks: rows (z, ez, chi2, sumpt2) in
    decreasing sumpt2.  Decisions in float32 as stated, sums in float64."""
    c = DEFAULT_VERTEX_CUTS
    order = np.argsort(z0, kind="stable")
    z0, ez, pt = z0[order], ez[order], pt[order]
    e2 = ez * ez
    dz = z0[:, None] - z0[None, :]
    near = (np.abs(dz) < np.float32(c["dz_cut"])) & (dz * dz < np.float32(c["chi2_max"]) * (e2[:, None] + e2[None, :]))
    np.fill_diagonal(near, False)
    rho, pos = 1 + near.sum(1), np.arange(len(z0))
    higher = near & ((rho[None, :] > rho[:, None]) | ((rho[None, :] == rho[:, None]) & (pos[None, :] < pos[:, None])))
    dist = np.where(higher, np.abs(dz), np.float32(np.inf))
    root = np.where(higher.any(1), dist.argmin(1), pos)
    while True:
        nxt = root[root]
        if (nxt == root).all():
            break
        root = nxt
    zz, w, rows = z0.astype(np.float64), 1.0 / ez.astype(np.float64) ** 2, []
    mean = lambda m: (w[m] * zz[m]).sum() / w[m].sum()
    for k in np.unique(root):
        m = np.nonzero(root == k)[0]
        if rho[k] <= 1 or len(m) < c["min_tracks"]:
            continue
        z = mean(m)
        parts = [m]
        if (w[m] * (zz[m] - z) ** 2).sum() / (len(m) - 1) > c["split_chi2"]:
            up = zz[m] >= z
            if up.any() and not up.all():
                ctr, last = (mean(m[~up]), mean(m[up])), None
                for _ in range(20):
                    up = np.abs(zz[m] - ctr[1]) < np.abs(zz[m] - ctr[0])
                    if last is not None and (up == last).all():
                        break
                    last = up
                    if not up.any() or up.all():
                        break
                    ctr = (mean(m[~up]), mean(m[up]))
                if min(up.sum(), (~up).sum()) >= c["min_tracks"]:
                    parts = [m[~up], m[up]]
        for q in parts:
            zv = mean(q)
            rows.append((zv, 1.0 / math.sqrt(w[q].sum()), (w[q] * (zz[q] - zv) ** 2).sum(), (pt[q].astype(np.float64) ** 2).sum()))
    rows.sort(key=lambda v: (-v[3], v[0]))
    return rows


def vertices64(s: dict, events: int, rows: int = 256) -> torch.Tensor:
    c, out = DEFAULT_VERTEX_CUTS, np.zeros((4, events, rows))
    a = {k: v.cpu().numpy() for k, v in s.items()}
    ok = (a["keep"] != 0) & (a["nhits"] >= c["min_hits"]) & (a["pt"] > np.float32(c["pt_min"])) & (a["ez0"] > 0) & \
         (a["ez0"] < np.float32(c["ez0_max"])) & np.isfinite(a["z0"])
    for e in range(events):
        m = ok & (a["ev"] == e)
        for i, v in enumerate(cluster(a["z0"][m], a["ez0"][m], a["pt"][m])[:rows]):
            out[:, e, i] = v
    return torch.as_tensor(out)


def values64(case: dict, seed: int):
    none = dict(n=None, members=None, track_vertex=None, status=None)
    if case["kind"] == "vertices":
        return dict(none, vertices=vertices64(make_summaries(case, seed), case["events"]))
    density = (case["pileup"] / 200.0) ** 2 * (1.5 if case["pt_min"] < 0.5 else 1.0) * (1.5 if case["ragged"] else 1.0)
    if case["events"] * density > 40.0:      # the pair loops over every event take too long
        return None
    b = make_events(case, seed)
    hits, n, alive = find_all(b, make_cuts(case["pt_min"], case["helices"] > 0))
    sel = fitted_order(n, alive)
    if case["kind"] == "chain":
        sel = sel.sort().values
    hits, n = hits[sel], n[sel]
    if case["kind"] == "chain":
        par, cov, chi2 = fit_all(b, hits, n)
        return dict(params=par, cov=cov, chi2=chi2, ndf=None, hits=None, counts=None)
    if case["kind"] == "postfit":
        par, cov, chi2 = (v.float() for v in fit_all(b, hits, n))
        ev = torch.searchsorted(b["ev_off"][1:].long(), hits[:, 0].contiguous(), right=True)
        pt = (np.float32(0.299792458e-2) * np.float32(BZ)).item() / par[:, 0].abs()
        s = dict(ev=ev, z0=par[:, 4], ez0=cov[:, 14].sqrt(), pt=pt, nhits=n, keep=resolve(hits, n, chi2, par[:, 3]))
        f = lambda v: v.to(F64)
        return dict(none, vertices=vertices64(s, case["events"]), ev=None, nhits=None, keep=None, z0=f(s["z0"]),
                    ez0=f(cov[:, 14]).sqrt(), pt=0.299792458e-2 * BZ / f(par[:, 0]).abs())
    xyz = [b[k].to(F64).requires_grad_() for k in "xyz"]
    if case["kind"] == "align":
        shift, rot = (t.to(F64).requires_grad_() for t in alignment(seed))
        mod, p = b["module"].long(), torch.stack([v.detach() for v in xyz], 1)
        moved = p + torch.cross(rot[mod], p - torch.as_tensor(module_centres(), device=DEV).float().to(F64)[mod], dim=1) + shift[mod]
        par, _, chi2 = fit_all(b, hits, n, list(moved.unbind(1)))
        gshift, grot = torch.autograd.grad(torch.log1p(chi2).sum(), (shift, rot))
        return dict(params=par, chi2=chi2, gshift=gshift, grot=grot)
    par, _, chi2 = fit_all(b, hits, n, xyz)
    if not case["grad"]:
        return dict(params=par, chi2=chi2)
    gp, gc = cotangents(seed, n.numel())
    gx, gy, gz = torch.autograd.grad((par, chi2), xyz, (gp.to(F64), gc.to(F64)))
    return dict(params=par, chi2=chi2, gx=gx, gy=gy, gz=gz)


def exact(case: dict, seed: int):
    values = values64(case, seed)
    if values is None:
        return None
    record = {k: v.to(F64) if v.is_floating_point() else v for k, v in make_record(case).items()}
    return fill(record, {k: v if v is None else v.detach() for k, v in values.items()})
