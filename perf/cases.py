"""Performance cases: the work a program has this library do, through its public entry points.

Four kinds of pass:
  fit     Kalman fit of tracks with known hit sequences (one small event; a batch of uneven events)
  index   hit-index build alone, over a batch of events
  events  event reconstruction: hit index, combinatorial finding, fit of the found tracks; on barrel
          layers or barrel + disks, plain or with the learned hit proposal, with the detector
          options (steering, material map, field map), with seed cleaning and duplicate removal
  net     the learned proposal's network: scoring rows, loss and gradient, a training step

Events are drawn here, on the GPU, in 64 bits: helices from the origin in a solenoid field, their
crossings with the surfaces, Highland scattering kicks, Gaussian smearing, uniform noise. Event sizes
depend on the case alone, the events themselves on the seed.
"""
import math
import os
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_1906_02253_gb300 as kf

CURV = 0.00299792458  # GeV / (T cm)
CHI2_CUT = 30.0
HALF_LENGTH, DISK_Z = 29.0, [30.0 + 11.25 * j for j in range(9)]


def listed():
    return [
        # one event's tracks refitted on their own: the smallest call, all latency
        dict(name="fit_event", kind="fit", events=1, lo=1000, hi=1000, layers=10, scatter=False),
        # a batch of uneven events refitted in one call
        dict(name="fit_batch", kind="fit", events=100, lo=2000, hi=20000, layers=17, scatter=True),
        # the hit index of a batch, as built before several finding passes
        dict(name="index_batch", kind="index", events=200, lo=3000, hi=8000, layers=17, disks=True, noise=1.0),
        # one event reconstructed as it arrives (online use)
        _events("event", 1, 5000, 5000, noise=0.3),
        # a batch of uneven events: the throughput of offline reconstruction
        _events("batch", 100, 2000, 20000),
        # high occupancy on barrel + disks, in two passes of candidate capacity
        _events("disks", 100, 3000, 8000, disks=True, noise=1.0, k=8, adaptive=2),
        # the same with the learned proposal, in its recommended setting
        _events("learned", 100, 3000, 8000, disks=True, noise=1.0, k=8, adaptive=2, top_n=2, margin=0.7),
        # a detector with a field map
        _events("field_map", 20, 3000, 8000, disks=True, noise=1.0, k=8, option="field"),
        # overlapping modules: several seeds per particle, cleaned before and after finding
        _events("duplicates", 20, 5000, 5000, noise=0.3, overlap=0.3),
        # candidate pairs scored with the network outside the finder
        dict(name="score_pairs", kind="net", call="score", rows=1000003),
        # one minibatch step of training: loss, gradient, Adam
        dict(name="train_step", kind="net", call="step", rows=4096),
        # loss and gradient over a whole training set, as at the end of every epoch
        dict(name="train_set", kind="net", call="loss", rows=2000003),
    ]


def _events(name, events, lo, hi, layers=17, disks=False, noise=0.0, overlap=0.0, k=6, adaptive=0, top_n=0, margin=0.0,
            option=""):
    case = dict(kind="events", events=events, lo=lo, hi=hi, layers=layers, disks=disks, noise=noise, overlap=overlap,
                k=k, adaptive=adaptive, top_n=top_n, margin=margin, option=option)
    return dict(case, name=name) if name else case


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "index", "barrel", "barrel", "disks", "disks", "learned", "option", "duplicates", "net"])
    if kind == "net":
        call = rng.choice(["score", "step", "loss"])
        top = {"score": 1000000, "step": 65536, "loss": 2000000}[call]
        return dict(kind="net", call=call, rows=_spread(rng, 1000, top))
    # about half the tracks of the largest batch at most, in events of ordinary sizes
    total = _spread(rng, 300, 500000)
    size = min(total, _spread(rng, 300, 12000))
    events, lo = max(1, total // size), max(100, size // 3)
    hi = max(lo, 2 * size - lo)
    layers = rng.randint(13, 17)
    if kind == "fit":
        return dict(kind="fit", events=events, lo=lo, hi=hi, layers=rng.randint(6, 17), scatter=rng.random() < 0.7)
    if kind == "index":
        return dict(kind="index", events=events, lo=lo, hi=hi, layers=layers, disks=rng.random() < 0.5,
                    noise=rng.choice([0.0, 0.3, 1.0]))
    if kind == "barrel":
        return _events("", events, lo, hi, layers, noise=rng.choice([0.0, 0.3]), k=rng.choice([2, 4, 5, 6]))
    if kind == "duplicates":
        return _events("", min(events, 100), min(lo, 4000), min(hi, 6000), layers, noise=0.3, overlap=0.3)
    events = min(events, 60)
    lo, hi = min(lo, 6000), min(hi, 9000)
    if kind == "option":
        return _events("", events, lo, hi, disks=True, noise=rng.choice([0.3, 1.0]), k=rng.choice([4, 6, 8]),
                       option=rng.choice(["field", "material", "steering", "all"]))
    top = rng.choice([1, 2, 4]) if kind == "learned" else 0
    return _events("", events, lo, hi, disks=True, noise=rng.choice([0.3, 1.0]), k=rng.choice([4, 6, 8]),
                   adaptive=rng.choice([0, 2, 4]), top_n=top, margin=rng.choice([0.0, 0.7, 1.0]) if top else 0.0)


# ---- detector -------------------------------------------------------------------------------------

def _detector(case):
    """Barrel layers every 4 cm (each long enough for |eta| <= 1, or of one half-length inside nine
    disks per side), 64 x 32 bins, in the form kf.Geometry takes."""
    f32 = lambda v: float(np.float32(v))  # noqa: E731  (the geometry is 32-bit; the events use the same numbers)
    disks, option = case.get("disks", False), case.get("option", "")
    x0 = f32(0.02) if case.get("scatter", True) else 0.0
    surf = []
    for i in range(case["layers"]):
        r = 4.0 + 4.0 * i
        h = f32(HALF_LENGTH if disks else 1.2 * r * math.sinh(1.0))
        surf.append(SimpleNamespace(type=0, r_or_z=r, lo=-h, hi=h, x_over_x0=x0, n_phi=64, n_2nd=32))
    for sign in (1.0, -1.0) if disks else ():
        for z in DISK_Z:
            surf.append(SimpleNamespace(type=1, r_or_z=sign * z, lo=4.0, hi=68.0, x_over_x0=x0, n_phi=64, n_2nd=32))
    d = SimpleNamespace(surfaces=surf, bz=f32(3.8), sigma_rphi=0.01, sigma_2nd=0.1, prior=(0.1, 1.0, 0.5, 0.05, 0.05),
                        ms_on=x0 > 0, disks=disks, barrels=case["layers"], eta=2.4 if disks else 1.0)
    d.lmax = case["layers"] + (len(DISK_Z) if disks else 0)
    if option in ("material", "all"):  # thicker towards the ends of each surface, with the loss in it
        d.material = [[x0 * (1 + 2 * ((s.lo + (s.hi - s.lo) * k / 7) / s.hi) ** 2) for k in range(8)] for s in surf]
        d.eloss = 0.0363
    if option in ("field", "all"):
        d.field_z2, d.field_r2 = -4e-6, -1e-6
    return d


def _steering(d):
    nb, nd = d.barrels, len(DISK_Z)
    b, p, m = list(range(nb)), list(range(nb, nb + nd)), list(range(nb + nd, nb + 2 * nd))
    return dict(c_barrel=float(np.float32(math.sinh(0.4))), c_endcap=float(np.float32(math.sinh(1.8))),
                lists=[b, b + p, b + m, b[:3] + p, b[:3] + m])


def _event_sizes(case):
    rng = random.Random(100000 * case["lo"] + case["hi"])
    return [rng.randint(case["lo"], case["hi"]) for _ in range(case["events"])]


def _total_hits(case, n):
    """Hits of the batch: the signal's (13.5 a track at most on barrel + disks) and the noise fraction."""
    return int(n * (13.5 if case["disks"] else case["layers"]) * (1 + case.get("overlap", 0)) * (1 + case["noise"]))


def _total_seeds(n):
    """Seeds of n tracks with overlap hits: 1.3^3 a track on average, with room below for chance."""
    return int(n * (1.3 ** 3 - 6.4 / math.sqrt(n)))


# ---- events ---------------------------------------------------------------------------------------

def _draw_events(case, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    U = lambda n, lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    N = lambda n: torch.randn(n, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    sizes = torch.tensor(_event_sizes(case), device="cuda")
    n, ns = int(sizes.sum()), len(d.surfaces)
    ev = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), sizes)
    th = 2 * torch.atan(torch.exp(-U(n, -d.eta, d.eta)))
    zero = torch.zeros(n, dtype=torch.float64, device="cuda")
    p = torch.stack([zero, zero, zero, torch.sign(U(n, -1, 1)) / U(n, 0.5, 10.0), U(n, -math.pi, math.pi), th])
    rec = []  # per surface: tracks, phi, second coordinate
    z2, r2, eloss = getattr(d, "field_z2", 0.0), getattr(d, "field_r2", 0.0), getattr(d, "eloss", 0.0)
    field = lambda p: d.bz * (1 + z2 * p[2] ** 2 + r2 * (p[0] ** 2 + p[1] ** 2))  # noqa: E731
    for s in d.surfaces:
        q, ok = _to_surface(s, field(p), p)
        if z2 or r2:  # the field halfway
            q, ok = _to_surface(s, field(torch.where(ok, 0.5 * (p + q), p)), p)
        v = q[2] if s.type == 0 else torch.hypot(q[0], q[1])
        ok &= (v >= s.lo) & (v <= s.hi)
        if s.x_over_x0 > 0:  # scattering: the direction turns, the momentum stays
            cos_a = torch.cos(q[5]).abs() if s.type else torch.sin(q[5]) * (q[0] * torch.cos(q[4]) + q[1] * torch.sin(q[4])) / s.r_or_z
            x = s.x_over_x0 * ((1 + 2 * (v / s.hi) ** 2) if eloss else 1.0) / cos_a.abs()
            t0 = _highland(q, x)
            th2 = q[5] + N(n) * t0
            q = torch.stack([q[0], q[1], q[2], q[3] * torch.sin(q[5]) / torch.sin(th2), _wrap(q[4] + N(n) * t0 / torch.sin(q[5])), th2])
            if eloss:  # of a pion
                mom = 1 / (q[3] * torch.sin(th2)).abs()
                left = (torch.sqrt(mom ** 2 + 0.13957 ** 2) - eloss * x).clamp(min=0.2)
                q[3] *= mom / torch.sqrt(left ** 2 - 0.13957 ** 2)
        at = torch.nonzero(ok).squeeze(1)
        rho = torch.hypot(q[0], q[1])
        phi = torch.atan2(q[1], q[0]) + N(n) * d.sigma_rphi / rho
        rec.append((at, phi[at], (v + N(n) * d.sigma_2nd)[at], rho[at]))
        p = torch.where(ok, q, p)
    trk, phi, v = (torch.cat([r[k] for r in rec]) for k in (0, 1, 2))
    surf = torch.cat([torch.full_like(r[0], s) for s, r in enumerate(rec)])
    own = torch.ones_like(trk)  # 1: first hit of its track on the surface, 2: overlap hit, 0: noise
    if case.get("overlap", 0):
        at = torch.nonzero(U(len(trk), 0, 1) < case["overlap"]).squeeze(1)
        rho = torch.cat([r[3] for r in rec])[at]
        off = U(len(at), 0.2, 0.5) * torch.sign(U(len(at), -1, 1)) / rho
        trk, phi, v, surf = (torch.cat([a, a[at]]) for a in (trk, phi, v, surf))
        phi = torch.cat([phi[:-len(at)], phi[-len(at):] + off])
        own = torch.cat([own, torch.full_like(at, 2)])
    slab = ev[trk] * ns + surf
    extra = _total_hits(case, n) - len(slab) if "noise" in case else 0
    if extra > 0:  # noise like the signal's occupancy, up to the batch's total
        count = torch.cumsum(torch.bincount(slab, minlength=len(sizes) * ns), 0)
        share = torch.diff(count * extra // count[-1], prepend=torch.zeros(1, dtype=torch.int64, device="cuda"))
        extra = torch.repeat_interleave(torch.arange(len(sizes) * ns, device="cuda"), share)
        lo = torch.tensor([s.lo for s in d.surfaces], device="cuda", dtype=torch.float64)[extra % ns]
        hi = torch.tensor([s.hi for s in d.surfaces], device="cuda", dtype=torch.float64)[extra % ns]
        disk = torch.tensor([s.type for s in d.surfaces], device="cuda")[extra % ns] == 1
        u = U(len(extra), 0, 1)
        w = torch.where(disk, torch.sqrt(lo * lo + u * (hi * hi - lo * lo)), lo + u * (hi - lo))
        slab, v, phi = torch.cat([slab, extra]), torch.cat([v, w]), torch.cat([phi, U(len(extra), -math.pi, math.pi)])
        trk, own = torch.cat([trk, torch.full_like(extra, -1)]), torch.cat([own, torch.zeros_like(extra)])
    # hits grouped by (event, surface), in random order within
    order = torch.argsort(slab * (1 << 32) + torch.randint(1 << 32, (len(slab),), generator=g, device="cuda"))
    slab, trk, own = slab[order], trk[order], own[order]
    hits = torch.stack([_wrap(phi[order]).clamp(-math.pi, math.pi), v[order]], 1).float().contiguous()
    offs = torch.zeros(len(sizes) * ns + 1, dtype=torch.int64, device="cuda")
    offs[1:] = torch.cumsum(torch.bincount(slab, minlength=len(sizes) * ns), 0)
    # hit lists in path order, a track's surfaces being crossed in index order
    table = torch.full((3, n, ns), -1, dtype=torch.int64, device="cuda")
    ids = torch.arange(len(slab), device="cuda")
    table[own, trk.clamp(min=0), slab % ns] = ids
    first, twin = table[1], table[2]
    rank = torch.argsort(torch.where(first >= 0, torch.arange(ns, device="cuda"), ns + torch.arange(ns, device="cuda")), 1)[:, :d.lmax]
    lists, twins = torch.gather(first, 1, rank), torch.gather(twin, 1, rank[:, :3])
    keep = torch.nonzero(lists[:, 2] >= 0).squeeze(1)
    lists, twins, ev = lists[keep], twins[keep], ev[keep]
    seeds, sev = lists[:, :3], ev
    if case.get("overlap", 0):  # one seed per combination of a track's hits on its first three surfaces
        pick = torch.stack([lists[:, :3], twins], 0)
        every = torch.stack([torch.stack([pick[(c >> k) & 1, :, k] for k in range(3)], 1) for c in range(8)], 1)
        valid = (every >= 0).all(2)
        seeds, sev = every[valid], ev[:, None].expand(-1, 8)[valid]
        some = torch.randperm(len(sev), generator=g, device="cuda")[:_total_seeds(len(ev))].sort()[0]
        seeds, sev = seeds[some], sev[some]
    i32 = lambda t: t.to(torch.int32).contiguous()  # noqa: E731
    return dict(hits=hits, surface=i32(slab % ns), offsets=i32(offs), lists=i32(lists.T), seeds=i32(seeds.T),
                seed_event=i32(sev), largest=int((offs[1:] - offs[:-1]).max()))


# ---- helix and filter in 64 bits (the inputs above, and exact() below) ----------------------------------

def _wrap(a):
    return torch.remainder(a + math.pi, 2 * math.pi) - math.pi


def _highland(p, x):
    return 0.0136 * p[3].abs() * torch.sin(p[5]) * torch.sqrt(x) * (1 + 0.038 * torch.log(x))


def _to_surface(s, bz, p):
    """State p [6, n] (x, y, z, q/pT, phi, theta) moved along its helix to surface s; and whether it gets there."""
    x, y, z, k, phi, th = p
    w, cot = -CURV * bz * k, torch.cos(th) / torch.sin(th)
    c, sn = torch.cos(phi), torch.sin(phi)
    if s.type:
        t = (s.r_or_z - z) / cot
        ok = (t > 0) & ((w * t).abs() < math.pi)
    else:
        d0 = x * x + y * y - s.r_or_z ** 2
        a, b = x * c + y * sn, y * c - x * sn
        disc = a * a - (1 + w * b) * d0
        t = -d0 / (a + torch.sqrt(disc.clamp(min=0)))
        for _ in range(8):
            h = 0.5 * w * t
            f = torch.sinc(h / math.pi)
            dx, dy = t * f * torch.cos(phi + h), t * f * torch.sin(phi + h)
            g = d0 + 2 * (x * dx + y * dy) + dx * dx + dy * dy
            t = t - g / (2 * ((x + dx) * torch.cos(phi + 2 * h) + (y + dy) * torch.sin(phi + 2 * h)))
        ok = (disc > 0) & (t > 0) & (g.abs() < 1e-3)
    h = 0.5 * w * t
    f = torch.sinc(h / math.pi)
    return torch.stack([x + t * f * torch.cos(phi + h), y + t * f * torch.sin(phi + h), z + t * cot, k, _wrap(phi + 2 * h), th]), ok


def _predict(s, d, p, C):
    """State and covariance [n, 6, 6] on the barrel layer s, with the layer's scattering."""
    q, ok = _to_surface(s, d.bz, p)
    a = -CURV * d.bz
    w, n = a * p[3], p.shape[1]
    st, cot = torch.sin(p[5]), torch.cos(p[5]) / torch.sin(p[5])
    t = torch.where(cot.abs() > 1e-9, (q[2] - p[2]) / torch.where(cot.abs() > 1e-9, cot, torch.ones_like(cot)), torch.zeros_like(cot))
    turn = _wrap(q[4] - p[4])
    t = torch.where(cot.abs() > 1e-6, t, turn / w)
    dx, dy = q[0] - p[0], q[1] - p[1]
    # d(dx, dy)/d omega at fixed t, by series in the turning angle where the closed form cancels
    D = w * t
    small = D.abs() < 1e-2
    Ds = torch.where(small, torch.ones_like(D), D)
    f1 = torch.where(small, D * (-1 / 3 + D ** 2 / 30 - D ** 4 / 840), (torch.cos(Ds) - torch.sin(Ds) / Ds) / Ds)
    f2 = torch.where(small, 0.5 - D ** 2 / 8 + D ** 4 / 144, (torch.sin(Ds) - (1 - torch.cos(Ds)) / Ds) / Ds)
    c, sn = torch.cos(p[4]), torch.sin(p[4])
    J = torch.eye(6, dtype=torch.float64, device=p.device).repeat(n, 1, 1)
    J[:, 0, 4], J[:, 1, 4], J[:, 2, 5], J[:, 4, 3] = -dy, dx, -t / st ** 2, a * t
    J[:, 0, 3], J[:, 1, 3] = a * t * t * (c * f1 - sn * f2), a * t * t * (sn * f1 + c * f2)
    tan = torch.stack([torch.cos(q[4]), torch.sin(q[4]), cot, torch.zeros_like(w), w, torch.zeros_like(w)], 1)
    grad = torch.stack([q[0], q[1]], 1)
    gt = (grad * tan[:, :2]).sum(1)
    P = torch.eye(6, dtype=torch.float64, device=p.device).repeat(n, 1, 1)
    P[:, :, :2] -= tan[:, :, None] * (grad / gt[:, None])[:, None, :]
    J = P @ J
    C = J @ C @ J.transpose(1, 2)
    if s.x_over_x0 > 0:
        var = _highland(q, s.x_over_x0 / (st * gt / s.r_or_z).abs()) ** 2
        C[:, 5, 5] += var
        C[:, 4, 4] += var / st ** 2
        C[:, 3, 5] -= q[3] * cot * var
        C[:, 5, 3] -= q[3] * cot * var
        C[:, 3, 3] += (q[3] * cot) ** 2 * var
    return q, C, ok


def _measure(s, d, p, C):
    """Rows of H over (x, y, z), C H^T and the innovation covariance on the barrel layer s."""
    H = torch.zeros(p.shape[1], 2, 6, dtype=torch.float64, device=p.device)
    rho2 = p[0] ** 2 + p[1] ** 2
    H[:, 0, 0], H[:, 0, 1], H[:, 1, 2] = -s.r_or_z * p[1] / rho2, s.r_or_z * p[0] / rho2, 1.0
    CH = C @ H.transpose(1, 2)
    S = H @ CH
    S[:, 0, 0] += float(np.float32(d.sigma_rphi)) ** 2
    S[:, 1, 1] += float(np.float32(d.sigma_2nd)) ** 2
    return H, CH, S


def _residual(s, p, phi, v):
    return torch.stack([s.r_or_z * _wrap(phi - torch.atan2(p[1], p[0])), v - p[2]], -1)


def _inverse2(S):
    det = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] * S[:, 1, 0]
    return torch.stack([S[:, 1, 1], -S[:, 0, 1], -S[:, 1, 0], S[:, 0, 0]], 1).reshape(-1, 2, 2) / det[:, None, None]


def _update(s, d, p, C, phi, v):
    H, CH, S = _measure(s, d, p, C)
    K, r = CH @ _inverse2(S), _residual(s, p, phi, v)
    q = p + (K @ r[:, :, None])[:, :, 0].T
    chi2 = (r[:, None, :] @ _inverse2(S) @ r[:, :, None])[:, 0, 0]
    return torch.cat([q[:4], _wrap(q[4:5]), q[5:]]), C - K @ CH.transpose(1, 2), chi2


def _seed(d, hits, surface, ids):
    """State and prior at the first of three hits: the circle through them, the line in arc length and z."""
    r = torch.tensor([s.r_or_z for s in d.surfaces], dtype=torch.float64, device="cuda")
    R = r[surface[ids].long()]
    x, y, z = R * torch.cos(hits[ids, 0]), R * torch.sin(hits[ids, 0]), hits[ids, 1]
    ax, ay, bx, by = x[1] - x[0], y[1] - y[0], x[2] - x[0], y[2] - y[0]
    lb = torch.hypot(bx, by)
    w = 2 * (ax * by - ay * bx) / (torch.hypot(ax, ay) * lb * torch.hypot(x[2] - x[1], y[2] - y[1]))
    half = torch.asin(0.5 * lb * w)
    arc = lb / torch.sinc(half / math.pi)
    p = torch.stack([x[0], y[0], z[0], -w / (CURV * d.bz), _wrap(torch.atan2(by, bx) - half), torch.atan2(arc, z[2] - z[0])])
    su, s2, *rest = (float(np.float32(v)) ** 2 for v in d.prior)
    C = torch.zeros(len(lb), 6, 6, dtype=torch.float64, device="cuda")
    u = torch.stack([-y[0], x[0]], 1) / torch.hypot(x[0], y[0])[:, None]
    C[:, :2, :2] = su * u[:, :, None] * u[:, None, :]
    for i, v in zip((2, 3, 4, 5), (s2, *rest)):
        C[:, i, i] = v
    return p, C


def _packed(C):
    i, j = torch.triu_indices(6, 6, device=C.device)
    return C[:, i, j].T


def _fit64(d, e, lists):
    """Fit over hit lists [lmax, n] on barrel layers; {state, cov, chi2}, 200,000 tracks at a time."""
    hits, out = e["hits"].double(), []
    for part in lists.long().split(200000, 1):
        p, C = _seed(d, hits, e["surface"], part[:3])
        chi2 = torch.zeros(part.shape[1], dtype=torch.float64, device="cuda")
        for k in range(len(part)):
            here = e["surface"][part[k].clamp(min=0)].long()
            for si in torch.unique(here[part[k] >= 0]).tolist():  # found lists may skip a layer
                at = torch.nonzero((part[k] >= 0) & (here == si)).squeeze(1)
                s, q, D = d.surfaces[si], p[:, at], C[at]
                if k:
                    q, D, _ = _predict(s, d, q, D)
                h = hits[part[k, at]]
                q, D, c = _update(s, d, q, D, h[:, 0], h[:, 1])
                p[:, at], C[at] = q, D
                chi2[at] += c
        out.append((p, _packed(C), chi2))
    return dict(state=torch.cat([o[0] for o in out], 1), cov=torch.cat([o[1] for o in out], 1), chi2=torch.cat([o[2] for o in out]))


def _find64(d, e, k_max):
    """Beam search of one event's barrel seeds against every hit of each layer: {hits, state, cov, chi2}."""
    hits, out = e["hits"].double(), []
    for ids in e["seeds"].long().split(500, 1):
        n, dev = ids.shape[1], "cuda"
        p, C = _seed(d, hits, e["surface"], ids)
        chi2 = torch.zeros(n, dtype=torch.float64, device=dev)
        for k in range(3):
            s = d.surfaces[k]
            if k:
                p, C, _ = _predict(s, d, p, C)
            p, C, c = _update(s, d, p, C, hits[ids[k], 0], hits[ids[k], 1])
            chi2 += c
        # candidates [n, k_max]: state, covariance, chi2, hits, misses, stopped, list; slot 0 is the seed's
        S = n * k_max
        P, V = p[:, :, None].repeat(1, 1, k_max).reshape(6, S), C[:, None].repeat(1, k_max, 1, 1).reshape(S, 6, 6)
        X = chi2[:, None].repeat(1, k_max).reshape(S)
        live = (torch.arange(S, device=dev) % k_max) == 0
        nh, nm = torch.full((S,), 3, device=dev), torch.zeros(S, dtype=torch.int64, device=dev)
        stop = torch.zeros(S, dtype=torch.bool, device=dev)
        lists = torch.full((S, d.lmax), -1, device=dev)
        lists[:, :3] = ids.T.repeat_interleave(k_max, 0)
        for step in range(3, d.lmax):
            s = d.surfaces[step]
            a, b = int(e["offsets"][step]), int(e["offsets"][step + 1])
            Q, W, ok = _predict(s, d, P, V)
            ok &= live & ~stop & (Q[2] >= s.lo) & (Q[2] <= s.hi)
            Q, W = torch.where(ok, Q, P), torch.where(ok[:, None, None], W, V)
            I = _inverse2(_measure(s, d, Q, W)[2])
            dphi = _wrap(hits[None, a:b, 0] - torch.atan2(Q[1], Q[0])[:, None]) * s.r_or_z
            dz = hits[None, a:b, 1] - Q[2][:, None]
            c2 = I[:, 0, 0, None] * dphi * dphi + 2 * I[:, 0, 1, None] * dphi * dz + I[:, 1, 1, None] * dz * dz
            c2 = torch.where((c2 < CHI2_CUT) & ok[:, None], c2, torch.full_like(c2, math.inf))
            kk = min(k_max, b - a)
            best, at = torch.topk(c2, kk, 1, largest=False)
            hit = torch.isfinite(best)
            none = ~hit[:, 0] & live
            miss = none & ok & (nm < 1)
            # children [S, kk + 1]: the hits, then a miss or the candidate carried on
            cn = torch.cat([nh[:, None] + hit.long(), nh[:, None]], 1)
            cx = torch.cat([X[:, None] + best, X[:, None]], 1)
            valid = torch.cat([hit, none[:, None]], 1)
            key = torch.where(valid, -1e9 * cn.double() + cx, torch.full_like(cx, math.inf)).reshape(n, -1)
            key, pick = torch.topk(key, k_max, 1, largest=False)
            par = (pick // (kk + 1) + k_max * torch.arange(n, device=dev)[:, None]).reshape(S)
            child = (pick % (kk + 1)).reshape(S)
            live = torch.isfinite(key).reshape(S)
            by_hit = live & (child < kk)
            gone = (live & ~by_hit & ~miss[par]) | (stop[par] & ~by_hit)
            h = torch.where(by_hit, at[par, child.clamp(max=kk - 1)] + a, torch.zeros_like(par))
            U, Y, _ = _update(s, d, Q[:, par], W[par], hits[h, 0], hits[h, 1])
            P = torch.where(by_hit, U, torch.where(gone, P[:, par], Q[:, par]))
            V = torch.where(by_hit[:, None, None], Y, torch.where(gone[:, None, None], V[par], W[par]))
            X, nh = cx[par, child], cn[par, child]
            nm = nm[par] + (live & ~by_hit & ~gone).long()
            stop = gone
            lists = lists[par]
            lists[:, step] = torch.where(by_hit, h, torch.full_like(h, -1))
        best = torch.arange(n, device=dev) * k_max
        out.append((lists[best].T, P[:, best], _packed(V[best]), X[best]))
    return dict(zip(("hits", "state", "cov", "chi2"), (torch.cat([o[i] for o in out], -1) for i in range(4))))


def _index64(d, e):
    """Search records (cos phi, sin phi, second coordinate) in the index's order: slab, bin, phi sub-bin, id."""
    phi, v = e["hits"][:, 0], e["hits"][:, 1]
    col = lambda f: torch.tensor([f(s) for s in d.surfaces], dtype=torch.float32, device="cuda")[e["surface"].long()]  # noqa: E731
    turn = phi + np.float32(math.pi).item()
    fine = (turn * np.float32(512 / (2 * math.pi)).item()).floor().long().clamp(0, 511)
    pb = (turn * np.float32(64 / (2 * math.pi)).item()).floor().long().clamp(0, 63)
    vb = ((v - col(lambda s: s.lo)) * col(lambda s: 32 / (float(np.float32(s.hi)) - float(np.float32(s.lo))))).floor().long().clamp(0, 31)
    slab = torch.bucketize(torch.arange(len(phi), device="cuda"), e["offsets"].long()[1:], right=True)
    order = torch.argsort(((slab * 64 + pb) * 32 + vb) * 8 + (fine - 8 * pb).clamp(0, 7), stable=True)
    return torch.stack([torch.cos(phi.double()), torch.sin(phi.double()), v.double()], 1)[order]


# ---- network ------------------------------------------------------------------------------------------

def _trained(disks):
    z = np.load(os.path.join(os.path.dirname(kf.__file__), "data", "mlp_hi_occ.npz" if disks else "mlp_learned.npz"))
    return z["weights"], z["mean"], z["sd"]


def _net_inputs(case, seed):
    """Rows around the normaliser's mean, labels, and a training state in mid-course."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    R = lambda *n: torch.randn(*n, generator=g, device="cuda")  # noqa: E731
    w, mean, sd = _trained(True)
    m, s = torch.from_numpy(mean).cuda(), torch.from_numpy(sd).cuda()
    rows = (m + s * R(case["rows"], 14)).contiguous()
    labels = (torch.rand(case["rows"], generator=g, device="cuda") < 0.4).float()
    m1 = 1e-3 * R(kf.MLP_PARAMS)
    m2 = (2e-3 * (0.5 + torch.rand(kf.MLP_PARAMS, generator=g, device="cuda"))) ** 2
    return dict(params=kf.mlp_buffer(w, mean, sd), rows=rows, labels=labels, m=m1, v=m2)


def _net64(params, rows, labels=None):
    """Logits; with labels the mean loss and its gradient too, 500,000 rows at a time."""
    f = params.double()
    W1, b1, W2, b2, W3, b3 = f[:896].reshape(64, 14), f[896:960], f[960:5056].reshape(64, 64), f[5056:5120], f[5120:5184], f[5184]
    mean, sd = f[5185:5199], f[5199:5213]
    logits, loss, grad = [], 0.0, 0.0
    for x, y in zip(rows.split(500000), labels.split(500000) if labels is not None else [None] * (len(rows) // 500000 + 1)):
        x = (x.double() - mean) / sd
        h1 = torch.relu(x @ W1.T + b1)
        h2 = torch.relu(h1 @ W2.T + b2)
        z = h2 @ W3 + b3
        logits.append(z)
        if y is None:
            continue
        y = y.double()
        loss = loss + (torch.nn.functional.softplus(z) - z * y).sum()
        g = torch.sigmoid(z) - y
        e2 = g[:, None] * W3 * (h2 > 0)
        e1 = (e2 @ W2) * (h1 > 0)
        grad = grad + torch.cat([(e1.T @ x).reshape(-1), e1.sum(0), (e2.T @ h1).reshape(-1), e2.sum(0), h2.T @ g, g.sum()[None]])
    return torch.cat(logits) if labels is None else (loss / len(rows), grad / len(rows))


# ---- the cases ----------------------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "net":
        s = _net_inputs(case, seed)
        s.update(call=case["call"], grad=torch.empty(kf.MLP_PARAMS, device="cuda"), loss=torch.empty(1, device="cuda"), step=100)
        return s
    d = _detector(case)
    e = _draw_events(case, d, seed)
    s = dict(e, kind=case["kind"], n_events=case["events"], geom=kf.Geometry(d))
    if case["kind"] == "fit":
        s["fit"] = _track_buffers(e["lists"].shape[1])
        return s
    s["index"] = kf.HitIndex(s["geom"], case["events"], len(e["hits"]))
    if case["kind"] == "events":
        n = e["seeds"].shape[1]
        net = kf.mlp_buffer(*_trained(case["disks"])) if case["top_n"] else None
        s["keep"] = torch.empty(n, dtype=torch.int32, device="cuda") if case["overlap"] else None
        steer = _steering(d) if case["option"] in ("steering", "all") else None
        s["params"] = kf.find_params(CHI2_CUT, case["k"], 1, d.lmax, mlp=net, top_n=case["top_n"], score_margin=case["margin"],
                                     adaptive_capacity=case["adaptive"], steering_tables=steer, seed_keep=s["keep"])
        s["found"], s["fit"] = _track_buffers(n, d.lmax), _track_buffers(n)
        s["space"] = torch.empty(max(256, kf.find_workspace_size(n, s["params"])), dtype=torch.uint8, device="cuda")
        if case["overlap"]:
            size = max(kf.dedup_workspace_size(n, 3, len(e["hits"])), kf.dedup_workspace_size(n, d.lmax, len(e["hits"])))
            s["dups"], s["unique"] = torch.empty(size, dtype=torch.uint8, device="cuda"), torch.empty_like(s["keep"])
    return s


def _track_buffers(n, lmax=0):
    f, i = dict(dtype=torch.float32, device="cuda"), dict(dtype=torch.int32, device="cuda")
    b = dict(state=torch.empty((6, n), **f), cov=torch.empty((21, n), **f), chi2=torch.empty(n, **f), status=torch.empty(n, **i))
    b.update(dict(hits=torch.empty((lmax, n), **i), nhits=torch.empty(n, **i)) if lmax else dict(ndof=torch.empty(n, **i)))
    return b


def _tracks(b):
    return {k: b[k] for k in b if k != "workspace"}


def run(s):
    if "call" in s:
        if s["call"] == "score":
            return kf.mlp_forward(s["params"], s["rows"])
        loss, grad = kf.mlp_loss_grad(s["params"], s["rows"], s["labels"], s["grad"], s["loss"])
        if s["call"] == "loss":
            return dict(loss=loss, grad=grad)
        s["step"] += 1
        kf.mlp_adam(s["params"], grad, s["m"], s["v"], s["step"])
        return dict(loss=loss, grad=grad, params=s["params"], m=s["m"], v=s["v"])
    if s["kind"] == "fit":
        return kf.fit_tracks(s["geom"], s["hits"], s["surface"], s["lists"], out=s["fit"])
    if s.get("keep") is not None:
        kf.clean_seeds(s["geom"], s["hits"], s["surface"], s["seeds"], s["seed_event"], keep=s["keep"], workspace=s["dups"])
    ix = kf.build_hit_index(s["geom"], s["hits"], s["offsets"], s["n_events"], s["largest"], index=s["index"])
    if s["kind"] == "index":
        return dict(bin_off=ix.bin_off, sub_off=ix.sub_off, sorted_hits=ix.sorted_hits, sorted_ids=ix.sorted_ids,
                    record=ix.sorted_rec[:, :3], record_id=ix.sorted_rec.view(torch.int32)[:, 3])
    found = kf.find_tracks(s["geom"], ix, s["hits"], s["surface"], s["seeds"], s["seed_event"], s["params"], out=s["found"],
                           workspace=s["space"])
    out = dict(found=_tracks(found))
    if s.get("keep") is not None:
        out["keep"] = s["keep"]
        out["unique"] = kf.remove_duplicates(found["hits"], found["nhits"], found["chi2"], found["state"], s["seed_event"],
                                             len(s["hits"]), keep=s["unique"], workspace=s["dups"])
    out["fit"] = kf.fit_tracks(s["geom"], s["hits"], s["surface"], found["hits"], out=s["fit"])
    return out


def work(case):
    if case["kind"] == "net":
        n = case["rows"]
        if case["call"] == "score":
            return dict(bytes=60 * n + 4 * 5213, flops=10112 * n)
        return dict(bytes=60 * n + 4 * 5213 * (2 if case["call"] == "loss" else 7), flops=28416 * n)
    n, disks = sum(_event_sizes(case)), case.get("disks", False)
    per = 12 if disks else case["layers"]  # hits of a track
    lmax = case["layers"] + (9 if disks else 0)
    fit = dict(bytes=n * (12 * per + 4 * lmax + 120), flops=n * (340 + 730 * (per - 1)))
    if case["kind"] == "fit":
        return fit
    hits = _total_hits(case, n)
    slabs = case["events"] * (case["layers"] + (18 if disks else 0))
    index = dict(bytes=36 * hits + slabs * (4 * 2049 + 16 * 2048), flops=20 * hits)
    if case["kind"] == "index":
        return index
    n = _total_seeds(n) if case["overlap"] else n
    # propagations a seed: every kept candidate at every layer, fewer where the network prunes
    props = (1.6 * per if case["top_n"] == 0 else per) if disks else min(case["k"], 4) * (per - 3)
    net = 3.6 * 10112 if case["top_n"] else 0
    find = dict(bytes=n * (4 * lmax + 16 + 120), flops=n * (800 + props * 470 + 1.1 * props * 260 + 40 * props + net))
    return {k: index[k] + find[k] + fit[k] for k in ("bytes", "flops")}


def tolerance(case):
    """About four times what 32-bit results measure against exact()."""
    if case["kind"] == "net":
        # measured: logits 6.6e-7, a step's state 1e-5 (its squares' moment), a set's gradient 2.3e-5
        return {"score": {"rel": 3e-6, "max": 2e-5}, "step": {"rel": 4e-5, "max": 1e-4}, "loss": {"rel": 1e-4, "max": 3e-4}}[case["call"]]
    if case["kind"] == "index":
        return {"rel": 2e-7, "max": 1e-6}
    if case["kind"] == "fit":
        return {"rel": 1e-4, "max": 1e-3}  # measured on chi2: 2.3e-5 and 2e-4
    # the same where every decision falls the same way; a seed whose candidates nearly tie may take
    # another track when a sum rounds otherwise (one in 10,000 and fewer)
    return {"rel": 1e-2, "max": 0.999, "differ": 1e-3}


def exact(case, seed):
    if case["kind"] == "net":
        s = _net_inputs(case, seed)
        if case["call"] == "score":
            return _net64(s["params"], s["rows"])
        loss, g = _net64(s["params"], s["rows"], s["labels"])
        out = dict(loss=loss[None], grad=g)
        if case["call"] == "step":
            m, v = 0.9 * s["m"].double() + 0.1 * g, 0.999 * s["v"].double() + 0.001 * g * g
            p = s["params"].double()
            p[:5185] -= 1e-3 * (m / (1 - 0.9 ** 101)) / (torch.sqrt(v / (1 - 0.999 ** 101)) + 1e-8)
            out.update(params=p, m=m, v=v)
        return out
    d = _detector(case)
    e = _draw_events(case, d, seed)
    if case["kind"] == "fit":
        return dict(_fit64(d, e, e["lists"]), ndof=None, status=None)
    if case["kind"] == "index":
        return dict(sorted_hits=None, record=_index64(d, e))
    # finding against every hit of a layer takes too long for more than one event, and is written
    # for barrel layers without options; the seeds of overlapping modules are cleaned first
    if case["events"] > 1 or case["disks"] or case["option"] or case["top_n"] or case["overlap"] or sum(_event_sizes(case)) > 6000:
        return None
    found = _find64(d, e, case["k"])
    fit = _fit64(d, e, found["hits"])
    return dict(found=dict(found, hits=None), fit=fit)
