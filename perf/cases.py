"""Performance cases of listmode TOF PET reconstruction with LM-SPDHG.

Each case is one call (or the calls of one step) that a reconstruction
program makes through the public binding, on the scanners and grids of this
repository's benchmark: the 2D ring (256 crystals on 300 mm, 128 x 128 voxels
of 2 mm) and the 3D scanner (36 rings x 672 crystals on 410 mm, 200 x 200 x 96
voxels of 2.5 mm), both with a 400 ps TOF kernel cut at 3 sigma.  The inputs are
made from the seed alone: a Monte Carlo of positron annihilations in an
ellipsoid with hot and cold spheres, detected with attenuation and timing
noise, plus 20 % of events uniform over (LOR, TOF bin).

Kinds of case:
  fwd    P^LM x of an event list              (operators: scatter estimates, checks, other algorithms)
  back   (P^LM)^T v of an event list
  sens   the sensitivity image P^T 1          (once per scanner and attenuation map)
  epoch  2n updates of Alg. 2 on one frame    (the reconstruction's loop)
  frame  set-up, initialisation, epochs and objective of one frame
  batch  one epoch of several frames together (dynamic studies, serving)
  emtv   one listmode EM-TV pass (Alg. 3)     (the warm start)
"""
import functools
import math

import numpy as np
import torch

from paper_2201_05497_gb300 import lm

MU = 0.0096  # 1/mm, attenuation of the body
F64 = torch.float64
TWO_D = {"rings": 1, "xtal": 256, "nx": 128, "ny": 128, "nz": 1}
THREE_D = {"rings": 36, "xtal": 672, "nx": 200, "ny": 200, "nz": 96}


def listed():
    d2, d3 = TWO_D, THREE_D
    return [
        # one subset of the 2D frame: the smallest call, where latency and launches count
        {"name": "fwd_2d_subset", "kind": "fwd", **d2, "events": 7143},
        # one subset of the 1e7-event frame through the operators, as other algorithms call them
        {"name": "fwd_3d_subset", "kind": "fwd", **d3, "events": 357143},
        {"name": "back_3d_subset", "kind": "back", **d3, "events": 357143},
        # P^T 1 of the 3D scanner with the attenuation of every LOR
        {"name": "sens_3d", "kind": "sens", **d3},
        # the 2D frame (launch-bound: 7143 events per update)
        {"name": "epoch_2d", "kind": "epoch", **d2, "events": 200000, "subsets": 28, "beta": 0.03, "dtv": False,
         "fwhm": 0.0},
        # a short dynamic frame on the 3D grid (mostly image passes)
        {"name": "epoch_3d_dynamic", "kind": "epoch", **d3, "events": 200000, "subsets": 28, "beta": 0.03, "dtv": False,
         "fwhm": 0.0},
        # the 3D short frame
        {"name": "epoch_3d_short", "kind": "epoch", **d3, "events": 10000000, "subsets": 28, "beta": 0.03, "dtv": False,
         "fwhm": 0.0},
        # a long acquisition: large subsets, 1.1e6 events per update
        {"name": "epoch_3d_long", "kind": "epoch", **d3, "events": 60000000, "subsets": 56, "beta": 0.01, "dtv": False,
         "fwhm": 0.0},
        # the options of the model: resolution in the projector, directional prior
        {"name": "epoch_3d_model", "kind": "epoch", **d3, "events": 2000000, "subsets": 28, "beta": 0.1, "dtv": True,
         "fwhm": 4.5},
        # a dynamic frame from its raw events to x: the median of a stream of 1e5 to 2e7 events, 10 epochs
        {"name": "frame_3d", "kind": "frame", **d3, "events": 1400000, "subsets": 28, "beta": 0.03, "epochs": 10},
        # eight dynamic frames advanced together
        {"name": "batch_3d", "kind": "batch", **d3, "events": 200000, "events_last": 3000000, "frames": 8, "subsets": 28,
         "beta": 0.03},
        # warm start of a 3D frame
        {"name": "emtv_3d", "kind": "emtv", **d3, "events": 3000000, "subsets": 28, "beta": 0.03, "iters": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, two_d):
    if two_d:
        n = rng.choice([rng.randrange(64, 129, 4), rng.randrange(65, 129)])
        return {**TWO_D, "nx": n, "ny": n + rng.randrange(-15, 1)}
    if rng.random() < 0.5:  # the scanner's own grid, or one that covers a part of it
        return dict(THREE_D)
    k = rng.choice([4, 1])  # rows a multiple of four voxels, or any
    return {**THREE_D, "nx": rng.randrange(25, 50) * 4 + rng.randrange(4) // k, "ny": rng.randrange(25, 50) * 4 + rng.randrange(4) // k,
            "nz": rng.randrange(48, 97)}


def draw(rng):
    kind = rng.choice(["fwd", "back", "sens", "epoch", "epoch", "epoch", "frame", "batch", "emtv"])
    two_d = rng.random() < 0.25
    c = {"kind": kind, **_grid(rng, two_d)}
    if kind == "sens":
        if not two_d:
            c["rings"], c["xtal"] = rng.randrange(8, 37), 4 * rng.randrange(64, 169)
        return c
    hi = {"fwd": 2000000, "back": 2000000, "epoch": 40000000, "frame": 4000000, "batch": 1000000, "emtv": 10000000}[kind]
    c["events"] = _log(rng, 5000, 50000) if two_d and kind in ("fwd", "back") else _log(
        rng, 50000, min(hi, 1000000) if two_d else hi)
    if kind in ("fwd", "back"):
        return c
    c["subsets"] = rng.choice([14, 28, 28, 56])
    c["beta"] = rng.choice([0.01, 0.03, 0.1])
    if kind == "epoch":
        c["dtv"] = rng.random() < 0.25
        c["fwhm"] = round(rng.uniform(3.5, 6.0), 2) if c["events"] < 5000000 and rng.random() < 0.25 else 0.0
    if kind == "frame":
        c["epochs"] = rng.randrange(2, 11)
    if kind == "batch":
        c["frames"] = rng.randrange(2, 9)
        c["events_last"] = 2 * c["events"] + rng.randrange(1000)
    if kind == "emtv":
        c["iters"] = 20
    return c


# ---- inputs ------------------------------------------------------------------
class _Setup:
    """Scanner, grid and TOF parameters of a case (host numbers, crystals on the device)."""

    def __init__(self, rings, xtal, nx, ny, nz):
        self.two_d = rings == 1
        self.rings, self.xtal, self.n = rings, xtal, (nx, ny, nz)
        self.radius = 300.0 if self.two_d else 410.0
        self.pitch = 1.0 if self.two_d else 250.0 / 36
        h = 2.0 if self.two_d else 2.5
        self.h = (h, h, h)
        self.origin = tuple(float(np.float32(-0.5 * (m - 1) * h)) for m in self.n)
        self.sigma = float(np.float32(400.0 * 0.299792458 / 2.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))))
        self.bin = float(np.float32(600.0 / 27))
        self.n_bins = 27 if self.two_d else 41
        phi = 2.0 * np.pi * np.arange(xtal) / xtal
        z = (np.arange(rings) - 0.5 * (rings - 1)) * self.pitch if rings > 1 else np.zeros(1)
        tab = np.stack([np.tile(self.radius * np.cos(phi), rings), np.tile(self.radius * np.sin(phi), rings),
                        np.repeat(z, xtal)], 1)
        self.crystals = torch.from_numpy(tab.astype(np.float32)).cuda()
        # the body: 0.38 x 0.26 of the grid's extent, attenuating a little further out
        self.body = (0.38 * nx * h, 0.26 * ny * h, 0.48 * nz * h)
        self.att = (0.42 * nx * h, 0.30 * ny * h)
        b = self.body
        self.spots = [((0.3 * b[0], 0.2 * b[1], 0.2 * b[2]), 0.20 * b[0], 4.0), ((-0.4 * b[0], 0.1 * b[1], -0.3 * b[2]), 0.25 * b[0], 0.2),
                      ((0.0, -0.4 * b[1], 0.1 * b[2]), 0.15 * b[0], 3.0), ((-0.1 * b[0], 0.4 * b[1], 0.4 * b[2]), 0.12 * b[0], 2.0)]
        self.V = nx * ny * nz
        self.n_lor = xtal * (xtal - 1) // 2 * rings * rings
        self.knorm = math.sqrt(sum(4 * math.sin(math.pi * (m - 1) / (2 * m)) ** 2 for m in self.n if m > 1))

    def geometry(self):
        return lm.Geometry(self.crystals, self.rings, self.xtal, self.n, self.h, self.origin, self.sigma, self.bin, 3.0,
                           self.n_bins)

    def activity(self, p):
        """Activity at points p [m, 3]."""
        r = (p[:, 0] / self.body[0]) ** 2 + (p[:, 1] / self.body[1]) ** 2
        if not self.two_d:
            r = r + (p[:, 2] / self.body[2]) ** 2
        act = (r <= 1).to(p.dtype)
        for c, rad, a in self.spots:
            q = (p[:, 0] - c[0]) ** 2 + (p[:, 1] - c[1]) ** 2
            if not self.two_d:
                q = q + (p[:, 2] - c[2]) ** 2
            act = torch.where((q <= rad * rad) & (r <= 1), torch.full_like(act, a), act)
        return act

    def chord(self, ax, ay, dx, dy):
        """Part of the line a + t d inside the attenuating cylinder, in units of t."""
        al = (dx / self.att[0]) ** 2 + (dy / self.att[1]) ** 2
        be = 2 * (ax * dx / self.att[0] ** 2 + ay * dy / self.att[1] ** 2)
        ga = (ax / self.att[0]) ** 2 + (ay / self.att[1]) ** 2 - 1
        return torch.sqrt(torch.clamp(be * be - 4 * al * ga, min=0)) / al

    def image(self):
        """Activity at the voxel centres (float32, x fastest)."""
        ax = [torch.arange(m, device="cuda", dtype=torch.float32) * h + o for m, h, o in zip(self.n, self.h, self.origin)]
        z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        return self.activity(torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1))


@functools.lru_cache(maxsize=4)
def _setup(rings, xtal, nx, ny, nz):
    return _Setup(rings, xtal, nx, ny, nz)


def _of(case):
    return _setup(case["rings"], case["xtal"], case["nx"], case["ny"], case["nz"])


def _pairs(xtal):
    """Transaxial crystal pairs in the library's canonical order."""
    q = torch.arange(xtal * (xtal - 1) // 2, device="cuda")
    base = xtal * ((xtal - 1) // 2)
    c1 = torch.where(q < base, q % xtal, q - base)
    c2 = (c1 + torch.where(q < base, 1 + q // xtal, torch.full_like(q, xtal // 2))) % xtal
    return c1, c2


@functools.lru_cache(maxsize=2)
def _lor_factor(S):
    """exp(-mu chord) of every canonical LOR (float32)."""
    c1, c2 = _pairs(S.xtal)
    a, b = S.crystals[c1].to(F64), S.crystals[c2].to(F64)
    d = b - a
    t, lxy = S.chord(a[:, 0], a[:, 1], d[:, 0], d[:, 1]), torch.hypot(d[:, 0], d[:, 1])
    z = S.crystals[:: S.xtal, 2].to(F64)
    dz = (z[None, :] - z[:, None]).reshape(-1)
    out = torch.empty(S.n_lor, dtype=torch.float32, device="cuda").view(-1, S.rings * S.rings)
    for s in range(0, len(t), 8192):
        out[s:s + 8192] = torch.exp(-MU * t[s:s + 8192, None] * torch.hypot(lxy[s:s + 8192, None], dz[None])).float()
    return out.view(-1)


@functools.lru_cache(maxsize=4)
def _sens_image(S):
    """The sensitivity image a program has at hand: P^T 1 with the axial part
    of the LORs tabulated over 48 positions along the line (within a few per
    cent of the exact one)."""
    nx, ny, nz = S.n
    nt = 48
    c1, c2 = _pairs(S.xtal)
    h = torch.zeros(nx * ny * nt, dtype=F64, device="cuda")
    for s in range(0, len(c1), 32768):
        a, b = S.crystals[c1[s:s + 32768], :2].to(F64), S.crystals[c2[s:s + 32768], :2].to(F64)
        d = b - a
        att = torch.exp(-MU * S.chord(a[:, 0], a[:, 1], d[:, 0], d[:, 1]) * torch.hypot(d[:, 0], d[:, 1]))
        for k in (0, 1):
            m = (d[:, 0].abs() >= d[:, 1].abs()) == (k == 0)
            ak, bk, dk = a[m], b[m], d[m]
            o = 1 - k
            i = torch.arange(S.n[k], device="cuda")
            t = (S.origin[k] + S.h[k] * i[None] - ak[:, k:k + 1]) / dk[:, k:k + 1]
            u = (ak[:, o:o + 1] + t * dk[:, o:o + 1] - S.origin[o]) / S.h[o]
            w = (att[m] * S.h[k] * torch.hypot(dk[:, 0], dk[:, 1]) / dk[:, k].abs())[:, None] * ((t >= 0) & (t <= 1))
            f = torch.floor(u)
            tb = torch.clamp((t * nt).long(), 0, nt - 1)
            for e, we in ((0, 1 - (u - f)), (1, u - f)):
                j = f.long() + e
                ok = (j >= 0) & (j < S.n[o])
                v = (i[None] + j * nx) if k == 0 else (j + i[None] * nx)
                h.index_add_(0, (v * nt + tb)[ok], (w * we)[ok])
    if S.two_d:
        return h.view(nx * ny, nt).sum(1).float()
    z = S.crystals[:: S.xtal, 2].to(F64)
    t = (torch.arange(nt, device="cuda", dtype=F64) + 0.5) / nt
    zz = z[None, :, None] + t[:, None, None] * (z[None, None, :] - z[None, :, None])
    obl = torch.hypot(z[None, None, :] - z[None, :, None], torch.tensor(0.9 * 2 * S.radius, dtype=F64, device="cuda"))
    u = (zz - S.origin[2]) / S.h[2]
    prof = torch.zeros(nt, nz, dtype=F64, device="cuda")
    for iz in range(nz):
        prof[:, iz] = (torch.clamp(1 - (u - iz).abs(), min=0) * obl / (0.9 * 2 * S.radius)).sum((1, 2))
    return (prof.t() @ h.view(nx * ny, nt).t()).reshape(-1).float().contiguous()


def _events(S, n, seed):
    """n listmode events (det1, det2, tof, corr, contam) on the device."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def U(m, lo, hi):
        return torch.rand(m, generator=g, device="cuda") * (hi - lo) + lo

    R, M = S.radius, S.n_bins // 2
    half = 0.5 * S.rings * S.pitch
    n_true = n - n // 5
    got, parts = 0, []
    m = 1 << (25 if n > 300000 else 22)
    while got < n_true:
        p = torch.stack([U(m, -S.body[0], S.body[0]), U(m, -S.body[1], S.body[1]), U(m, -S.body[2], S.body[2])], 1)
        if S.two_d:
            p[:, 2] = 0
        p = p[U(m, 0.0, 4.0) < S.activity(p)]
        phi = U(len(p), 0.0, math.pi)
        ux, uy = torch.cos(phi), torch.sin(phi)
        pu = p[:, 0] * ux + p[:, 1] * uy
        sq = torch.sqrt(pu * pu - p[:, 0] ** 2 - p[:, 1] ** 2 + R * R)
        lo, hi = -pu - sq, sq - pu
        keep = U(len(p), 0.0, 1.0)
        if S.two_d:
            uz = torch.zeros_like(ux)
        else:
            # slope of the line: uniform over those that hit the scanner at both ends, weighted to isotropic directions
            z = p[:, 2]
            s_lo = torch.maximum((-half - z) / hi, (half - z) / lo)
            s_hi = torch.minimum((half - z) / hi, (-half - z) / lo)
            uz = s_lo + U(len(p), 0.0, 1.0) * (s_hi - s_lo)
            keep = keep / torch.clamp((s_hi - s_lo) / 0.8 * (1 + uz * uz) ** -1.5, min=1e-6)
        keep = keep < torch.exp(-MU * S.chord(p[:, 0], p[:, 1], ux, uy) * torch.sqrt(1 + uz * uz))
        ends = []
        for s in (lo, hi):
            ang = torch.atan2(p[:, 1] + s * uy, p[:, 0] + s * ux) * (S.xtal / (2 * math.pi))
            c = torch.round(ang).int() % S.xtal
            r = torch.zeros_like(c) if S.two_d else torch.clamp(((p[:, 2] + s * uz + half) / S.pitch).int(), 0, S.rings - 1)
            ends.append(r * S.xtal + c)
        keep &= ends[0] % S.xtal != ends[1] % S.xtal
        p, a, b = p[keep], ends[0][keep], ends[1][keep]
        A, B = S.crystals[a], S.crystals[b]
        t = ((p - 0.5 * (A + B)) * (B - A)).sum(1) / (B - A).norm(dim=1)
        t = t + S.sigma * torch.randn(len(t), generator=g, device="cuda")
        parts.append((a, b, torch.clamp(torch.round(t / S.bin), -M, M).short()))
        got += len(a)
    det1, det2, tof = (torch.cat([q[k] for q in parts])[:n_true] for k in range(3))
    # contamination, uniform over (LOR, TOF bin), shuffled in
    k = n - n_true
    c1 = torch.randint(0, S.xtal, (k,), generator=g, device="cuda", dtype=torch.int32)
    c2 = (c1 + torch.randint(1, S.xtal, (k,), generator=g, device="cuda", dtype=torch.int32)) % S.xtal
    r = [torch.randint(0, S.rings, (k,), generator=g, device="cuda", dtype=torch.int32) for _ in range(2)]
    order = torch.randperm(n, generator=g, device="cuda")
    det1 = torch.cat([det1, r[0] * S.xtal + c1])[order]
    det2 = torch.cat([det2, r[1] * S.xtal + c2])[order]
    tof = torch.cat([tof, torch.randint(-M, M + 1, (k,), generator=g, device="cuda").short()])[order]
    swap = U(n, 0.0, 1.0) < 0.5  # the detector order of an event is arbitrary
    det1, det2 = torch.where(swap, det2, det1), torch.where(swap, det1, det2)
    tof = torch.where(swap, -tof, tof)
    corr = torch.empty(n, device="cuda")
    for s in range(0, n, 1 << 22):
        A, B = S.crystals[det1[s:s + (1 << 22)]].to(F64), S.crystals[det2[s:s + (1 << 22)]].to(F64)
        D = B - A
        corr[s:s + (1 << 22)] = torch.exp(-MU * S.chord(A[:, 0], A[:, 1], D[:, 0], D[:, 1]) * D.norm(dim=1)).float()
    contam = torch.full((n,), k / (S.n_lor * S.n_bins), device="cuda")
    return lm.DeviceEvents(det1.contiguous(), det2.contiguous(), tof.contiguous(), corr, contam)


def _noisy_image(S, seed):
    """An image on the way to convergence: the activity with 20 % noise."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return S.image() * (0.8 + 0.4 * torch.rand(S.V, generator=g, device="cuda")) + 0.01


def _start_image(S, n):
    """Uniform x0: the expected true counts spread over the sensitivity."""
    return torch.full((S.V,), float(np.float32(0.8 * n / float(_sens_image(S).double().sum()))), device="cuda")


def _sequence(n, seed):
    """2n selections: the prior (n) or a data subset with equal probability."""
    rng = np.random.default_rng(seed)
    return np.where(rng.random(2 * n) < 0.5, n, rng.integers(0, n, 2 * n)).astype(np.uint16)


def _counts(case):
    f = case["frames"]
    r = case["events_last"] / case["events"]
    return [int(round(case["events"] * r ** (i / max(1, f - 1)))) for i in range(f)]


def _structure(S):
    """Structural image of the directional prior: the activity, contrast flipped."""
    img = S.image()
    return img.max() - img


def _eta(S):
    return 0.04  # 1 % of the largest step of the structural image


class _State:
    pass


def prepare(case, seed):
    S = _of(case)
    s = _State()
    s.kind, s.geo = case["kind"], S.geometry()
    if s.kind == "sens":
        # another seed: another patient (the attenuation scaled by a per cent or so)
        s.lf = _lor_factor(S) * (1.0 + 0.01 * (seed % 97) / 97)
        return s
    if s.kind == "batch":
        evs = [_events(S, k, seed + i) for i, k in enumerate(_counts(case))]
    else:
        evs = [_events(S, case["events"], seed)]
    if s.kind in ("fwd", "back"):
        s.ev = evs[0]
        if s.kind == "fwd":
            s.x = _noisy_image(S, seed)
        else:  # the dual change of an update: both signs, a few large ones
            g = torch.Generator(device="cuda")
            g.manual_seed(seed + 1)
            s.v = torch.randn(s.ev.n, generator=g, device="cuda") ** 3
        return s
    n = case["subsets"]
    sens = _sens_image(S)
    s.seq = [_sequence(n, seed + 7 * i) for i in range(max(case.get("epochs", 1), case.get("frames", 1)))]
    if s.kind == "emtv":
        s.pe, s.x0, s.sens = lm.event_setup(s.geo, evs[0], n), _start_image(S, evs[0].n), sens
        s.beta, s.iters, s.knorm = case["beta"], case["iters"], S.knorm
        s.ws = lm._emtv_ws(s.geo, None, sens.device)
        return s
    xi = None
    if case.get("dtv"):
        xi = lm.dtv_field(s.geo, _structure(S), _eta(S))
    s.rec = []
    for ev in evs:
        pe = lm.event_setup(s.geo, ev, n)
        # the frames of a batch share one lane-group width (the server's); a lone frame's is found at creation
        s.rec.append(lm.LMSPDHG(s.geo, pe, sens, _start_image(S, ev.n), beta=case["beta"], n_subsets=n, knorm=S.knorm, xi=xi,
                                res_fwhm=case.get("fwhm", 0.0), group=32 if s.kind == "batch" else 0))
    if s.kind == "frame":
        s.ev, s.x0, s.n = evs[0], _start_image(S, evs[0].n), n
        s.ws = torch.empty(int(lm.load_library().lm_setup_workspace_bytes(s.ev.n)), dtype=torch.uint8, device="cuda")
    if s.kind == "batch":
        s.batch = lm.Batch(len(evs), n)
        for i, r in enumerate(s.rec):
            s.batch.set(i, r)
    return s


def _updated(r):
    return {"x": r.x(), "y": r.y(), "z": r.z(), "w": r.w()}


def run(s):
    if s.kind == "fwd":
        return lm.fwd(s.geo, s.x, s.ev)
    if s.kind == "back":
        return lm.back(s.geo, s.v, s.ev)
    if s.kind == "sens":
        return lm.sens(s.geo, s.lf)
    if s.kind == "emtv":
        return lm.emtv_epoch(s.geo, s.pe, s.sens, s.x0.clone(), beta=s.beta, pdhg_iters=s.iters, knorm=s.knorm, ws=s.ws)
    if s.kind == "batch":
        s.batch.epoch(np.stack(s.seq))
        return [_updated(r) for r in s.rec]
    r = s.rec[0]
    if s.kind == "epoch":
        r.epoch(s.seq[0])
        return _updated(r)
    # frame: the raw events of a new frame into the buffers of the last one
    pe = lm.event_setup(s.geo, s.ev, s.n, into=r.pe, ws=s.ws)
    r.reinit(s.x0)
    for q in s.seq:
        r.epoch(q)
    return {"objective": r.objective(), "mu": pe.mu, **_updated(r)}


# ---- what a pass cannot do without ---------------------------------------------
def _samples(S):
    """Samples of an event: the planes of its 6 sigma TOF window inside the grid,
    on average over directions (0.74 of the window's length in voxels: measured
    46 of 62 on the 3D grid)."""
    return 0.74 * 6 * S.sigma / S.h[0]


def work(case):
    S = _of(case)
    V, kind = S.V, case["kind"]
    taps = 2 if S.two_d else 4
    nd = 2 if S.two_d else 3
    sample = 12 + 2 * taps  # flops of a sample's position and weights
    proj = _samples(S) * (sample + 2 * taps)
    if kind == "sens":
        # the LORs that meet the grid (about 0.6), over its extent along them
        return {"bytes": 4.0 * S.n_lor + 4.0 * V, "flops": 0.6 * S.n_lor * 0.6 * S.n[0] * (sample + 2 * taps)}
    N = float(sum(_counts(case)) if kind == "batch" else case["events"])
    if kind in ("fwd", "back"):
        return {"bytes": 18.0 * N + 4.0 * V, "flops": N * proj}
    n = case["subsets"]
    frames = case.get("frames", 1)
    # an event of a data update: detectors, TOF bin, c, s, mu, y read, y written; both projections share the weights
    ev_b, ev_f = 28.0, _samples(S) * (sample + 4 * taps) + 20
    if kind == "emtv":
        # z, w, u, ubar, q read, u, ubar, q written by each inner iteration
        it = n * case["iters"] * V
        return {"bytes": 22.0 * N + n * 16.0 * V + it * 4.0 * (6 + 2 * nd), "flops": N * ev_f + it * 8.0 * nd}
    # an epoch: n data and n prior updates on average; x, z and its compensation read and written, T, w
    img_b = n * V * 4.0 * (7 + 7 + 2 * nd) * frames
    img_f = n * V * (20.0 + 20.0 * nd) * frames
    if case.get("dtv"):
        img_b += n * V * 4.0 * nd
    if case.get("fwhm"):
        taps_r = 2 * int(3 * case["fwhm"] / 2.3548 / S.h[0] + 0.5) + 1
        img_b += 3 * n * V * 8.0  # G x after every update, G A^T v of the data updates
        img_f += 3 * n * V * 2.0 * taps_r * nd
    if kind == "frame":
        e = case["epochs"]
        return {"bytes": N * (18 + 20) + e * (N * ev_b + img_b), "flops": N * (2 + e) * ev_f + e * img_f}
    return {"bytes": N * ev_b + img_b, "flops": N * ev_f + img_f}


# ---- the same in 64 bits ---------------------------------------------------------
class _Exact:
    """Projector, TV and the updates of Alg. 2 and 3 in float64 with torch."""

    def __init__(self, case):
        self.S = S = _of(case)
        self.xy = S.crystals.to(F64)
        self.h = [float(np.float32(v)) for v in S.h]
        self.W = 3.0 * S.sigma
        self.axes = [d for d in range(3) if S.n[d] > 1]

    def _window(self, det1, det2, m, nk):
        """Traversal of the events: per (event, plane) voxel base, weights."""
        S = self.S
        a, b = self.xy[det1], self.xy[det2]
        d = b - a
        ad = (S.crystals[det2] - S.crystals[det1]).abs()
        k = torch.where(ad[:, 1] > ad[:, 0], 1, 0)
        k = torch.where(ad[:, 2] > torch.maximum(ad[:, 0], ad[:, 1]), 2, k)
        ka, kb = torch.where(k == 0, 1, 0), torch.where(k == 2, 1, 2)
        take = lambda v, j: v.gather(1, j[:, None])[:, 0]  # noqa: E731
        h, o = torch.tensor(self.h, dtype=F64, device="cuda"), torch.tensor(S.origin, dtype=F64, device="cuda")
        n = torch.tensor(S.n, device="cuda")
        st = torch.tensor([1, S.n[0], S.n[0] * S.n[1]], device="cuda")
        c = a + 0.5 * d
        L = d.norm(dim=1)
        dk = take(d, k)
        mu0, dmu = (o[k] - take(c, k)) / dk, h[k] / dk
        tau0, dtau = mu0 * L - m * S.bin, dmu * L
        lo = torch.floor(torch.minimum((-self.W - tau0) / dtau, (self.W - tau0) / dtau)).long()
        i = lo[:, None] + torch.arange(nk, device="cuda")[None]
        tau = tau0[:, None] + i * dtau[:, None]
        s2 = math.sqrt(2.0) * S.sigma
        w = 0.5 * (torch.erf((tau + 0.5 * S.bin) / s2) - torch.erf((tau - 0.5 * S.bin) / s2))
        w *= (tau.abs() <= self.W) & (i >= 0) & (i < n[k][:, None])
        w *= (h[k] * L / dk.abs())[:, None]
        mu = mu0[:, None] + i * dmu[:, None]
        out = [(i * st[k][:, None], w)]
        for j in (ka, kb):
            u = (take(c, j)[:, None] + mu * take(d, j)[:, None] - o[j][:, None]) / h[j][:, None]
            f = torch.floor(u)
            fi, r = f.long(), u - f
            nxt = []
            for base, wt in out:
                for e, we in ((0, 1 - r), (1, r)):
                    g = fi + e
                    ok = (g >= 0) & (g < n[j][:, None])
                    nxt.append((base + torch.where(ok, g, 0) * st[j][:, None], wt * we * ok))
            out = nxt
            if S.two_d:
                break
        return [(torch.where(w != 0, base, 0), w) for base, w in out]

    def chunks(self, ev, lo=0, hi=None):
        hi = ev.n if hi is None else hi
        nk = int(2 * self.W / min(self.h)) + 3
        for s in range(lo, hi, 1 << 18):
            e = slice(s, min(hi, s + (1 << 18)))
            yield e, self._window(ev.det1[e].long(), ev.det2[e].long(), ev.tof[e].to(F64), nk)

    def project(self, ev, win, e, x):
        return ev.corr[e].to(F64) * sum((w * x[b]).sum(1) for b, w in win)

    def spread(self, ev, win, e, v, img):
        cv = (ev.corr[e].to(F64) * v)[:, None]
        for b, w in win:
            img.index_add_(0, b.reshape(-1), (w * cv).reshape(-1))

    def grad(self, x):
        S = self.S
        v = x.view(S.n[2], S.n[1], S.n[0])
        out = []
        for d in self.axes:
            g = torch.zeros_like(v)
            k = 2 - d
            g.narrow(k, 0, S.n[d] - 1).copy_(v.narrow(k, 1, S.n[d] - 1) - v.narrow(k, 0, S.n[d] - 1))
            out.append(g.reshape(-1))
        return torch.stack(out)

    def grad_t(self, q):
        S = self.S
        out = torch.zeros(S.n[2], S.n[1], S.n[0], dtype=F64, device="cuda")
        for c, d in enumerate(self.axes):
            v = q[c].view(S.n[2], S.n[1], S.n[0])
            k = 2 - d
            g = v.narrow(k, 0, S.n[d] - 1)
            out.narrow(k, 0, S.n[d] - 1).sub_(g)
            out.narrow(k, 1, S.n[d] - 1).add_(g)
        return out.reshape(-1)

    def blur(self, x, fwhm):
        """Separable Gaussian, mirrored about the outer faces."""
        S = self.S
        v = x.view(S.n[2], S.n[1], S.n[0])
        for d in self.axes:
            sd = fwhm / (2 * math.sqrt(2 * math.log(2))) / self.h[d]
            r = min(int(3 * sd + 0.5), S.n[d] - 1)
            t = torch.exp(-0.5 * (torch.arange(-r, r + 1, dtype=F64) / sd) ** 2)
            t = t / t.sum()
            i = torch.arange(-r, S.n[d] + r, device="cuda")
            i = torch.where(i < 0, -1 - i, torch.where(i >= S.n[d], 2 * S.n[d] - 1 - i, i))
            p = v.index_select(2 - d, i)
            v = sum(float(t[j]) * p.narrow(2 - d, j, S.n[d]) for j in range(2 * r + 1))
        return v.reshape(-1)

    def field(self):
        g = self.grad(_structure(self.S).to(F64))
        eta = float(np.float32(_eta(self.S)))
        return g / torch.sqrt((g * g).sum(0) + eta * eta)


class _ExactFrame:
    """Alg. 2 on one frame."""

    def __init__(self, X, ev, pe, case, x0):
        self.X, self.n = X, case["subsets"]
        n_ev = ev.n
        order = torch.cat([torch.arange(i, n_ev, self.n, device="cuda") for i in range(self.n)])
        self.ev = lm.DeviceEvents(ev.det1[order], ev.det2[order], ev.tof[order], ev.corr[order], ev.contam[order])
        self.off = np.cumsum([0] + [len(range(i, n_ev, self.n)) for i in range(self.n)])
        lo, hi = torch.minimum(ev.det1, ev.det2).long(), torch.maximum(ev.det1, ev.det2).long()
        tb = torch.where(ev.det1 < ev.det2, ev.tof, -ev.tof).long()
        key = (lo * X.S.rings * X.S.xtal + hi) * 256 + tb + 128
        srt, at = torch.sort(key)
        _, cnt = torch.unique_consecutive(srt, return_counts=True)
        mu = torch.empty_like(key)
        mu[at] = torch.repeat_interleave(cnt, cnt)
        self.mu = mu[order]
        self.fwhm = case.get("fwhm", 0.0)
        self.xi = X.field() if case.get("dtv") else None
        self.beta = float(np.float32(case["beta"]))
        rho, kn = float(np.float32(0.999)), X.S.knorm
        self.gamma = 3.0 / float(x0.max())
        self.rho, self.kn = rho, kn
        sens = _sens_image(X.S).to(F64)
        self.sens = sens
        n = self.n
        self.T = torch.clamp(rho / (2 * n) / self.gamma / (sens / n), max=0.5 * rho / (self.gamma * kn))
        x0 = x0.to(F64)
        self.y = torch.empty(n_ev, dtype=F64, device="cuda")
        back = torch.zeros(X.S.V, dtype=F64, device="cuda")
        gx = self.G(x0)
        for e, w in X.chunks(self.ev):
            u = X.project(self.ev, w, e, gx) + self.ev.contam[e]
            self.y[e] = 1 - self.mu[e] / u
            X.spread(self.ev, w, e, -1 / u, back)
        self.z = sens + self.G(back)
        self.zbar = self.z
        self.w = torch.zeros(len(X.axes), X.S.V, dtype=F64, device="cuda")
        self.xn, self.x = x0, x0

    def G(self, x):
        return self.X.blur(x, self.fwhm) if self.fwhm else x

    def K(self, x):
        g = self.X.grad(x)
        return g if self.xi is None else g - self.xi * (self.xi * g).sum(0)

    def KT(self, q):
        return self.X.grad_t(q if self.xi is None else q - self.xi * (self.xi * q).sum(0))

    def epoch(self, seq):
        X, ev, n = self.X, self.ev, self.n
        for k in seq:
            x = self.x = self.xn = torch.clamp(self.xn - self.T * self.zbar, min=0)
            if k == n:
                v = self.w + self.gamma * self.rho / self.kn * self.K(x)
                r = v.norm(dim=0)
                wn = v / torch.clamp(r / self.beta, min=1)
                dz, p = self.KT(wn - self.w), 0.5
                self.w = wn
            else:
                dz, p = torch.zeros_like(x), 1 / (2 * n)
                gx = self.G(x)
                for e, win in X.chunks(ev, int(self.off[k]), int(self.off[k + 1])):
                    p1 = ev.corr[e].to(F64) * sum(w.sum(1) for _, w in win)
                    Se = torch.where(p1 > 0, self.gamma * self.rho / p1, 0)
                    a = self.y[e] + Se * (X.project(ev, win, e, gx) + ev.contam[e])
                    yn = 0.5 * (a + 1 - torch.sqrt((a - 1) ** 2 + 4 * self.mu[e] * Se))
                    X.spread(ev, win, e, (yn - self.y[e]) / self.mu[e], dz)
                    self.y[e] = yn
                dz = self.G(dz)
            self.z = self.z + dz
            self.zbar = self.z + dz / p

    def out(self):
        return {"x": self.x, "y": self.y, "z": self.z, "w": self.w.reshape(-1)}

    def objective(self):
        gx = self.G(self.x)
        lg = sum(float(torch.log(self.X.project(self.ev, w, e, gx) + self.ev.contam[e]).sum()) for e, w in self.X.chunks(self.ev))
        return float((self.sens * self.x).sum()) - lg + self.beta * float(self.K(self.x).norm(dim=0).sum())


def _exact_emtv(X, ev, case, x):
    S, n = X.S, case["subsets"]
    sens, x = _sens_image(S).to(F64), x.to(F64)
    beta = float(np.float32(case["beta"]))
    for i in range(n):
        sub = lm.DeviceEvents(ev.det1[i::n], ev.det2[i::n], ev.tof[i::n], ev.corr[i::n], ev.contam[i::n])
        b = torch.zeros(S.V, dtype=F64, device="cuda")
        for e, w in X.chunks(sub):
            X.spread(sub, w, e, 1 / (X.project(sub, w, e, x) + sub.contam[e]), b)
        z = torch.where(sens > 0, x * n / sens * b, 0)
        free = (x > 0) & (sens > 0)
        w = torch.where(free, sens / (beta * x), 0)
        gam = float(w[free].min())
        u = ub = torch.where(free, z, 0)
        q = torch.zeros(len(X.axes), S.V, dtype=F64, device="cuda")
        tau = sigma = 0.99 / S.knorm
        for _ in range(case["iters"]):
            q = q + sigma * X.grad(ub)
            q = q / torch.clamp(q.norm(dim=0), min=1)
            th = 1 / math.sqrt(1 + 2 * gam * tau)
            un = torch.where(free, torch.clamp((u - tau * X.grad_t(q) + tau * w * z) / (1 + tau * w), min=0), 0)
            un = torch.nan_to_num(un)  # weights that overflow belong to voxels that vanish
            ub, u = un + th * (un - u), un
            tau, sigma = tau * th, sigma / th
        x = u
    return x


def _exact_sens(S, lf):
    """P^T 1 over every LOR and TOF bin."""
    X = torch.zeros(S.V, dtype=F64, device="cuda")
    c1, c2 = _pairs(S.xtal)
    R, M, W = S.rings, S.n_bins // 2, 3.0 * S.sigma
    s2 = math.sqrt(2.0) * S.sigma
    nx, ny, nz = S.n
    z = S.crystals[:: S.xtal, 2].to(F64)
    z1, z2 = z.repeat_interleave(R), z.repeat(R)
    lf = lf.view(-1, R * R).to(F64)
    step = max(1, (1 << 20) // (R * R))
    h = S.h[0]
    for s in range(0, len(c1), step):
        a, b = S.crystals[c1[s:s + step], :2].to(F64), S.crystals[c2[s:s + step], :2].to(F64)
        d = b - a
        ky = (S.crystals[c2[s:s + step], 1] - S.crystals[c1[s:s + step], 1]).abs() > (
            S.crystals[c2[s:s + step], 0] - S.crystals[c1[s:s + step], 0]).abs()
        for k in (0, 1):
            m = ky == (k == 1)
            if not bool(m.any()):
                continue
            ak, dk, o = a[m], d[m], 1 - k
            i = torch.arange(S.n[k], device="cuda")
            t = (S.origin[k] + h * i[None] - ak[:, k:k + 1] - 0.5 * dk[:, k:k + 1]) / dk[:, k:k + 1]  # [q, plane] from the centre
            u = (ak[:, o:o + 1] + (t + 0.5) * dk[:, o:o + 1] - S.origin[o]) / h
            f = torch.floor(u)
            near = ((f >= -1) & (f < S.n[o])).nonzero(as_tuple=True)
            qi, ii = near
            tt, uu, ff = t[near], u[near], f[near].long()
            L = torch.sqrt((dk ** 2).sum(1)[:, None] + (z2 - z1)[None] ** 2)[qi]   # [sample, ring pair]
            tau = tt[:, None] * L
            lo = torch.clamp(torch.ceil((tau - W) / S.bin), min=-M)
            hi = torch.clamp(torch.floor((tau + W) / S.bin), max=M)
            w = 0.5 * (torch.erf((tau - (lo - 0.5) * S.bin) / s2) - torch.erf((tau - (hi + 0.5) * S.bin) / s2)) * (lo <= hi)
            w *= lf[s:s + step][m][qi] * h * L / dk[qi, k].abs()[:, None]
            uz = (z1[None] + (tt + 0.5)[:, None] * (z2 - z1)[None] - S.origin[2]) / S.h[2]
            if nz == 1:
                prof = w.sum(1, keepdim=True)
            else:
                fz = torch.floor(uz)
                prof = torch.zeros(len(tt), nz + 2, dtype=F64, device="cuda")
                iz = torch.clamp(fz.long() + 1, 0, nz + 1)
                prof.scatter_add_(1, iz, w * (1 - (uz - fz)) * ((fz >= 0) & (fz < nz)))
                prof.scatter_add_(1, torch.clamp(iz + 1, max=nz + 1), w * (uz - fz) * ((fz >= -1) & (fz < nz - 1)))
                prof = prof[:, 1:nz + 1]
            for e, we in ((0, 1 - (uu - ff)), (1, uu - ff)):
                j = ff + e
                ok = (j >= 0) & (j < S.n[o])
                v = (i[ii] + j * nx) if k == 0 else (j + i[ii] * nx)
                X.view(nz, nx * ny).index_add_(1, v[ok], (prof * we[:, None])[ok].t().contiguous())
    return X


def exact(case, seed):
    S, kind = _of(case), case["kind"]
    if kind == "sens":
        if S.n_lor * max(S.n) > 1.5e10:  # too long in 64 bits
            return None
        return _exact_sens(S, _lor_factor(S) * (1.0 + 0.01 * (seed % 97) / 97))
    X = _Exact(case)
    if kind == "batch":
        evs = [_events(S, k, seed + i) for i, k in enumerate(_counts(case))]
    else:
        evs = [_events(S, case["events"], seed)]
    ev = evs[0]
    if kind == "fwd":
        x = _noisy_image(S, seed).to(F64)
        return torch.cat([X.project(ev, w, e, x) for e, w in X.chunks(ev)])
    if kind == "back":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        v = torch.randn(ev.n, generator=g, device="cuda") ** 3
        img = torch.zeros(S.V, dtype=F64, device="cuda")
        for e, w in X.chunks(ev):
            X.spread(ev, w, e, v[e].to(F64), img)
        return img
    if kind == "emtv":
        return _exact_emtv(X, ev, case, _start_image(S, ev.n))
    n = case["subsets"]
    seqs = [_sequence(n, seed + 7 * i) for i in range(max(case.get("epochs", 1), case.get("frames", 1)))]
    if kind == "batch":
        out = []
        for e, q in zip(evs, seqs):
            f = _ExactFrame(X, e, None, case, _start_image(S, e.n))
            f.epoch(q)
            out.append(f.out())
        return out
    f = _ExactFrame(X, ev, None, case, _start_image(S, ev.n))
    for q in (seqs if kind == "frame" else seqs[:1]):
        f.epoch(q)
    if kind == "frame":
        return {"objective": f.objective(), "mu": f.mu, **f.out()}
    return f.out()
