"""Workloads by which the speed of the map-maker is judged, and their results in
plain 64-bit torch.

A case is one call (or one short sequence of calls) that a user of the library
makes, on a synthetic scan of the kind the library is for: constant-elevation
drift scans with a rising and a setting half, 0.3 pixels per sample, detectors on
a hexagonal focal plane, noise 1 + (f/f_knee)^-3.5 with scattered levels, flat-sky
TQU (or T) maps.  The detector angles, noise levels, skies and data all come from
the seed.

kinds
  apply         A m = P^T N^-1 P m, the product every solver iteration makes
  solve         a preconditioned conjugate-gradient solve, as a user calls it
  rhs           P^T N^-1 d of stored time-ordered data, once per data set
  project       P m, synthesis of time-ordered data from a map
  precon_build  the circulant preconditioner built for a scan, and applied
  precon_apply  the circulant preconditioner applied
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

DEV = "cuda:0"
PX_PER_SAMPLE = 0.3      # 1 deg/s at 400 Hz on 0.5' pixels
F_SAMP = 400.0
ALPHA = 3.5
PREC = {"f64": 0, "f32": 1}


def _case(name, kind, n_det, log_nt, ny, nx, **more):
    c = {"kind": kind, "n_det": n_det, "log_nt": log_nt, "ny": ny, "nx": nx, "ncomp": 3, "prec": "f32",
         "corr": 0, "table": False, "precon": "circulant", "taper": 10.0, "iters": 0, "tol": 0.0}
    assert set(more) <= set(c)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest patch (32 detectors, 64 x 64): one operator product, bound by latency
        _case("tiny_apply", "apply", 32, 16, 64, 64),
        # the same patch solved to 1e-6 in double precision, the plain FP64 PCG of small studies
        _case("tiny_solve_f64", "solve", 32, 16, 64, 64, prec="f64", taper=8.0, iters=200, tol=1e-6),
        # the small corner of the Monte-Carlo batches: one product, and 20 iterations of a solve
        _case("patch_apply", "apply", 128, 18, 256, 256),
        _case("patch_solve", "solve", 128, 18, 256, 256, iters=20),
        # a mid-size patch after detector cuts: an odd number of detectors
        _case("ragged_apply", "apply", 301, 19, 360, 480),
        # double precision on a mid-size patch: the product that checks the FP32 modes
        _case("apply_f64", "apply", 48, 18, 240, 320, prec="f64"),
        # atmosphere: noise correlated between the detectors through three focal-plane modes
        _case("corr_apply", "apply", 192, 19, 450, 600, corr=3),
        # the data of a mid-size patch into the right-hand side, and a sky into data
        _case("rhs", "rhs", 256, 19, 450, 600),
        _case("project", "project", 512, 19, 600, 800),
        # the set-up every solve pays, and the preconditioner of the full-size map by itself
        _case("precon_build", "precon_build", 256, 19, 450, 600),
        _case("precon_apply", "precon_apply", 64, 20, 900, 1200),
        # the full-size patch (1024 detectors x 2^20 samples, 1200 x 900): ten iterations
        _case("act_solve", "solve", 1024, 20, 900, 1200, iters=10),
    ]


def _smooth(lo, hi):
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


SIDES = _smooth(45, 1200)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "rhs", "project", "precon_build", "precon_apply"])
    prec = "f64" if kind in ("apply", "solve") and rng.random() < 0.25 else "f32"
    n_det = int(round(math.exp(rng.uniform(math.log(24), math.log(320)))))
    log_nt = rng.randint(14, 17 if prec == "f64" else 19)
    if prec == "f64":
        n_det = min(n_det, 96)
    # 60 to 1500 samples on a pixel, sides of 2, 3 and 5 between 45 and 900 x 1200
    npix = n_det * 2 ** log_nt / math.exp(rng.uniform(math.log(60), math.log(1500)))
    npix = min(max(npix, 48.0 ** 2), 900.0 * 1200.0)
    aspect = math.exp(rng.uniform(math.log(0.75), math.log(1.4)))
    near = lambda v, hi: min((s for s in SIDES if s <= hi), key=lambda s: abs(s - v))  # noqa: E731
    ny, nx = near(math.sqrt(npix / aspect), 900), near(math.sqrt(npix * aspect), 1200)
    ncomp = 1 if rng.random() < 0.2 else 3
    more = {}
    if kind == "apply":
        if prec == "f32" and ncomp == 3 and rng.random() < 0.2:
            more["corr"] = rng.randint(1, 3)
        elif rng.random() < 0.25:
            more["table"] = True
    if kind == "solve":
        more["precon"] = rng.choice(["circulant", "circulant", "binned"])
        more["iters"] = rng.randint(5, 20)
    if kind in ("solve", "precon_build", "precon_apply"):
        more["taper"] = float(rng.choice([6.0, 8.0, 10.0]))
    return _case(None, kind, n_det, log_nt, ny, nx, ncomp=ncomp, prec=prec, **more)


# ---------------------------------------------------------------- inputs

@dataclasses.dataclass
class Scan:
    """The pointing tables the library takes (integers, see include/cmm.h)."""
    ny: int
    nx: int
    bore: np.ndarray
    det_off: np.ndarray
    det_pol: np.ndarray
    ncomp: int
    f_samp: float = F_SAMP
    periodic: bool = False

    @property
    def n_t(self):
        return self.bore.shape[0]

    @property
    def n_det(self):
        return self.det_off.shape[0]

    @property
    def npix(self):
        return self.ny * self.nx


@dataclasses.dataclass
class Noise:
    sigma: np.ndarray
    fknee: np.ndarray
    alpha: np.ndarray


@dataclasses.dataclass
class Corr:
    modes: np.ndarray
    amp: np.ndarray
    fknee: np.ndarray
    alpha: np.ndarray


def _focal(n_det, spacing):
    rings = 1
    while 3 * rings * (rings + 1) + 1 < n_det:
        rings += 1
    a, b = np.meshgrid(np.arange(-rings, rings + 1), np.arange(-rings, rings + 1), indexing="ij")
    keep = np.maximum(np.maximum(abs(a), abs(b)), abs(a + b)) <= rings
    x, y = (a + 0.5 * b)[keep], (math.sqrt(0.75) * b)[keep]
    order = np.lexsort((np.round(np.arctan2(y, x), 9), np.round(np.hypot(x, y), 9)))[:n_det]
    return np.stack([x[order], y[order]], 1) * spacing, rings


def _scan(c, rng):
    ny, nx, n_t, n_det = c["ny"], c["nx"], 1 << c["log_nt"], c["n_det"]
    focal, rings = _focal(n_det, 1.0)
    focal *= min(10.0 / 3.0, 0.25 * min(ny, nx) / rings)   # 1.667' apart, or half of a small map across
    margin = float(np.abs(focal).max()) + 2.0
    throw = 0.8 * nx
    t = np.arange(n_t)
    ph = np.mod(t * (PX_PER_SAMPLE / (2.0 * throw)), 1.0)
    a = 0.5 * throw * np.where(ph < 0.5, -1.0 + 4.0 * ph, 3.0 - 4.0 * ph)
    u = (np.mod(t, n_t // 2) + 0.5) / (n_t // 2)
    rising = t < n_t // 2
    phi = np.deg2rad(np.where(rising, 10.0 + 30.0 * u, -10.0 - 30.0 * u))
    half = ny / 2.0 + margin
    drift = np.where(rising, -half + 2.0 * half * u, half - 2.0 * half * u)
    bx, by = (nx - 1) / 2.0 + np.cos(phi) * a, (ny - 1) / 2.0 + np.sin(phi) * a + drift
    bore = np.stack([np.round(bx * 65536), np.round(by * 65536), np.round(np.cos(phi) * 32768),
                     np.round(np.sin(phi) * 32768)], 1).astype(np.int32)
    psi = rng.uniform(0.0, np.pi, n_det)
    pol = np.stack([np.cos(2 * psi), np.sin(2 * psi)], 1)
    return Scan(ny, nx, bore, np.round(focal * 128).astype(np.int32), pol, c["ncomp"])


def _noise(c, rng):
    n = c["n_det"]
    s = math.sqrt(math.log(1.04))   # 20 % scatter of the levels about 1
    return Noise(np.exp(rng.normal(-0.5 * s * s, s, n)), rng.uniform(1.0, 5.0, n), np.full(n, ALPHA))


def _corr(c, scan):
    off = scan.det_off / 128.0
    v = np.stack([np.ones(scan.n_det), off[:, 0] - off[:, 0].mean(), off[:, 1] - off[:, 1].mean()], 1)[:, :c["corr"]]
    return Corr(v / np.linalg.norm(v, axis=0), np.array([3.0, 1.0, 1.0])[:c["corr"]],
                np.array([2.0, 1.0, 1.0])[:c["corr"]], np.array([3.0, 2.5, 2.5])[:c["corr"]])


def _table(c, noise, rng):
    """Measured spectra: the law times a smooth ripple of each detector's own."""
    k = np.arange((1 << c["log_nt"]) // 2 + 1)
    f = np.maximum(k, 1) * (F_SAMP / (1 << c["log_nt"]))
    w = 1.0 / (noise.sigma[:, None] ** 2 * (1.0 + (f / noise.fknee[:, None]) ** -ALPHA))
    return w * (1.0 + 0.2 * np.sin(0.05 * f + rng.uniform(0, 6.28, (c["n_det"], 1))))


def _sky(c, gen):
    """A Gaussian sky with C_l ~ l^-2, T of unit rms and Q, U of 0.1."""
    ny, nx = c["ny"], c["nx"]
    ell = torch.hypot(torch.fft.fftfreq(ny, dtype=torch.float64, device=DEV)[:, None],
                      torch.fft.fftfreq(nx, dtype=torch.float64, device=DEV)[None])
    amp = torch.where(ell > 0, 1.0 / ell.clamp_min(1e-12), torch.zeros_like(ell))
    white = torch.randn((c["ncomp"], ny, nx), dtype=torch.float64, device=DEV, generator=gen)
    m = torch.fft.ifft2(torch.fft.fft2(white) * amp).real
    m = m / m.std(dim=(1, 2), keepdim=True)
    m[1:] *= 0.1
    return m.contiguous()


def _inputs(c, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    scan = _scan(c, rng)
    noise = _noise(c, rng)
    table = _table(c, noise, rng) if c["table"] else None
    sky = _sky(c, gen)
    # what A and the preconditioner meet inside a solve are residuals and search
    # directions: sky-like large scales together with pixel-scale structure
    m = sky + 0.3 * torch.randn(sky.shape, dtype=torch.float64, device=DEV, generator=gen)
    return scan, noise, table, sky, m, gen


def _detector_noise(c, noise, gen):
    """The detectors' white noise levels (the data of the right-hand side are sky + white noise)."""
    d = torch.randn((c["n_det"], 1 << c["log_nt"]), dtype=torch.float32, device=DEV, generator=gen)
    return d * torch.as_tensor(noise.sigma, dtype=torch.float32, device=DEV)[:, None]


def prepare(case, seed):
    from paper_1309_7473_gb300 import cmm
    c = case
    scan, noise, table, sky, m, gen = _inputs(c, seed)
    ctx = cmm.Context(0)
    op = cmm.Operator(ctx, scan, noise, precision=PREC[c["prec"]], corr=_corr(c, scan) if c["corr"] else None)
    if table is not None:
        op.noise.set_table(table)
    s = {"case": c, "op": op, "m": m, "cmm": cmm, "out": op.new_map()}
    if c["kind"] == "rhs":
        s["tod"] = op.project(sky).add_(_detector_noise(c, noise, gen))
        del s["m"]
    if c["kind"] == "solve":
        s["pc"] = _precon(cmm, c, op)
        s["b"] = op.apply(sky)
        del s["m"]
    if c["kind"] == "precon_apply":
        s["pc"] = _precon(cmm, c, op)
    return s


def _precon(cmm, c, op):
    if c["precon"] == "binned":
        return cmm.Precon(op, cmm.PRECON_BINNED)
    return cmm.Precon(op, cmm.PRECON_CIRCULANT, taper_sigma_px=c["taper"])


def run(state):
    c, op, cmm = state["case"], state["op"], state["cmm"]
    kind = c["kind"]
    if kind == "apply":
        return op.apply(state["m"], state["out"])
    if kind == "rhs":
        return op.rhs(state["tod"], state["out"])
    if kind == "project":
        return op.project(state["m"])
    if kind == "precon_apply":
        return state["pc"].apply(state["m"], state["out"])
    if kind == "precon_build":
        return _precon(cmm, c, op).apply(state["m"], state["out"])
    x, info, _, _ = cmm.solve(op, state["pc"], state["b"], tol=c["tol"], maxit=c["iters"])
    return {"x": x, "iterations": int(info.iterations)}


def work(case):
    """Tables, maps and stored data once each; the arithmetic of P, N^-1 and P^T per
    sample (two real FFTs of 2.5 log2 n a sample, projection, weights and binning)
    and of the preconditioner's transforms."""
    c = case
    n_t, npix = 1 << c["log_nt"], c["ny"] * c["nx"]
    ns, nc = c["n_det"] * n_t, c["ncomp"]
    word = 8 if c["prec"] == "f64" else 4
    maps = 2 * 8.0 * nc * npix
    tables = 16.0 * n_t
    a = ns * (5.0 * c["log_nt"] + 20.0)
    blocks = (6 + 9 if nc == 3 else 2) * word * float(npix)
    m = npix * nc * (10.0 * math.log2(npix) + 30.0)
    if c["kind"] == "apply":
        return {"bytes": tables + maps + (2 * ns // 2 * 4.0 if c["table"] else 0.0), "flops": a}
    if c["kind"] == "rhs":
        return {"bytes": 4.0 * ns + tables + maps / 2, "flops": ns * (5.0 * c["log_nt"] + 14.0)}
    if c["kind"] == "project":
        return {"bytes": 4.0 * ns + tables + maps / 2, "flops": 6.0 * ns}
    if c["kind"] == "precon_apply":
        return {"bytes": blocks + maps, "flops": m}
    if c["kind"] == "precon_build":
        return {"bytes": blocks + maps + tables, "flops": nc * a + 12.0 * ns + m}
    its = c["iters"] if c["tol"] == 0 else 26   # the small patch takes about 26
    return {"bytes": tables + maps + (blocks if c["precon"] == "circulant" else 0.0),
            "flops": (its + 1) * (a + (m if c["precon"] == "circulant" else 15.0 * npix))}


# ---------------------------------------------------------------- results in 64 bits

class _Exact:
    """P, N^-1, P^T and the preconditioners of one case in FP64 torch."""

    def __init__(self, c, scan, noise, table):
        self.c, self.scan = c, scan
        self.shape = (c["ncomp"], c["ny"], c["nx"])
        dev = dict(device=DEV, dtype=torch.float64)
        b = torch.as_tensor(scan.bore, device=DEV)
        self.bore = b.to(torch.int64).T.contiguous()
        cf, sf = b[:, 2].double(), b[:, 3].double()
        r2 = cf * cf + sf * sf
        self.c2, self.s2 = (cf * cf - sf * sf) / r2, 2.0 * cf * sf / r2
        self.off = torch.as_tensor(scan.det_off, device=DEV).to(torch.int64)
        self.pol = torch.as_tensor(scan.det_pol, **dev)
        n_t = scan.n_t
        k = torch.arange(n_t // 2 + 1, **dev).clamp_min(1.0) * (F_SAMP / n_t)
        self.freq = k
        self.noise = [torch.as_tensor(v, **dev) for v in (noise.sigma, noise.fknee, noise.alpha)]
        self.table = None if table is None else torch.as_tensor(table, **dev)
        self.step = max(1, min(scan.n_det, (1 << 25) // n_t))
        self.chunks = [range(d, min(d + self.step, scan.n_det)) for d in range(0, scan.n_det, self.step)]
        self.mask = torch.ones(scan.npix, dtype=torch.bool, device=DEV)
        hits = self.blocks(None)
        if c["ncomp"] == 1:
            self.mask = hits[:, 0, 0] > 0
        else:
            lam = self.eigh(hits)[0]
            self.mask = (lam[:, 2] > 0) & (lam[:, 0] >= 1e-3 * lam[:, 2])

    def weights(self, dets):
        if self.table is not None:
            return self.table[dets.start:dets.stop]
        s, f, a = (v[dets.start:dets.stop, None] for v in self.noise)
        return 1.0 / (s * s * (1.0 + (self.freq / f) ** -a))

    def diag(self):
        out = []
        for d in self.chunks:
            w = self.weights(d)
            out.append((w[:, 0] + w[:, -1] + 2.0 * w[:, 1:-1].sum(1)) / self.scan.n_t)
        return torch.cat(out)

    def point(self, dets):
        """Pixels (npix: none) and response of a chunk, [chunk, n_t] each."""
        bx, by, c, s = self.bore
        ox, oy = self.off[dets.start:dets.stop, 0, None], self.off[dets.start:dets.stop, 1, None]
        ix = (bx + ((c * ox - s * oy) >> 6) + 32768) >> 16
        iy = (by + ((s * ox + c * oy) >> 6) + 32768) >> 16
        ny, nx = self.scan.ny, self.scan.nx
        ok = (ix >= 0) & (ix < nx) & (iy >= 0) & (iy < ny)
        p = torch.where(ok, iy * nx + ix, self.scan.npix)
        pc, ps = self.pol[dets.start:dets.stop, 0, None], self.pol[dets.start:dets.stop, 1, None]
        return p, pc * self.c2 - ps * self.s2, ps * self.c2 + pc * self.s2

    def project(self, m, dets):
        p, c, s = self.point(dets)
        g = torch.cat([m.reshape(self.shape[0], -1) * self.mask, torch.zeros((self.shape[0], 1), dtype=m.dtype, device=DEV)], 1)
        return g[0][p] if self.shape[0] == 1 else g[0][p] + c * g[1][p] + s * g[2][p]

    def bin(self, tod, dets, out):
        p, c, s = self.point(dets)
        p = p.reshape(-1)
        for k, r in enumerate((None, c, s)[:self.shape[0]]):
            out[k].index_add_(0, p, (tod if r is None else r * tod).reshape(-1))

    def filter_bin(self, data):
        """P^T N^-1 d, data(dets) giving the chunk's time-ordered data."""
        n_t, npix = self.scan.n_t, self.scan.npix
        out = torch.zeros((self.shape[0], npix + 1), dtype=torch.float64, device=DEV)
        if self.c["corr"]:
            co = _corr(self.c, self.scan)
            v, amp, fk, al = (torch.as_tensor(x, dtype=torch.float64, device=DEV) for x in (co.modes, co.amp, co.fknee, co.alpha))
            minv = torch.diag_embed(1.0 / (amp ** 2 * (1.0 + (self.freq[:, None] / fk) ** -al)))
            t = torch.zeros((len(self.freq), v.shape[1]), dtype=torch.complex128, device=DEV)
            for d in self.chunks:
                w, vd = self.weights(d), v[d.start:d.stop]
                t += torch.einsum("dk,dj->kj", w * torch.fft.rfft(data(d)), vd.to(torch.complex128))
                minv += torch.einsum("dk,di,dj->kij", w, vd, vd)
            sol = torch.linalg.solve(minv.to(torch.complex128), t[..., None])[..., 0]
        for d in self.chunks:
            x = torch.fft.rfft(data(d))
            if self.c["corr"]:
                x = x - torch.einsum("kj,dj->dk", sol, v[d.start:d.stop].to(torch.complex128))
            self.bin(torch.fft.irfft(self.weights(d) * x, n=n_t), d, out)
        return (out[:, :npix] * self.mask).reshape(self.shape)

    def apply(self, m):
        return self.filter_bin(lambda d: self.project(m, d))

    def blocks(self, u):
        """sum_t u_d P_t P_t^T per pixel, [npix, nc, nc]."""
        nc, npix = self.shape[0], self.scan.npix
        acc = torch.zeros((6, npix + 1), dtype=torch.float64, device=DEV)
        for d in self.chunks:
            p, c, s = self.point(d)
            w = torch.ones_like(c) if u is None else u[d.start:d.stop, None].expand_as(c)
            p = p.reshape(-1)
            for k, v in enumerate((w, w * c, w * s, w * c * c, w * c * s, w * s * s)[:1 if nc == 1 else 6]):
                acc[k].index_add_(0, p, v.reshape(-1))
        acc = acc[:, :npix] * self.mask
        idx = [[0]] if nc == 1 else [[0, 1, 2], [1, 3, 4], [2, 4, 5]]
        return torch.stack([torch.stack([acc[j] for j in row], 1) for row in idx], 1)

    @staticmethod
    def eigh(a):
        parts = [torch.linalg.eigh(x) for x in a.cpu().split(1 << 15)]
        return torch.cat([p[0] for p in parts]).to(DEV), torch.cat([p[1] for p in parts]).to(DEV)

    def binned(self):
        b = self.blocks(self.diag())
        one = torch.eye(self.shape[0], dtype=torch.float64, device=DEV)
        inv = torch.linalg.inv(torch.where(self.mask[:, None, None], b, one)) * self.mask[:, None, None]
        return lambda r: torch.einsum("pab,bp->ap", inv, r.reshape(self.shape[0], -1)).reshape(self.shape)

    def circulant(self, taper):
        nc, ny, nx = self.shape
        b = self.blocks(self.diag())
        one = torch.eye(nc, dtype=torch.float64, device=DEV)
        lam, vec = self.eigh(torch.where(self.mask[:, None, None], b, one))
        si = torch.einsum("pak,pk,pbk->pab", vec, lam ** -0.5, vec) * self.mask[:, None, None]
        ref = (ny // 2) * nx + nx // 2
        if not bool(self.mask[ref]):
            good = torch.nonzero(self.mask)[:, 0]
            d2 = (good // nx - ny // 2) ** 2 + (good % nx - nx // 2) ** 2
            ref = int(good[d2 == d2.min()].min())
        rows = torch.zeros((nc, nc, ny * nx), dtype=torch.float64, device=DEV)
        for g in range(nc):
            e = torch.zeros(self.shape, dtype=torch.float64, device=DEV)
            e.reshape(nc, -1)[g, ref] = 1.0
            rows[g] = self.apply(e).reshape(nc, -1)
        q = torch.einsum("ga,gdj,jdb->abj", si[ref], rows, si).reshape(nc, nc, ny, nx)
        q = torch.roll(q, (-(ref // nx), -(ref % nx)), (-2, -1))
        q = 0.5 * (q + torch.roll(q.flip(-2, -1), (1, 1), (-2, -1)).transpose(0, 1))
        wrap = lambda n: torch.where(torch.arange(n, device=DEV) < (n + 1) // 2, torch.arange(n, device=DEV), torch.arange(n, device=DEV) - n).double()  # noqa: E731
        q = q * torch.exp(-(wrap(ny)[:, None] ** 2 + wrap(nx)[None] ** 2) / (2.0 * taper * taper))
        h = torch.conj(torch.fft.fft2(q)).permute(2, 3, 0, 1).reshape(ny * nx, nc, nc)
        lam, vec = self.eigh(0.5 * (h + torch.conj(h.transpose(1, 2))))
        lam = torch.clamp(lam, min=1e-6 * float(lam.max())).to(torch.complex128)
        hinv = torch.einsum("pak,pk,pbk->pab", vec, 1.0 / lam, torch.conj(vec))

        def apply(r):
            y = torch.einsum("pab,bp->ap", si, r.reshape(nc, -1)).reshape(self.shape)
            f = torch.einsum("pab,bp->ap", hinv, torch.fft.fft2(y).reshape(nc, -1)).reshape(self.shape)
            z = torch.fft.ifft2(f).real
            return torch.einsum("pab,bp->ap", si, z.reshape(nc, -1)).reshape(self.shape)
        return apply


def exact(case, seed):
    c = case
    scan, noise, table, sky, m, gen = _inputs(c, seed)
    e = _Exact(c, scan, noise, table)
    kind = c["kind"]
    if kind == "apply":
        return e.apply(m)
    if kind == "project":
        return torch.cat([e.project(m, d).float() for d in e.chunks]) if c["prec"] == "f32" else None
    if kind == "rhs":
        # the stored data are single precision: sky as the library projects it, plus the noise
        white = _detector_noise(c, noise, gen)
        return e.filter_bin(lambda d: e.project(sky, d) + white[d.start:d.stop].double())
    if kind in ("precon_apply", "precon_build"):
        return e.circulant(c["taper"])(m)
    apply_m = e.binned() if c["precon"] == "binned" else e.circulant(c["taper"])
    b = e.apply(sky)
    x, r = torch.zeros_like(b), b.clone()
    z = apply_m(r)
    p, rho, k = z.clone(), torch.sum(r * z), 0
    while k < c["iters"] and float(torch.linalg.norm(r)) > c["tol"] * float(torch.linalg.norm(b)):
        q = e.apply(p)
        alpha = rho / torch.sum(p * q)
        x, r, k = x + alpha * p, r - alpha * q, k + 1
        z = apply_m(r)
        new = torch.sum(r * z)
        p, rho = z + (new / rho) * p, new
    return {"x": x, "iterations": None}
