"""The workloads whose speed is tracked: what a program that uses the library
has it do, through the entry points of ``paper_2002_12471_gb300.lmosem``.

Every kind of case is one of the calls (or the short fixed sequence of calls)
that a reconstruction program makes, over the sizes of the repository's own
workloads (``synthetic.workload``, the benchmark's arms) and of grids and
event counts between them.  Inputs are made on the GPU from the seed alone: a
first-order photon simulation of the DaT-like phantom (about half the events
scattered, energies and positions blurred as by the scanner), so that the
positions, energies and angles are distributed as in earnest.

``exact`` evaluates the same quantities in 64 bits from the definitions (path
sums pair by pair, line integrals by sorted crossings), with torch alone.
"""
import math

import numpy as np
import torch

import paper_2002_12471_gb300.lmosem as L
from paper_2002_12471_gb300 import synthetic as S

MEC2 = 510.99895
FW2S = 1.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
CHUNK = 1 << 24


def listed():
    return [
        # the smallest whole call: the 16 x 16 parity workload from host
        # buffers (launches, allocations and host work count)
        dict(name="tiny16_whole", kind="whole", n=16, angles=32, events=2000, subsets=4, iters=5, fmt="fp32"),
        # a ragged whole call: 50 x 50 pixels, 90 angles, an odd event count
        dict(name="odd50_whole", kind="whole", n=50, angles=90, events=37013, subsets=6, iters=4, fmt="bf16"),
        # the plain-method workload: 64 x 64, 200k events, 8 x 10
        dict(name="dat64_whole", kind="whole", n=64, angles=120, events=200000, subsets=8, iters=10, fmt="fp32"),
        # the largest single-set workload: 128 x 128, 1M events, FP16 cache
        dict(name="dat128_whole", kind="whole", n=128, angles=120, events=1000000, subsets=8, iters=10, fmt="fp16"),
        # the system model itself, built and read back (analysis of rows)
        dict(name="rows50", kind="rows", n=50, angles=60, events=60000, subsets=6, fmt="fp32"),
        # iterations on a cached model: more iterations of an open data set
        dict(name="iterate64_fp32", kind="iterate", n=64, angles=120, events=200000, subsets=8, iters=10, fmt="fp32"),
        dict(name="iterate128_fp16", kind="iterate", n=128, angles=120, events=500000, subsets=8, iters=10,
             fmt="fp16"),
        # noise realisations of one object in one batch, built and iterated
        dict(name="batch64", kind="batch", n=64, angles=120, events=3600000, reals=16, subsets=8, iters=10),
        # the binned form of one realisation, built and iterated
        dict(name="binned64", kind="binned", n=64, angles=120, events=200000, ebins=3, subsets=8, iters=10),
        # the scatter surrogate: inference of 2M pairs, and a training run
        dict(name="infer_2m", kind="infer", rows=2000003),
        dict(name="train_100", kind="train", rows=2000000, steps=100, batch=8192),
        # the smallest call of all: one sub-iteration on the caller's rows
        dict(name="subiter_small", kind="subiter", rows=1667, cols=1540),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["whole", "whole", "whole", "rows", "iterate", "iterate", "batch", "binned", "infer", "train",
                       "subiter", "subiter"])
    if kind == "infer":
        return dict(kind=kind, rows=_log(rng, 100, 2000000))
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 20000, 2000000), steps=rng.randrange(20, 100),
                    batch=64 * _log(rng, 4, 128))
    if kind == "subiter":
        return dict(kind=kind, rows=_log(rng, 200, 60000), cols=_log(rng, 100, 6000))
    n = _log(rng, 16, 128 if kind in ("whole", "iterate") else 64)
    angles = rng.randrange(32, 121)
    subsets = rng.choice([1, 2, 4, 6, 8])
    iters = rng.randrange(2, 11)
    fmt = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind == "whole":
        return dict(kind=kind, n=n, angles=angles, events=_log(rng, 2000, 1000000), subsets=subsets, iters=iters,
                    fmt=fmt)
    if kind == "rows":
        return dict(kind=kind, n=n, angles=angles, events=_log(rng, 1000, 100000), subsets=subsets, fmt=fmt)
    if kind == "iterate":
        return dict(kind=kind, n=n, angles=angles, events=_log(rng, 2000, 500000), subsets=subsets, iters=iters,
                    fmt=fmt)
    if kind == "batch":
        reals = rng.randrange(2, 17)
        return dict(kind=kind, n=n, angles=angles, events=_log(rng, 20000, 3600000), reals=reals, subsets=subsets,
                    iters=iters)
    return dict(kind=kind, n=n, angles=angles, events=_log(rng, 20000, 400000), ebins=rng.randrange(1, 4),
                subsets=subsets, iters=iters)


# ---------------------------------------------------------------- inputs

_PH = {}


def _phantom(n):
    if n not in _PH:
        _PH[n] = S.brain_phantom(n, 256.0 / n) if n > 16 else S.disk_phantom()
    return _PH[n]


def _problem(case):
    n = case["n"]
    ph = _phantom(n)
    g = S.geometry(case["angles"], n, ph.pixel_mm, 80.0 if n <= 16 else 150.0)
    return ph, g


def _events(ph, g, count, seed):
    """First-order list-mode events on the GPU: (angle int32, u float32, E float32)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    act = torch.from_numpy(ph.activity.reshape(-1).astype(np.float64)).to(dev)
    mu = torch.from_numpy(ph.mu.reshape(-1).astype(np.float32)).to(dev)
    cdf = torch.cumsum(act, 0) / act.sum()
    n, d = ph.mu.shape[0], ph.pixel_mm
    e0, half = g["e0_kev"], 0.5 * g["n_bins"] * g["bin_mm"]
    parts, got = [], 0
    while got < count:
        k = min(1 << 21, 2 * count + 1024)

        def rnd():
            return torch.rand(k, generator=gen, device=dev)

        def gauss():
            return torch.randn(k, generator=gen, device=dev)

        pix = torch.searchsorted(cdf, rnd().double()).clamp(max=n * n - 1)
        x = ((pix % n) + rnd() - 0.5 * n) * d
        y = (torch.div(pix, n, rounding_mode="floor") + rnd() - 0.5 * n) * d
        a = (rnd() * g["n_angles"]).long().clamp(max=g["n_angles"] - 1)
        th = g["angle0_rad"] + 2 * math.pi * a / g["n_angles"]
        ct, st = torch.cos(th), torch.sin(th)
        # half of the photons interact once on the way, at an exponential
        # distance along another direction
        scat = rnd() < 0.5
        phi = 2 * math.pi * rnd()
        step = -torch.log(rnd() + 1e-20) / 0.016
        xs, ys = x + step * torch.cos(phi), y + step * torch.sin(phi)
        ix, iy = torch.floor(xs / d + 0.5 * n).long(), torch.floor(ys / d + 0.5 * n).long()
        inside = (ix >= 0) & (ix < n) & (iy >= 0) & (iy < n)
        m = mu[(iy.clamp(0, n - 1) * n + ix.clamp(0, n - 1))]
        cp = torch.cos(phi) * ct + torch.sin(phi) * st
        p = 1.0 / (1.0 + e0 / MEC2 * (1.0 - cp))
        kn = 0.5 * p * p * (p + 1.0 / p - (1.0 - cp * cp))
        keep = ~scat | (inside & (rnd() < kn) & (rnd() * 0.025 < m))
        x, y = torch.where(scat, xs, x), torch.where(scat, ys, y)
        e1 = torch.where(scat, e0 * p, torch.full_like(p, e0))
        depth = g["radius_mm"] - (x * ct + y * st)
        u = -x * st + y * ct + (g["coll_fwhm0_mm"] + g["coll_fwhm_slope"] * depth) * FW2S * gauss()
        e = e1 + g["fwhm_frac_e0"] * torch.sqrt(e0 * e1) * FW2S * gauss()
        keep &= (u.abs() <= half) & (e >= g["e_lo_kev"]) & (e <= g["e_hi_kev"])
        parts.append((a[keep].int(), u[keep], e[keep]))
        got += int(keep.sum())
    return tuple(torch.cat([q[i] for q in parts])[:count].contiguous() for i in range(3))


def _offsets(case, seed):
    """Uneven event counts of the realisations (a factor of about eight apart)."""
    rng = np.random.default_rng(seed)
    w = 1.0 + 7.0 * rng.uniform(0.0, 1.0, case["reals"])
    cnt = np.floor(w / w.sum() * case["events"]).astype(np.int64)
    return np.concatenate([[0], np.cumsum(cnt)])


def _edges(g, k):
    return [[100.0, 175.0], [100.0, 143.0, 175.0], [100.0, 120.0, 143.0, 175.0]][k - 1]


def _counts(g, ev, k):
    """Counts [angle, position bin, energy bin] (float32) of the events."""
    a, u, e = ev
    nb, half = g["n_bins"], 0.5 * g["n_bins"] * g["bin_mm"]
    b = torch.floor((u.double() + half) / g["bin_mm"]).long().clamp(0, nb - 1)
    edges = torch.tensor(_edges(g, k), dtype=torch.float64, device=u.device)
    q = (torch.searchsorted(edges, e.double(), right=True) - 1).clamp(0, k - 1)
    idx = (a.long() * nb + b) * k + q
    return torch.bincount(idx, minlength=g["n_angles"] * nb * k).float().reshape(g["n_angles"], nb, k).contiguous()


def _weights(seed):
    return torch.from_numpy(L.surrogate_init(seed)).cuda()


def _features(rows, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return torch.randn(rows, L.SURROGATE_INPUTS, generator=gen, device="cuda") * 0.6, gen


class _State:
    """What a program keeps between calls; gives the context back with itself."""

    ctx = None

    def __del__(self):
        if self.ctx is not None:
            torch.cuda.synchronize()
            L.lmosem_destroy(self.ctx)


def prepare(case, seed):
    s = _State()
    s.case, k = case, case["kind"]
    s.stream = torch.cuda.Stream()
    if k == "subiter":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        ld = (case["cols"] + 31) // 32 * 32
        s.rows = torch.zeros(case["rows"], ld, device="cuda")
        s.rows[:, :case["cols"]] = torch.rand(case["rows"], case["cols"], generator=gen, device="cuda") ** 8
        s.f0 = 0.5 + torch.rand(case["cols"], generator=gen, device="cuda")
        s.f = s.f0.clone()
        s.sens = (0.5 + torch.rand(case["cols"], generator=gen, device="cuda")).double() * case["rows"] / 9.0
    elif k in ("infer", "train"):
        ph, g = _problem(dict(n=16, angles=32))
        s.ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=s.stream)
        s.x, gen = _features(case["rows"], seed)
        if k == "infer":
            s.w, s.y = _weights(seed), torch.empty(case["rows"], device="cuda")
        else:  # targets of a smooth law, each pair's log offset from its row's largest
            s.w0 = _weights(seed)
            s.w = s.w0.clone()
            s.rel = -torch.rand(case["rows"], generator=gen, device="cuda") ** 2 * 18.0
            s.t = s.rel - 9.0 + torch.sin(s.x[:, 0] * 2) * s.x[:, 4] + 0.3 * s.x[:, 5] * s.x[:, 7]
    else:
        ph, g = _problem(case)
        s.ph, s.g = ph, g
        ev = _events(ph, g, case["events"], seed)
        if k == "whole":
            s.ev = [t.cpu().pin_memory() for t in ev]
            return s
        s.ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=s.stream)
        nsup = L.lmosem_n_support(s.ctx)
        torch.cuda.synchronize()
        L.lmosem_sensitivity(s.ctx, case["subsets"])
        if k == "rows":
            s.ev = ev
            s.ids = torch.arange(case["events"], dtype=torch.int64, device="cuda")
            s.out = torch.empty(case["events"], nsup, device="cuda")
        elif k == "iterate":
            L.lmosem_build_model(s.ctx, *ev, case["subsets"], case["fmt"])
            s.f = torch.empty(nsup, device="cuda")
        elif k == "batch":
            s.ev, s.off = ev, _offsets(case, seed)
            s.f = torch.empty(case["reals"], nsup, device="cuda")
        else:
            s.counts = _counts(g, ev, case["ebins"])
            s.f = torch.empty(nsup, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    c, k = s.case, s.case["kind"]
    if k == "whole":
        # mu-map, scanner and host events in; image and log-likelihood out (a
        # number: an FP32 sum's worth of digits)
        ctx = L.lmosem_create(s.ph.mu, s.ph.pixel_mm, s.g, stream=s.stream)
        try:
            f, ll = L.lmosem_reconstruct(ctx, *s.ev, c["subsets"], c["iters"], 1.0, c["fmt"])
        finally:
            L.lmosem_destroy(ctx)
        return {"image": f, "loglik": float(ll[0])}
    if k == "rows":
        L.lmosem_build_model(s.ctx, *s.ev, c["subsets"], c["fmt"])
        L.lmosem_model_rows(s.ctx, s.ids, s.out)
        return s.out
    if k == "iterate":
        L.lmosem_init_image(s.ctx, 1.0, s.f)
        L.lmosem_iterate(s.ctx, c["iters"], 1.0, s.f)
        return s.f
    if k == "batch":
        L.lmosem_sensitivity(s.ctx, c["subsets"])
        L.lmosem_build_model_batch(s.ctx, *s.ev, s.off, c["subsets"])
        L.lmosem_init_image_batch(s.ctx, 1.0, s.f)
        L.lmosem_iterate_batch(s.ctx, c["iters"], 1.0, s.f)
        return s.f
    if k == "binned":
        L.lmosem_sensitivity(s.ctx, c["subsets"])
        L.lmosem_build_model_binned(s.ctx, s.counts, _edges(s.g, c["ebins"]), c["subsets"])
        L.lmosem_init_image(s.ctx, 1.0, s.f)
        L.lmosem_iterate(s.ctx, c["iters"], 1.0, s.f)
        return s.f
    if k == "infer":
        L.lmosem_surrogate_infer(s.ctx, s.w, s.x, s.y)
        return s.y
    if k == "train":
        with torch.cuda.stream(s.stream):
            s.w.copy_(s.w0)
        curve = L.lmosem_surrogate_train(s.ctx, s.x, s.t, s.w, steps=c["steps"], batch=c["batch"], target_floor=14.0,
                                         residual_fit=True, d_rel_log=s.rel, magnitude_power=1.0)
        return {"weights": s.w, "loss": curve.astype(np.float32)}  # losses of FP32 residuals
    with torch.cuda.stream(s.stream):
        s.f.copy_(s.f0)
    L.lmosem_osem_subiter_noalloc(s.rows, c["cols"], s.f, s.sens, 1.0, stream=s.stream)
    return s.f


# ---------------------------------------------------------------- needed work

def work(case):
    """Bytes in and out, and the operations of the sums as they are defined:
    one multiply-add per kept path term (a scatter pixel within the position
    cut of the event, 0.3 of them), two per model entry and sub-iteration."""
    k = case["kind"]
    if k == "subiter":
        return dict(bytes=4.0 * case["rows"] * case["cols"] + 16.0 * case["cols"],
                    flops=4.0 * case["rows"] * case["cols"])
    if k == "infer":
        return dict(bytes=36.0 * case["rows"] + 8e5, flops=case["rows"] * 2.0 * (8 * 256 + 3 * 65536 + 256))
    if k == "train":
        return dict(bytes=40.0 * case["rows"] + 1.6e6,
                    flops=6.0 * case["steps"] * case["batch"] * (8 * 256 + 3 * 65536 + 256))
    ph = _phantom(case["n"])
    q = float((ph.mu > 0).sum())
    if k == "binned":
        bins = float(case["angles"] * case["n"] * case["ebins"])
        rows = min(0.7 * bins, float(case["events"]))
        return dict(bytes=4.0 * bins + 4.0 * q, flops=2.0 * rows * q * (0.3 * q) + 4.0 * rows * q * case["iters"])
    j = float(case["events"])
    if k == "iterate":
        size = 4.0 if case["fmt"] == "fp32" else 2.0
        return dict(bytes=j * q * size * case["iters"], flops=4.0 * j * q * case["iters"])
    if k == "rows":
        return dict(bytes=12.0 * j + 4.0 * j * q, flops=2.0 * j * q * (0.3 * q))
    return dict(bytes=12.0 * j + 4.0 * q * case.get("reals", 1),
                flops=2.0 * j * q * (0.3 * q) + 4.0 * j * q * case["iters"])


# ---------------------------------------------------------------- 64 bits

def _line(mu, n, d, x0, y0, x1, y1):
    """Integral of the pixel map along segments: crossings with every grid
    line, sorted; each piece in the pixel of its midpoint."""
    out = torch.empty_like(x0)
    lines = (torch.arange(n + 1, dtype=torch.float64, device=mu.device) - 0.5 * n) * d
    step = max(1, CHUNK // (2 * n + 4))
    for b in range(0, x0.numel(), step):
        e = slice(b, b + step)
        ax, ay, dx, dy = x0[e, None], y0[e, None], (x1 - x0)[e, None], (y1 - y0)[e, None]
        tx = torch.where(dx.abs() > 1e-12, (lines - ax) / dx, torch.zeros_like(dx))
        ty = torch.where(dy.abs() > 1e-12, (lines - ay) / dy, torch.zeros_like(dy))
        t = torch.cat([tx, ty, torch.zeros_like(dx), torch.ones_like(dx)], 1).clamp(0.0, 1.0).sort(1).values
        mid, seg = 0.5 * (t[:, 1:] + t[:, :-1]), t[:, 1:] - t[:, :-1]
        ix = torch.floor((ax + mid * dx) / d + 0.5 * n).long()
        iy = torch.floor((ay + mid * dy) / d + 0.5 * n).long()
        ok = (ix >= 0) & (ix < n) & (iy >= 0) & (iy < n)
        v = mu[iy.clamp(0, n - 1) * n + ix.clamp(0, n - 1)] * ok
        out[e] = (v * seg).sum(1) * torch.sqrt(dx * dx + dy * dy)[:, 0]
    return out


def _kn_total(e):
    k = e / MEC2
    lg = torch.log1p(2 * k)
    return ((1 + k) / k ** 2 * (2 * (1 + k) / (1 + 2 * k) - lg / k) + lg / (2 * k) - (1 + 3 * k) / (1 + 2 * k) ** 2)


def _mass(lo, hi, c, sig):
    r = math.sqrt(0.5) / sig
    return 0.5 * (torch.erfc((lo - c) * r) - torch.erfc((hi - c) * r))


class _Exact:
    """The first-order path model of one object and scanner in 64 bits."""

    def __init__(self, ph, g):
        self.g, self.n, self.d = g, ph.mu.shape[0], ph.pixel_mm
        n, d = self.n, self.d
        self.mu = torch.from_numpy(np.ascontiguousarray(ph.mu.reshape(-1), dtype=np.float64)).cuda()
        self.pix = torch.nonzero(self.mu > 0)[:, 0]
        self.x = ((self.pix % n) + 0.5 - 0.5 * n) * d
        self.y = (torch.div(self.pix, n, rounding_mode="floor") + 0.5 - 0.5 * n) * d
        self.x, self.y = self.x.double(), self.y.double()
        q = self.pix.numel()
        # [m, n]: from emission pixel n to scatter pixel m
        self.vx, self.vy = self.x[:, None] - self.x[None, :], self.y[:, None] - self.y[None, :]
        self.r = torch.sqrt(self.vx ** 2 + self.vy ** 2)
        xs, ys = self.x[None, :].expand(q, q).reshape(-1), self.y[None, :].expand(q, q).reshape(-1)
        xe, ye = self.x[:, None].expand(q, q).reshape(-1), self.y[:, None].expand(q, q).reshape(-1)
        self.pair = _line(self.mu, n, d, xs.contiguous(), ys.contiguous(), xe.contiguous(), ye.contiguous())
        self.pair = self.pair.reshape(q, q)
        e0 = g["e0_kev"]
        c = torch.cos(2 * math.pi * torch.arange(4096, dtype=torch.float64, device="cuda") / 4096)
        self.kbar = float(self._kn(c)[1].mean())
        self.se0 = g["fwhm_frac_e0"] * e0 * FW2S

    def _kn(self, c):
        p = 1.0 / (1.0 + self.g["e0_kev"] / MEC2 * (1.0 - c))
        return p, 0.5 * p * p * (p + 1.0 / p - (1.0 - c * c))

    def angle(self, a):
        """u, sigma_u, primary weight per pixel; path weight, E', sigma_E [m, n]."""
        g, d = self.g, self.d
        th = g["angle0_rad"] + 2 * math.pi * a / g["n_angles"]
        ct, st = math.cos(th), math.sin(th)
        far = 2.0 * self.n * d
        ledge = _line(self.mu, self.n, d, self.x, self.y, self.x + far * ct, self.y + far * st)
        u = -self.x * st + self.y * ct
        sig = (g["coll_fwhm0_mm"] + g["coll_fwhm_slope"] * (g["radius_mm"] - (self.x * ct + self.y * st))) * FW2S
        eye = torch.eye(len(self.x), dtype=torch.bool, device="cuda")
        r = torch.where(eye, torch.ones_like(self.r), self.r)
        c = ((self.vx * ct + self.vy * st) / r).clamp(-1.0, 1.0)
        p, kn = self._kn(c)
        e1 = g["e0_kev"] * p
        ratio = _kn_total(e1) / _kn_total(torch.tensor(g["e0_kev"], dtype=torch.float64))
        w = (d * d * self.mu[self.pix][:, None] * kn / self.kbar / (2 * math.pi * r)
             * torch.exp(-self.pair - ratio * ledge[:, None]))
        w = torch.where(eye, torch.zeros_like(w), w)
        return u, sig, torch.exp(-ledge), w, e1, g["fwhm_frac_e0"] * torch.sqrt(g["e0_kev"] * e1) * FW2S

    def sens(self, tab):
        g = self.g
        half = 0.5 * g["n_bins"] * g["bin_mm"]
        u, sig, w0, w, e1, se = tab
        du = _mass(-half, half, u, sig)
        e0 = torch.tensor(g["e0_kev"], dtype=torch.float64)
        return w0 * du * _mass(g["e_lo_kev"], g["e_hi_kev"], e0, self.se0) + (
            du[:, None] * w * _mass(g["e_lo_kev"], g["e_hi_kev"], e1, se)).sum(0)

    def rows(self, tab, uj, ej):
        """Rows of events of one angle, in blocks of neighbours in position
        (scatter pixels over 9 sigma away from the whole block left out)."""
        u, sig, w0, w, e1, se = tab
        out = torch.empty(len(uj), len(u), dtype=torch.float64, device="cuda")
        lw, r2 = w / (se * math.sqrt(2 * math.pi)), math.sqrt(0.5) / se
        order = torch.argsort(uj)
        for b in range(0, len(uj), 32):
            j = order[b:b + 32]
            z = (uj[j][:, None] - u) / sig
            pos = torch.exp(-0.5 * z * z) / (sig * math.sqrt(2 * math.pi))
            k = torch.nonzero((z.abs() < 9.0).any(0))[:, 0]
            t = (ej[j][:, None, None] - e1[k]) * r2[k]
            te = (ej[j] - self.g["e0_kev"]) / self.se0
            prim = w0 * pos * (torch.exp(-0.5 * te * te) / (self.se0 * math.sqrt(2 * math.pi)))[:, None]
            out[j] = prim + torch.bmm(pos[:, None, k], lw[k] * torch.exp(-t * t))[:, 0]
        return out

    def binned(self, tab, k_edges):
        """[position bin, energy bin, n]"""
        g = self.g
        u, sig, w0, w, e1, se = tab
        nb = g["n_bins"]
        lo = -0.5 * nb * g["bin_mm"] + g["bin_mm"] * torch.arange(nb, dtype=torch.float64, device="cuda")
        mb = _mass(lo[:, None], lo[:, None] + g["bin_mm"], u[None, :], sig[None, :])
        e0 = torch.tensor(g["e0_kev"], dtype=torch.float64)
        res = []
        for a, b in zip(k_edges[:-1], k_edges[1:]):
            res.append(mb @ (w * _mass(a, b, e1, se)) + mb * w0 * _mass(a, b, e0, self.se0))
        return torch.stack(res, 1)


def _em(rows, of, weight, sens, subsets, iters, total):
    """OS-EM (T = 1): image, and log-likelihood of the last one."""
    f = torch.full_like(sens[0], total / float(sens.sum()))
    for _ in range(iters):
        for i in range(subsets):
            p, c = rows[of == i], weight[of == i]
            y = p @ f
            b = torch.where(y > 0, c / y, torch.zeros_like(y)) @ p
            f = torch.where(sens[i] > 0, f * b / sens[i], torch.zeros_like(f))
    y = rows @ f
    return f, float((weight * torch.log(y))[y > 0].sum() - (sens.sum(0) * f).sum())


def exact(case, seed):
    k = case["kind"]
    if k == "subiter":
        s = prepare(case, seed)
        p, f = s.rows[:, :case["cols"]].double(), s.f0.double()
        y = p @ f
        return f * ((1.0 / y) @ p) / s.sens
    if k == "infer":
        w, at, par = _weights(seed).double(), 0, []
        for fi, fo in ((8, 256), (256, 256), (256, 256), (256, 256), (256, 1)):
            par.append((w[at:at + fi * fo].reshape(fo, fi), w[at + fi * fo:at + fi * fo + fo]))
            at += fi * fo + fo
        x, out = _features(case["rows"], seed)[0], []
        for b in range(0, case["rows"], 1 << 18):
            h = x[b:b + (1 << 18)].double()
            for i, (m, bias) in enumerate(par):
                h = h @ m.T + bias
                h = torch.relu(h) if i < 4 else h
            out.append(h[:, 0])
        return torch.cat(out)
    if k not in ("whole", "rows", "binned"):
        return None
    ph, g = _problem(case)
    q = int((ph.mu > 0).sum())
    pairs = float(case["events"]) * q * q if k != "binned" else 40.0 * case["angles"] * q * q
    if pairs > 6e10 or q > 2000:
        return None
    X = _Exact(ph, g)
    ns = case["subsets"]
    sens = torch.zeros(ns, q, dtype=torch.float64, device="cuda")
    ev = _events(ph, g, case["events"], seed)
    if k == "binned":
        c = _counts(g, ev, case["ebins"]).double()
        rows, of, wt = [], [], []
        for a in range(g["n_angles"]):
            tab = X.angle(a)
            sens[a % ns] += X.sens(tab)
            m = X.binned(tab, _edges(g, case["ebins"]))
            hit = c[a] > 0
            rows.append(m[hit])
            wt.append(c[a][hit])
            of.append(torch.full((int(hit.sum()),), a % ns, device="cuda"))
        return _em(torch.cat(rows), torch.cat(of), torch.cat(wt), sens, ns, case["iters"], float(c.sum()))[0]
    rows = torch.empty(case["events"], q, dtype=torch.float64, device="cuda")
    aj, uj, ej = ev[0].long(), ev[1].double(), ev[2].double()
    for a in range(g["n_angles"]):
        tab = X.angle(a)
        sens[a % ns] += X.sens(tab)
        at = torch.nonzero(aj == a)[:, 0]
        if len(at):
            rows[at] = X.rows(tab, uj[at], ej[at])
    if k == "rows":
        return rows
    f, ll = _em(rows, aj % ns, torch.ones_like(uj), sens, ns, case["iters"], float(case["events"]))
    return {"image": f, "loglik": ll}
