"""Performance cases of the messenger mapmaker: what its users run, through the public calls.

A case is one pass of a user's program on the GPU: a cooled messenger solve, PCG on the same
kernels, a gradient through the solver, the set-up of a new data set, the operators P, P^T and
F on their own, or the allocation-free binned map.  The sizes are those of the repository's
configurations (64^2 T-only, 256^2 / 512^2 / 2048^2 IQU rasters, uneven chunks on 1024^2, the
differencing instrument on 512^2) plus the short ragged chunks of its tests; ``draw`` spreads
over the ranges between them.

Inputs are made on the GPU from the seed: a Gaussian random sky with power ~ l^-2, raster
pointing, a rotating half-wave plate, exactly circulant 1/f noise per chunk.  The solver works
in FP32 timestreams with FP64 pixel sums, so a solved map carries FP32 accuracy (1e-7 and up)
in a float64 tensor; a program keeps such maps, their chi^2 and the noise gradients as float32
products, and so do the passes here.  What is FP64 throughout (hit weights, P^T, the
allocation-free binned map) is returned as float64.
"""
import math
import random

import numpy as np
import torch

from paper_1705_01893_gb300 import binding

INF = float("inf")


# ------------------------------------------------------------------------------- the cases
def _case(name, op, **kw):
    c = dict(op=op, width=512, ncomp=3, scan="alternating", spp=4, chunks=8, n=1 << 22, n_max=0, layout=0,
             half=False, fs=200.0, levels=1, iters=1, graph=False, theta=False, tune=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest solve: one detector, 64^2 T-only, the whole 10 x 10 cooling schedule as
        # graph launches; one iteration is about 20 us, so latency and launches are what counts
        _case("t64_schedule", "messenger", width=64, ncomp=1, scan="square", chunks=1, n=1 << 15, fs=100.0,
              levels=10, iters=10, graph=True),
        # short ragged chunks (2-3-5-smooth, odd lengths among them): a quick look at a few
        # minutes of data, launch-bound
        _case("ragged_small", "messenger", width=24, scan="angled", spp=2, chunks=12, n=1500, n_max=12000, layout=6,
              levels=4, iters=5, graph=True),
        # an ordinary small-patch solve: 256^2 IQU, 4 detectors x 2^20
        _case("iqu256_graph", "messenger", width=256, chunks=4, n=1 << 20, levels=4, iters=5, graph=True),
        # the production patch: 512^2 IQU, 8 detectors x 2^22, launched from the host
        _case("iqu512_messenger", "messenger", levels=2, iters=5),
        # the largest single-GPU run: 2048^2 IQU, 32 detectors x 2^24 samples, FP16 weights
        _case("iqu2048_messenger", "messenger", width=2048, scan="angled", spp=2, chunks=32, n=1 << 24, half=True,
              levels=1, iters=3),
        # batched uneven chunks on 1024^2 IQU, each with its own noise and raster angle
        _case("uneven1024_graph", "messenger", width=1024, scan="angled", spp=2, chunks=64, n=1 << 16, n_max=1 << 20,
              layout=2, levels=2, iters=5, graph=True, tune=True),
        # a differencing instrument: two beams per sample, 9 orientations on 512^2 T-only
        _case("differential512", "composite", ncomp=1, scan="angled", spp=2, chunks=9, n=1 << 21, levels=2, iters=2,
              tune=True),
        # the comparison solver on the production patch
        _case("pcg512", "pcg", iters=8),
        # a gradient step: 20 iterations and their adjoint for the data and the noise parameters
        _case("adjoint256", "adjoint", width=256, chunks=4, n=1 << 20, levels=4, iters=5, theta=True),
        # opening a new data set: pointing plan, noise tables, data spectrum, first binned map
        _case("setup512", "setup"),
        # P, P^T and the chunk rffts on their own (a caller's own solver)
        _case("operators512", "operators"),
        # quick-look binned map by a caller that must not allocate
        _case("quicklook512", "noalloc", chunks=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: operation, chunk lengths, detectors, map, scan and types at random; at most
    2^27 samples a pass of the solvers and 12 iterations, below the largest listed case."""
    op = rng.choice(["messenger"] * 6 + ["pcg", "pcg", "adjoint", "composite", "setup", "operators", "noalloc"])
    scan = rng.choice(["alternating", "angled", "angled"])
    ncomp = 1 if op == "composite" else rng.choice([1, 3, 3, 3])
    smooth = op not in ("adjoint", "noalloc") and rng.random() < 0.4
    if smooth:
        n = _log_int(rng, 1000, 300000)
        n_max = min(1 << 20, _log_int(rng, n + n // 3, 8 * n))
        most = 1 << 25
    else:
        n, n_max = 1 << rng.randint(11, 22 if op == "adjoint" else 24), 0
        most = {"adjoint": 1 << 23, "composite": 1 << 24, "noalloc": 1 << 25, "setup": 1 << 26}.get(op, 1 << 27)
    top = max(n, n_max)
    chunks = max(1, min(48, _log_int(rng, 1, 48), most // top))
    total = chunks * n
    side = int(math.sqrt(total / rng.uniform(8, 60)))
    width = max(12, min(2048 if op != "noalloc" else 512, side + rng.randint(0, 3)))
    if op == "messenger":
        levels, iters = rng.randint(1, 3), rng.randint(1, 4)
    elif op == "adjoint":
        levels, iters = rng.randint(1, 3), rng.randint(1, 4)
    elif op == "pcg":
        levels, iters = 1, rng.randint(2, 8)
    else:
        levels, iters = 1, rng.randint(1, 4)
    return _case(None, op, width=width, ncomp=ncomp, scan=scan, spp=rng.choice([2, 4]), chunks=chunks, n=n, n_max=n_max,
                 layout=rng.randint(1, 1 << 20), half=ncomp == 3 and op != "adjoint" and rng.random() < 0.4,
                 levels=levels, iters=iters, graph=op == "messenger" and rng.random() < 0.5,
                 theta=op == "adjoint" and rng.random() < 0.5, tune=smooth and rng.random() < 0.5)


# ------------------------------------------------------------------------------ the inputs
def _lengths(case):
    """Chunk lengths: all n, or drawn from the 2-3-5-smooth integers of [n, n_max]."""
    if not case["n_max"]:
        return [case["n"]] * case["chunks"]
    cand = []
    for a in range(21):
        for b in range(13):
            for c in range(10):
                v = 2 ** a * 3 ** b * 5 ** c
                if case["n"] <= v <= case["n_max"]:
                    cand.append(v)
    cand.sort()
    rng = random.Random(case["layout"])
    return [rng.choice(cand) for _ in range(case["chunks"])]


def _sky(width, ncomp, gen, dev):
    """[width^2, ncomp] float64: T with unit rms and power ~ l^-2, Q and U at a tenth of it."""
    fy = torch.fft.fftfreq(width, device=dev, dtype=torch.float64)[:, None] * width
    fx = torch.fft.rfftfreq(width, device=dev, dtype=torch.float64)[None, :] * width
    ell = torch.sqrt(fx * fx + fy * fy)
    amp = torch.where(ell > 0, 1.0 / torch.where(ell > 0, ell, 1.0), 0.0)
    out = []
    for k in range(ncomp):
        w = torch.randn(width, width, generator=gen, device=dev, dtype=torch.float64)
        m = torch.fft.irfft2(torch.fft.rfft2(w) * amp, s=(width, width))
        m = m - m.mean()
        out.append((m * ((1.0 if k == 0 else 0.1) / m.std())).reshape(-1))
    return torch.stack(out, 1)


def _pointing(case, n, angle, phase, dev, offset=0.0):
    """int32 pixels of one chunk; rows of the map are scanned back and forth."""
    w, spp = case["width"], case["spp"]
    s = torch.arange(n, device=dev)
    if case["scan"] == "square":          # every row once, then every column once, and again
        sweep, j = s // (w * spp), (s % (w * spp)) // spp
        line = sweep % w
        pix = torch.where((sweep // w) % 2 == 0, line * w + j, j * w + line)
    elif case["scan"] == "alternating":   # rows and columns in turn
        sweep, j = s // (w * spp), (s % (w * spp)) // spp
        line = (sweep // 2 + phase) % w
        pix = torch.where(sweep % 2 == 0, line * w + j, j * w + line)
    else:                                 # sweeps through the map at `angle`, -1 outside it
        ca, sa = math.cos(angle), math.sin(angle)
        span = int(math.ceil(w * (abs(ca) + abs(sa)) - 1e-9))
        sweep, j = s // (span * spp), s % (span * spp)
        xi = -0.5 * span + (j.double() + 0.5) / spp
        xi = torch.where(sweep % 2 == 0, xi, -xi)
        eta = -0.5 * span + ((sweep // 2 + phase) % span).double() + 0.5 + offset
        x, y = 0.5 * w + xi * ca - eta * sa, 0.5 * w + xi * sa + eta * ca
        inside = (x >= 0) & (x < w) & (y >= 0) & (y < w)
        pix = torch.where(inside, x.floor().long() + w * y.floor().long(), -1)
    return pix.to(torch.int32)


def _psd(n, q, dev):
    """N on the rfft bins: sigma^2 (1 + (f_knee / f)^alpha), DC floored to bin 1."""
    sigma, fk, alpha, fs = q
    f = torch.arange(n // 2 + 1, device=dev, dtype=torch.float64)
    f[0] = 1.0
    return sigma * sigma * (1.0 + (fk / (f * (fs / n))) ** alpha)


def _inputs(case, seed, dev):
    rng = random.Random(seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    lens = _lengths(case)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    total, w, nc, C = int(off[-1]), case["width"], case["ncomp"], len(lens)
    sky = _sky(w, nc, gen, dev)
    wt = torch.float16 if case["half"] else torch.float32
    pix = torch.empty(total, dtype=torch.int32, device=dev)
    tod = torch.empty(total, dtype=torch.float32, device=dev)
    cos = torch.empty(total, dtype=wt, device=dev) if nc == 3 else None
    sin = torch.empty(total, dtype=wt, device=dev) if nc == 3 else None
    two = case["op"] == "composite"
    pix_b = torch.empty(total, dtype=torch.int32, device=dev) if two else None
    params = np.zeros((C, 4))
    shift = rng.randint(0, 1 << 20)
    for c, n in enumerate(lens):
        a, b = int(off[c]), int(off[c + 1])
        if case["scan"] == "square":
            q = (1.0, 1.0, 2.0, case["fs"])
        elif case["n_max"]:
            q = (rng.uniform(0.5, 2.0), rng.uniform(0.05, 3.0), rng.uniform(1.0, 3.0), case["fs"])
        else:
            q = (1.0, rng.uniform(0.1, 2.0), rng.uniform(1.0, 3.0), case["fs"])
        if case["n_max"]:
            angle = rng.uniform(0.0, math.pi)
        elif two:
            angle = math.pi * c / C
        else:
            angle = math.radians(45.0 * (c % 4))
        phase = (shift + c * max(1, w // C)) if case["scan"] != "square" else 0
        params[c] = q
        p = _pointing(case, n, angle, phase, dev, 1.5 if two else 0.0)
        pix[a:b] = p
        hit = p >= 0
        rows = torch.where(hit, p, 0).long()
        if nc == 3:
            psi = math.radians(180.0 * c / C) + math.pi * torch.arange(n, device=dev, dtype=torch.float64) / case["fs"]
            cos[a:b] = torch.cos(2 * psi).to(wt)
            sin[a:b] = torch.sin(2 * psi).to(wt)
            m = sky[rows]
            sig = m[:, 0] + m[:, 1] * cos[a:b].double() + m[:, 2] * sin[a:b].double()
        else:
            sig = sky[rows, 0]
        sig = torch.where(hit, sig, 0.0)
        if two:
            pb = _pointing(case, n, angle, phase, dev, -1.5)
            pix_b[a:b] = pb
            sig = sig - torch.where(pb >= 0, sky[torch.where(pb >= 0, pb, 0).long(), 0], 0.0)
        white = torch.randn(n, generator=gen, device=dev, dtype=torch.float32).double()
        noise = torch.fft.irfft(torch.sqrt(_psd(n, q, dev)) * torch.fft.rfft(white), n)
        tod[a:b] = (sig + noise).float()
    # cooling: one lambda = inf step (not for two beams, whose update starts from the map),
    # then geometric levels from max Nbar / tau down to 1
    lmax = max(1.0, max((q[1] / (q[3] / n)) ** q[2] for q, n in zip(params, lens)))
    lam = binding.cooling_schedule(lmax, case["levels"], case["iters"])
    return dict(off=off, lens=lens, npix=w * w, nc=nc, pix=pix, cos=cos, sin=sin, tod=tod, pix_b=pix_b, params=params,
                sky=sky, lam=lam[1:] if two else lam)


def _plan(d):
    second = None if d["pix_b"] is None else (d["pix_b"], None, None, 1.0, -1.0)
    plan = binding.Plan(d["off"], d["pix"], d["cos"], d["sin"], d["npix"], d["nc"], second=second)
    plan.set_noise(d["tod"], params=d["params"])
    return plan


def prepare(case, seed):
    dev = torch.device("cuda:0")
    d = _inputs(case, seed, dev)
    op = case["op"]
    if op not in ("setup", "noalloc"):
        d["plan"] = _plan(d)
        if case["tune"]:
            d["plan"].autotune()
    if op == "adjoint":
        d["fn"] = binding.messenger_fn()
        d["tod_leaf"] = d["tod"].clone().requires_grad_(True)
        d["theta_leaf"] = torch.from_numpy(d["params"][:, :3].copy()).to(dev).requires_grad_(case["theta"])
    if op == "operators":
        d["bins"] = int(sum(n // 2 + 1 for n in d["lens"]))
    d["case"] = case
    return d


# -------------------------------------------------------------------------------- one pass
def run(d):
    case, plan, dev = d["case"], d.get("plan"), d["pix"].device
    op, shape = case["op"], (d["npix"], d["nc"])
    if op in ("messenger", "composite"):
        m = torch.zeros(shape, dtype=torch.float64, device=dev)
        chi = torch.zeros(len(d["lam"]), dtype=torch.float64, device=dev)
        (plan.messenger_graph if case["graph"] else plan.messenger)(m, d["lam"], chi)
        return {"map": m.float(), "chi2": chi.float()}
    if op == "pcg":
        m = torch.zeros(shape, dtype=torch.float64, device=dev)
        chi = torch.zeros(case["iters"], dtype=torch.float64, device=dev)
        plan.pcg(m, case["iters"], chi2_out=chi)
        return {"map": m.float(), "chi2": chi.float()}
    if op == "adjoint":
        m0 = torch.zeros(shape, dtype=torch.float64, device=dev)
        wanted = (d["tod_leaf"], d["theta_leaf"]) if case["theta"] else (d["tod_leaf"],)
        m = d["fn"].apply(plan, d["lam"], m0, d["tod_leaf"], d["theta_leaf"])
        grads = torch.autograd.grad(0.5 * torch.sum((m - d["sky"]) ** 2), wanted)
        return {"map": m.detach().float(), "grad_tod": grads[0],
                "grad_theta": grads[1].float() if case["theta"] else None}
    if op == "setup":
        plan = _plan(d)
        m = torch.zeros(shape, dtype=torch.float64, device=dev)
        plan.messenger(m, [INF])
        hits = torch.empty(d["npix"], dtype=torch.int32, device=dev)
        weight = torch.empty(d["npix"], d["nc"] ** 2, dtype=torch.float64, device=dev)
        plan.maps(hits=hits, weight=weight)
        return {"map": m.float(), "hits": hits, "weight": weight, "lambda_max": plan.lambda_max()}
    if op == "operators":
        tod = torch.empty_like(d["tod"])
        acc = torch.empty(shape, dtype=torch.float64, device=dev)
        spec = torch.empty(d["bins"], 2, dtype=torch.float32, device=dev)
        plan.apply_pointing(d["sky"], tod)
        plan.apply_pointing_T(d["tod"], acc)
        plan.rfft(d["tod"], spec)
        return {"Pm": tod, "PTd": acc, "spectrum": spec}
    m = torch.empty(shape, dtype=torch.float64, device=dev)
    binding.binned_map_noalloc(d["pix"], d["cos"], d["sin"], d["tod"], d["npix"], d["nc"], m)
    return {"map": m}


def work(case):
    """Bytes and flops one pass cannot do without: per iteration the pointing once for P and once
    for P^T, the data spectrum, and per pixel the map, the sums and the weights; per transform
    2.5 n log2 n flops of a real FFT of n samples and about 30 for gather, filter and sums."""
    lens, w = _lengths(case), (4 if case["half"] else 8) if case["ncomp"] == 3 else 0
    N, px, nc = sum(lens), case["width"] ** 2, case["ncomp"]
    beams = 2 if case["op"] == "composite" else 1
    per_px = 104 if nc == 3 else 28
    fft = sum(2.5 * n * math.log2(n) for n in lens)
    step_b = 2 * beams * N * (4 + w) + 4 * N + per_px * px
    step_f = 2 * fft + 30.0 * N * beams
    its = case["levels"] * case["iters"] + (1 if case["op"] in ("messenger", "adjoint") else 0)
    op = case["op"]
    if op in ("messenger", "composite"):
        return {"bytes": its * step_b, "flops": its * step_f}
    if op == "pcg":
        return {"bytes": (case["iters"] + 1) * (step_b - 4 * N) + case["iters"] * 9 * 8 * nc * px,
                "flops": (case["iters"] + 1) * step_f}
    if op == "adjoint":
        return {"bytes": 2 * its * step_b + 4 * N, "flops": 2 * its * step_f}
    if op == "setup":
        return {"bytes": N * (4 + w) + 4 * N + step_b + 8 * nc * nc * px, "flops": fft + step_f + 30.0 * N}
    if op == "operators":
        return {"bytes": 2 * N * (4 + w) + 3 * 4 * N + 4 * N + 2 * 8 * nc * px, "flops": fft + 10.0 * N}
    return {"bytes": N * (4 + w) + 4 * N + 8 * nc * px, "flops": 20.0 * N}


# --------------------------------------------------------------- the same in 64 bits, plainly
class _Exact:
    """P, P^T, the weight blocks and the noise of one data set in float64 torch."""

    def __init__(self, case, seed):
        self.dev = torch.device("cuda:0" if torch.cuda.is_available() else "cpu")
        self.d = d = _inputs(case, seed, self.dev)
        self.case, self.nc, self.npix, self.lens, self.off = case, d["nc"], d["npix"], d["lens"], d["off"]
        self.tau = [q[0] ** 2 for q in d["params"]]

    def span(self, c):
        return slice(int(self.off[c]), int(self.off[c + 1]))

    def entries(self, c):
        """(rows, [weights], gain) of chunk c's pointing, excluded samples on row npix."""
        s, d = self.span(c), self.d
        out = []
        for pix, gain in ((d["pix"], 1.0),) + (((d["pix_b"], -1.0),) if d["pix_b"] is not None else ()):
            p = pix[s].long()
            w = [torch.ones((), dtype=torch.float64, device=self.dev)]
            if self.nc == 3:
                w += [d["cos"][s].double(), d["sin"][s].double()]
            out.append((torch.where(p >= 0, p, self.npix), w, gain))
        return out

    def P(self, c, m):
        pad = torch.cat([m, torch.zeros(1, self.nc, dtype=m.dtype, device=self.dev)])
        t = 0.0
        for p, w, gain in self.entries(c):
            for k in range(self.nc):
                t = t + gain * pad[:, k][p] * w[k]
        return t

    def PT(self, c, t):
        cols = []
        for k in range(self.nc):
            col = torch.zeros(self.npix + 1, dtype=torch.float64, device=self.dev)
            for p, w, gain in self.entries(c):
                col = col.index_add(0, p, gain * t * w[k])
            cols.append(col[:-1])
        return torch.stack(cols, 1)

    def hits(self):
        h = torch.zeros(self.npix + 1, dtype=torch.int64, device=self.dev)
        for c in range(len(self.lens)):
            for p, _, _ in self.entries(c):
                h += torch.bincount(p, minlength=self.npix + 1)
        return h[:-1]

    def blocks(self, scale):
        """Upper triangles [npix, 6 or 1] of sum_c scale_c P_c^T P_c (gains squared)."""
        idx = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)] if self.nc == 3 else [(0, 0)]
        cols = [torch.zeros(self.npix + 1, dtype=torch.float64, device=self.dev) for _ in idx]
        for c in range(len(self.lens)):
            for p, w, gain in self.entries(c):
                for i, (a, b) in enumerate(idx):
                    cols[i] = cols[i].index_add(0, p, (w[a] * w[b]).expand(p.shape) * (gain * gain * scale[c]))
        return torch.stack([x[:-1] for x in cols], 1)

    def keep(self, A, hits):
        """Pixels with a hit whose block has eigmin / eigmax >= 1e-3."""
        if self.nc == 1:
            return (hits > 0) & (A[:, 0] > 0)
        a, b, c, d, e, f = (A[:, i] for i in range(6))
        q = (a + d + f) / 3
        x, y, z = a - q, d - q, f - q
        r = torch.sqrt((x * x + y * y + z * z + 2 * (b * b + c * c + e * e)) / 6).clamp_min(1e-300)
        det = x * (y * z - e * e) - b * (b * z - e * c) + c * (b * e - y * c)
        phi = torch.acos((det / (2 * r ** 3)).clamp(-1, 1)) / 3
        top, low = q + 2 * r * torch.cos(phi), q + 2 * r * torch.cos(phi + 2 * math.pi / 3)
        return (hits > 0) & (top > 0) & (low >= 1e-3 * top)

    def inverse(self, A, ok):
        """[npix, nc, nc] inverses on kept pixels, 0 elsewhere."""
        if self.nc == 1:
            return torch.where(ok, 1 / torch.where(ok, A[:, 0], 1.0), 0.0).reshape(-1, 1, 1)
        eye = torch.tensor([1.0, 0, 0, 1, 0, 1], dtype=torch.float64, device=self.dev)
        a, b, c, d, e, f = torch.where(ok[:, None], A, eye).unbind(1)
        i = [d * f - e * e, c * e - b * f, b * e - c * d, a * f - c * c, b * c - a * e, a * d - b * b]
        det = a * i[0] + b * i[1] + c * i[2]
        W = torch.stack([i[0], i[1], i[2], i[1], i[3], i[4], i[2], i[4], i[5]], 1) / det[:, None]
        return torch.where(ok[:, None], W, 0.0).reshape(-1, 3, 3)

    def weights(self, tau=None):
        two = 2.0 if self.d["pix_b"] is not None else 1.0
        A = self.blocks([two / t for t in (self.tau if tau is None else tau)])
        self.ok = self.keep(A.detach(), self.hits())
        return self.inverse(A, self.ok)

    def cut(self, m):
        return torch.where(self.ok[:, None], m, 0.0)

    def mult(self, n):
        w = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device=self.dev)
        w[0] = 1.0
        if n % 2 == 0:
            w[-1] = 1.0
        return w


def _apply(W, v):
    return torch.einsum("pij,pj->pi", W, v)


def _exact_messenger(x, tod, theta=None):
    """(map, chi^2 of each iteration's input) of the cooled schedule; theta: [C, 3] or None."""
    d, C = x.d, len(x.lens)
    q = [tuple(d["params"][c]) if theta is None else (theta[c, 0], theta[c, 1], theta[c, 2], d["params"][c, 3])
         for c in range(C)]
    tau = [v[0] ** 2 for v in q]
    W = x.weights(tau)
    two = d["pix_b"] is not None
    m = torch.zeros(x.npix, x.nc, dtype=torch.float64, device=x.dev)
    chi = []
    for lam in d["lam"]:
        acc, x2 = 0.0, 0.0
        for c, n in enumerate(x.lens):
            N = _psd(n, q[c], x.dev)
            D, X = torch.fft.rfft(tod[x.span(c)]), torch.fft.rfft(x.P(c, x.cut(m)))
            x2 = x2 + torch.sum(x.mult(n) * (D - X).detach().abs() ** 2 / N.detach()) / n
            if two:
                Y = (D - X) / (tau[c] if math.isinf(lam) else (N - tau[c]) / lam + tau[c])
            elif math.isinf(lam):
                Y = D / tau[c]
            else:
                Y = (lam * tau[c] * D + (N - tau[c]) * X) / (lam * tau[c] + N - tau[c]) / tau[c]
            acc = acc + x.PT(c, torch.fft.irfft(Y, n))
        m = m + _apply(W, acc) if two else _apply(W, acc)
        chi.append(x2)
    return m, torch.stack(chi)


def _exact_pcg(x):
    d, C, iters = x.d, len(x.lens), x.case["iters"]
    x.weights()
    N = [_psd(n, tuple(d["params"][c]), x.dev) for c, n in enumerate(x.lens)]
    Minv = x.inverse(x.blocks([float(torch.sum(x.mult(n) / N[c])) / n for c, n in enumerate(x.lens)]), x.ok)

    def filtered(of):
        return x.cut(sum(x.PT(c, torch.fft.irfft(torch.fft.rfft(of(c)) / N[c], n)) for c, n in enumerate(x.lens)))

    b = filtered(lambda c: d["tod"][x.span(c)].double())
    dd = sum(float(torch.sum(x.mult(n) * torch.fft.rfft(d["tod"][x.span(c)].double()).abs() ** 2 / N[c])) / n
             for c, n in enumerate(x.lens))
    m, r = torch.zeros_like(b), b.clone()
    p = z = _apply(Minv, r)
    rz, chi = torch.sum(r * z), []
    for _ in range(iters):
        chi.append(dd - torch.sum(m * b) - torch.sum(m * r))
        v = filtered(lambda c: x.P(c, p))
        a = rz / torch.sum(p * v)
        m, r = m + a * p, r - a * v
        z = _apply(Minv, r)
        rz, old = torch.sum(r * z), rz
        p = z + (rz / old) * p
    return m, torch.stack(chi)


def exact(case, seed):
    x, op = _Exact(case, seed), case["op"]
    d, C = x.d, len(x.lens)
    if op in ("messenger", "composite"):
        m, chi = _exact_messenger(x, d["tod"].double())
        return {"map": m, "chi2": chi}
    if op == "pcg":
        m, chi = _exact_pcg(x)
        return {"map": m, "chi2": chi}
    if op == "adjoint":
        tod = d["tod"].double().requires_grad_(True)
        theta = torch.from_numpy(d["params"][:, :3].copy()).to(x.dev).requires_grad_(True)
        m, _ = _exact_messenger(x, tod, theta)
        gt, gth = torch.autograd.grad(0.5 * torch.sum((m - d["sky"]) ** 2), (tod, theta))
        return {"map": m.detach(), "grad_tod": gt, "grad_theta": gth if case["theta"] else None}
    if op == "setup":
        W = x.weights()
        acc = sum(x.PT(c, d["tod"][x.span(c)].double() / x.tau[c]) for c in range(C))
        lmax = max(float((_psd(n, tuple(d["params"][c]), x.dev).max() - x.tau[c]) / x.tau[c])
                   for c, n in enumerate(x.lens))
        return {"map": _apply(W, acc), "hits": x.hits().to(torch.int32), "weight": W.reshape(x.npix, -1),
                "lambda_max": lmax}
    if op == "operators":
        x.weights()
        spec = torch.cat([torch.fft.rfft(d["tod"][x.span(c)].double()) for c in range(C)])
        return {"Pm": torch.cat([x.P(c, x.cut(d["sky"])) for c in range(C)]),
                "PTd": sum(x.PT(c, d["tod"][x.span(c)].double()) for c in range(C)),
                "spectrum": torch.view_as_real(spec)}
    A = x.blocks([1.0] * C)
    W = x.inverse(A, x.keep(A, x.hits()))
    return {"map": _apply(W, sum(x.PT(c, d["tod"][x.span(c)].double()) for c in range(C)))}
