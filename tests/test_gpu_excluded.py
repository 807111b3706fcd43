"""GPU: an excluded sample (pixel -1) counts as 0 whatever its orientation weights: NaN and infinite
weights there give what finite ones give, through every kernel that gathers P m and every solver
entry point, for excluded runs of one sample and longer, beside kept samples on either side of a pair.

Two calls on the same inputs may differ in the order of their FP64 additions, hence by rounding of
the FP32 map (6e-8) passed on by later iterations: 1e-6 for solves; the gathers themselves are
compared bit for bit."""
import math

import numpy as np
import pytest

from paper_1705_01893_gb300 import binding

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
INF = math.inf


def _plans(lens, half, two=False):
    """(plan with weight 0, plan with NaN / inf weights on excluded samples, pixels, data)."""
    rng = np.random.default_rng(11)
    n, npix = int(sum(lens)), 101
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    wt = np.float16 if half else np.float32
    bad = np.array([np.nan, np.inf, -np.inf], dtype=wt)

    def beam():
        pix = np.repeat(rng.integers(0, npix, size=n // 3 + 1), 3)[:n].astype(np.int32)
        pix[rng.random(n) < 0.2] = -1
        pix[n // 3: n // 3 + n // 10] = -1
        psi = rng.uniform(0, np.pi, n)
        w = [np.cos(2 * psi).astype(wt), np.sin(2 * psi).astype(wt)]
        clean = [np.where(pix < 0, wt(0), x).astype(wt) for x in w]
        dirty = [np.where(pix < 0, bad[rng.integers(0, 3, n)], x).astype(wt) for x in w]
        return pix, clean, dirty
    beams = [beam() for _ in range(2 if two else 1)]
    tod = torch.from_numpy(rng.standard_normal(n).astype(np.float32)).cuda()
    params = np.array([[1.0 + 0.1 * c, 0.5, 1.5, 20.0] for c in range(len(lens))])
    plans = []
    for which in (1, 2):
        t = [[torch.from_numpy(x).cuda() for x in (b[0], b[which][0], b[which][1])] for b in beams]
        plan = binding.Plan(off, *t[0], npix, 3, second=(*t[1], 1.0, -0.9) if two else None)
        plan.set_noise(tod, params=params)
        plan.tod, plan.weights = tod, t
        plans.append(plan)
    return plans[0], plans[1], npix, n


def _same(a, b, tol):
    a, b = a.double(), b.double()
    assert torch.isfinite(a).all() and torch.isfinite(b).all()
    assert (a - b).norm() <= tol * a.norm()


# one launch (small), compile-time passes, general passes (even and odd), fused launch
ROUTES = {"small": [4096, 4096, 8192], "passes": [1 << 18], "general": [200000, 3125], "fused": [1 << 22]}


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("route", ROUTES)
def test_solves(route, half):
    a, b, npix, n = _plans(ROUTES[route], half)
    lam = [INF, 30.0, 1.0]
    out = []
    for p in (a, b):
        m = torch.zeros(npix, 3, dtype=torch.float64, device="cuda")
        g, x, md = torch.zeros_like(m), torch.zeros_like(m), torch.zeros_like(m)
        chi, cx = (torch.zeros(3, dtype=torch.float64, device="cuda") for _ in range(2))
        p.messenger(m, lam, chi)
        p.messenger_graph(g, lam)
        p.pcg(x, 3, chi2_out=cx)
        p.messenger_md(md, lam)
        tot, modes = p.chi2_modes(m, 2.0)
        w = torch.empty(npix, 9, dtype=torch.float64, device="cuda")
        p.maps(weight=w)
        out.append((m, g, x, md, chi, cx, p.chi2(m, 2.0), tot, modes, w))
    for u, v in zip(*out):
        _same(u, v, 1e-6)


@pytest.mark.parametrize("lens", [[1 << 18], [200000, 3125]])
def test_two_beams(lens):
    a, b, npix, _ = _plans(lens, False, two=True)
    out = []
    for p in (a, b):
        m = torch.zeros(npix, 3, dtype=torch.float64, device="cuda")
        chi = torch.zeros(3, dtype=torch.float64, device="cuda")
        p.messenger(m, [INF, 30.0, 1.0], chi)
        out.append((m, chi, p.chi2(m, 2.0)))
    for u, v in zip(*out):
        _same(u, v, 1e-6)


def test_gradient():
    a, b, npix, n = _plans([1 << 16, 1 << 16], False)
    out = []
    for p in (a, b):
        m0 = torch.zeros(npix, 3, dtype=torch.float64, device="cuda")
        gm = torch.ones_like(m0)
        gt = torch.empty(n, dtype=torch.float32, device="cuda")
        gth = torch.empty(2, 3, dtype=torch.float64, device="cuda")
        p.adjoint([INF, 30.0, 30.0, 1.0], m0, gm, gt, gth, ckpt_every=2)
        out.append((gt, gth))
    _same(out[0][0], out[1][0], 1e-6)
    # sums over 1e5 modes of terms of either sign, known to FP32 rounding each
    _same(out[0][1], out[1][1], 1e-5)


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("lens", [[1 << 16, 5], [1 << 22, 5]])   # one sample a thread; four, and a tail
def test_operators(lens, half):
    a, b, npix, n = _plans(lens, half)
    m = torch.from_numpy(np.random.default_rng(1).standard_normal((npix, 3))).cuda()
    tod = torch.randn(n, device="cuda")
    out = []
    for p in (a, b):
        t = torch.empty(n, dtype=torch.float32, device="cuda")
        acc = torch.empty(npix, 3, dtype=torch.float64, device="cuda")
        q = torch.empty(npix, 3, dtype=torch.float64, device="cuda")
        p.apply_pointing(m, t)
        p.apply_pointing_T(tod, acc)
        binding.binned_map_noalloc(*p.weights[0], tod, npix, 3, q)
        out.append((t, acc, q))
    assert torch.equal(out[0][0], out[1][0])
    _same(out[0][1], out[1][1], 1e-12)
    _same(out[0][2], out[1][2], 1e-10)
