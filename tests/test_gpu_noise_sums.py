"""GPU: c0 = (1/n) sum_k w_k / N_k of every chunk, on its own, through the PCG preconditioner of the
starting state z = Minv r (Minv = (sum_c c0_c P_c^T P_c)^-1 pixel by pixel): chunks of different noise
that share pixels, long enough for the power-law tables, even and odd, slopes and levels on both sides
of the ranges in which tables and refined reciprocals are used."""
import numpy as np
import pytest

from paper_1705_01893_gb300 import binding

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _c0(n, q):
    sigma, fk, alpha, fs = q
    f = np.maximum(np.arange(n // 2 + 1), 1) * fs / n
    N = sigma ** 2 * (1.0 + (fk / f) ** alpha) if fk > 0 else np.full(len(f), sigma ** 2 * (2.0 if alpha == 0 else 1.0))
    w = np.full(len(f), 2.0)
    w[0] = 1.0
    if n % 2 == 0:
        w[-1] = 1.0
    return np.sum(w / N) / n


LEVELS = {"unit": (1.0, 1.0), "tiny": (3e-16, 1.0), "huge": (3e15, 1.0)}


@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("level", LEVELS)
@pytest.mark.parametrize("alpha,fknee", [(0.0, 1.0), (-0.5, 0.3), (-4.0, 30.0), (0.7, 2.0), (2.0, 0.5), (4.0, 0.01),
                                         (4.5, 0.01), (2.5, 0.0)])
def test_c0(alpha, fknee, level, ncomp):
    """Positive terms: the sums and the two reciprocals carry a few ulps each, 1e-12 in all for the
    T-only quotient; 3 x 3 blocks of condition up to 1e3 carry 1e-9."""
    lens = [1 << 15, 20000, 16875, 1 << 17]
    rng = np.random.default_rng(2)
    n, npix = int(sum(lens)), 64
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    pix = np.repeat(rng.integers(0, npix, size=n // 2 + 1), 2)[:n].astype(np.int32)
    psi = rng.uniform(0, np.pi, n)
    cos, sin = np.cos(2 * psi).astype(np.float32), np.sin(2 * psi).astype(np.float32)
    s = LEVELS[level][0]
    params = np.array([[s * (1.0 + c), fknee * (1.0 + 0.5 * c), alpha, 100.0] for c in range(len(lens))])
    up = [torch.from_numpy(x).cuda() for x in (pix, cos, sin)]
    plan = binding.Plan(off, up[0], *(up[1:] if ncomp == 3 else (None, None)), npix, ncomp)
    plan.set_noise(torch.from_numpy(rng.standard_normal(n).astype(np.float32)).cuda(), params=params)
    x = torch.zeros(npix, ncomp, dtype=torch.float64, device="cuda")
    plan.pcg(x, 0)                                      # r = b - A x and z = Minv r, no iteration
    first = plan.pcg_state() - plan._pcg_state_t.data_ptr()
    state = plan._pcg_state_t[first:first + 2 * 8 * npix * ncomp].view(torch.float64).cpu().numpy()
    r, z = state.reshape(2, npix, ncomp)
    w = np.stack([np.ones(n), cos, sin], 1)[:, :ncomp].astype(np.float64)
    A = np.zeros((npix, ncomp, ncomp))
    for c, k in enumerate(lens):
        sl = slice(off[c], off[c + 1])
        for i in range(ncomp):
            for j in range(ncomp):
                A[:, i, j] += _c0(k, params[c]) * np.bincount(pix[sl], w[sl, i] * w[sl, j], npix)
    back = np.einsum("pij,pj->pi", A, z)
    assert np.abs(r).min() > 0
    assert np.linalg.norm(back - r) <= (1e-12 if ncomp == 1 else 1e-9) * np.linalg.norm(r)
    if ncomp == 1:
        assert np.abs(back / r - 1.0).max() <= 1e-12
