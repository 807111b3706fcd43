"""GPU: the run-wise binning kernels (P^T, weight blocks, allocation-free binned map, hit counts)
and the power-law noise tables at the sizes where they can go wrong: totals around the tile of
1024 samples, runs longer than a warp round, excluded samples, chunk boundaries inside a tile,
unaligned arrays; slopes on both sides of the tables' range."""
import numpy as np
import pytest

import oracle.messenger as O

pytestmark = pytest.mark.gpu


def _pointing(n, npix, run, seed):
    rng = np.random.default_rng(seed)
    pix = np.repeat(rng.integers(-1, npix, size=n // run + 1), run)[:n].astype(np.int32)
    psi = rng.uniform(0, np.pi, n)
    return pix, np.cos(2 * psi).astype(np.float32), np.sin(2 * psi).astype(np.float32), \
        rng.standard_normal(n).astype(np.float32)


def _plan(offsets, pix, cos, sin, npix, skip=0):
    import torch
    from paper_1705_01893_gb300 import binding

    def up(a):   # `skip` elements in front: arrays off the 16-byte boundary
        return torch.cat([torch.zeros(skip, dtype=torch.from_numpy(a).dtype), torch.from_numpy(a)]).cuda()[skip:]
    return binding.Plan(offsets, up(pix), None if cos is None else up(cos),
                        None if sin is None else up(sin), npix, 1 if cos is None else 3)


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("n,run", [(4, 1), (1000, 3), (1024, 1), (1080, 40), (5000, 1024), (8192, 2)])
def test_p_transpose_and_p(n, run, ncomp, skip):
    """FP64 sums: exact products of FP32 inputs, so only the order of the additions differs (at
    most n terms: n eps); P m is one FP32 rounding chain of three terms."""
    import torch
    npix = 257
    pix, cos, sin, tod = _pointing(n, npix, run, n + run)
    plan = _plan([0, n], pix, cos if ncomp == 3 else None, sin if ncomp == 3 else None, npix, skip)
    acc = torch.empty(npix, ncomp, dtype=torch.float64, device="cuda")
    plan.apply_pointing_T(torch.from_numpy(tod).cuda(), acc)
    w = np.stack([np.ones(n), cos, sin], 1)[:, :ncomp].astype(np.float64)
    good = pix >= 0
    ref = np.zeros((npix, ncomp))
    np.add.at(ref, pix[good], w[good] * tod[good, None].astype(np.float64))
    assert np.abs(acc.cpu().numpy() - ref).max() <= n * 2.3e-16 * max(1.0, np.abs(tod).max()) * 2
    hits = torch.empty(npix, dtype=torch.int32, device="cuda")
    plan.maps(hits=hits)
    assert np.array_equal(hits.cpu().numpy(), np.bincount(pix[good], minlength=npix))


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("lens", [[500, 600], [1024, 1024], [24, 3000, 10, 1500]])
def test_weight_blocks_across_chunks(lens, skip):
    """W of chunks with different tau whose boundaries fall inside a tile, and P m at the tails
    of vector accesses, against the oracle (FP64: 1e-10 for blocks of condition up to 1e3)."""
    import torch
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n, npix = int(off[-1]), 37
    pix, cos, sin, tod = _pointing(n, npix, 5, 3)
    params = np.array([[0.5 + c, 0.5, 1.5, 50.0] for c in range(len(lens))])
    prob = O.problem_from_synth(dict(pix=pix, cos=cos, sin=sin, tod=tod, offsets=off, npix=npix,
                                     ncomp=3, params=params))
    plan = _plan(off, pix, cos, sin, npix, skip)
    plan.set_noise(torch.from_numpy(tod).cuda(), params=params)
    W = torch.empty(npix, 3, 3, dtype=torch.float64, device="cuda")
    plan.maps(weight=W)
    assert np.linalg.norm(W.cpu().numpy() - prob.W) <= 1e-10 * np.linalg.norm(prob.W)
    m = np.random.default_rng(1).standard_normal((npix, 3))
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    plan.apply_pointing(torch.from_numpy(m).cuda(), out)
    ref = np.concatenate([prob.P(m, a, b) for a, b in prob.chunks()])
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("alpha,fknee", [(0.0, 1.0), (-0.5, 0.3), (0.7, 2.0), (2.0, 0.5), (4.0, 0.01),
                                         (4.5, 0.01), (2.5, 0.0)])
@pytest.mark.parametrize("n", [1 << 14, 16875, 20000, 1 << 16])
def test_noise_tables(n, alpha, fknee):
    """lambda_max to FP64 accuracy and a step at lambda = 3 (reads every Nbar), plus PCG's second
    iterate (reads c0), chunks long enough for the tables and slopes in and out of their range."""
    import torch
    npix = 64
    pix, _, _, tod = _pointing(n, npix, 3, 7)
    params = np.array([[1.3, fknee, alpha, 100.0]])
    prob = O.problem_from_synth(dict(pix=pix, cos=None, sin=None, tod=tod, offsets=np.array([0, n]),
                                     npix=npix, ncomp=1, params=params))
    plan = _plan([0, n], pix, None, None, npix)
    plan.set_noise(torch.from_numpy(tod).cuda(), params=params)
    lam = O.lambda_max(prob)
    assert abs(plan.lambda_max() - lam) <= 1e-12 * max(lam, 1.0)
    m0 = np.random.default_rng(2).standard_normal((npix, 1))
    ref, chi = O.messenger_step(prob, m0, 3.0)
    m = torch.from_numpy(m0.copy()).cuda()
    x2 = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan.messenger(m, [3.0], x2)
    assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
    assert abs(x2.item() - chi) <= 1e-5 * chi
    x = torch.zeros(npix, 1, dtype=torch.float64, device="cuda")
    plan.pcg(x, 2)
    pref, _ = O.pcg(prob, 2)
    assert np.linalg.norm(x.cpu().numpy() - pref) <= 1e-4 * np.linalg.norm(pref)
