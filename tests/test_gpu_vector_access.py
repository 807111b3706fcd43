"""GPU: the operators and the set-up from 2^22 samples on, where they read four samples at a time and
a CTA bins four rounds: totals that are no multiple of 4, chunk boundaries inside a tile, arrays off
the 16-byte boundary, FP32 and FP16 weights, short and long runs, against FP64 torch on the device."""
import numpy as np
import pytest

from paper_1705_01893_gb300 import binding

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LENS = [2187, 1 << 22, 3000]      # 4199491 samples: 3 past a multiple of 4; boundaries inside tiles
N = sum(LENS)


def _runs(n, npix, run, gen):
    """Pixels in runs of `run` samples (0: of 1 to 64), a tenth of them excluded."""
    if run:
        p = torch.randint(0, npix, (n // run + 1,), generator=gen, device="cuda").repeat_interleave(run)
    else:
        k = torch.randint(1, 65, (n // 16,), generator=gen, device="cuda")
        p = torch.randint(0, npix, (n // 16,), generator=gen, device="cuda").repeat_interleave(k)
    assert p.numel() >= n
    p = p[:n]
    drop = torch.rand((n + 6) // 7, generator=gen, device="cuda").repeat_interleave(7)[:n] < 0.1
    return torch.where(drop, -1, p).to(torch.int32)


def _up(x, skip):
    return torch.cat([torch.zeros(skip, dtype=x.dtype, device="cuda"), x])[skip:]


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("ncomp,half", [(1, False), (3, False), (3, True)])
@pytest.mark.parametrize("run", [1, 5, 40, 0])
def test_operators_and_blocks(run, ncomp, half, skip):
    """FP64 sums of exact products: only the order of the additions differs (1e-12 of the sums of
    magnitudes); P m is an FP32 chain of three terms (4 roundings of 6e-8 of their magnitudes)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(run + 7 * ncomp)
    npix = 1000
    pix = _up(_runs(N, npix, run, gen), skip)
    wt = torch.float16 if half else torch.float32
    psi = torch.rand(N, generator=gen, device="cuda", dtype=torch.float64) * np.pi
    cos, sin = (_up(torch.cos(2 * psi).to(wt), skip), _up(torch.sin(2 * psi).to(wt), skip)) if ncomp == 3 else (None, None)
    tod = _up(torch.randn(N, generator=gen, device="cuda"), 2 * skip)
    off = np.concatenate([[0], np.cumsum(LENS)])
    params = np.array([[1.0, 0.5, 1.5, 50.0], [2.0, 0.5, 1.5, 50.0], [0.5, 0.5, 1.5, 50.0]])
    plan = binding.Plan(off, pix, cos, sin, npix, ncomp)
    plan.set_noise(tod, params=params)

    row = torch.where(pix >= 0, pix, npix).long()
    w = [torch.ones(N, dtype=torch.float64, device="cuda")] + ([cos.double(), sin.double()] if ncomp == 3 else [])

    def binned(v):
        return torch.zeros(npix + 1, dtype=torch.float64, device="cuda").index_add(0, row, v)[:-1]
    # P^T
    acc = torch.empty(npix, ncomp, dtype=torch.float64, device="cuda")
    plan.apply_pointing_T(tod, acc)
    for k in range(ncomp):
        assert ((acc[:, k] - binned(tod.double() * w[k])).abs() <= 1e-12 * binned((tod.double() * w[k]).abs())).all()
    # hits and W
    hits = torch.empty(npix, dtype=torch.int32, device="cuda")
    W = torch.empty(npix, ncomp, ncomp, dtype=torch.float64, device="cuda")
    plan.maps(hits=hits, weight=W)
    assert torch.equal(hits, torch.bincount(row, minlength=npix + 1)[:-1].to(torch.int32))
    tau = torch.repeat_interleave(torch.tensor([1.0, 4.0, 0.25], dtype=torch.float64, device="cuda"),
                                  torch.tensor(LENS, device="cuda"))
    A = torch.stack([torch.stack([binned(w[i] * w[j] / tau) for j in range(ncomp)], 1) for i in range(ncomp)], 1)
    assert (torch.linalg.inv(A) - W).norm() <= 1e-10 * W.norm()
    # P m on both sides of an output's alignment
    m = torch.randn(npix, ncomp, generator=gen, device="cuda", dtype=torch.float64)
    out = torch.full((N + 8,), 7.0, device="cuda")
    for first in (0, 1):
        t = out[first:first + N]
        plan.apply_pointing(m, t)
        pad = torch.cat([m.float().double(), torch.zeros(1, ncomp, dtype=torch.float64, device="cuda")])
        terms = [pad[:, k][row] * w[k] for k in range(ncomp)]
        assert ((t.double() - sum(terms)).abs() <= 2.4e-7 * sum(x.abs() for x in terms)).all()
        assert (out[first + N:] == 7.0).all()
    # the allocation-free map
    q = torch.empty(npix, ncomp, dtype=torch.float64, device="cuda")
    binding.binned_map_noalloc(pix, cos, sin, tod, npix, ncomp, q)
    A1 = torch.stack([torch.stack([binned(w[i] * w[j]) for j in range(ncomp)], 1) for i in range(ncomp)], 1)
    want = torch.linalg.solve(A1, torch.stack([binned(tod.double() * w[k]) for k in range(ncomp)], 1))
    assert (q - want).norm() <= 1e-10 * want.norm()
