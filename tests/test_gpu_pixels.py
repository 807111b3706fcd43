"""GPU: per-pixel solves at their edges: which pixels are counted as kept, and quotients that are not
finite."""
import numpy as np
import pytest

from paper_1705_01893_gb300 import binding

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix", [32, 33, 300])
@pytest.mark.parametrize("filler", ["cut", "unhit", "mixed"])
def test_one_kept_pixel_is_enough(npix, filler):
    """A plan is refused only when every pixel is cut: one well cross-linked pixel keeps it, in any
    lane of a warp, beside pixels that are unhit or cut by their eigenvalues."""
    rng = np.random.default_rng(npix)
    for keep in [*range(32), npix - 1]:
        others = np.delete(np.arange(npix), keep)
        hit = {"cut": others, "unhit": others[:0], "mixed": others[rng.random(len(others)) < 0.5]}[filler]
        # the kept pixel at 4 angles, the others four times at one angle each (singular blocks)
        pix = np.concatenate([np.full(4, keep), np.repeat(hit, 4)]).astype(np.int32)
        psi = np.concatenate([np.arange(4) * np.pi / 4, np.repeat(rng.uniform(0, np.pi, len(hit)), 4)])
        n = 1 << int(np.ceil(np.log2(max(len(pix), 8))))
        pad = n - len(pix)
        pix, psi = np.pad(pix, (0, pad), constant_values=-1), np.pad(psi, (0, pad))
        up = [torch.from_numpy(x).cuda() for x in
              (pix, np.cos(2 * psi).astype(np.float32), np.sin(2 * psi).astype(np.float32))]
        plan = binding.Plan([0, n], *up, npix, 3)
        plan.set_noise(torch.zeros(n, device="cuda"), params=np.array([[1.0, 0.5, 1.5, 20.0]]))
        valid = torch.empty(npix, dtype=torch.uint8, device="cuda")
        plan.maps(valid=valid)
        want = np.zeros(npix, np.uint8)
        want[keep] = 1
        assert np.array_equal(valid.cpu().numpy(), want)


def test_no_kept_pixel_is_refused():
    pix = torch.zeros(8, dtype=torch.int32, device="cuda")
    one = torch.ones(8, device="cuda")
    plan = binding.Plan([0, 8], pix, one, 0 * one, 40, 3)
    with pytest.raises(binding.MMError) as e:
        plan.set_noise(one, params=np.array([[1.0, 0.5, 1.5, 20.0]]))
    assert e.value.code == binding.MM_ERR_SINGULAR


def test_binned_map_of_infinite_samples():
    """One infinite sample in a pixel: each component of the allocation-free map is +inf, -inf or NaN
    as the FP64 formula adj(A) b / det gives it, and the other pixels stay finite."""
    rng = np.random.default_rng(8)
    npix, per = 64, 12
    pix = np.repeat(np.arange(npix), per).astype(np.int32)
    n = len(pix)
    psi = rng.uniform(0, np.pi, n)
    cos, sin = np.cos(2 * psi).astype(np.float32), np.sin(2 * psi).astype(np.float32)
    tod = rng.standard_normal(n).astype(np.float32)
    bad = np.arange(0, npix, 2)
    tod[bad * per + 3] = np.where(bad % 4 == 0, np.inf, -np.inf)
    w = np.stack([np.ones(n), cos, sin], 1).astype(np.float64).reshape(npix, per, 3)
    t = tod.astype(np.float64).reshape(npix, per)
    A = np.einsum("psi,psj->pij", w, w)
    adj = np.linalg.inv(A) * np.linalg.det(A)[:, None, None]
    with np.errstate(invalid="ignore"):
        want = sum(adj[:, :, k] * (t * w[:, :, k]).sum(1)[:, None] for k in range(3)) / np.linalg.det(A)[:, None]
    assert np.isinf(want).any() and np.isnan(want).any() and np.isfinite(want).any()
    out = torch.empty(npix, 3, dtype=torch.float64, device="cuda")
    up = [torch.from_numpy(x).cuda() for x in (pix, cos, sin, tod)]
    binding.binned_map_noalloc(*up, npix, 3, out, rcond_min=0.0)
    got = out.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf])
    good = np.isfinite(want)
    assert np.allclose(got[good], want[good], rtol=1e-9, atol=1e-12)
