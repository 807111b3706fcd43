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
