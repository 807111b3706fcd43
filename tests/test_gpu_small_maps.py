"""GPU: the one-launch path of small plans is taken for maps that its own CTAs update quickly, and not
for large ones, whose map step belongs on the whole GPU."""
import math

import numpy as np
import pytest

import oracle.messenger as O
from paper_1705_01893_gb300 import binding

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plan(lens, npix, ncomp, seed=3):
    rng = np.random.default_rng(seed)
    n = int(sum(lens))
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    seen = rng.choice(npix, size=min(npix, 50), replace=False)          # the map is mostly unhit
    seen[:2] = (0, npix - 1)
    pix = seen[rng.integers(0, len(seen), n // 2 + 1)].repeat(2)[:n].astype(np.int32)
    psi = rng.uniform(0, np.pi, n)
    cos, sin = (np.cos(2 * psi).astype(np.float32), np.sin(2 * psi).astype(np.float32)) if ncomp == 3 else (None, None)
    s = dict(pix=pix, cos=cos, sin=sin, tod=rng.standard_normal(n).astype(np.float32), npix=npix, ncomp=ncomp,
             offsets=off, params=np.array([[1.0 + 0.1 * c, 0.5, 1.5, 20.0] for c in range(len(lens))]))
    return binding.plan_from_synth(s), O.problem_from_synth(s)


@pytest.mark.parametrize("ncomp,npix", [(1, 1 << 22), (3, 1 << 20)])
def test_large_maps_keep_the_full_gpu_map_step(ncomp, npix):
    """Only the one-launch path waits on other CTAs in a plan like this one (no chunk is long enough
    for the fused launch), so that a one-poll limit would run out in it."""
    plan, prob = _plan([1 << 13] * 6, npix, ncomp)
    assert plan.n_fused_batches() == 0
    plan.set_wait_policy(1, True)
    m = torch.zeros(npix, ncomp, dtype=torch.float64, device="cuda")
    plan.messenger(m, [math.inf, 5.0])
    assert plan.fault_flags() == 0
    ref, _ = O.run_messenger(prob, [math.inf, 5.0])
    assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)


# 8 CTAs: the limit lies at 8 x 20480 (T) and 8 x 4096 (IQU) pixels
@pytest.mark.parametrize("ncomp,limit", [(1, 163840), (3, 32768)])
@pytest.mark.parametrize("over", [0, 1])
def test_both_sides_of_the_limit(ncomp, limit, over):
    npix = limit + over
    plan, prob = _plan([1 << 12], npix, ncomp)
    m = torch.zeros(npix, ncomp, dtype=torch.float64, device="cuda")
    plan.messenger(m, [math.inf, 5.0, 1.0])
    ref, _ = O.run_messenger(prob, [math.inf, 5.0, 1.0])
    assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("over", [0, 1, 255, 511])
def test_two_pixels_a_thread(ncomp, over):
    """The map step's two-pixel form, from 2^19 pixels on, at the ends of its last block."""
    npix = (1 << 19) + over
    plan, prob = _plan([1 << 12], npix, ncomp, seed=over)
    m = torch.ones(npix, ncomp, dtype=torch.float64, device="cuda")
    plan.messenger(m, [math.inf, 5.0])
    ref, _ = O.run_messenger(prob, [math.inf, 5.0])
    assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
