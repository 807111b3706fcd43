"""GPU: the one-launch path of small plans (thread-block clusters, distributed shared memory)
against the FP64 oracle: shortest chunks, odd and prime-power lengths, one and several clusters,
more chunks than clusters, T-only and IQU, FP32 and FP16 weights, schedules longer than one
launch's 128 iterations, a grid barrier that runs out."""
import math

import numpy as np
import pytest

import oracle.messenger as O
from paper_1705_01893_gb300 import synth

pytestmark = pytest.mark.gpu


def _data(lens, npix, ncomp, seed, half=False):
    rng = np.random.default_rng(seed)
    n = int(sum(lens))
    pix = np.repeat(rng.integers(-1, npix, size=n // 3 + 1), 3)[:n].astype(np.int32)
    pix[:npix] = np.arange(npix)[:n]
    psi = rng.uniform(0, np.pi, n)
    wt = np.float16 if half else np.float32
    m = rng.standard_normal((npix, ncomp))
    cos, sin = np.cos(2 * psi).astype(wt), np.sin(2 * psi).astype(wt)
    w = np.stack([np.ones(n), cos.astype(np.float64), sin.astype(np.float64)], 1)[:, :ncomp]
    tod = np.where(pix >= 0, np.sum(w * m[np.maximum(pix, 0)], 1), 0.0) + rng.standard_normal(n)
    return dict(pix=pix, cos=cos if ncomp == 3 else None, sin=sin if ncomp == 3 else None,
                tod=tod.astype(np.float32), npix=npix, ncomp=ncomp,
                offsets=np.concatenate([[0], np.cumsum(lens)]).astype(np.int64),
                params=np.array([[1.0 + 0.1 * c, 0.5, 1.5 + 0.01 * c, 20.0] for c in range(len(lens))]))


CASES = [([512], 16), ([4, 5, 6, 8, 9, 10], 5), ([625, 729, 2187, 1000, 6000], 40), ([1 << 15], 64),
         ([8192] * 40, 300), ([600] * 200, 100), ([45000, 30375], 64), ([1 << 14, 3000, 1 << 13], 50)]


@pytest.mark.parametrize("ncomp,half", [(1, False), (3, False), (3, True)])
@pytest.mark.parametrize("lens,npix", CASES)
def test_small_plan_matches_oracle(lens, npix, ncomp, half):
    """Three cooled iterations through both entry points: map <= 1e-5, chi^2 <= 1e-5 of the
    oracle (the tolerances of the other paths' step tests)."""
    import torch
    from paper_1705_01893_gb300 import binding
    s = _data(lens, npix, ncomp, 5, half)
    prob = O.problem_from_synth(s)
    if not prob.valid.any():
        pytest.skip("every pixel cut")
    lam = [math.inf, max(2.0, math.sqrt(O.lambda_max(prob))), 1.0]
    ref, chi_ref = O.run_messenger(prob, lam)
    plan = binding.plan_from_synth(s)
    for call in (plan.messenger, plan.messenger_graph, plan.messenger):
        m = torch.zeros(npix, ncomp, dtype=torch.float64, device="cuda")
        chi = torch.zeros(3, dtype=torch.float64, device="cuda")
        call(m, lam, chi)
        assert plan.fault_flags() == 0
        scale = max(np.linalg.norm(ref), 1e-30)
        # cut blocks down to rcond 1e-3 amplify FP32 errors of poorly hit pixels
        assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * scale
        assert np.max(np.abs(chi.cpu().numpy() - chi_ref) / chi_ref) <= 1e-5


def test_long_schedule_spans_launches():
    """300 iterations (three launches) end in the iterate of the oracle."""
    import torch
    from paper_1705_01893_gb300 import binding
    s = _data([2048, 1500], 20, 1, 9)
    prob = O.problem_from_synth(s)
    lam = O.cooling_schedule(O.lambda_max(prob), 13, 23)
    ref, chi_ref = O.run_messenger(prob, lam)
    plan = binding.plan_from_synth(s)
    m = torch.zeros(20, 1, dtype=torch.float64, device="cuda")
    chi = torch.zeros(len(lam), dtype=torch.float64, device="cuda")
    plan.messenger(m, lam, chi)
    assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
    assert np.max(np.abs(chi.cpu().numpy() - chi_ref) / chi_ref) <= 1e-5


def test_expired_barrier_is_reported_and_cleared():
    """A one-poll limit lets the grid barrier of several clusters run out: MM_ERR_TIMEOUT; with
    the default limit the same plan gives the right iteration again."""
    import torch
    from paper_1705_01893_gb300 import binding
    s = synth.config_iqu(16, 6, 1 << 13, 60)
    prob = O.problem_from_synth(s)
    lam = [math.inf, 50.0, 5.0]
    ref, _ = O.run_messenger(prob, lam)
    plan = binding.plan_from_synth(s)
    plan.set_wait_policy(1, True)
    m = torch.zeros(s["npix"], 3, dtype=torch.float64, device="cuda")
    with pytest.raises(binding.MMError) as e:
        plan.messenger(m, lam)
    assert e.value.code == binding.MM_ERR_TIMEOUT
    plan.set_wait_policy()
    m.zero_()
    plan.messenger(m, lam)
    assert plan.fault_flags() == 0
    assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
