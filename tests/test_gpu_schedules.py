"""GPU: the three-kernel route of plans that are not run as one launch: every tile width, thread
count and radix order of the general kernels, the compile-time kernels of short chunks, and graph
replay with its separately launched last iteration.  Short chunks come through the stage calls, which
never take the one-launch route; the solver calls on plans too long for it."""
import math

import numpy as np
import pytest

import oracle.messenger as O
from paper_1705_01893_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
INF = math.inf


def _problem(lens, ncomp, half=False, seed=5, npix=61):
    rng = np.random.default_rng(seed)
    n = int(sum(lens))
    pix = np.repeat(rng.integers(-1, npix, size=n // 3 + 1), 3)[:n].astype(np.int32)
    psi = rng.uniform(0, np.pi, n)
    wt = np.float16 if half else np.float32
    cos, sin = (np.cos(2 * psi).astype(wt), np.sin(2 * psi).astype(wt)) if ncomp == 3 else (None, None)
    return dict(pix=pix, cos=cos, sin=sin, tod=rng.standard_normal(n).astype(np.float32), npix=npix, ncomp=ncomp,
                offsets=np.concatenate([[0], np.cumsum(lens)]).astype(np.int64),
                params=np.array([[1.0 + 0.1 * c, 0.5, 1.5, 50.0] for c in range(len(lens))]))


def _stages(plan, m0, lam, ncomp):
    """One step through the stage calls: (map, chi^2)."""
    m, out = torch.from_numpy(m0.copy()).cuda(), torch.zeros(*m0.shape, dtype=torch.float64, device="cuda")
    chi = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan.stage(binding.MM_STAGE_LOAD, map_inout=m)
    for b in range(plan.n_batches()):
        plan.stage(binding.MM_STAGE_GATHER_FFT, b)
        plan.stage(binding.MM_STAGE_FILTER, b, lam, chi2_slot=chi)
        plan.stage(binding.MM_STAGE_IFFT_BIN, b)
    plan.stage(binding.MM_STAGE_MAP, map_inout=out)
    return out.cpu().numpy(), chi.item()


def _check_stages(plan, prob, shape):
    m0 = np.random.default_rng(4).standard_normal(shape) * prob.valid[:, None]
    for lam in (INF, 3.0, 1.0):
        ref, chi_ref = O.messenger_step(prob, m0, lam)
        got, chi = _stages(plan, m0, lam, shape[1])
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref), lam
        assert abs(chi - chi_ref) <= 1e-5 * chi_ref, lam


@pytest.mark.parametrize("ncomp,half", [(1, False), (3, False), (3, True)])
@pytest.mark.parametrize("tune", [(8, 256, 256, 0), (16, 512, 1024, 1), (8, 512, 512, 2), (16, 256, 256, 2),
                                  (16, 512, 512, 0), (8, 256, 1024, 1)])
def test_general_schedules(tune, ncomp, half):
    """Even, odd and ragged tiles (M2 not a multiple of the tile) of every width: a step at three
    lambdas within 1e-5 of the oracle."""
    s = _problem([3125, 4500, 6561, 9000, 11520], ncomp, half)
    prob = O.problem_from_synth(s)
    plan = binding.plan_from_synth(s)
    plan.set_tune(*tune)
    assert plan.tune == tune
    _check_stages(plan, prob, (s["npix"], ncomp))


@pytest.mark.parametrize("ncomp,half", [(1, False), (3, False), (3, True)])
@pytest.mark.parametrize("log_n", range(9, 19))
def test_compile_time_shapes(log_n, ncomp, half):
    """Every column and row length of the compile-time kernels up to 2^18 samples, two chunks."""
    s = _problem([1 << log_n] * 2, ncomp, half, seed=log_n)
    _check_stages(binding.plan_from_synth(s), O.problem_from_synth(s), (s["npix"], ncomp))


# each holds a chunk above the one-launch route's largest (16 x 6144 complex samples)
@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("lens", [[1 << 18], [1 << 18, 1 << 12, 1 << 12], [200000, 3125, 4500], [1 << 18, 202500]])
def test_graph_replay(lens, ncomp):
    """Graph replay and host launches give the iterate and chi^2 of the oracle, whatever the number of
    iterations (the last one is launched by itself, with the caller's map and chi^2 slot), twice on one
    plan; the two differ by the order of FP64 additions, hence by FP32 rounding of a map at most."""
    s = _problem(lens, ncomp)
    prob = O.problem_from_synth(s)
    plan = binding.plan_from_synth(s)
    assert plan.n_fused_batches() == 0
    lam = [INF, 40.0, 5.0, 1.0]
    for k in (1, 2, 4):
        ref, chi_ref = O.run_messenger(prob, lam[:k])
        for call in (plan.messenger, plan.messenger_graph, plan.messenger_graph):
            m = torch.zeros(s["npix"], ncomp, dtype=torch.float64, device="cuda")
            chi = torch.zeros(k, dtype=torch.float64, device="cuda")
            call(m, lam[:k], chi)
            assert np.linalg.norm(m.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref), k
            assert np.max(np.abs(chi.cpu().numpy() - chi_ref) / chi_ref) <= 1e-5, k
