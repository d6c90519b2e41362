"""The lists of a Metropolis move (exact ratios, refactorisations) and the
kernels that take the pairs beyond their length, with determinants that enter
and leave the conditioning test.
Float64 state, where a lemma ratio and a float64 LU agree to 1e-10, so that
every choice of the conditioning tolerance and of the lists' length has to
give the same decisions; the carried log|Psi| against the rebuild at the end
shows a wrong inverse, which every later lemma ratio would use."""
import numpy as np
import pytest
import torch

from paper_2504_06087_gb300 import fire, synth

pytestmark = pytest.mark.gpu
W, D, SEED = 48, 16, 4242


def _sweeps(monkeypatch, system, arch, p, r0, tol, cap, prec="fp64", sweeps=3):
    monkeypatch.setenv("FIRE_MCMC_KAPPA_TOL", repr(tol))
    if cap:
        monkeypatch.setenv("FIRE_MCMC_LIST", str(cap))
    else:
        monkeypatch.delenv("FIRE_MCMC_LIST", raising=False)
    f = fire.Fire(system, arch, p, prec)
    r = torch.as_tensor(r0, device=f.device).clone()
    out = f.mcmc_step(r, 0.4, sweeps, refresh_every=0, seed=SEED, n_global=2)
    # refactorised pairs of the last move
    out["last"] = int(f.ws_view(W, fire.OP_MCMC, "mc_xcnt", torch.int32, (1,))[0])
    kap = f.ws_view(W, fire.OP_MCMC, "mc_kap", torch.float32, (W * D,)).double().cpu().numpy()
    return r.cpu().numpy(), out, kap


@pytest.fixture(scope="module")
def case():
    s = synth.water()
    arch = synth.Arch(width=64, n_layers=1, n_det=D)
    return s, arch, synth.init_params(s, arch, 8), synth.walkers(s, W, 9)


# conditioning tolerance in units of the median kappa u
@pytest.mark.parametrize("share", [0.5, 0.05, 0.0])
@pytest.mark.parametrize("cap", [1, 5, 0])
def test_lists_and_conditioning_test_leave_the_chain_alone(case, share, cap, monkeypatch):
    s, arch, p, r0 = case
    r_ref, ref, kap = _sweeps(monkeypatch, s, arch, p, r0, -1.0, 0)
    tol = share * float(np.median(kap)) * 2.0 ** -53
    r, out, _ = _sweeps(monkeypatch, s, arch, p, r0, tol, cap)
    assert out["n_accepted"] == ref["n_accepted"]
    np.testing.assert_array_equal(out["accepted"].cpu().numpy(), ref["accepted"].cpu().numpy())
    np.testing.assert_allclose(r, r_ref, rtol=0, atol=1e-11)
    la, la_ref = out["logabs"].cpu().numpy(), ref["logabs"].cpu().numpy()
    np.testing.assert_allclose(la, la_ref, rtol=1e-10, atol=1e-10)
    assert out["max_drift"] < 1e-8, out["max_drift"]
    pairs = W * D * 3 * (s.n_el + 2)
    assert out["n_exact"] > ref["n_exact"] and out["n_repair"] > ref["n_repair"]
    if share == 0.0:
        assert out["n_exact"] >= pairs * 0.99        # every pair, every move
    else:
        assert 0.02 * pairs < out["n_exact"] < 0.98 * pairs
    if cap:
        assert out["last"] > cap                     # more refactorisations than the list holds


@pytest.mark.parametrize("cap", [1, 0])
def test_float32_state_with_short_lists(case, cap, monkeypatch):
    """The bound of the float32 sampler tests on the carried log|Psi|."""
    s, arch, p, r0 = case
    _, _, kap = _sweeps(monkeypatch, s, arch, p, r0, 1e-4, 0, prec="fp32", sweeps=1)
    tol = 0.05 * float(np.median(kap)) * 2.0 ** -24
    _, out, _ = _sweeps(monkeypatch, s, arch, p, r0, tol, cap, prec="fp32", sweeps=1)
    assert out["n_exact"] > 0 and out["max_drift"] < 2e-3, out["max_drift"]
