"""The low-rank update at the edges of its kernels: systems up to and beyond
192 electrons, update sets up to and beyond 64 and 192 members.  A float64
state carried through a sweep has to make the decisions of one that is rebuilt
after every move, and its log|Psi| may leave the rebuild's by what first-order
perturbation allows: n kappa u per move (kappa the Frobenius condition estimate of
the worst determinant)."""
import numpy as np
import pytest
import torch

from paper_2504_06087_gb300 import fire, synth

pytestmark = pytest.mark.gpu
W = 3

# n, cutoff, smallest and largest |U| that the case is there for
CASES = [
    (64, 4.0, 1, 64), (65, 4.0, 1, 64), (65, 200.0, 65, 65), (129, 4.0, 1, 64), (150, 200.0, 150, 150),
    (192, 4.0, 1, 64), (193, 4.0, 1, 64), (193, 14.0, 65, 192), (200, 200.0, 200, 200),
]


def _model(n, cutoff):
    pos = np.array([[2.2 * k, 0.6 * (k % 2), 0.0] for k in range(max(1, n // 4))])
    s = synth.System(pos, np.full(pos.shape[0], 4.0), n, (n + 1) // 2, cutoff=cutoff)
    arch = synth.Arch(width=32, n_layers=1, n_det=2, n_env=4, jastrow_width=32, n_reg=4, d_reg=8)
    return s, arch, synth.init_params(s, arch, 3), synth.walkers(s, W, 4)


@pytest.mark.parametrize("n,cutoff,lo,hi", CASES)
def test_float64_update_follows_the_rebuilds(n, cutoff, lo, hi):
    s, arch, p, r0 = _model(n, cutoff)
    near = (np.linalg.norm(r0[:, :, None] - r0[:, None], axis=-1) <= cutoff).sum(-1)   # electron itself included
    assert near.max() <= hi and (near >= lo).any()
    out = []
    for refresh in (1, 0):
        f = fire.Fire(s, arch, p, "fp64", k_cap=n)
        r = torch.as_tensor(r0, device=f.device).clone()
        o = f.mcmc_step(r, 0.2, 1, refresh_every=refresh, seed=6)
        kap = f.ws_view(W, fire.OP_MCMC, "mc_kap", torch.float32, (W * 2,)).max().item()
        out.append((r.cpu().numpy(), o, kap))
    (ra, oa, _), (rb, ob, kap) = out
    assert 0 < ob["n_accepted"]
    np.testing.assert_array_equal(oa["accepted"].cpu().numpy(), ob["accepted"].cpu().numpy())
    np.testing.assert_allclose(ra, rb, rtol=0, atol=1e-11)
    bound = n * n * kap * 2.0 ** -53
    assert ob["max_drift"] <= bound < 1e-2, (ob["max_drift"], bound)


@pytest.mark.parametrize("n,cutoff,lo,hi", [c for c in CASES if c[0] in (65, 192, 193, 200)])
def test_float32_update_keeps_the_state(n, cutoff, lo, hi):
    """Rebuilt every 32 moves: the conditioning test bounds what a move can bring
    into log|Psi| by 1e-4 (1e-2 is the bound of the sampler's own test)."""
    s, arch, p, r0 = _model(n, cutoff)
    f = fire.Fire(s, arch, p, "fp32", k_cap=n)
    r = torch.as_tensor(r0, device=f.device).clone()
    o = f.mcmc_step(r, 0.2, 1, refresh_every=32, seed=6)
    assert 0 < o["n_accepted"] and o["max_drift"] < 1e-2, o["max_drift"]
