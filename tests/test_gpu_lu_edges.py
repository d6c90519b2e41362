"""Factorisations and inverses at the edges of their kernels (4 rows, 32
columns, the whole-matrix limits of 119 in float64 and 169 in float32), on
well-conditioned matrices, so that the bounds are far below one.

One electron sits near each nucleus of a chain, in an order that makes every
column search for its pivot; orbital l is exp(-|r - R_l|) around nucleus l, so
Phi is a row-permuted, diagonally dominant matrix (kappa_F about n).

The Metropolis state holds Phi and A = Phi^-1 rounded to its type from a
float64 Phi and inverse: Phi A - I is at most 2 u kappa_F (u of the type, first order)
and log|det| of the rounded Phi differs by at most u kappa_F; the factor 1.1 and
the float64 term cover the rest.  fire_logpsi in float32 factorises in
float32: max(t max(|l|, 1), n kappa u), t = 1e-10 or 1e-5, the bound of the parity
tests (a wrong pivot or column changes |l| by far more)."""
import numpy as np
import pytest
import torch

from oracle import fire_oracle as O
from paper_2504_06087_gb300 import fire, synth
from recipes import const_h_params

pytestmark = pytest.mark.gpu


def _model(n):
    pos = np.array([[3.0 * k, 0.0, 0.0] for k in range(n)])
    s = synth.System(pos, np.ones(n), n, (n + 1) // 2)
    arch = synth.Arch(width=32, n_layers=1, n_det=2, n_env=1, jastrow_width=32, flags=0)
    p = const_h_params(s, arch, 1)
    p["orb_w"][:] = 1.0
    p["env_pi"][:] = 0.0
    for q in range(n):
        p["env_pi"][:, :, q, q, 0] = 1.0
    p["env_sigma"][:] = 1.0
    g = np.random.default_rng(n)
    r = np.stack([pos[g.permutation(n)] for _ in range(2)]) + 0.2 * g.standard_normal((2, n, 3))
    return s, arch, p, r


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 64, 65, 119, 120, 130])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_state_factorisation_and_inverse(n, prec):
    s, arch, p, r0 = _model(n)
    f = fire.Fire(s, arch, p, prec, k_cap=130)
    r = torch.as_tensor(r0, device=f.device).clone()
    f.mcmc_step(r, 0.3, 0)
    dt = torch.float64 if prec == "fp64" else torch.float32
    view = lambda k, t, sh: f.ws_view(2, fire.OP_MCMC, k, t, sh).double().cpu().numpy()  # noqa: E731
    phi, at = view("PhiS", dt, (4, n, n)), view("Ainv", dt, (4, n, n))
    la, sg = view("ldabs", torch.float64, (4,)), view("lsign", torch.float64, (4,))
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    for m in range(4):
        kappa = np.linalg.norm(phi[m]) * np.linalg.norm(np.linalg.inv(phi[m]))
        lu = 16 * n * 2.0 ** -53 * kappa      # the float64 factorisation itself
        bound = 1.1 * 2 * u * kappa + lu
        assert bound < 1e-3
        assert np.abs(phi[m] @ at[m].T - np.eye(n)).max() <= bound
        sr, lr = np.linalg.slogdet(phi[m])
        assert sr == sg[m] and abs(lr - la[m]) <= 1.1 * u * kappa + lu + 1e-14 * abs(lr)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 119, 120, 168, 169, 170, 171])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_log_determinant(n, prec):
    s, arch, p, r = _model(n)
    la, sg = O.logpsi_np(s, arch, p, r)
    out = fire.Fire(s, arch, p, prec, k_cap=n).logpsi(r)
    pt, rt = O.params_to_torch(p), torch.as_tensor(r)
    phi = O.orbitals(s, arch, pt, rt, O.embeddings(s, arch, pt, rt)[2]).numpy()
    kappa = np.linalg.cond(phi[:, 0])
    assert kappa.max() < 100
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    np.testing.assert_array_equal(out["sign"].cpu().numpy(), sg)
    err = np.abs(out["logabs"].cpu().numpy() - la)
    t = 1e-10 if prec == "fp64" else 1e-5
    assert (err <= np.maximum(t * np.maximum(np.abs(la), 1.0), n * kappa * u)).all(), err


@pytest.mark.parametrize("n", [58, 119, 120])
def test_second_stream_factorises_alike(n, monkeypatch):
    """FIRE_LU_SIDE moves the float64 LU to another stream: the same kernel, the same bits."""
    s, arch, p, r = _model(n)
    f = fire.Fire(s, arch, p, "bf16", k_cap=n)
    ref = f.logpsi(r)["logabs"].cpu().numpy()
    monkeypatch.setenv("FIRE_LU_SIDE", "1")
    np.testing.assert_array_equal(f.logpsi(r)["logabs"].cpu().numpy(), ref)
