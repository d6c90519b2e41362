"""The float64 factorisation and inverse of the Metropolis state at the edges
of their tiles (4 rows, 32 columns, the whole-matrix limit of 119), against
numpy.  For A computed from an LU with partial pivoting, ||Phi A - I|| is
bounded by a modest multiple of n u ||Phi||_F ||A||_F (u = 2^-53; the factor 16
covers the pivot growth), and log|det| by n u ||Phi||_F ||A||_F."""
import numpy as np
import pytest
import torch

from paper_2504_06087_gb300 import fire, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 58, 64, 65, 119, 120, 130])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_refresh_factorisation_and_inverse(n, precision):
    pos = np.array([[1.7 * k, 0.4 * (k % 2), 0.0] for k in range(max(1, n // 6))])
    z = np.full(pos.shape[0], 6.0)
    system = synth.System(pos, z, n, (n + 1) // 2)
    arch = synth.Arch(width=64, n_layers=1, n_det=3)
    f = fire.Fire(system, arch, synth.init_params(system, arch, 3), precision, k_cap=130)
    W = 2
    r = torch.as_tensor(synth.walkers(system, W, 5), device="cuda")
    f.mcmc_step(r, 0.3, 0)
    dt = torch.float64 if precision == "fp64" else torch.float32
    view = lambda k, t, s: f.ws_view(W, fire.OP_MCMC, k, t, s).double().cpu().numpy()  # noqa: E731
    phi, at = view("PhiS", dt, (W * 3, n, n)), view("Ainv", dt, (W * 3, n, n))
    la, sg = view("ldabs", torch.float64, (W * 3,)), view("lsign", torch.float64, (W * 3,))
    u = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24   # A is stored in the state's type
    for m in range(W * 3):
        A = at[m].T
        kappa = np.linalg.norm(phi[m]) * np.linalg.norm(A)
        # Phi itself is kept rounded to the state's type too, the factors are of the unrounded matrix
        assert np.abs(phi[m] @ A - np.eye(n)).max() <= 16 * n * u * kappa
        s, l = np.linalg.slogdet(phi[m])
        assert s == sg[m]
        assert abs(l - la[m]) <= 16 * n * u * kappa + 1e-12 * abs(l)
