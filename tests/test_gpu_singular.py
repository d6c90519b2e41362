"""A batch in which one walker's orbital matrices are exactly singular: an
electron beyond every cutoff has a zero embedding and a zero row.  Its
neighbours in the batch keep their results, and the call comes back (the
float32 inverse of such a matrix meets columns without a pivot)."""
import numpy as np
import pytest
import torch

from oracle import fire_oracle as O
from paper_2504_06087_gb300 import fire, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 5, 13, 24, 40])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_singular_walker_leaves_the_others_alone(n, prec):
    pos = np.array([[2.0 * k, 0.5 * (k % 2), 0.0] for k in range(max(1, n // 3))])
    s = synth.System(pos, np.full(pos.shape[0], 3.0), n, (n + 1) // 2, cutoff=2.0, cutoff_nuc=4.0)
    arch = synth.Arch(width=64, n_layers=0, n_det=2, n_env=4, jastrow_width=32)
    p = synth.init_params(s, arch, 6)
    r = np.random.default_rng(7).standard_normal((3, n, 3)) * 0.5 + pos[np.arange(n) % pos.shape[0]]
    r[1, n // 2] = [0.0, 40.0, 0.0]
    keep = [0, 2]
    f = fire.Fire(s, arch, p, prec)
    g = f.grad_logpsi(r, check=False)
    torch.cuda.synchronize()
    assert g["status"] in (0, 3)
    assert g["sign"][1] == 0 and g["logabs"][1] == -np.inf
    ref = f.grad_logpsi(r[keep])
    a, b = g["grad"][keep].double().cpu().numpy(), ref["grad"].double().cpu().numpy()
    assert (np.linalg.norm(a - b, axis=1) <= 1e-5 * np.linalg.norm(b, axis=1)).all()
    la, sg = O.logpsi_np(s, arch, p, r[keep])
    np.testing.assert_array_equal(g["sign"][keep].cpu().numpy(), sg)
    np.testing.assert_allclose(g["logabs"][keep].cpu().numpy(), ref["logabs"].cpu().numpy(), rtol=0, atol=0)
    e = f.local_energy(r, check=False)
    torch.cuda.synchronize()
    assert e["status"] in (0, 3) and e["sign"][1] == 0
    e2 = f.local_energy(r[keep])
    np.testing.assert_array_equal(e["logabs"][keep].cpu().numpy(), e2["logabs"].cpu().numpy())
