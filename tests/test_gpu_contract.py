"""The float32 log-det contraction at the edges of its member buckets (24, 36,
60) and for every alignment of its rows (n a multiple of 4, even, odd), with
c beyond the molecule so that every neighbourhood has n members."""
import numpy as np
import pytest

from oracle import fire_oracle as O
from paper_2504_06087_gb300 import fire, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 5, 6, 24, 25, 33, 35, 36, 37, 38, 59, 60])
@pytest.mark.parametrize("variant", [None, "v2"])
def test_contraction_matches_oracle(n, variant, monkeypatch):
    """E_L within 1e-4 of the sum of its kinetic terms' magnitudes (the float32
    bound of the parity tests: a sum's rounding is relative to its summands)."""
    pos = np.array([[2.1 * k, 0.4 * (k % 2), 0.3 * (k % 3)] for k in range(max(1, n // 5))])
    s = synth.System(pos, np.full(pos.shape[0], 5.0), n, (n + 1) // 2, cutoff=100.0)
    arch = synth.Arch(width=64, n_layers=1, n_det=2)
    p = synth.init_params(s, arch, 5)
    r = synth.walkers(s, 2, 17)
    e, la, sg, kin, v, g, lap = O.local_energy(s, arch, p, r, return_parts=True)
    if variant:
        monkeypatch.setenv("FIRE_CONTRACT", variant)
    out = fire.Fire(s, arch, p, "fp32").local_energy(r)
    scale = np.maximum(np.maximum(np.abs(e), 1.0), np.abs(np.asarray(lap)) + (np.asarray(g) ** 2).sum(axis=(1, 2)))
    np.testing.assert_array_equal(out["sign"].cpu().numpy(), np.asarray(sg))
    assert (np.abs(out["e_loc"].cpu().numpy() - np.asarray(e)) <= 1e-4 * scale).all()
