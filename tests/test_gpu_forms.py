"""Every precision form in one process, in an order in which each first call
meets kernels whose shared-memory limit another form has or has not raised."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import numpy as np, torch
from paper_2504_06087_gb300 import fire, synth
s = synth.zigzag_polyene(14, terminal_h=False)
a = synth.Arch(width=64, n_layers=1, n_det=2)
p, r = synth.init_params(s, a, 1), synth.walkers(s, 2, 2)
ref = None
for prec in "{order}".split():
    f = fire.Fire(s, a, p, prec)
    l = f.logpsi(r)["logabs"].double().cpu().numpy()
    assert np.isfinite(f.local_energy(r)["e_loc"].cpu().numpy()).all()
    rr = torch.as_tensor(r, device="cuda").clone()
    f.mcmc_step(rr, 0.1, 0)
    torch.cuda.synchronize()
    ref = l if ref is None else ref
    assert np.allclose(l, ref, rtol=1e-3), (prec, l, ref)
print("all forms ran")
"""


@pytest.mark.parametrize("order", ["fp32 bf16 fp64", "bf16 fp32 fp64", "fp64 fp32 bf16"])
def test_every_form_after_every_other(order):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    q = subprocess.run([sys.executable, "-c", CHILD.format(order=order)], cwd=root, capture_output=True, text=True,
                       timeout=600)
    assert q.returncode == 0 and "all forms ran" in q.stdout, q.stderr[-2000:]
