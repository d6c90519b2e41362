"""The widest network of each form: 512 columns in float32 and BF16_FP64, 256
in float64 and in the gradient of every form (the kernels with one thread per
column are launched at the limit of their registers there).  Wider ones are
refused by the plan, before anything is launched."""
import ctypes
import os

import numpy as np
import pytest
import torch

from oracle import fire_oracle as O
from oracle import mcmc_oracle as M
from oracle import spin_oracle as S
from paper_2504_06087_gb300 import fire, synth

FORWARD = {"fp64": 256, "fp32": 512, "bf16": 512}
GRAD = 256


def _model(width):
    s = synth.System(np.array([[0.0, 0.0, 0.0], [1.6, 0.0, 0.3]]), np.array([2.0, 2.0]), 4, 2)
    arch = synth.Arch(width=width, n_layers=1, n_det=2, jastrow_width=64)
    return s, arch, synth.init_params(s, arch, 11), synth.walkers(s, 3, 12)


@pytest.mark.parametrize("prec", list(FORWARD))
def test_plan_takes_the_widest_and_refuses_the_next(prec):
    if not os.path.exists(fire.LIB_PATH):
        from paper_2504_06087_gb300 import build
        build.build()
    L = fire.lib()
    s, arch, _, _ = _model(32)
    sys_c = fire.System(s.n_el, s.n_up, s.n_nuc, 0, None, None, s.cutoff, s.cutoff_nuc)
    for op, widest in ((fire.OP_LOGPSI, FORWARD[prec]), (fire.OP_LOCAL_ENERGY, FORWARD[prec]),
                       (fire.OP_MCMC, FORWARD[prec]), (fire.OP_GRAD_LOGPSI, GRAD)):
        for width, ok in ((32, True), (widest, True), (widest + 32, False), (1024, False)):
            arch.width = width
            a = fire.make_arch(arch)
            size = L.fire_workspace_size(ctypes.byref(sys_c), ctypes.byref(a), 3, fire.PREC[prec], 64, op)
            n, wc = ctypes.c_int32(0), ctypes.c_int64(0)
            rc = L.fire_workspace_layout(ctypes.byref(sys_c), ctypes.byref(a), 3, fire.PREC[prec], 64, op, None,
                                         ctypes.byref(n), ctypes.byref(wc))
            assert (size > 0) == ok and rc == (0 if ok else 7), (op, width, size, rc)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", list(FORWARD))
def test_widest_forward_calls_match_oracle(prec):
    """The bounds that include/fire.h states: E_L within tau of the magnitudes
    of its kinetic terms, log|Psi| within tau_l (3e-5 for BF16_FP64 at small
    |log|Psi||, about 10 here); moves and swaps as in their own tests."""
    s, arch, p, r = _model(FORWARD[prec])
    tau, tau_l = {"fp64": (1e-10, 1e-10), "fp32": (1e-4, 1e-5), "bf16": (1e-4, 3e-5)}[prec]
    f = fire.Fire(s, arch, p, prec)
    e, la, sg, _, _, g, lap = O.local_energy(s, arch, p, r, return_parts=True)
    out = f.local_energy(r)
    scale = np.maximum(np.maximum(np.abs(e), 1.0), np.abs(np.asarray(lap)) + (np.asarray(g) ** 2).sum(axis=(1, 2)))
    np.testing.assert_array_equal(out["sign"].cpu().numpy(), np.asarray(sg))
    assert (np.abs(out["e_loc"].cpu().numpy() - np.asarray(e)) <= tau * scale).all()
    for got in (out["logabs"], f.logpsi(r)["logabs"]):
        assert (np.abs(got.cpu().numpy() - np.asarray(la)) <= tau_l * np.maximum(np.abs(la), 1.0)).all()
    ref = M.mcmc_sweeps(s, arch, p, r, 0.3, 1, 7, 0)
    rr = torch.as_tensor(r, device=f.device).clone()
    acc = f.mcmc_step(rr, 0.3, 1, seed=7)["accepted"].cpu().numpy()
    safe = ref["margin"] > (1e-8 if prec == "fp64" else 1e-3)
    assert safe.any()
    np.testing.assert_array_equal(acc[safe], ref["accepted"][safe])
    np.testing.assert_allclose(rr.cpu().numpy()[safe], ref["r"][safe], rtol=0, atol=1e-9)
    sw, _ = S.swap_ratios(s, arch, p, r, 3)
    got = f.spin_ratios(r, 3)["ratios"].cpu().numpy()
    assert (np.abs(got - sw) <= (1e-10 if prec == "fp64" else 1e-3) * np.maximum(np.abs(sw), 1.0)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", list(FORWARD))
def test_widest_gradient_matches_oracle(prec):
    """FP64: 1e-9 of max(|g|, 1) per entry.  Float32 forms: 1e-4 + 2 kappa u of
    a walker's gradient norm, kappa the condition number of its worst orbital
    matrix (the bound of the stored-oracle test)."""
    s, arch, p, r = _model(GRAD)
    f = fire.Fire(s, arch, p, prec)
    g = f.grad_logpsi(r)["grad"].cpu().numpy().astype(np.float64)
    refd = O.grad_logpsi(s, arch, p, r)
    ref = np.concatenate([np.asarray(refd[name]).reshape(3, -1) for name, _, _ in f.layout], 1)
    if prec == "fp64":
        assert (np.abs(g - ref) <= 1e-9 * np.maximum(np.abs(ref), 1.0)).all()
        return
    pt = O.params_to_torch(p)
    rt = torch.as_tensor(r)
    phi = O.orbitals(s, arch, pt, rt, O.embeddings(s, arch, pt, rt)[2]).numpy()
    kappa = np.linalg.cond(phi).reshape(3, -1).max(1)
    norm = np.linalg.norm(g - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert (norm <= 1e-4 + 2.0 * kappa * 2.0 ** -24).all(), (norm, kappa)
