"""Gradient rows where the launch shapes change: a spin without electrons
(its orbital and envelope weights are not written by any product), batches
large enough for several electrons per CTA of the message adjoint, and more
(walker, determinant) products than a grid's third dimension holds.

Tolerances as in the gradient tests: FP64 1e-9 max(|g|, 1) per entry; float32
1e-4 + 2 kappa u of a walker's gradient norm.  Large float32 batches are
compared with the rows of small ones, 1e-4 of a walker's norm: the forward
values have the same bits there, only sums are taken in another order (against
float64, single walkers near a zero of the determinant sum or of a Jastrow
factor are further off than any kappa of one matrix says, in every batch)."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import fire_oracle as O
from paper_2504_06087_gb300 import fire, synth

pytestmark = pytest.mark.gpu


def _model(n, n_up, n_det, seed, width=32):
    s = synth.System(np.array([[0.0, 0.0, 0.0], [2.0, 0.0, 0.5]]), np.array([3.0, 3.0]), n, n_up)
    arch = synth.Arch(width=width, n_layers=1, n_det=n_det, n_env=2, jastrow_width=32)
    return s, arch, synth.init_params(s, arch, seed)


def _rows(f, r):
    """grad_logpsi into a buffer of NaNs: an entry that nothing writes stays one."""
    r = torch.as_tensor(r, dtype=torch.float64, device=f.device).contiguous()
    W = r.shape[0]
    g = torch.full((W, f.n_params), float("nan"), dtype=f.theta.dtype, device=f.device)
    la, sg = (torch.empty(W, dtype=torch.float64, device=f.device) for _ in range(2))
    ws, info, vp = f.workspace(W, fire.OP_GRAD_LOGPSI), fire.Info(), ctypes.c_void_p
    rc = fire.lib().fire_grad_logpsi(ctypes.byref(f.sys_c), ctypes.byref(f.arch_c), ctypes.byref(f.params_c), W,
                                     vp(r.data_ptr()), f.k_cap, f.prec, vp(g.data_ptr()), vp(la.data_ptr()),
                                     vp(sg.data_ptr()), ctypes.byref(info), vp(ws.data_ptr()), ws.numel(),
                                     vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    return g.double().cpu().numpy()


def _oracle(f, s, arch, p, r):
    ref = O.grad_logpsi(s, arch, p, r)
    return np.concatenate([np.asarray(ref[name]).reshape(r.shape[0], -1) for name, _, _ in f.layout], 1)


def _close64(g, ref):
    assert (np.abs(g - ref) <= 1e-9 * np.maximum(np.abs(ref), 1.0)).all()


@pytest.mark.parametrize("n_up", [0, 3])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_one_spin_alone(n_up, prec):
    s, arch, p = _model(3, n_up, 2, 21)
    r = np.random.default_rng(22).standard_normal((3, 3, 3)) * 1.5
    f = fire.Fire(s, arch, p, prec)
    g, ref = _rows(f, r), _oracle(f, s, arch, p, r)
    if prec == "fp64":
        return _close64(g, ref)
    _norm32(g, ref, s, arch, p, r)
    # the absent spin's weights get exactly zero
    for name, off, sh in f.layout:
        if name in ("orb_w", "env_pi"):
            half = int(np.prod(sh)) // 2
            z = g[:, off:off + half] if n_up == 0 else g[:, off + half:off + 2 * half]
            assert (z == 0).all()


def _norm32(g, ref, s, arch, p, r):
    pt, rt = O.params_to_torch(p), torch.as_tensor(r)
    phi = O.orbitals(s, arch, pt, rt, O.embeddings(s, arch, pt, rt)[2]).numpy()
    kappa = np.linalg.cond(phi).reshape(r.shape[0], -1).max(1)
    norm = np.linalg.norm(g - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert (norm <= 1e-4 + 2.0 * kappa * 2.0 ** -24).all()


def _same(g, parts, prec):
    if prec == "fp64":
        _close64(g, parts)
    else:
        assert (np.linalg.norm(g - parts, axis=1) <= 1e-4 * np.linalg.norm(parts, axis=1)).all()


# n W / 608 electrons a CTA, at most 8 and at most n: 4 + 1, 8 + 2 and 8 of 8 electrons
@pytest.mark.parametrize("n,W", [(5, 500), (10, 700), (8, 700)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_several_electrons_per_cta(n, W, prec):
    s, arch, p = _model(n, (n + 1) // 2, 2, 31)
    r = synth.walkers(s, W, 32)
    f = fire.Fire(s, arch, p, prec)
    parts = np.concatenate([_rows(f, r[k:k + 50]) for k in range(0, W, 50)])   # one electron a CTA
    _same(_rows(f, r), parts, prec)
    if prec == "fp64":
        _close64(parts[-2:], _oracle(f, s, arch, p, r[-2:]))


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_more_products_than_a_grid_dimension(prec):
    """64 determinants x 1030 walkers = 65920 batched products."""
    s, arch, p = _model(3, 2, 64, 41)
    r = synth.walkers(s, 1030, 42)
    f = fire.Fire(s, arch, p, prec)
    parts = np.concatenate([_rows(f, r[k:k + 515]) for k in (0, 515)])
    _same(_rows(f, r), parts, prec)
    if prec == "fp64":
        _close64(parts[-2:], _oracle(f, s, arch, p, r[-2:]))
