"""The framework's work as a variational Monte Carlo program calls it, as timed cases.

One case is one call (or, for the differentiable log|Psi|, one forward and
backward pass) through ``paper_2504_06087_gb300.fire`` on seeded walkers and
weights.  The molecules are the ones of ``synth``: water with the width-64
network, and the zigzag chains C_k H_(k+2) with the width-128 network of C8H10
or the width-256 network of C26H24.

``exact`` evaluates the same quantities densely in float64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2504_06087_gb300 import fire, synth

# (width, layers, determinants) of the three networks the framework is used with
NETS = {"s": (64, 2, 4), "m": (128, 3, 8), "l": (256, 4, 16)}


def _case(name, op, mol, net, precision, walkers, **more):
    c = {"op": op, "mol": mol, "net": net, "precision": precision, "walkers": walkers, "flags": synth.J_ALL}
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a handful of walkers of a small molecule: what one call costs at least
        _case("logpsi_water_fp32_16", "logpsi", "water", "s", "fp32", 16),
        # the plain float64 reference run
        _case("energy_water_fp64_256", "energy", "water", "s", "fp64", 256),
        # single precision, middle-sized molecule
        _case("energy_c8h10_fp32_512", "energy", "C8", "m", "fp32", 512),
        # the production form on 180 electrons: tensor-core products, float64 determinants
        _case("energy_c26h24_bf16_200", "energy", "C26-", "l", "bf16", 200),
        # the same molecule in single precision
        _case("energy_c26h24_fp32_128", "energy", "C26-", "l", "fp32", 128),
        # rows of d log|Psi| / d theta for the natural-gradient optimiser
        _case("grad_c26h24_fp32_128", "grad", "C26-", "l", "fp32", 128),
        # log|Psi| as a differentiable function in a training loop
        _case("autograd_c8h10_bf16_256", "autograd", "C8", "m", "bf16", 256),
        # a sweep of single-electron moves on a chain of 100 electrons
        _case("sweep_c14h16_fp32_128", "mcmc", "C14", "l", "fp32", 128, sweeps=1, jumps=0),
        # sweeps with global jumps, float64 state
        _case("sweep_water_fp64_256", "mcmc", "water", "s", "fp64", 256, sweeps=2, jumps=5),
        # the non-local pseudopotential of an energy evaluation
        _case("ecp_c8h10_fp32_64", "ecp", "C8", "m", "fp32", 64),
        # spin-operator swap ratios
        _case("spin_c8h10_fp32_256", "spin", "C8", "m", "fp32", 256),
        # the SPRING update of one optimisation step: N rows of P parameters
        {"name": "spring_1024x1e6", "op": "spring", "rows": 1024, "params": 1000000, "momentum": True},
    ]


# Estimated seconds of a pass, to keep drawn cases below the largest listed ones.
_RATE = {"fp64": 0.15e12, "fp32": 14e12, "bf16": 60e12}
_MOST_S = 0.3


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        op = rng.choice(["logpsi", "energy", "energy", "energy", "grad", "grad", "autograd", "mcmc", "mcmc", "ecp",
                         "spin", "spring"])
        if op == "spring":
            c = {"op": op, "rows": _log_int(rng, 64, 1500), "params": _log_int(rng, 50000, 2000000),
                 "momentum": rng.random() < 0.7}
            if c["rows"] * c["params"] <= 1.2e9:
                return c
            continue
        precision = rng.choice({"mcmc": ["fp32", "fp32", "fp64"], "ecp": ["fp32"], "spin": ["fp32"],
                                "grad": ["fp32", "fp32", "bf16"]}.get(op, ["fp32", "bf16", "fp64"]))
        net = "s" if precision == "fp64" else rng.choice(["m", "l"])
        k = _log_int(rng, 2, 6 if net == "s" else 14 if op in ("mcmc", "ecp", "spin") else 26)
        mol = "water" if net == "s" and rng.random() < 0.5 else "C%d%s" % (k, rng.choice(["", "-"]))
        c = _case(None, op, mol, net, precision, _log_int(rng, 8, 1024),
                  flags=synth.J_ALL if rng.random() < 0.8 else synth.J_CUSP | synth.J_MLP)
        if op == "mcmc":
            c.update(sweeps=1, jumps=rng.choice([0, 0, 5]))
        s = _system(c)
        if op in ("grad", "autograd") and c["walkers"] * _n_params(s, _arch(c)) > 6.6e8:
            continue
        if op in ("mcmc", "ecp", "spin"):
            moves = {"mcmc": s.n_el, "ecp": 4 * s.n_el, "spin": s.n_up}[op]
            # a move of a batch takes a good part of a millisecond however small it is
            if moves * (1e-3 + work(c)["flops"] / moves / _RATE["fp32"] * 8) > _MOST_S:
                continue
        elif work(c)["flops"] / _RATE[precision] > _MOST_S:
            continue
        if op == "energy" and c["walkers"] * _scratch(s, _arch(c)) > 7e10:
            continue
        return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _system(c):
    if c["mol"] == "water":
        return synth.water()
    k = int(c["mol"].strip("C-"))
    return synth.zigzag_polyene(k, terminal_h=not c["mol"].endswith("-"))


def _arch(c):
    d, layers, dets = NETS[c["net"]]
    return synth.Arch(width=d, n_layers=layers, n_det=dets, flags=c["flags"])


def _scratch(s, a):
    """Bytes of workspace per walker of an energy call, about: rows for up to 64 neighbours of every electron."""
    rows = s.n_el * (2.0 + 3.0 * min(s.n_el, 65))
    return rows * (16.0 * s.n_el + 30.0 * a.width)


def _n_params(s, a):
    return sum(int(np.prod(shape)) for _, shape in synth.param_spec(s, a))


def _ecp(s):
    return [{"n_quad": 4, "r_cut": 1.2, "terms": [[(4.0, 0, 1.0)], [], [(1.5, 0, 0.6)]]} if z == 6.0 else None
            for z in s.nuc_charge]


def _inputs(c, seed):
    s, a = _system(c), _arch(c)
    return s, a, synth.init_params(s, a, 2 * seed + 1), synth.walkers(s, c["walkers"], 2 * seed)


def _spring_inputs(c, seed):
    """Rows with a spread of norms over orders of magnitude (walkers near a node have large gradients)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    o = torch.randn((c["rows"], c["params"]), generator=g, device="cuda")
    o *= torch.exp(1.5 * torch.randn((c["rows"], 1), generator=g, device="cuda"))
    e = torch.randn(c["rows"], generator=g, device="cuda", dtype=torch.float64) * 3.0 - 100.0
    d = torch.randn(c["params"], generator=g, device="cuda") * 1e-3 if c["momentum"] else None
    return o, e, d


def prepare(case, seed):
    if case["op"] == "spring":
        o, e, d = _spring_inputs(case, seed)
        return {"op": "spring", "o": o, "e": e, "d": d}
    s, a, p, r = _inputs(case, seed)
    st = {"op": case["op"], "model": fire.Fire(s, a, p, case["precision"], device="cuda:0"),
          "r": torch.as_tensor(r, device="cuda:0"), "seed": seed}
    if case["op"] == "autograd":
        st["theta"] = st["model"].theta.clone().requires_grad_(True)
        st["weight"] = _weights(case, seed).cuda()
    if case["op"] == "mcmc":
        st["sweeps"], st["jumps"] = case["sweeps"], case["jumps"]
    if case["op"] == "ecp":
        st["ecp"] = _ecp(s)
    return st


def _weights(case, seed):
    """Centred per-walker weights of the score-function gradient, as E_L - <E_L> gives them."""
    w = torch.from_numpy(np.random.default_rng(seed + 77).standard_normal(case["walkers"]))
    return (w - w.mean()) / case["walkers"]


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    op = state["op"]
    if op == "spring":
        return fire.spring_step(state["o"], state["e"], state["d"])["delta"]
    m, r = state["model"], state["r"]
    if op == "logpsi":
        o = m.logpsi(r)
        return {k: o[k] for k in ("logabs", "sign")}
    if op == "energy":
        o = m.local_energy(r)
        return {k: o[k] for k in ("e_loc", "logabs", "sign", "e_kin", "e_pot")}
    if op == "grad":
        o = m.grad_logpsi(r)
        return {k: o[k] for k in ("grad", "logabs", "sign")}
    if op == "autograd":
        t = state["theta"]
        t.grad = None
        la = fire.logpsi(t, r, m)
        (state["weight"] * la).sum().backward()
        return {"logabs": la.detach(), "grad": t.grad}
    if op == "mcmc":
        r = r.clone()   # the call moves the walkers in place
        o = m.mcmc_step(r, 0.3, state["sweeps"], seed=state["seed"], n_global=state["jumps"])
        return {"r": r, "accepted": o["accepted"], "n_accepted": o["n_accepted"], "logabs": o["logabs"],
                "sign": o["sign"]}
    if op == "ecp":
        return m.ecp_nonlocal(r, state["ecp"], seed=state["seed"])["v_nl"]
    o = m.spin_ratios(r, m.system.n_el - 1)
    return {k: o[k] for k in ("ratios", "r_beta")}


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------

_mean_nbr = {}


def _neighbours(c):
    """(mean |N_i|, mean (|N_i| + 1)^2) of the molecule's walkers."""
    if c["mol"] not in _mean_nbr:
        s = _system(c)
        r = synth.walkers(s, 16, 1)
        d = np.linalg.norm(r[:, :, None] - r[:, None], axis=-1)
        k = (d <= s.cutoff).sum(-1) - 1
        _mean_nbr[c["mol"]] = (float(k.mean()), float(((k + 1.0) ** 2).mean()))
    return _mean_nbr[c["mol"]]


def work(case):
    if case["op"] == "spring":
        n, p = case["rows"], case["params"]
        return {"bytes": 4.0 * p * (n + 1 + case["momentum"]) + 8.0 * n,
                "flops": 2.0 * p * n * (n / 2 + 2) + n ** 3 / 3}
    s, a = _system(case), _arch(case)
    n, N, d, D, J, RD = s.n_el, s.n_nuc, a.width, a.n_det, a.jw, a.n_reg * a.d_reg
    kbar, m2 = _neighbours(case)
    W, P = case["walkers"], _n_params(s, a)
    dense = 2.0 * d * d * a.n_layers + 2.0 * d * n * D     # per row of h
    if case["flags"] & synth.J_MLP:
        dense += 4.0 * (d * J + J * J)
    if case["flags"] & synth.J_ATT:
        dense += 2.0 * d * (a.n_reg + RD)
    once = 14.0 * d * d + 2.0 * N * a.n_env * D * n + 2.0 * 52 * d * (N + kbar)   # per electron (and derivative)
    value = n * (dense + once) + 2.0 / 3 * n ** 3 * D
    size = 8 if case["precision"] == "fp64" else 4
    r_bytes = 24.0 * W * n
    op = case["op"]
    if op == "logpsi":
        return {"bytes": size * P + r_bytes + 16.0 * W, "flops": W * value}
    if op == "energy":
        per = n * (2 + 3 * (kbar + 1)) * dense + 5 * n * once + (2.0 / 3 + 2) * n ** 3 * D + 6.0 * n * m2 * n * D
        return {"bytes": size * P + r_bytes + 40.0 * W, "flops": W * per}
    if op in ("grad", "autograd"):
        rows = W if op == "grad" else 1
        return {"bytes": size * P * (1.0 + rows) + r_bytes + 16.0 * W, "flops": W * (3 * value + 2.0 * n ** 3 * D)}
    u = min(n, 1.5 * kbar + 1)
    move = u * dense + once + 2.0 * 52 * d * (kbar + 2 * u) + D * (2 * u * n + 2 * u * u * n)
    if op == "mcmc":
        update = D * (4.0 * u * n * n)
        per = 2 * value + 2 * 2.0 * n ** 3 * D + case["sweeps"] * (n + case["jumps"]) * (move + 0.7 * update)
        return {"bytes": size * P + 2 * r_bytes + 20.0 * W, "flops": W * per}
    if op == "ecp":
        return {"bytes": size * P + r_bytes + 8.0 * W, "flops": W * (value + 2.0 * n ** 3 * D + 4 * n * move)}
    return {"bytes": size * P + r_bytes + 8.0 * W * (s.n_up + 1),
            "flops": W * (value + 2.0 * n ** 3 * D + s.n_up * 1.5 * move)}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _filter(e, w1, b1, w2, wenv, sigma, cut):
    hid = torch.nn.functional.silu(e @ w1 + b1) @ w2
    x = e[..., 0]
    s = (x / cut).clamp(max=1.0)
    fc = 1 - 28 * s ** 6 + 48 * s ** 7 - 21 * s ** 8
    return hid * ((fc[..., None] * torch.exp(-(sigma * x[..., None]) ** 2)) @ wenv)


def _readout(x, p, pre):
    x = torch.nn.functional.silu(x @ p[pre + "_w1"] + p[pre + "_b1"])
    x = torch.nn.functional.silu(x @ p[pre + "_w2"] + p[pre + "_b2"])
    return x @ p[pre + "_w3"] + p[pre + "_b3"][0]


class _Dense:
    """log|Psi| over all pairs, masked by the cutoff, in float64 on the GPU."""

    def __init__(self, s, a, params, size):
        self.s, self.a = s, a
        # weights as the call holds them (rounded to its type), then in float64
        self.p = {k: torch.as_tensor(v.astype("f8" if size == 8 else "f4").astype("f8"), device="cuda")
                  for k, v in params.items()}
        self.R = torch.as_tensor(s.nuc_pos, device="cuda")
        n = s.n_el
        self.off = ~torch.eye(n, dtype=torch.bool, device="cuda")
        up = torch.arange(n, device="cuda") < s.n_up
        self.same = up[:, None] == up[None, :]

    def logpsi(self, r, p=None):
        s, a = self.s, self.a
        p = p or self.p
        silu = torch.nn.functional.silu
        n, nu, B, d = s.n_el, s.n_up, r.shape[0], a.width
        # h^0
        de = r[:, :, None] - self.R
        dist = de.norm(dim=-1)
        e = torch.cat([dist[..., None], de], -1)                                  # [B, n, N, 4]
        x = e.permute(2, 0, 1, 3).reshape(s.n_nuc, B * n, 4)
        gam = _filter(x, p["en_w1"], p["en_b1"][:, None], p["en_w2"], p["en_wenv"], p["en_sigma"], s.cutoff_nuc)
        eb = (torch.log1p(x[..., :1]) / x[..., :1]) * x
        h = (gam * (p["nuc_emb"][:, None] + eb @ p["en_wfeat"])).sum(0).reshape(B, n, d)
        y = torch.nn.functional.layer_norm(h, (d,), p["ln_gamma"], p["ln_beta"], 1e-5)
        h0 = (silu(y @ p["glu_wg"]) * (y @ p["glu_wv"])) @ p["glu_wo"]
        # h^1
        dr = r[:, :, None] - r[:, None]
        d2 = (dr ** 2).sum(-1)
        rij = torch.sqrt(torch.where(self.off, d2, torch.ones_like(d2)))
        e = torch.cat([rij[..., None], dr], -1)
        near = self.off & (rij <= s.cutoff)
        h1 = h0
        if n > 1:
            gam = _filter(e, p["ee_w1"], p["ee_b1"], p["ee_w2"], p["ee_wenv"], p["ee_sigma"], s.cutoff)
            eb = (torch.log1p(rij) / rij)[..., None] * e
            for al, sel in ((0, self.same), (1, ~self.same)):
                w = p["msg_w"][al]
                z = (h0 @ w[:d])[:, :, None] + (h0 @ w[d:2 * d])[:, None] + eb @ w[2 * d:] + p["msg_b"][al]
                h1 = h1 + ((near & sel)[..., None] * gam * silu(z)).sum(2)
        h = h1
        for k in range(a.n_layers):
            h = h + silu(h @ p["mlp_w"][k] + p["mlp_b"][k])
        # determinants
        D = a.n_det
        q = torch.exp(-p["env_sigma"] * dist[..., None]).reshape(B, n, -1)
        phi = []
        for sp, sl in ((0, slice(0, nu)), (1, slice(nu, n))):
            m = h[:, sl].shape[1]
            o = h[:, sl] @ p["orb_w"][sp].permute(1, 0, 2).reshape(d, D * n)
            env = q[:, sl] @ p["env_pi"][sp].reshape(D * n, -1).T
            phi.append((o * env).reshape(B, m, D, n))
        sg, la = torch.linalg.slogdet(torch.cat(phi, 1).transpose(1, 2))
        top = la.max(1, keepdim=True).values.detach()
        tot = (sg * torch.exp(la - top)).sum(1)
        out, sign = top[:, 0] + torch.log(tot.abs()), torch.sign(tot)
        # Jastrow factors
        if a.flags & synth.J_CUSP and n > 1:
            iu, ju = torch.triu_indices(n, n, 1, device="cuda")
            x, same = rij[:, iu, ju], self.same[iu, ju]
            c = p["cusp"]
            om, al = torch.where(same, c[0], c[1]), torch.where(same, c[2], c[3])
            out = out + (om * al ** 2 / (al + x)).sum(-1)
        if a.flags & synth.J_MLP:
            f2 = _readout(h, p, "jm2").sum(-1)
            out, sign = out + _readout(h, p, "jm1").sum(-1) + torch.log(f2.abs()), sign * torch.sign(f2)
        if a.flags & synth.J_ATT:
            w = torch.softmax(h @ p["att_q"].T, dim=1)                             # over electrons
            v = torch.einsum("bir,bik->brk", w, h)
            v = torch.einsum("brk,rkc->brc", v, p["att_wv"]).reshape(B, -1)
            g2 = _readout(v, p, "ja2")
            out, sign = out + _readout(v, p, "ja1") + torch.log(g2.abs()), sign * torch.sign(g2)
        return out, sign

    def batches(self, r, copies):
        """r in batches whose pair tensors (so many at once) stay within a few GB."""
        step = max(1, int(8e9 / (8.0 * copies * r.shape[1] ** 2 * self.a.width)))
        return torch.split(r, step)

    def values(self, r):
        with torch.no_grad():
            got = [self.logpsi(x) for x in self.batches(r, 12)]
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])

    def kinetic(self, r):
        out = []
        for x in self.batches(r, 200):
            x = x.clone().requires_grad_(True)
            (g,) = torch.autograd.grad(self.logpsi(x)[0].sum(), x, create_graph=True)
            lap = torch.zeros_like(g[:, 0, 0])
            for i in range(x.shape[1]):
                for t in range(3):
                    (gg,) = torch.autograd.grad(g[:, i, t].sum(), x, retain_graph=True)
                    lap = lap + gg[:, i, t].detach()
            out.append(-0.5 * (lap + (g.detach() ** 2).sum((1, 2))).detach())
        return torch.cat(out)

    def potential(self, r):
        z = torch.as_tensor(self.s.nuc_charge, device="cuda")
        n, N = self.s.n_el, self.s.n_nuc
        i, j = torch.triu_indices(n, n, 1, device="cuda")
        v = (1 / (r[:, i] - r[:, j]).norm(dim=-1)).sum(-1) - (z / (r[:, :, None] - self.R).norm(dim=-1)).sum((1, 2))
        i, j = torch.triu_indices(N, N, 1, device="cuda")
        return v + (z[i] * z[j] / (self.R[i] - self.R[j]).norm(dim=-1)).sum()

    def grads(self, r, weight=None):
        """Rows d log|Psi| / d theta (weight None) or their weighted sum, flat in the order of the parameters."""
        names = [k for k, _ in synth.param_spec(self.s, self.a)]
        p = {k: v.clone().requires_grad_(True) for k, v in self.p.items()}

        def flat(g):
            return torch.cat([(torch.zeros_like(p[k]) if x is None else x).reshape(-1) for k, x in zip(names, g)])

        if weight is not None:
            tot = 0.0
            for x, w in zip(self.batches(r, 60), self.batches_like(r, weight, 60)):
                tot = tot + flat(torch.autograd.grad((w * self.logpsi(x, p)[0]).sum(), [p[k] for k in names],
                                                     allow_unused=True))
            return tot
        return torch.stack([flat(torch.autograd.grad(self.logpsi(r[k:k + 1], p)[0].sum(), [p[q] for q in names],
                                                     allow_unused=True)) for k in range(r.shape[0])])

    def batches_like(self, r, w, copies):
        at = 0
        for x in self.batches(r, copies):
            yield w[at:at + x.shape[0]]
            at += x.shape[0]


def _philox_uniform(c0, c2, stream, seed):
    """Three uniforms of Philox4x32-10 at counter (c0, 0, c2[...], stream); c2 an int64 tensor."""
    mask = 0xFFFFFFFF
    c = [torch.full_like(c2, c0), torch.zeros_like(c2), c2, torch.full_like(c2, stream)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(m, x):   # 32 x 32 -> (high, low), without overflow of int64
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        t = lo + ((hi & 0xFFFF) << 16)
        return ((hi >> 16) + (t >> 32)) & mask, t & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return [(x.double() + 0.5) / 2.0 ** 32 for x in c[:3]]


def _exact_ecp(m, r, entries, seed):
    W, n = r.shape[0], r.shape[1]
    la, sg = m.values(r)
    base = torch.tensor([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], dtype=torch.float64, device="cuda")
    base = base / math.sqrt(3.0)
    out = torch.zeros(W, dtype=torch.float64, device="cuda")
    has = torch.tensor([e is not None for e in entries], device="cuda")
    (s0, p0, a0), (s2, p2, a2) = (4.0, 0, 1.0), (1.5, 0, 0.6)
    for k in range(n):
        dist = (r[:, k, None] - m.R).norm(dim=-1)
        ok = has & (dist < 1.2)
        sel = torch.nonzero(ok.any(1))[:, 0]
        if not sel.numel():
            continue
        nuc = ok[sel].to(torch.uint8).argmax(1)
        rad = dist[sel, nuc]
        rhat = (r[sel, k] - m.R[nuc]) / rad[:, None]
        u1, u2, u3 = _philox_uniform(k, sel, 3, seed)
        x, y = torch.sqrt(1 - u1) * torch.sin(2 * math.pi * u2), torch.sqrt(1 - u1) * torch.cos(2 * math.pi * u2)
        z, w = torch.sqrt(u1) * torch.sin(2 * math.pi * u3), torch.sqrt(u1) * torch.cos(2 * math.pi * u3)
        rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                           2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                           2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(-1, 3, 3)
        dirs = torch.einsum("wab,qb->wqa", rot, base)
        cos = torch.einsum("wqa,wa->wq", dirs, rhat)
        q = r[sel][:, None].repeat(1, 4, 1, 1)
        q[:, :, k] = m.R[nuc][:, None] + rad[:, None, None] * dirs
        ln, sn = m.values(q.reshape(-1, n, 3))
        ratio = (sn.reshape(-1, 4) * sg[sel, None]) * torch.exp(ln.reshape(-1, 4) - la[sel, None])
        v = s0 * torch.exp(-a0 * rad ** 2)[:, None] + 5 * s2 * torch.exp(-a2 * rad ** 2)[:, None] * (1.5 * cos ** 2 - 0.5)
        out[sel] += (v * ratio).sum(1) / 4
    return out


def exact(case, seed):
    op = case["op"]
    if op == "spring":
        o, e, d = _spring_inputs(case, seed)
        n = o.shape[0]
        parts = o.split(65536, 1)
        gram = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        proj = torch.zeros(n, dtype=torch.float64, device="cuda")
        for k, c in enumerate(parts):
            c = c.double()
            c = c - c.mean(0)
            gram += c @ c.T
            if d is not None:
                proj += c @ d[k * 65536:k * 65536 + c.shape[1]].double()
        rhs = e - e.mean() - 0.99 * proj
        x = torch.linalg.solve(gram + 1e-3 * torch.eye(n, dtype=torch.float64, device="cuda"), rhs)
        out = []
        for c in parts:
            c = c.double()
            out.append((c - c.mean(0)).T @ x)
        out = torch.cat(out)
        return out + 0.99 * d.double() if d is not None else out
    if op == "mcmc":
        return None   # a chain of accept / reject decisions: the path, not a number, is the result
    s, a, params, r = _inputs(case, seed)
    m = _Dense(s, a, params, 8 if case["precision"] == "fp64" else 4)
    r = torch.as_tensor(r, device="cuda")
    n, W = s.n_el, case["walkers"]
    if op == "logpsi":
        la, sg = m.values(r)
        return {"logabs": la, "sign": sg}
    if op == "energy":
        la, sg = m.values(r)
        v = m.potential(r)
        # the Laplacian takes 3 n second-derivative passes of the dense function
        kin = m.kinetic(r) if 3.0 * n * W * n * n * a.width < 1.5e10 else None
        return {"e_loc": None if kin is None else kin + v, "logabs": la, "sign": sg, "e_kin": kin, "e_pot": v}
    if op == "grad":
        la, sg = m.values(r)
        rows = m.grads(r) if W * m.a.width * n * n < 3e9 else None
        return {"grad": rows, "logabs": la, "sign": sg}
    if op == "autograd":
        la, _ = m.values(r)
        return {"logabs": la, "grad": m.grads(r, _weights(case, seed).cuda())}
    if op == "ecp":
        if 4.0 * n * W * n * n * a.width > 1e11:
            return None
        return _exact_ecp(m, r, _ecp(s), seed)
    if s.n_up * W * n * n * a.width > 1e11:
        return None
    la, sg = m.values(r)
    beta, ratios = n - 1, []
    for al in range(s.n_up):
        q = r.clone()
        q[:, al], q[:, beta] = r[:, beta], r[:, al]
        ln, sn = m.values(q)
        ratios.append(sn * sg * torch.exp(ln - la))
    ratios = torch.stack(ratios, 1)
    return {"ratios": ratios, "r_beta": 1 - ratios.sum(1)}
