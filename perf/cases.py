"""Timed cases of the open-GRAPE library: what a pulse-optimisation program asks of it.

Each case is one call (or one short chain of calls) through the public Python
front end.  The sizes are those of the repository's problem families
(workloads.py, bench.py): the dispersive qubit/qutrit reset, the driven
transmon x resonator, the Jaynes-Cummings scaling problem, the uneven batch,
the long checkpointed pulse, and the control filter.

Fields of a case
  kind    gradient   P.gradient(u)                     -> Phi, dPhi/du
          filtered   P.gradient_filtered(u, omega0)    -> Phi, dPhi/du (App. A)
          autograd   grape_phi(u, P).backward()        -> Phi, u.grad
          forward    P.forward(u)                      -> Phi, rho(T)
          batch      GrapeBatch.gradient(us)           -> Phi, dPhi/du of every problem
          filter     GaussianFilter.apply and .adjoint -> s, g_u
  model   dispersive (resonator drives), driven (and a transmon drive, T1 and
          dephasing), jc (Jaynes-Cummings coupling)
  Q, N    transmon levels and resonator Fock states, d = Q N
  start   levels: state q is |q>|alpha_q>, one state per transmon level up to
          `states`; mixed: the transmon starts in a superposition of its levels
  slices, n_rk, dt   control slices, RK4 substeps per slice, slice length (1/kappa)
  first_order, fp64, ckpt, penalty, steps   the options of the problem
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_1609_03170_gb300 import (GRAPE_GRAD_EXACT, GRAPE_GRAD_FIRST_ORDER, GRAPE_PREC_DF64,
                                    GRAPE_PREC_FP64, GaussianFilter, GrapeBatch, GrapeProblem,
                                    band_model, grape_phi)

# 3 dB bandwidth of the control line over kappa (the paper's reset parameters:
# 100 MHz over 1.1 MHz), as the reference bandwidth of the erf transfer matrix
OMEGA0 = (100.0 / 1.1) / math.sqrt(-math.log(1.0 / math.sqrt(2.0)))

_BASE = dict(kind="gradient", model="dispersive", Q=2, N=10, start="levels", states=2, slices=200,
             n_rk=4, dt=0.003, alpha=(0.0, 3.0), u_bound=1.0, kerr=0.0, first_order=False, fp64=False,
             ckpt=0, penalty=False, steps=0)


def _case(name, **kw):
    c = dict(_BASE)
    c.update(kw)
    c["alpha_lo"], c["alpha_hi"] = c.pop("alpha")
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # shaping one set of drives for the signal line and pulling a gradient back through
        # the filter: the shortest call a program makes, 200 controls on 2000 subpixels
        _case("filter_200x2000", kind="filter", model="driven", Q=3, N=40, slices=2000, steps=200),
        # the introductory problem: one qubit, ten Fock states, 200 slices - the gradient that an
        # optimiser asks for hundreds of times, where launches and stage latency are everything
        _case("qubit_d20", Q=2, N=10, slices=200, dt=0.02, alpha=(1.5, 1.6)),
        # an odd size with every coherence between the levels present at the start
        _case("qutrit_d111_mixed", Q=3, N=37, start="mixed", states=2, slices=333, u_bound=2.0),
        # the headline problem: driven transmon x resonator, three states, 2000 slices
        _case("transmon_d120", model="driven", Q=3, N=40, states=3, slices=2000, kerr=-0.01,
              alpha=(2.0, 4.0)),
        # the same system as it is optimised in practice: filtered controls and the
        # photon-number penalty
        _case("transmon_d120_filtered_penalty", kind="filtered", model="driven", Q=3, N=40, states=3,
              slices=500, kerr=-0.01, alpha=(2.0, 4.0), steps=50, penalty=True),
        # propagation alone: checking a pulse, and the trial points of a line search
        _case("transmon_d120_forward", kind="forward", model="driven", Q=3, N=40, states=3,
              slices=500, kerr=-0.01, alpha=(2.0, 4.0)),
        # a served job of the large kind at a tenth of its slices
        _case("qutrit_d300", Q=3, N=100, states=3, slices=1000, kerr=-0.01, alpha=(1.5, 2.3)),
        # the long pulse on the largest space, with states kept every 200 slices
        _case("ququart_d600_ckpt", Q=4, N=150, states=1, slices=1000, dt=1.5e-4, kerr=-0.005,
              alpha=(2.0, 2.1), ckpt=200),
        # many uneven problems in one launch: N 10..60, Q 2..3, slices 50..400
        _case("batch_24", kind="batch", Q=3, N=60, slices=400, u_bound=2.0, steps=24),
        # the scaling study's first-order gradient at its middle and its largest size
        _case("jc_d128_first_order", model="jc", Q=2, N=64, states=1, slices=200, n_rk=1,
              dt=math.pi / 100.0 / 200, first_order=True),
        _case("jc_d512_first_order", model="jc", Q=2, N=256, states=1, slices=200, n_rk=1,
              dt=math.pi / 100.0 / 200, first_order=True),
        # native FP64, differentiated by torch
        _case("transmon_d60_fp64_autograd", kind="autograd", model="driven", Q=3, N=20, states=3,
              slices=200, kerr=-0.01, alpha=(1.0, 2.5), fp64=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gradient"] * 8 + ["forward", "filtered", "autograd", "batch", "filter"])
    if kind == "filter":
        steps = _log(rng, 8, 400)
        return _case(None, kind="filter", model="driven", Q=3, N=_log(rng, 8, 60), steps=steps,
                     slices=steps * rng.randint(3, 12) + rng.randint(0, 7))
    if kind == "batch":
        return _case(None, kind="batch", Q=3, N=60, slices=_log(rng, 60, 400), u_bound=2.0,
                     steps=rng.randint(3, 24), Q_seed=rng.randint(1, 10 ** 6))
    model = rng.choice(["dispersive", "dispersive", "driven", "driven", "jc"])
    if model == "jc":
        c = _case(None, kind="gradient" if kind == "filtered" else kind, model="jc", Q=2,
                  N=_log(rng, 3, 256), states=1, slices=rng.randint(60, 400), n_rk=rng.choice([1, 1, 2]),
                  dt=math.pi / 100.0 / 200, first_order=rng.random() < 0.7)
    else:
        top = 120 if model == "dispersive" else 50
        Q = rng.choice([2, 2, 3, 3, 4]) if model == "dispersive" else rng.choice([2, 3])
        c = _case(None, kind=kind, model=model, Q=Q, N=_log(rng, 6, top), states=rng.randint(1, Q),
                  start="mixed" if rng.random() < 0.3 else "levels", slices=_log(rng, 40, 2000),
                  n_rk=rng.choice([2, 4, 4]), dt=0.003 if rng.random() < 0.7 else 0.0015,
                  kerr=rng.choice([0.0, -0.01]), u_bound=rng.choice([1.0, 2.0]),
                  fp64=rng.random() < 0.15, first_order=rng.random() < 0.15,
                  penalty=rng.random() < 0.2)
        if c["N"] < 12:
            c["alpha_hi"] = 1.5
        if kind == "gradient" and rng.random() < 0.2:
            c["ckpt"] = max(4, c["slices"] // rng.randint(3, 9))
        if kind == "filtered":
            c["steps"] = max(2, c["slices"] // rng.randint(4, 12))
    # no dearer than the headline problem (native FP64 is several times as dear per operation)
    cap = _dense_work(listed()[3]) / (8.0 if c["fp64"] else 1.0)
    while c["slices"] > 8 and _dense_work(c) > cap:
        c["slices"] = max(8, int(0.7 * c["slices"]))
        c["ckpt"] = min(c["ckpt"], c["slices"])
        c["steps"] = min(c["steps"], c["slices"])
    return c


# ---------------------------------------------------------------------------- inputs

def _phys(c):
    """The model's parameters, in units of kappa."""
    Q, N = c["Q"], c["N"]
    if c["model"] == "jc":
        return types.SimpleNamespace(Q=Q, N=N, chi=(0.0,) * Q, kerr=0.0, delta=0.0, kappa=1.0, gamma1=0.0,
                                     gamma_phi=0.0, qubit_energy=(0.0, 10.0), g=100.0,
                                     controls=("res_x", "res_y"))
    driven = c["model"] == "driven"
    chi = {2: (-0.5, 0.5), 3: (0.0, 1.0, 2.6), 4: (0.0, 1.0, 2.2, 3.6)}[Q]
    return types.SimpleNamespace(Q=Q, N=N, chi=chi, kerr=c["kerr"], delta=0.0, kappa=1.0,
                                 gamma1=0.002 if driven else 0.0, gamma_phi=0.001 if driven else 0.0,
                                 qubit_energy=(), g=0.0,
                                 controls=("res_x", "res_y", "qub_x") if driven else ("res_x", "res_y"))


def _controls(c):
    return 3 if c["model"] == "driven" else 2


def _subproblems(c):
    """The problems of a batch (sizes from the case, not from the seed)."""
    rng = np.random.default_rng(c.get("Q_seed", 1609))
    out = []
    for _ in range(c["steps"]):
        Q = int(rng.integers(2, 4))
        out.append(_case(None, Q=Q, N=int(rng.integers(10, c["N"] + 1)), states=Q, u_bound=2.0,
                         slices=int(rng.integers(max(8, c["slices"] // 8), c["slices"] + 1))))
    return out


def _inputs(c, seed):
    """Initial states, target and controls (host arrays)."""
    Q, N = c["Q"], c["N"]
    d = Q * N
    rng = np.random.default_rng([seed, d, c["slices"]])
    n = np.arange(1, N)
    ns = max(1, c["states"])
    rho0 = np.zeros((ns, d, d), dtype=np.complex128)
    for s in range(ns):
        if c["model"] == "jc":
            alpha = math.sqrt(d / 8.0) * np.exp(1j * rng.uniform(-0.2, 0.2))
        else:
            alpha = rng.uniform(c["alpha_lo"], c["alpha_hi"]) * np.exp(2j * np.pi * rng.uniform())
        ket = np.ones(N, dtype=np.complex128)
        ket[1:] = np.cumprod(alpha / np.sqrt(n))
        ket /= np.linalg.norm(ket)
        if c["start"] == "mixed":
            amp = rng.normal(size=Q) + 1j * rng.normal(size=Q)
            amp /= np.linalg.norm(amp)
        else:
            amp = np.zeros(Q, dtype=np.complex128)
            amp[1 if c["model"] == "jc" or ns == 1 else s % Q] = 1.0
        psi = np.kron(ket, amp)
        rho0[s] = np.outer(psi, psi.conj())
    sigma = np.zeros((d, d), dtype=np.complex128)
    if c["model"] == "jc":
        sigma[1, 1] = 1.0                          # |0> (x) |e>
    else:
        sigma[np.arange(Q), np.arange(Q)] = 1.0    # the resonator's vacuum
    rows = c["steps"] if c["kind"] == "filtered" else c["slices"]
    u = rng.uniform(-c["u_bound"], c["u_bound"], size=(rows, _controls(c)))
    return rho0, sigma, u


def _problem(c, rho0, sigma):
    P = GrapeProblem(band_model(_phys(c)), rho0, sigma, c["dt"] * c["slices"], c["slices"], c["n_rk"],
                     grad_mode=GRAPE_GRAD_FIRST_ORDER if c["first_order"] else GRAPE_GRAD_EXACT,
                     ckpt_stride=c["ckpt"], precision=GRAPE_PREC_FP64 if c["fp64"] else GRAPE_PREC_DF64)
    if c["penalty"]:
        P.set_photon_penalty(c["Q"], c["N"], 0.2 / (c["dt"] * c["slices"]))
    return P


def _filter_inputs(c, seed):
    rng = np.random.default_rng([seed, c["steps"], c["slices"]])
    R = _controls(c)
    return rng.uniform(-1, 1, size=(c["steps"], R)), rng.normal(size=(c["slices"], R)) * 1e-3


def prepare(case, seed):
    c = case
    if c["kind"] == "filter":
        u, g = _filter_inputs(c, seed)
        R = _controls(c)
        return dict(kind="filter", filt=GaussianFilter(c["steps"], c["slices"], c["dt"] * c["slices"], OMEGA0, R),
                    u=torch.from_numpy(u).cuda(), g=torch.from_numpy(g).cuda())
    if c["kind"] == "batch":
        subs = _subproblems(c)
        ins = [_inputs(s, seed + 1000 * i) for i, s in enumerate(subs)]
        probs = [_problem(s, r, sg) for s, (r, sg, _) in zip(subs, ins)]
        return dict(kind="batch", batch=GrapeBatch(probs), us=[torch.from_numpy(u).cuda() for _, _, u in ins])
    rho0, sigma, u = _inputs(c, seed)
    ut = torch.from_numpy(u).cuda()
    if c["kind"] == "autograd":
        ut.requires_grad_(True)
    return dict(kind=c["kind"], P=_problem(c, rho0, sigma), u=ut, omega0=[OMEGA0] * _controls(c))


def run(state):
    kind = state["kind"]
    stream = torch.cuda.current_stream()
    if kind == "filter":
        f = state["filt"]
        return f.apply(state["u"], stream=stream), f.adjoint(state["g"], stream=stream)
    if kind == "batch":
        return state["batch"].gradient(state["us"], stream=stream)
    P, u = state["P"], state["u"]
    if kind == "forward":
        return P.forward(u, stream=stream)
    if kind == "filtered":
        return P.gradient_filtered(u, state["omega0"], stream=stream)
    if kind == "autograd":
        u.grad = None
        phi = grape_phi(u, P)
        phi.backward()
        return phi.detach(), u.grad
    return P.gradient(u, stream=stream)


# ---------------------------------------------------------------------------- work

def _stage_flops(c):
    """Operations per entry and RK stage: two complex multiply-adds per
    off-diagonal Hamiltonian band, the own-entry term, one real coefficient
    per dissipator with an offset, the two stage combinations; and of the
    gradient's trace, two complex products per control band offset."""
    bands, jumps, offs = {"dispersive": (2, 1, 2), "driven": (4, 2, 4), "jc": (4, 1, 2)}[c["model"]]
    return 16.0 * bands + 8.0 + 4.0 * jumps + 8.0, 16.0 * offs


def _dense_work(c):
    d = c["Q"] * c["N"]
    lin, tr = _stage_flops(c)
    sweeps = 1 if c["kind"] == "forward" else 2
    return 0.5 * d * (d + 1) * max(1, c["states"]) * c["slices"] * c["n_rk"] * 4 * (sweeps * lin + tr)


def work(case):
    c = case
    if c["kind"] == "batch":
        parts = [work(s) for s in _subproblems(c)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    R = _controls(c)
    if c["kind"] == "filter":
        band = min(c["steps"], 2 + int(13.0 / OMEGA0 / (c["dt"] * c["slices"] / c["steps"])))
        return {"bytes": 16.0 * R * (c["steps"] + c["slices"]), "flops": 2 * 2.0 * 30 * R * c["slices"] * band}
    # a resonator drive keeps the transmon's level, so a state that starts in
    # one level stays in its N x N block: only those entries are ever not zero
    d = c["N"] if c["model"] == "dispersive" and c["start"] == "levels" else c["Q"] * c["N"]
    ns = max(1, c["states"])
    entries = 0.5 * d * (d + 1) * ns
    stages = c["slices"] * c["n_rk"] * 4
    lin, tr = _stage_flops(c)
    rows = c["steps"] if c["kind"] == "filtered" else c["slices"]
    full = (c["Q"] * c["N"]) ** 2
    if c["kind"] == "forward":
        return {"bytes": 16.0 * entries * 2 + 8.0 * rows * R + 16.0 * ns * full, "flops": entries * stages * lin}
    flops = entries * stages * 2 * lin
    flops += entries * tr * (c["slices"] if c["first_order"] else stages)
    return {"bytes": 16.0 * entries * 2 + 16.0 * rows * R, "flops": flops}


# ---------------------------------------------------------------------------- 64-bit values

def _operators(c):
    """Dense H0, controls and jump operators in the basis i = n Q + q."""
    p = _phys(c)
    aN = np.diag(np.sqrt(np.arange(1.0, p.N)), 1)
    bQ = np.diag(np.sqrt(np.arange(1.0, p.Q)), 1)
    a, b = np.kron(aN, np.eye(p.Q)).astype(complex), np.kron(np.eye(p.N), bQ).astype(complex)
    n = np.repeat(np.arange(p.N), p.Q).astype(float)
    q = np.tile(np.arange(p.Q), p.N)
    diag = np.asarray(p.chi)[q] * n + p.kerr * n ** 2
    if p.qubit_energy:
        diag = diag + np.asarray(p.qubit_energy)[q]
    H0 = np.diag(diag).astype(complex)
    if p.g:
        H0 = H0 + p.g * (a @ b.T + a.T @ b)
    Hs = {"res_x": a + a.T, "res_y": 1j * (a.T - a), "qub_x": b + b.T}
    jumps = [math.sqrt(p.kappa) * a]
    if p.gamma1:
        jumps.append(math.sqrt(p.gamma1) * b)
    if p.gamma_phi:
        jumps.append(math.sqrt(p.gamma_phi) * np.diag(q).astype(complex))
    return H0, [Hs[k] for k in p.controls], jumps


def _diagonals(M):
    i, j = np.nonzero(M)
    d = M.shape[0]
    out = {}
    for o in np.unique(j - i):
        v = np.zeros(d, dtype=complex)
        r = np.arange(max(0, -o), d - max(0, o))
        v[r] = M[r, r + o]
        out[int(o)] = v
    return out


class _Exact:
    """The discrete problem on a GPU (or the host) in complex128: the Lindblad
    action as a sum of shifted copies of rho, one coefficient matrix each."""

    def __init__(self, c, device):
        self.c, self.dev = c, device
        d = c["Q"] * c["N"]
        self.d = d
        H0, Hc, jumps = _operators(c)
        A0 = H0 - 0.5j * sum(J.conj().T @ J for J in jumps)
        self.R = len(Hc)
        parts = []                                  # [A0 and jumps, H_1, ..., H_R]
        offs = set()
        for k, A in enumerate([A0] + Hc):
            for adj in (0, 1):
                B = -A.conj().T if adj else A
                terms = {}
                for o, v in _diagonals(B).items():
                    terms[(o, 0)] = terms.get((o, 0), 0) + (-1j * v)[:, None] * np.ones(d)[None, :]
                    terms[(0, o)] = terms.get((0, o), 0) + np.ones(d)[:, None] * (1j * v.conj())[None, :]
                if k == 0:
                    for J in jumps:
                        dg = _diagonals(J.conj().T if adj else J)
                        for oL, vL in dg.items():
                            for oR, vR in dg.items():
                                terms[(oL, oR)] = terms.get((oL, oR), 0) + vL[:, None] * vR.conj()[None, :]
                parts.append(terms)
                offs |= set(terms)
        offs = sorted(offs)
        i, j = np.meshgrid(np.arange(d), np.arange(d), indexing="ij")
        idx = np.zeros((len(offs), d * d), dtype=np.int64)
        ok = np.zeros((len(offs), d, d))
        for t, (a, b) in enumerate(offs):
            r, s = i + a, j + b
            inside = (r >= 0) & (r < d) & (s >= 0) & (s < d)
            idx[t] = np.where(inside, r * d + s, 0).reshape(-1)
            ok[t] = inside
        C = np.zeros((self.R + 1, 2, len(offs), d * d), dtype=complex)
        for k in range(self.R + 1):
            for adj in (0, 1):
                for o, v in parts[2 * k + adj].items():
                    t = offs.index(o)
                    C[k, adj, t] = (v * ok[t]).reshape(-1)
        self.T = len(offs)
        self.idx = torch.from_numpy(idx.reshape(-1)).to(device)
        self.C = torch.from_numpy(C).to(device)
        self.control_terms = []
        for k in range(self.R):
            terms = np.flatnonzero(np.abs(C[k + 1, 0]).max(axis=1))
            self.control_terms.append((torch.from_numpy(terms).to(device), self.C[k + 1, 0, terms]))

    def coefficients(self, uj, sel):
        C = self.C[0, sel]
        for k in range(self.R):
            C = C + float(uj[k]) * self.C[k + 1, sel]
        return C[:, None]                           # [dirs, 1, T, d d]

    def apply(self, C, X):
        """X [dirs, states, d d] -> L X (the dual for dirs of the adjoint)."""
        g = X.index_select(2, self.idx).view(X.shape[0], X.shape[1], self.T, -1)
        return g.mul_(C).sum(2)

    def traces(self, kb, y):
        """sum over the pairs of Re Tr(kb (-i)[H_k, y]) per control, for kb, y [pairs, d d]."""
        out = []
        for terms, C in self.control_terms:
            g = y.index_select(1, self.idx.view(self.T, -1)[terms].reshape(-1)).view(y.shape[0], len(terms), -1)
            out.append((kb.conj() * g.mul_(C).sum(1)).sum().real)
        return torch.stack(out)


def _exact_sweeps(c, seed, device):
    rho0, sigma, u = _inputs(c, seed)
    if c["kind"] == "filtered":
        Tm = _transfer(c, device)
        s = (Tm @ torch.from_numpy(u).to(device)).cpu().numpy()
    else:
        s = u
    E = _Exact(c, device)
    d, ns, n_rk, N = E.d, rho0.shape[0], c["n_rk"], c["slices"]
    h = c["dt"] / n_rk
    beta_dt = 0.2 / N if c["penalty"] else 0.0
    num = torch.from_numpy(np.repeat(np.arange(float(c["N"])), c["Q"])).to(device)
    sg = torch.from_numpy(sigma).to(device)
    x = torch.from_numpy(rho0).to(device).view(1, ns, d * d)
    bounds = [x]
    for j in range(N):
        C = E.coefficients(s[j], slice(0, 1))
        for _ in range(n_rk):
            k1 = E.apply(C, x)
            k2 = E.apply(C, torch.add(x, k1, alpha=h / 2))
            k3 = E.apply(C, torch.add(x, k2, alpha=h / 2))
            k4 = E.apply(C, torch.add(x, k3, alpha=h))
            x = x + (h / 6) * (k1 + 2 * k2 + 2 * k3 + k4)
        bounds.append(x)
    rhoT = x[0].view(ns, d, d)
    F = (sg.conj().reshape(-1) * x[0]).sum().real
    if beta_dt:
        for b in bounds:
            F = F - beta_dt * (torch.diagonal(b[0].view(ns, d, d), dim1=1, dim2=2).real * num).sum()
    if c["kind"] == "forward":
        return [F.reshape(1), rhoT]
    src = (torch.diag(num) * -beta_dt).to(torch.complex128).reshape(-1)
    mu = sg.reshape(1, 1, -1).repeat(1, ns, 1) + src
    G = torch.zeros((N, E.R), dtype=torch.float64, device=device)
    first = c["first_order"]
    for j in range(N - 1, -1, -1):
        if first:
            G[j] = c["dt"] * E.traces(mu[0], bounds[j + 1][0])
            C = E.coefficients(s[j], slice(1, 2))
        else:
            C = E.coefficients(s[j], slice(0, 2))
        ys, kbs = [], []
        x = bounds[j]
        for _ in range(n_rk):
            # the slice's forward stages again and, in the same tensors, the adjoint's:
            # row 0 walks the substeps up, row 1 walks them down
            if first:
                yb4 = E.apply(C, (h / 6) * mu)
                yb3 = E.apply(C, (h / 3) * mu + h * yb4)
                yb2 = E.apply(C, (h / 3) * mu + (h / 2) * yb3)
                yb1 = E.apply(C, (h / 6) * mu + (h / 2) * yb2)
                mu = mu + yb1 + yb2 + yb3 + yb4
                continue
            z1 = torch.cat([x, (h / 6) * mu])
            w1 = E.apply(C, z1)
            z2 = torch.cat([x + (h / 2) * w1[:1], (h / 3) * mu + h * w1[1:]])
            w2 = E.apply(C, z2)
            z3 = torch.cat([x + (h / 2) * w2[:1], (h / 3) * mu + (h / 2) * w2[1:]])
            w3 = E.apply(C, z3)
            z4 = torch.cat([x + h * w3[:1], (h / 6) * mu + (h / 2) * w3[1:]])
            w4 = E.apply(C, z4)
            ys.append(torch.cat([z1[0], z2[0], z3[0], z4[0]]))
            kbs.append(torch.cat([z4[1], z3[1], z2[1], z1[1]]))
            x = x + (h / 6) * (w1[:1] + 2 * w2[:1] + 2 * w3[:1] + w4[:1])
            mu = mu + w1[1:] + w2[1:] + w3[1:] + w4[1:]
        if not first:
            G[j] = E.traces(torch.cat(kbs[::-1]), torch.cat(ys))
        mu = mu + src
    if c["kind"] == "filtered":
        G = Tm.T @ G
    F = F.reshape(()) if c["kind"] == "autograd" else F.reshape(1)
    return [F, G]


def _transfer(c, device):
    n = torch.arange(c["slices"], dtype=torch.float64, device=device)[:, None] * c["dt"]
    Dt = c["dt"] * c["slices"] / c["steps"]
    j = torch.arange(c["steps"], dtype=torch.float64, device=device)[None, :]
    return 0.5 * (torch.erf(0.5 * OMEGA0 * (n - j * Dt)) - torch.erf(0.5 * OMEGA0 * (n - (j + 1) * Dt)))


def _exact_seconds(c):
    """Rough seconds of _exact_sweeps (launches and memory)."""
    d2 = (c["Q"] * c["N"]) ** 2
    stages = c["slices"] * c["n_rk"] * 4
    per = 60e-6 + 3 * 13 * d2 * max(1, c["states"]) * 16 * 3 / 2.5e12
    return stages * (1 if c["kind"] == "forward" else 3) * per


def exact(case, seed):
    c = case
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if c["kind"] == "filter":
        u, g = _filter_inputs(c, seed)
        Tm = _transfer(c, device)
        return [Tm @ torch.from_numpy(u).to(device), Tm.T @ torch.from_numpy(g).to(device)]
    subs = _subproblems(c) if c["kind"] == "batch" else [c]
    if sum(_exact_seconds(s) for s in subs) > 25.0:
        return None
    if c["kind"] == "batch":
        out = [_exact_sweeps(s, seed + 1000 * i, device) for i, s in enumerate(subs)]
        return [torch.cat([f for f, _ in out]), [g for _, g in out]]
    return _exact_sweeps(c, seed, device)
