"""Problems whose states never leave a part of the Hilbert space (no operator
of the Lindbladian leads out of the basis states they start in) run on that
part alone: the restricted operators, one table set per state where the
states live in different parts.  Results against the dense oracle on the
full space, and against the same problem made irreducible by a transmon drive
that is always off, for the forms a restriction can take: one level per
state, states that share a set, sets of different sizes (relaxation without a
drive), an irregular set (levels 0 and 2 of three), jump values that differ
between the parts (dephasing), controls on dissipation rates, the penalty
with a level-dependent operator, both gradient modes, precisions and every
propagation kernel, checkpoints, the batch and the no-allocation call.

Tolerance 1e-10 relative against the oracle (the library's parity bar) and
1e-11 between two runs of the library that are each within it by a margin of
the double-float rounding (2^-48 per operation, a few thousand operations).
"""
import os

import numpy as np
import pytest

import workloads
from oracle import dense, operators, penalty

pytestmark = pytest.mark.gpu

TOL = 1e-10


def rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


@pytest.fixture(scope="module")
def gp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import problem
    return problem


class env:
    def __init__(self, **kv):
        self.kv = kv

    def __enter__(self):
        self.old = {k: os.environ.get(k) for k in self.kv}
        os.environ.update({k: str(v) for k, v in self.kv.items()})

    def __exit__(self, *a):
        for k, v in self.old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


def build(form, n_slices=7):
    """(workload, basis size of the part its states stay in)"""
    Q, N = 3, 9
    kw = dict(Q=Q, N=N, chi=(0.0, 1.0, 2.6), kerr=-0.02, kappa=1.0, controls=("res_x", "res_y"))
    states = [(0, 0.8 + 0.1j), (1, 0.5 - 0.4j), (2, 0.3j)]
    part = N
    if form == "shared":
        states = [(1, 0.8), (1, -0.5j)]
    elif form == "relaxation":                   # level q decays: sets of q + 1 levels, run on their union
        kw["gamma1"] = 0.3
        states, part = states[:2], 2 * N
    elif form == "dephasing":
        kw["gamma_phi"] = 0.4
    elif form == "rate":
        kw["controls"] = ("res_x", "rate_a")
    w = workloads.make(form, workloads.Physics(**kw), T=0.5, n_slices=n_slices, n_rk=3, states=states, u_bound=1.0)
    if form == "irregular":                      # a superposition of levels 0 and 2
        psi = np.zeros(Q * N, dtype=np.complex128)
        psi[np.arange(N) * Q] = workloads.coherent_ket(N, 0.7) * 0.6
        psi[np.arange(N) * Q + 2] = workloads.coherent_ket(N, 0.7) * 0.8j
        w.rho0 = np.outer(psi, psi.conj())[None]
        w.states = [(0, 0.7)]
        # a target with coherences between the levels
        s = w.sigma.copy()
        s[0, 2], s[2, 0] = 0.3 + 0.2j, 0.3 - 0.2j
        w.sigma = s
        part = 2 * N
    if "rate" in form:
        w.u[:, 1] = np.abs(w.u[:, 1])
    return w, part


FORMS = ["levels", "shared", "relaxation", "irregular", "dephasing", "rate"]


def reference(w, first_order, A=None, beta=0.0):
    m = operators.build(w.phys)
    _, r = dense.forward(m, w.u, w.rho0, w.sigma, w.T, w.n_rk)
    if A is not None:
        F, G = penalty.phi_and_gradient(m, w.u, w.rho0, w.sigma, w.T, w.n_rk, A, beta, first_order)
    else:
        f = dense.gradient_first_order if first_order else dense.gradient_exact
        F, G = f(m, w.u, w.rho0, w.sigma, w.T, w.n_rk)
    return F, G, r


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("first_order", [False, True])
@pytest.mark.parametrize("kernel", ["hermitian", "full", "grid"])
def test_matches_the_oracle_on_the_full_space(gp, form, prec, first_order, kernel):
    w, _ = build(form)
    F_ref, G_ref, r_ref = reference(w, first_order)
    kv = {"hermitian": {}, "full": {"GRAPE_HERMITIAN": 0}, "grid": {"GRAPE_KERNEL": "grid"}}[kernel]
    with env(**kv):
        P = gp.GrapeProblem.from_workload(w, grad_mode=int(first_order), precision=prec)
    F, r = P.forward(w.u)
    assert r.shape == r_ref.shape and rel(r, r_ref) < TOL
    assert np.all(r[np.abs(r_ref) == 0.0] == 0.0)
    F2, G = P.gradient(w.u)
    assert abs(F - F_ref) < TOL * abs(F_ref) and abs(F2 - F_ref) < TOL * abs(F_ref)
    assert rel(G, G_ref) < TOL


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("first_order", [False, True])
def test_penalty_with_a_level_dependent_operator(gp, form, first_order):
    w, _ = build(form)
    diag = np.repeat(np.arange(w.phys.N, dtype=float), w.phys.Q) + 0.3 * np.tile(np.arange(w.phys.Q), w.phys.N)
    F_ref, G_ref, _ = reference(w, first_order, np.diag(diag).astype(complex), 0.4)
    P = gp.GrapeProblem.from_workload(w, grad_mode=int(first_order))
    P.set_penalty(diag, 0.4)
    F, G = P.gradient(w.u)
    assert abs(F - F_ref) < TOL * abs(F_ref) and rel(G, G_ref) < TOL
    assert abs(P.forward(w.u)[0] - F_ref) < TOL * abs(F_ref)


@pytest.mark.parametrize("N", [1, 2, 11, 40])
@pytest.mark.parametrize("prec", [0, 1])
def test_equals_the_same_problem_with_a_drive_that_is_off(gp, prec, N):
    phys = workloads.Physics(Q=2, N=N, chi=(-0.5, 0.5), kappa=1.0)
    w = workloads.make("levels", phys, T=0.2, n_slices=9, n_rk=4, states=[(0, 0.9), (1, 0.4j)], u_bound=1.0)
    full = workloads.make("off", workloads.Physics(Q=2, N=N, chi=(-0.5, 0.5), kappa=1.0,
                                                   controls=("res_x", "res_y", "qub_x")),
                          T=0.2, n_slices=9, n_rk=4, states=w.states, u_bound=1.0)
    full.u[:, :2], full.u[:, 2] = w.u, 0.0
    P = gp.GrapeProblem.from_workload(w, precision=prec)
    Pf = gp.GrapeProblem.from_workload(full, precision=prec)
    F, G = P.gradient(w.u)
    Ff, Gf = Pf.gradient(full.u)
    assert abs(F - Ff) < 1e-11 * abs(Ff)
    assert np.max(np.abs(G - Gf[:, :2])) <= 1e-11 * max(np.max(np.abs(Gf)), 1e-3)
    r, rf = P.forward(w.u)[1], Pf.forward(full.u)[1]
    assert rel(r, rf) < 1e-11
    if N == 40:
        assert P.memory_bytes() < 0.6 * Pf.memory_bytes()      # the smaller problem is the one that ran


@pytest.mark.parametrize("form", ["levels", "relaxation"])
def test_checkpoints_batch_static_and_tiles_give_the_same_bits(gp, form):
    torch = pytest.importorskip("torch")
    w, _ = build(form, n_slices=13)
    P = gp.GrapeProblem.from_workload(w)
    F, G = P.gradient(w.u)
    Pc = gp.GrapeProblem.from_workload(w, ckpt_stride=5)
    Fc, Gc = Pc.gradient(w.u)
    assert Fc == F and np.array_equal(Gc, G)
    for tile in ((2, 64), (16, 512), (1, 96)):
        P.set_tile(*tile)
        Ft, Gt = P.gradient(w.u)
        assert Ft == F and np.array_equal(Gt, G)
    u = torch.from_numpy(w.u).cuda()
    Fs = torch.empty(1, dtype=torch.float64, device="cuda")
    Gs = torch.empty_like(u)
    gp._lib.grape_gradient_static(P.handle, u.data_ptr(), Fs.data_ptr(), Gs.data_ptr(), 0)
    torch.cuda.synchronize()
    assert Fs.item() == F and np.array_equal(Gs.cpu().numpy(), G)
    B = gp.GrapeBatch([P, Pc], n_lanes=2)
    Fb, Gb = B.gradient([u, u])
    torch.cuda.synchronize()
    for i in range(2):
        assert Fb[i].item() == F and np.array_equal(Gb[i].cpu().numpy(), G)


def superposed(Q, N, controls=("res_x", "res_y"), n_slices=7, **kw):
    """Two states over all levels, no operator between the levels."""
    phys = workloads.Physics(Q=Q, N=N, chi=tuple(0.7 * q for q in range(Q)), kerr=-0.02, kappa=1.0,
                             controls=controls, **kw)
    w = workloads.make("superposed", phys, T=0.4, n_slices=n_slices, n_rk=3, states=[(0, 0.8), (1, 0.5j)], u_bound=1.0)
    rng = np.random.default_rng(Q * 100 + N)
    for s in range(2):
        amp = rng.normal(size=Q) + 1j * rng.normal(size=Q)
        if s == 1:
            amp[0] = 0.0                               # the second state leaves level 0 empty
        psi = np.kron(workloads.coherent_ket(N, 0.6 + 0.3j * s), amp / np.linalg.norm(amp))
        w.rho0[s] = np.outer(psi, psi.conj())
    return w


@pytest.mark.parametrize("Q,N", [(2, 1), (2, 7), (3, 9), (4, 5)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("first_order", [False, True])
@pytest.mark.parametrize("kernel", ["hermitian", "full", "grid"])
def test_sectors_of_a_superposition(gp, Q, N, prec, first_order, kernel):
    """Phi and the gradient from the levels' blocks, rho(T) with its coherences."""
    w = superposed(Q, N)
    F_ref, G_ref, r_ref = reference(w, first_order)
    kv = {"hermitian": {}, "full": {"GRAPE_HERMITIAN": 0}, "grid": {"GRAPE_KERNEL": "grid"}}[kernel]
    with env(**kv):
        P = gp.GrapeProblem.from_workload(w, grad_mode=int(first_order), precision=prec)
    F2, G = P.gradient(w.u)
    F, r = P.forward(w.u)
    F3, none = P.forward(w.u, want_rho=False)
    assert none is None and F3 == F2
    assert rel(r, r_ref) < TOL
    assert abs(F - F_ref) < TOL * abs(F_ref) and abs(F2 - F_ref) < TOL * abs(F_ref)
    assert np.max(np.abs(G - G_ref)) < TOL * max(np.max(np.abs(G_ref)), 1e-3)


@pytest.mark.parametrize("first_order", [False, True])
@pytest.mark.parametrize("form", ["penalty", "dephasing", "rate", "between"])
def test_sectors_with_options(gp, form, first_order):
    kw = {}
    controls = ("res_x", "res_y")
    if form == "dephasing":
        kw["gamma_phi"] = 0.4
    if form == "rate":
        controls = ("res_x", "rate_a")
    w = superposed(3, 7, controls=controls, **kw)
    if form == "rate":
        w.u[:, 1] = np.abs(w.u[:, 1])
    if form == "between":                              # a target between levels: nothing may be split
        s = w.sigma.copy()
        s[0, 1], s[1, 0] = 0.4 - 0.1j, 0.4 + 0.1j
        w.sigma = s
    diag = np.repeat(np.arange(7.0), 3) + 0.3 * np.tile(np.arange(3), 7)
    A = np.diag(diag).astype(complex) if form == "penalty" else None
    F_ref, G_ref, _ = reference(w, first_order, A, 0.4)
    P = gp.GrapeProblem.from_workload(w, grad_mode=int(first_order))
    if form == "penalty":
        P.set_penalty(diag, 0.4)
    F, G = P.gradient(w.u)
    assert abs(F - F_ref) < TOL * abs(F_ref) and rel(G, G_ref) < TOL
    for want in (True, False):
        assert abs(P.forward(w.u, want_rho=want)[0] - F_ref) < TOL * abs(F_ref)
    if form == "penalty":
        P.set_penalty(None, 0.0)
        F0, G0, _ = reference(w, first_order)
        F, G = P.gradient(w.u)
        assert abs(F - F0) < TOL * abs(F0) and rel(G, G0) < TOL
        assert abs(P.forward(w.u)[0] - F0) < TOL * abs(F0)


def test_sectors_in_checkpoints_batch_and_static_give_the_same_bits(gp):
    torch = pytest.importorskip("torch")
    w = superposed(3, 9, n_slices=13)
    P, Pc = gp.GrapeProblem.from_workload(w), gp.GrapeProblem.from_workload(w, ckpt_stride=4)
    F, G = P.gradient(w.u)
    Fc, Gc = Pc.gradient(w.u)
    assert Fc == F and np.array_equal(Gc, G)
    for tile in ((2, 64), (16, 512)):
        P.set_tile(*tile)
        r0 = P.forward(w.u)[1]
        Ft, Gt = P.gradient(w.u)
        assert Ft == F and np.array_equal(Gt, G) and np.array_equal(P.forward(w.u)[1], r0)
    u = torch.from_numpy(w.u).cuda()
    Fs, Gs = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(u)
    gp._lib.grape_gradient_static(P.handle, u.data_ptr(), Fs.data_ptr(), Gs.data_ptr(), 0)
    B = gp.GrapeBatch([P, Pc], n_lanes=2)
    Fb, Gb = B.gradient([u, u])
    torch.cuda.synchronize()
    assert Fs.item() == F and np.array_equal(Gs.cpu().numpy(), G)
    for i in range(2):
        assert Fb[i].item() == F and np.array_equal(Gb[i].cpu().numpy(), G)
