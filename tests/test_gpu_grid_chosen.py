"""Problems that the library itself places on the grid kernel: one irreducible
block that no cluster holds, in the band layouts the kernel is built for (five
bands: Jaynes-Cummings, the scaling study's sizes; three bands: one level) and in
the run-time layout (a transmon y drive; a control on a dissipation rate).  Both
gradient modes, both precisions, checkpoints, the penalty and several states,
against the plain-C oracle."""
import functools

import numpy as np
import pytest

import workloads
from oracle import sparse

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def gp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import problem
    return problem


@functools.lru_cache(maxsize=None)
def make(name):
    if name.startswith("jc"):
        w = workloads.jaynes_cummings(int(name[2:]), n_rk=2 if name == "jc256" else 1).with_slices(5)
        w.sigma = np.diag(np.repeat(np.arange(w.phys.N) / w.phys.N, 2)).astype(complex)   # a photon number: no tiny Phi
        return w
    Q, N, controls, ns, kw = {
        "one_level": (1, 300, ("res_x", "res_y"), 1, {}),
        "two_states": (3, 82, ("res_x", "res_y", "qub_x"), 2, dict(gamma1=0.1, gamma_phi=0.05)),
        "y_drive": (3, 80, ("res_x", "res_y", "qub_x", "qub_y"), 1, dict(gamma1=0.1)),
        "rate": (2, 130, ("res_x", "qub_x", "rate_a"), 1, {})}[name]
    phys = workloads.Physics(Q=Q, N=N, chi=tuple(0.7 * q for q in range(Q)), kerr=-0.001, kappa=1.0, controls=controls, **kw)
    w = workloads.make(name, phys, T=0.01, n_slices=5, n_rk=2, states=[(s % Q, 0.9 + 0.3j * s) for s in range(ns)], u_bound=1.0)
    if name == "rate":
        w.u[:, 2] = np.abs(w.u[:, 2])
    return w


@functools.lru_cache(maxsize=None)
def reference(name, first_order):
    w = make(name)
    return sparse.run_workload(w, mode=sparse.MODE_FIRST_ORDER if first_order else 1, threads=w.n_states)[:3]


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("first_order", [0, 1])
@pytest.mark.parametrize("name", ["jc256", "jc512", "one_level", "two_states", "y_drive", "rate"])
def test_matches_the_oracle(gp, name, first_order, prec):
    w = make(name)
    F_ref, G_ref, r_ref = reference(name, first_order)
    out = []
    for ckpt in (0, 2):
        P = gp.GrapeProblem.from_workload(w, grad_mode=first_order, precision=prec, ckpt_stride=ckpt)
        assert P.running()[:3] == (w.d, w.n_states, "grid")
        out.append(P.gradient(w.u))
        P.status()
    F, G = out[0]
    assert out[1][0] == F and np.array_equal(out[1][1], G)
    assert abs(F - F_ref) < TOL * abs(F_ref) and rel(G, G_ref) < TOL
    F2, r = P.forward(w.u)
    assert F2 == F and rel(r, r_ref) < TOL


@pytest.mark.parametrize("prec", [0, 1])
def test_grid_and_cluster_kernel_agree_at_the_limit_between_them(gp, prec):
    """d=216 is the last Jaynes-Cummings problem on clusters; GRAPE_KERNEL=grid
    forces the grid kernel: the same bits."""
    import os
    w = workloads.jaynes_cummings(216).with_slices(4)
    P = gp.GrapeProblem.from_workload(w, precision=prec)
    os.environ["GRAPE_KERNEL"] = "grid"
    try:
        Pg = gp.GrapeProblem.from_workload(w, precision=prec)
    finally:
        os.environ.pop("GRAPE_KERNEL")
    assert P.running()[2] == "hermitian-cluster" and Pg.running()[2] == "grid"
    (F, G), (Fg, Gg) = P.gradient(w.u), Pg.gradient(w.u)
    assert F == Fg and np.array_equal(G, Gg)
