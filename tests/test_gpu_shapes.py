"""The propagation kernels for band layouts known at compile time take every
problem with three or five bands and up to three jump terms: fewer jump terms
than the layout has room for, bands that happen to be real, no dissipation.
They run the operations of the run-time-layout kernels (GRAPE_SHAPE=0) in the
same order, so the bits are equal; the values are checked against the dense
oracle to the library's 1e-10.  N = 11 has several entries per thread on 64
threads and one per thread by default; N = 40 (d = 120) spreads over 16 CTAs.
"""
import os

import numpy as np
import pytest

import workloads
from oracle import dense, operators

pytestmark = pytest.mark.gpu

TOL = 1e-10

MODELS = {
    "driven_relaxation": dict(controls=("res_x", "res_y", "qub_x"), gamma1=0.2),
    "driven": dict(controls=("res_x", "res_y", "qub_x")),
    "real_drives": dict(controls=("res_x", "qub_x")),
    "one_real_drive": dict(controls=("res_x",)),
    "dephasing": dict(controls=("res_x", "res_y"), gamma_phi=0.3),
    "no_dissipation": dict(controls=("res_x", "res_y", "qub_x"), kappa=0.0),
}


@pytest.fixture(scope="module")
def gp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import problem
    return problem


def make(model, N, n_slices):
    kw = dict(Q=3, N=N, chi=(0.0, 1.0, 2.6), kerr=-0.01, kappa=1.0)
    kw.update(MODELS[model])
    w = workloads.make(model, workloads.Physics(**kw), T=0.02 * n_slices, n_slices=n_slices, n_rk=2,
                       states=[(0, 0.8), (1, 0.5j)], u_bound=1.0)
    psi = np.zeros(3 * N, dtype=np.complex128)          # a superposition of the levels: nothing to leave out
    for q, a in enumerate((0.6, 0.64, 0.48j)):
        psi[np.arange(N) * 3 + q] = a * workloads.coherent_ket(N, 0.7)
    w.rho0[1] = np.outer(psi, psi.conj())
    return w


def problems(gp, w, **kw):
    out = []
    for shape in (None, "0"):
        if shape:
            os.environ["GRAPE_SHAPE"] = shape
        try:
            out.append(gp.GrapeProblem.from_workload(w, **kw))
        finally:
            os.environ.pop("GRAPE_SHAPE", None)
    return out


@pytest.mark.parametrize("model", list(MODELS))
@pytest.mark.parametrize("prec", [0, 1])
def test_equals_the_runtime_layout_and_the_oracle(gp, model, prec):
    w = make(model, 11, 5)
    m = operators.build(w.phys)
    F_ref, G_ref = dense.gradient_exact(m, w.u, w.rho0, w.sigma, w.T, w.n_rk)
    P1, P0 = problems(gp, w, precision=prec)
    F0, G0 = P0.gradient(w.u)
    assert abs(F0 - F_ref) < TOL * abs(F_ref)
    assert np.max(np.abs(G0 - G_ref)) < TOL * np.max(np.abs(G_ref))
    for tile in (None, (1, 64), (2, 96), (16, 512)):
        if tile:
            P1.set_tile(*tile)
        F1, G1 = P1.gradient(w.u)
        assert F1 == F0 and np.array_equal(G1, G0)
        assert np.array_equal(P1.forward(w.u)[1], P0.forward(w.u)[1])


@pytest.mark.parametrize("model", ["driven", "real_drives", "dephasing"])
def test_sixteen_cta_clusters(gp, model):
    w = make(model, 40, 3)
    P1, P0 = problems(gp, w)
    F1, G1 = P1.gradient(w.u)
    F0, G0 = P0.gradient(w.u)
    assert np.all(np.isfinite(G1)) and F1 == F0 and np.array_equal(G1, G0)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("model,N,tile", [("driven", 33, (8, 352)),          # 619 entries: two per thread
                                          ("dephasing", 46, (16, 320)),      # 600 on 320: the second pass ragged
                                          ("driven_relaxation", 23, (4, 320)),   # 604, windows 32 KB apart
                                          ("dephasing", 30, (16, 256))])     # 256 on 256: exactly one each
def test_two_entries_per_thread(gp, model, N, tile, prec):
    w = make(model, N, 3)
    P1, P0 = problems(gp, w, precision=prec)
    F0, G0 = P0.gradient(w.u)
    for t in (tile, None):                              # and the tile chosen at create
        P = P1 if t else gp.GrapeProblem.from_workload(w, precision=prec)
        if t:
            P.set_tile(*t)
        F1, G1 = P.gradient(w.u)
        assert np.all(np.isfinite(G1)) and F1 == F0 and np.array_equal(G1, G0)
        assert np.array_equal(P.forward(w.u)[1], P0.forward(w.u)[1])
