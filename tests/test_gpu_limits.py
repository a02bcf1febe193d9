"""The largest problems that each kernel's shared memory holds: what the
kernels keep per entry and per CTA decides them, so they are pinned here, with
the values of one slice against the oracle.  The sizes are computed from the
kernels' shared-memory layout; the next size of each family is refused or, for
the cluster kernel, runs on the grid kernel."""
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


def one_slice(Q, N, controls, ns=1, g=0.0, n_rk=1, **kw):
    phys = workloads.Physics(Q=Q, N=N, chi=tuple(0.7 * q for q in range(Q)), kerr=-0.001, kappa=1.0, g=g,
                             controls=controls, **kw)
    return workloads.make("limit", phys, T=0.002, n_slices=1, n_rk=n_rk,
                          states=[(s % Q, 0.9 + 0.3j * s) for s in range(ns)], u_bound=1.0)


def check(gp, w, kernel):
    P = gp.GrapeProblem.from_workload(w)
    assert P.kernel() == kernel
    F, G = P.gradient(w.u)
    F_ref, G_ref, r_ref, _ = sparse.run_workload(w, threads=w.n_states)
    assert abs(F - F_ref) < TOL * abs(F_ref)
    assert np.max(np.abs(G - G_ref)) < TOL * np.max(np.abs(G_ref))
    r = P.forward(w.u)[1]
    assert np.max(np.abs(r - r_ref)) < TOL * np.max(np.abs(r_ref))


RES, ALL = ("res_x", "res_y"), ("res_x", "res_y", "qub_x", "qub_y")


@pytest.mark.parametrize("Q,N,controls", [(1, 762, RES),     # three bands
                                          (3, 219, RES),     # three bands, run on 219 x 219 blocks
                                          (3, 201, ALL)])    # five complex bands
def test_grid_kernel_takes_its_largest_problems(gp, Q, N, controls):
    check(gp, one_slice(Q, N, controls), "grid")


@pytest.mark.parametrize("N,ns,kernel", [(319, 1, "grid"), (254, 2, "grid"), (108, 1, "hermitian-cluster")])
def test_fewer_jump_terms_than_the_layout_has_room_for(gp, N, ns, kernel):
    """Jaynes-Cummings has one jump term in a band layout built for three: where
    the room for three does not fit, the run-time layout keeps one."""
    check(gp, one_slice(2, N, RES, ns=ns, g=10.0, qubit_energy=(0.0, 1.0)), kernel)


@pytest.mark.parametrize("n_slices", [14, 15])
def test_first_order_static_call_at_the_last_byte_of_its_scratch(gp, n_slices):
    """At d=512 the states of 14 or 15 slices in segments of 3, with their
    checkpoints, are exactly the 64 MiB of the no-allocation call; the partial
    traces lie in a state that is no longer needed."""
    torch = pytest.importorskip("torch")
    w = workloads.jaynes_cummings(512, n_slices=n_slices)
    P = gp.GrapeProblem.from_workload(w, grad_mode=gp._lib.GRAPE_GRAD_FIRST_ORDER)
    F, G = P.gradient(w.u)
    u = torch.from_numpy(w.u).cuda()
    Fs, Gs = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(u)
    gp._lib.grape_gradient_static(P.handle, u.data_ptr(), Fs.data_ptr(), Gs.data_ptr(), 0)
    torch.cuda.synchronize()
    P.status()
    assert Fs.item() == F and np.array_equal(Gs.cpu().numpy(), G)
