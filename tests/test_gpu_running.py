"""What a problem launches, which for a problem on a part of the space is not
what its full size would (P.geometry and P.kernel): the part's dimension, its
kernel, and that tiles set on the problem, tuned by a batch or narrowed by a
server are set on the part, come back afterwards and change no bit."""
import time

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_03170_gb300 as gp
    return gp


def superposed():
    w = workloads.make("superposed", workloads.Physics(Q=3, N=12, chi=(0.0, 0.7, 1.4), kappa=1.0), T=0.2, n_slices=6,
                       n_rk=2, states=[(0, 0.5), (1, 0.5j)], u_bound=1.0)
    psi = np.kron(workloads.coherent_ket(12, 0.7), np.array([0.6, 0.48, 0.64j]))
    w.rho0[:] = np.outer(psi, psi.conj())
    return w


@pytest.mark.parametrize("make,grad,rho", [
    (lambda: workloads.qubit_resonator_d20(n_slices=2), (10, 2), (10, 2)),            # a block per level
    (lambda: workloads.transmon_resonator_d600(n_slices=2), (150, 1), (150, 1)),      # one level of four
    (lambda: workloads.transmon_resonator_d120(n_slices=2), (120, 3), (120, 3)),      # the transmon is driven
    (lambda: workloads.jaynes_cummings(64, n_slices=2), (64, 1), (64, 1)),
    (superposed, (12, 6), (36, 2))], ids=["d20", "d600", "d120", "jc64", "superposed"])
def test_the_part_that_runs(gp, make, grad, rho):
    P = gp.GrapeProblem.from_workload(make())
    for want, (d, ns) in ((False, grad), (True, rho)):
        r = P.running(want)
        assert r[:3] == (d, ns, "hermitian-cluster")
        if d == P.d and ns == P.n_states:
            assert r[2] == P.kernel() and r[3:] == P.geometry()[:2]


def test_tiles_are_set_on_the_part(gp):
    w = workloads.qubit_resonator_d20(n_slices=9)
    P = gp.GrapeProblem.from_workload(w)
    F, G = P.gradient(w.u)
    own = P.running()[3:]
    for tile in ((2, 96), (16, 512), own):
        P.set_tile(*tile)
        assert P.running()[3:] == tile and P.running(True)[3:] == tile
        F1, G1 = P.gradient(w.u)
        assert F1 == F and np.array_equal(G1, G)
    with pytest.raises(gp._lib.GrapeError):
        P.set_tile(3, 64)
    assert P.running()[3:] == own


def driven(i):
    """Problems with a transmon drive, which run at their full size."""
    rng = np.random.default_rng(i)
    N = int(rng.integers(8, 22))
    phys = workloads.Physics(Q=3, N=N, chi=(0.0, 1.0, 2.2), kappa=1.0, gamma1=0.1, controls=("res_x", "res_y", "qub_x"))
    return workloads.make(f"driven{i}", phys, T=0.05, n_slices=12 + i, n_rk=2, states=[(0, 0.7), (1, 0.4j)], u_bound=1.0)


@pytest.mark.parametrize("make", [lambda i: workloads.batch_problem(i, n_slices=12 + i), driven],
                         ids=["blocks", "whole"])
def test_the_batch_tunes_what_runs_and_gives_it_back(gp, make):
    import torch
    ws = [make(i) for i in range(10)]
    probs = [gp.GrapeProblem.from_workload(w) for w in ws]
    refs = [P.gradient(w.u) for P, w in zip(probs, ws)]
    own = [P.running() for P in probs]
    B = gp.GrapeBatch(probs)
    tuned = [P.running() for P in probs]
    assert [t[:3] for t in tuned] == [o[:3] for o in own]
    buckets = {}
    for t, o in zip(tuned, own):
        if t != o:
            buckets.setdefault((t[0] - 1) // 32, set()).add(t[3:])
    assert buckets and all(len(v) == 1 for v in buckets.values())
    F, Gs = B.gradient([torch.from_numpy(w.u).cuda() for w in ws])
    torch.cuda.synchronize()
    for i, (Fr, Gr) in enumerate(refs):
        assert F[i].item() == Fr and np.array_equal(Gs[i].cpu().numpy(), Gr)
    B.close()
    assert [P.running() for P in probs] == own


@pytest.mark.parametrize("make", [lambda i: workloads.batch_problem(i, n_slices=8), driven], ids=["blocks", "whole"])
def test_the_server_gives_tiles_back(gp, make):
    ws = [make(i) for i in range(12)]
    probs = [gp.GrapeProblem.from_workload(w) for w in ws]
    own = [P.running() for P in probs]
    out = []
    for slots in (1, 12):
        srv = gp.GrapeServer(max_slots=slots)
        tickets = [srv.submit(P, w.u, max_iters=40) for P, w in zip(probs, ws)]
        narrowed, t0, res = False, time.time(), {}
        while len(res) < len(tickets) and time.time() - t0 < 120:
            narrowed = narrowed or any(P.running()[3] < o[3] for P, o in zip(probs, own))
            for t in tickets:
                if t not in res:
                    r = srv.poll(t)
                    if r is not None:
                        res[t] = r
        srv.close()
        assert len(res) == len(tickets)
        out.append([res[t][:3] for t in tickets])
        assert narrowed == (slots > 1)                   # the tiles of jobs that share the GPU
        assert [P.running() for P in probs] == own
    for a, b in zip(*out):
        assert np.array_equal(a[0], b[0]) and a[1:] == b[1:]
