"""A problem serves one job at a time: jobs of one problem submitted together,
more of them than run at once and with other problems between, wait for one
another and give the results of a job that runs alone."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: workloads.qubit_resonator_d20(n_slices=12),
                                  lambda: workloads.transmon_resonator_d120(n_slices=4)], ids=["blocks", "whole"])
def test_jobs_of_one_problem_wait_for_one_another(make):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_03170_gb300 as gp
    w, other = make(), workloads.batch_problem(3, n_slices=10)
    P, O = gp.GrapeProblem.from_workload(w), gp.GrapeProblem.from_workload(other)
    starts = [w.u, 0.5 * w.u, -w.u]
    own = P.running()

    def run(slots, jobs):
        srv = gp.GrapeServer(max_slots=slots)
        tickets = [srv.submit(p, u, max_iters=5) for p, u in jobs]
        out = []
        for t in tickets:
            r = None
            for _ in range(240):
                r = srv.poll(t, timeout_s=0.5)
                if r is not None:
                    break
            assert r is not None
            out.append(r[:3])
        srv.close()
        return out

    jobs = [(P, starts[0]), (P, starts[1]), (O, other.u), (P, starts[2])]
    alone = [run(1, [j])[0] for j in jobs]
    for _ in range(3):
        for a, b in zip(alone, run(8, jobs)):
            assert np.array_equal(a[0], b[0]) and a[1:] == b[1:]
    assert P.running() == own
