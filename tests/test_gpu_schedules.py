"""How a gradient's launches are scheduled changes no bit: the sweeps side by
side or one after the other (GRAPE_CONCURRENT=0) in the first-order mode, and
with checkpoints (each segment's recomputation beside its adjoint; lengths
that divide the pulse, leave a short last segment, and one slice per segment),
with and without the penalty.  The exact mode without checkpoints is covered
by test_gpu_concurrent.py; the kernels and the order of every sum are the same
in both schedules, so the results are compared for equality.
"""
import os

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


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


def gradients(P, u):
    out = []
    for c in (1, 0):
        with env(GRAPE_CONCURRENT=c):
            out += [P.gradient(u), P.gradient(u)]     # twice: streams and events are reused
    P.status()
    return out


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("penalty", [False, True])
@pytest.mark.parametrize("make", [lambda: workloads.transmon_resonator_d120(n_slices=9),
                                  lambda: workloads.jaynes_cummings(30, n_slices=21),
                                  lambda: workloads.qubit_resonator_d20(n_slices=1)],
                         ids=["d120", "jc30", "one_slice"])
def test_first_order_sweeps_side_by_side(gp, make, penalty, prec):
    w = make()
    P = gp.GrapeProblem.from_workload(w, grad_mode=gp._lib.GRAPE_GRAD_FIRST_ORDER, precision=prec)
    if penalty:
        P.set_photon_penalty(w.phys.Q, w.phys.N, 0.3)
    out = gradients(P, w.u)
    assert np.all(np.isfinite(out[0][1]))
    for F, G in out[1:]:
        assert F == out[0][0] and np.array_equal(G, out[0][1])


@pytest.mark.parametrize("first_order", [False, True])
@pytest.mark.parametrize("penalty", [False, True])
@pytest.mark.parametrize("stride", [1, 6, 7, 20])
def test_checkpointed_segments_side_by_side(gp, first_order, penalty, stride):
    w = workloads.transmon_resonator_d120(n_slices=24)
    out = []
    for ck in (0, stride):
        P = gp.GrapeProblem.from_workload(w, grad_mode=int(first_order), ckpt_stride=ck)
        if penalty:
            P.set_photon_penalty(w.phys.Q, w.phys.N, 0.3)
        out += gradients(P, w.u)
        P.set_profiling(True)
        P.gradient(w.u)
        counted = sum(n for _, n in P.phase_times().values())
        assert counted <= P.gradient_launches() and (penalty or counted == P.gradient_launches())
    assert np.all(np.isfinite(out[0][1]))
    for F, G in out[1:]:
        assert F == out[0][0] and np.array_equal(G, out[0][1])
