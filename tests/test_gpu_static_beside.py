"""grape_gradient_static keeps every buffer it writes in its own array, the
cost's partial sums and their ticket among them, so on a cluster-kernel problem
it is independent of a grape_forward or grape_gradient of the same problem on
another stream.  Both in flight at once, with costs of one CTA (d=20) and of
many (d=120: 22 CTAs), several rounds of each: every Phi and every gradient has
the bits of a call that ran alone."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("make", [lambda: workloads.qubit_resonator_d20(n_slices=3),
                                  lambda: workloads.transmon_resonator_d120(n_slices=2)], ids=["d20", "d120"])
def test_static_call_beside_the_other_calls(make, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import GrapeProblem, _lib
    w = make()
    P = GrapeProblem.from_workload(w, precision=prec)
    u = torch.from_numpy(w.u).cuda()
    F0, G0 = P.gradient(u)
    f0 = P.forward(u, want_rho=False)[0]
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    n = 12
    Fs = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    Gs = torch.zeros((n, 2) + tuple(u.shape), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for i in range(n):
        _lib.grape_gradient(P.handle, u.data_ptr(), Fs[i, 0].data_ptr(), Gs[i, 0].data_ptr(), a.cuda_stream)
        _lib.grape_forward(P.handle, u.data_ptr(), Fs[i, 1].data_ptr(), 0, a.cuda_stream)
        _lib.grape_gradient_static(P.handle, u.data_ptr(), Fs[i, 2].data_ptr(), Gs[i, 1].data_ptr(), b.cuda_stream)
    torch.cuda.synchronize()
    P.status()
    assert f0.item() == F0.item()
    assert torch.all(Fs == F0) and torch.all(Gs == G0)
