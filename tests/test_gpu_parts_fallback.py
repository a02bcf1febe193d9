"""Parts of the space that cannot be built leave a problem at its full size.

The states here occupy nine of 24 basis states whose distances differ: a jump
operator with one band (offset 6) becomes one with three on that part, and with
its rate under a control its nine products are more than the gradient's traces
hold, although the part has fewer products in all (a fixed jump outside it
drops out).  The problem itself is within every limit and runs on the whole
space; against the dense oracle."""
import numpy as np
import pytest

from oracle import dense, operators

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("first_order", [0, 1])
def test_a_part_beyond_the_limits_runs_at_full_size(prec, first_order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import BandModel, BandOp, GrapeProblem
    d, n_slices, n_rk, T = 24, 5, 2, 0.3
    rng = np.random.default_rng(4)
    I = [0, 6, 7, 8, 13, 14, 15, 16, 20]
    row = lambda i, v: np.where(np.arange(d) == i, v, 0.0).astype(complex)
    hop = sum(row(i, v) for i, v in ((0, 0.9), (7, 1.1), (14, 0.7)))
    out = [(o, row(1, 0.3 + 0.1 * o)) for o in (1, 2, 3)]
    H0, H1 = rng.normal(size=d).astype(complex), rng.normal(size=d).astype(complex)
    model = BandModel(d=d, H0=BandOp.make(d, [(0, H0)]), Hc=[BandOp.make(d, []), BandOp.make(d, [(0, H1)])],
                      jumps=[BandOp.make(d, [(6, hop)]), BandOp.make(d, out)], rates=np.array([1.0, 0.5]),
                      jump_control=[0, -1])

    def full(bands):
        A = np.zeros((d, d), dtype=complex)
        for o, v in bands:
            for i in range(max(0, -o), d - max(0, o)):
                A[i, i + o] += v[i]
        return A

    dm = operators.DenseModel(d=d, H0=np.diag(H0), Hc=[np.zeros((d, d), dtype=complex), np.diag(H1)],
                              jumps=[(0.5, full(out))], rate_ctl=[(0, 1.0, full([(6, hop)]))])
    psi = np.zeros(d, dtype=complex)
    psi[I] = rng.normal(size=len(I)) + 1j * rng.normal(size=len(I))
    psi /= np.linalg.norm(psi)
    rho0 = np.outer(psi, psi.conj())[None]
    A = rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))
    sigma = (A + A.conj().T) / 2
    u = np.abs(rng.normal(size=(n_slices, 2)))
    P = GrapeProblem(model, rho0, sigma, T, n_slices, n_rk, grad_mode=first_order, precision=prec)
    F_ref, G_ref = (dense.gradient_first_order if first_order else dense.gradient_exact)(dm, u, rho0, sigma, T, n_rk)
    r_ref = dense.forward(dm, u, rho0, sigma, T, n_rk)[1]
    F, G = P.gradient(u)
    assert abs(F - F_ref) < TOL * abs(F_ref)
    assert np.max(np.abs(G - G_ref)) < TOL * np.max(np.abs(G_ref))
    assert np.max(np.abs(P.forward(u)[1] - r_ref)) < TOL
