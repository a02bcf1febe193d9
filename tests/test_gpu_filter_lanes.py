"""The filter kernels let fewer lanes share an output where there are outputs
enough to fill the chip and their bands are short: every group width, with
numbers of outputs that leave groups of the last warp idle, one control and
several of equal and unequal bandwidth (1, 2, 4, 8 and 16 lanes of the adjoint,
1, 4 and 8 of apply).  Against the terms within the band, which are all that are not
zero (erf is +-1 beyond 6.5).  Dt = 1/4 and M a power of two times N, so every
edge t - j Dt is exact; erf to 1e-16 and a few dozen roundings of sums leave
1e-14, so 1e-13 of the largest value as for the other sizes."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def erf(x):
    out = np.sign(x)
    near = np.abs(x) < 6.5
    out[near] = [math.erf(v) for v in x[near]]
    return out


def band(n_out, n_in, step_out, step_in, w, v, adjoint):
    """sum over the terms near each output of T times v."""
    lo, hi = (-2 * 6.5 / w, 2 * 6.5 / w)
    out = np.zeros(n_out)
    width = int(math.ceil(((hi - lo) + (step_out if adjoint else 0.0)) / step_in)) + 6
    o = np.arange(n_out)
    first = np.floor((o * step_out + lo) / step_in).astype(int) - 2
    for k in range(width):
        i = first + k
        ok = (i >= 0) & (i < n_in)
        ic = np.clip(i, 0, n_in - 1)
        n, j = (ic, o) if adjoint else (o, ic)
        dt, Dt = (step_in, step_out) if adjoint else (step_out, step_in)
        T = 0.5 * (erf(0.5 * w * (n * dt - j * Dt)) - erf(0.5 * w * (n * dt - (j + 1) * Dt)))
        out += np.where(ok, T * v[ic], 0.0)
    return out


@pytest.mark.parametrize("N,sub,w0", [(30011, 1, [1e6]), (9001, 1, [1e6]), (4001, 1, [1e6]), (2003, 1, [1e6]),
                                      (1201, 1, [52.0]), (9001, 1, [52.0, 52.0]), (1001, 4, [56.0]), (7001, 4, [50.0]),
                                      (13001, 8, [1e3]), (6007, 8, [60.0, 90.0, 90.0]), (2111, 16, [31.0])])
def test_narrow_groups(N, sub, w0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import GaussianFilter
    M, R, T = N * sub, len(w0), 0.25 * N
    rng = np.random.default_rng(N + M)
    u, gs = rng.uniform(-2, 2, size=(N, R)), rng.uniform(-1, 1, size=(M, R))
    f = GaussianFilter(N, M, T, w0, R)
    s = f.apply(torch.from_numpy(u).cuda()).cpu().numpy()
    gu = f.adjoint(torch.from_numpy(gs).cuda()).cpu().numpy()
    for k in range(R):
        ref = band(M, N, T / M, T / N, w0[k], u[:, k], False)
        assert np.max(np.abs(s[:, k] - ref)) <= 1e-13 * np.max(np.abs(ref))
        ref = band(N, M, T / N, T / M, w0[k], gs[:, k], True)
        assert np.max(np.abs(gu[:, k] - ref)) <= 1e-13 * np.max(np.abs(ref))
