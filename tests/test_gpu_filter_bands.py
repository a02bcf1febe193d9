"""The filter kernels share an output's band between lanes and the matrix
entries between controls of equal bandwidth: bands shorter and longer than the
15 (apply) and 32 (adjoint) terms of one pass, numbers of outputs that leave
half-warps and lanes idle, runs of equal and unequal bandwidths, one to eight
controls, fewer subpixels than controls.  Against the dense transfer matrix;
every term and sum is FP64, so 1e-13 of the largest value (some hundred
roundings of 1e-16), as in test_gpu_filter.py."""
import numpy as np
import pytest

from oracle import filter as gf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M", [(1, 33), (15, 16), (16, 15), (17, 240), (64, 31), (200, 1999)])
@pytest.mark.parametrize("w0", [[3.0], [5.0, 5.0, 2.0], [40.0, 0.5, 0.5, 90.0], [12.0] * 8])
def test_bands_and_bandwidth_runs(N, M, w0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_03170_gb300 import GaussianFilter
    T, R = 2.9, len(w0)
    rng = np.random.default_rng(N * 1000 + M + R)
    u, gs = rng.uniform(-2, 2, size=(N, R)), rng.uniform(-1, 1, size=(M, R))
    f = GaussianFilter(N, M, T, w0, R)
    s = f.apply(torch.from_numpy(u).cuda()).cpu().numpy()
    gu = f.adjoint(torch.from_numpy(gs).cuda()).cpu().numpy()
    for got, ref in ((s, gf.apply(u, M, T / N, T / M, w0)), (gu, gf.adjoint(gs, N, T / N, T / M, w0))):
        assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))
