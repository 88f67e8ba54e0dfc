"""Point kernels at the edges of their inputs (GPU, through the C ABI)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _acr():
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr
    return acr


def test_codi_stencil_of_nan_and_infinite_velocities():
    """The upwind terms are those of fmax(b, 0) and fmin(b, 0), which a NaN leaves at zero;
    whole coefficients equal (an infinite one included)."""
    acr = _acr()
    n = 5
    N = n ** 3
    beta = np.random.default_rng(3).uniform(-3.0, 3.0, (3, N))
    beta[:, 31] = [np.nan, -np.nan, 0.0]
    beta[:, 62] = [np.inf, -np.inf, -0.0]
    coef = torch.empty(7 * N, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_codi(n, torch.tensor(beta.ravel(), device="cuda:0"), coef)
    got = coef.cpu().numpy().reshape(7, n, n, n)
    h = 1.0 / (n + 1)
    ih, ih2 = 1.0 / h, 1.0 / (h * h)
    for a in range(3):
        b = beta[a].reshape(n, n, n)
        axis = 2 - a
        for k, want in ((2 * a + 1, -ih2 - np.fmax(b, 0.0) * ih), (2 * a + 2, -ih2 + np.fmin(b, 0.0) * ih)):
            edge = [slice(None)] * 3
            edge[axis] = 0 if k % 2 else n - 1
            want[tuple(edge)] = 0.0
            # (one rounding less where the multiply-add is fused)
            fin = np.isfinite(want)
            assert np.array_equal(np.isfinite(got[k]), fin), k
            assert np.array_equal(got[k][~fin], want[~fin]), k
            assert np.abs(got[k][fin] - want[fin]).max() <= 2.3e-16 * np.abs(want[fin]).max(), k


@pytest.mark.parametrize("n", [7, 33])
def test_spmv_of_vectors_that_are_results(n):
    """y = x + N: each vector is the result of the one before; equal to single products."""
    acr = _acr()
    N = n ** 3
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(5)
    kappa = 1.0 + torch.rand(N, dtype=torch.float64, device="cuda:0", generator=gen)
    coef = torch.empty(7 * N, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_poisson(n, kappa, coef)
    v = torch.zeros(7, N, dtype=torch.float64, device="cuda:0")
    v[0] = kappa / n ** 2
    want = v.clone()
    for k in range(6):
        acr.acr_spmv(n, coef, want[k], want[k + 1], 1)
    acr.acr_spmv(n, coef, v.reshape(-1), v.reshape(-1)[N:], 6)
    assert torch.equal(v, want)
