"""The fused recompression stages of the float forms (basis and core kernels)
at the edges of their range (GPU, through the C ABI): leaf sizes that are no
multiple of a warp, sketches of every width up to the widest (rank cap 48), and
weak admissibility, whose largest sketch (1152 x 56 floats) does not fit shared
memory.  And 32 right-hand sides at once at several leaf sizes.

The float factors differ from the FP64 form's by rounding, far below eps, so
GMRES preconditioned with them takes the FP64 form's iterations, give or take
one; the residual is confirmed by the oracle's SpMV.
"""
import numpy as np
import pytest

from inputs import codi_beta, gaussian_field_kappa, uniform_rhs
from oracle.assembly import stencil_apply, stencil_codi, stencil_poisson

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pde,n,eta,eps,cap", [
    ("poisson", 20, 2.0, 1e-2, 19),     # 50-point leaves, 27-column sketches
    ("codi", 24, 2.0, 1e-2, 24),        # 36-point leaves
    ("poisson", 28, 2.0, 1e-5, 48),     # 49-point leaves, 56-column sketches
    ("codi", 48, 96.0, 0.3, 48),        # one 1152 x 1152 admissible block per half
])
def test_float_cores(pde, n, eta, eps, cap):
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    def dev(x):
        return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda:0")

    coef = torch.empty(7 * n ** 3, dtype=torch.float64, device="cuda:0")
    if pde == "codi":
        beta = codi_beta(n)
        acr.acr_stencil_codi(n, dev(beta.ravel()), coef)
        st = stencil_codi(beta, n)
    else:
        kappa = gaussian_field_kappa(n, 3)
        acr.acr_stencil_poisson(n, dev(kappa), coef)
        st = stencil_poisson(kappa, n)
    f = uniform_rhs(n, 5)
    its = {}
    for prec in (acr.ACR_FP64, acr.ACR_FP32):
        h = acr.Handle(n, coef, eps, eta, 64, prec, cap)
        u = torch.zeros(n ** 3, dtype=torch.float64, device="cuda:0")
        info, _ = acr.acr_krylov_solve(h.h, coef, acr.ACR_GMRES, 30, 1e-9, 200, dev(f), u)
        h.close()
        its[prec] = info.iterations
        res = np.linalg.norm(f - stencil_apply(st, n, u.cpu().numpy())) / np.linalg.norm(f)
        assert res <= 1.0001e-9, (prec, res)
    assert abs(its[acr.ACR_FP32] - its[acr.ACR_FP64]) <= 1, its


@pytest.mark.parametrize("n,leaf,prec", [(8, 64, 1), (16, 64, 2), (20, 25, 1), (24, 64, 2), (28, 64, 1)])
@pytest.mark.parametrize("trans", [False, True])
def test_apply_32_vectors_any_leaf(n, leaf, prec, trans):
    """33 right-hand sides, the first 32 in one pass, against the same vectors in
    groups of 8 and one: leaves of 64 (alone, without low-rank blocks, and 4 of them),
    25, 36 and 49 points.  The same factors and float vectors (rounding 6e-8) in
    other summation orders: float sums of at most 64 products err by less than
    8 * 6e-8 of their norm, through a chain of at most 2 log2 n products that mostly
    average out: 1e-6.  The 33rd vector takes the same path in both."""
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    beta = torch.full((3 * n ** 3,), 30.0, dtype=torch.float64, device="cuda:0")
    coef = torch.empty(7 * n ** 3, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_codi(n, beta, coef)
    h = acr.Handle(n, coef, 1e-2, 2.0, leaf, prec, 24)
    fn = h.apply_transpose if trans else h.apply
    r = torch.tensor(np.stack([uniform_rhs(n, k) for k in range(33)]), device="cuda:0")
    z = torch.empty_like(r)
    fn(r.reshape(-1), z.reshape(-1), nrhs=33)
    for k in range(0, 33, 8):
        q = r[k:k + 8].contiguous()
        w = torch.empty_like(q)
        fn(q.reshape(-1), w.reshape(-1), nrhs=q.shape[0])
        err = ((z[k:k + 8] - w).norm(dim=1) / w.norm(dim=1)).max().item()
        assert err <= (0.0 if k == 32 else 1e-6), (k, err)
    h.close()


@pytest.mark.parametrize("n,prec", [(2, 0), (3, 1), (8, 1), (20, 0), (28, 1), (32, 2)])
def test_inverse_beside_updates(n, prec):
    """A profiled setup times every launch and so runs on one stream; the default one
    inverts the next level's planes beside the other planes' updates.  The same kernels
    on the same operands, whose sums do not depend on the batch: equal results."""
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    beta = torch.full((3 * n ** 3,), 20.0, dtype=torch.float64, device="cuda:0")
    coef = torch.empty(7 * n ** 3, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_codi(n, beta, coef)
    r = torch.tensor(uniform_rhs(n, 5), device="cuda:0")
    out = []
    for flags in (acr.ACR_FLAG_PROFILE, 0, 0):
        h = acr.Handle(n, coef, 1e-2, 2.0, 64, prec, 24, flags=flags)
        z, i = torch.empty_like(r), h.info()
        h.apply(r, z)
        out.append((z.cpu(), i.max_rank, i.lr_truncations, i.sketch_overflows, i.factor_bytes))
        h.close()
    for o in out[1:]:
        assert torch.equal(o[0], out[0][0]) and o[1:] == out[0][1:], o[1:]


@pytest.mark.parametrize("n,prec,nr", [(12, 0, 3), (16, 1, 9), (20, 1, 33)])
def test_pcg_in_lockstep(n, prec, nr):
    """Several right-hand sides by PCG, one of them zero: every residual by the
    oracle's SpMV meets the tolerance (slack for the final residual's own rounding), the
    zero one's solution is zero, and the count is the largest single one, give or take
    the one step that rounding can move at the tolerance."""
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    def dev(x):
        return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda:0")

    kappa = gaussian_field_kappa(n, 4)
    st = stencil_poisson(kappa, n)
    coef = torch.empty(7 * n ** 3, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_poisson(n, dev(kappa), coef)
    F = np.stack([uniform_rhs(n, 60 + k) for k in range(nr)])
    F[1] = 0.0
    h = acr.Handle(n, coef, 1e-2, 2.0, 64, prec, 24)
    u = torch.ones(nr * n ** 3, dtype=torch.float64, device="cuda:0")
    info, _ = acr.acr_krylov_solve(h.h, coef, acr.ACR_PCG, 30, 1e-9, 200, dev(F.ravel()), u, nrhs=nr)
    single = 0
    for k in range(nr):
        v = torch.ones(n ** 3, dtype=torch.float64, device="cuda:0")
        one, _ = acr.acr_krylov_solve(h.h, coef, acr.ACR_PCG, 30, 1e-9, 200, dev(F[k]), v)
        single = max(single, one.iterations)
    h.close()
    U = u.cpu().numpy().reshape(nr, -1)
    assert not U[1].any()
    for k in range(nr):
        if k != 1:
            res = np.linalg.norm(F[k] - stencil_apply(st, n, U[k])) / np.linalg.norm(F[k])
            assert res <= 1.001e-9, (k, res)
    assert abs(info.iterations - single) <= 1, (info.iterations, single)


@pytest.mark.parametrize("n", [1, 7, 33])
@pytest.mark.parametrize("nr", [1, 2, 3, 4, 5, 7])
def test_spmv_vector_groups(n, nr):
    """The SpMV reads the coefficients once per up to four vectors: every count of
    vectors against the oracle's (seven products and their sum, so 8 units of
    rounding of the terms' magnitudes)."""
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    kappa = gaussian_field_kappa(n, 4)
    st = stencil_poisson(kappa, n)
    coef = torch.empty(7 * n ** 3, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_poisson(n, torch.tensor(np.ascontiguousarray(kappa), dtype=torch.float64,
                                            device="cuda:0"), coef)
    X = np.stack([uniform_rhs(n, k) for k in range(nr)])
    x = torch.tensor(X, device="cuda:0").reshape(-1)
    y = torch.empty_like(x)
    acr.acr_spmv(n, coef, x, y, nr)
    Y = y.cpu().numpy().reshape(nr, -1)
    for k in range(nr):
        ref = stencil_apply(st, n, X[k]).ravel()
        mag = np.abs(st["c"]).max() * 2 * np.abs(X[k]).max()
        assert np.abs(Y[k] - ref).max() <= 8 * 2.3e-16 * mag, k
