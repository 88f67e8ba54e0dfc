"""Rounding of the 32-vector apply beside that of groups of 8 (GPU, through the C ABI).
Both add float sums of a few products (at most 8 in the one, 16 in the other) into
compensated pairs, so by the count of roundings per sum the 32-vector form errs no more:
the relative defect of linearity, M(sum c_k x_k) - sum c_k M x_k over 31 random
vectors, may exceed that of the groups by what two samples of 31 x N errors differ, a few
per cent; half as much again is allowed.  (Sums of 64 products gave 2.6 times as much.)"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec", [(32, 1), (64, 1), (64, 2), (24, 1), (40, 1), (56, 2)])
@pytest.mark.parametrize("trans", [False, True])
def test_wide_apply_rounds_as_groups_of_8(n, prec, trans):
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    N = n ** 3
    coef = torch.empty(7 * N, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_codi(n, torch.full((3 * N,), 30.0, dtype=torch.float64, device="cuda:0"), coef)
    h = acr.Handle(n, coef, 1e-2, 2.0, 64, prec, 24)
    fn = h.apply_transpose if trans else h.apply
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(n)
    c = torch.randn(31, 1, dtype=torch.float64, device="cuda:0", generator=gen)
    r = torch.randn(32, N, dtype=torch.float64, device="cuda:0", generator=gen)
    r[31] = (c * r[:31]).sum(0)

    def defect(group):
        z = torch.empty_like(r)
        for k in range(0, 32, group):
            fn(r[k:k + group].reshape(-1), z[k:k + group].reshape(-1), nrhs=group)
        y = c * z[:31]
        return ((z[31] - y.sum(0)).norm() / y.norm()).item()

    wide, eights = defect(32), defect(8)
    h.close()
    assert wide <= 1.5 * eights, (wide, eights)
