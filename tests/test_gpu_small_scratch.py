"""A setup whose scratch holds one plane of a small operation at a time pushes so many
pointer tables that the ring that holds them comes round within one H-inverse; the
leaf inverses must not read a table that has been overwritten.  The same operator with
all of its scratch: equal ranks, and the applies differ by the float sums' order only."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_setup_with_little_scratch(monkeypatch):
    from paper_1712_08872_gb300 import _build
    _build.build()
    import paper_1712_08872_gb300 as acr

    n = 64
    N = n ** 3
    coef = torch.empty(7 * N, dtype=torch.float64, device="cuda:0")
    acr.acr_stencil_codi(n, torch.full((3 * N,), 30.0, dtype=torch.float64, device="cuda:0"), coef)
    r = torch.rand(N, dtype=torch.float64, device="cuda:0")
    out = []
    for mb in (None, "1"):
        if mb:
            monkeypatch.setenv("ACR_SCRATCH_MB", mb)
        h = acr.Handle(n, coef, 1e-2, 2.0, 64, acr.ACR_FP32, 24)
        z = torch.empty_like(r)
        h.apply(r, z)
        out.append((z, h.info().max_rank))
        h.close()
    assert out[0][1] == out[1][1]
    # rounding of the factors' float sums (6e-8 each) through the setup's levels, as the parity
    # of the float form with the oracle's float32 model: 1e-5
    assert ((out[0][0] - out[1][0]).norm() / out[0][0].norm()).item() <= 1e-5
