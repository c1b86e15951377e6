"""The read-outs and the preparation of systems of at most 1024 points (one launch each) against plain
torch in FP64, either side of the sizes where the launches change: N = 1024 / 2048, a state below
and above the one-launch preparation's 4 MiB, the smallest rows, and repeated calls (the block
counter of the sums returns to zero)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hhl():
    import torch
    assert torch.cuda.is_available()
    import paper_2307_00391_gb300 as pkg
    pkg.load()
    return pkg


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n_s,n_c", [(1, 1), (1, 9), (4, 6), (7, 11), (10, 4), (10, 9), (11, 4)])
def test_preparation_and_read_outs(hhl, prec, n_s, n_c):
    import torch
    n, r = 1 << n_s, 1 << n_c
    diag, off = hhl.laplacian(n)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision=prec, expm="trotter", trotter_dt=1e9, nu=0.3, walls=(0.5, -0.25))
    gen = torch.Generator(device="cuda").manual_seed(n_s * 31 + n_c)
    b = torch.randn((n, 2), dtype=torch.float64, device="cuda", generator=gen)
    st = plan.new_state()
    plan.prepare_rhs(torch.view_as_complex(b), st)
    bn = b.square().sum().sqrt()
    want = (torch.view_as_complex(b) / (bn * r ** 0.5)).to(st.dtype)
    view = st.view(2, r, n)
    # the scaled row is one FP64 product rounded once: half an ulp, two for the norm's own rounding
    tol = (2.4e-7 if prec == "c64" else 1e-15) * float(want.abs().max())
    assert (view[0] - want).abs().max().item() <= tol and view[1].abs().max().item() == 0.0
    torch.view_as_real(st).normal_(generator=gen)
    big = st.to(torch.complex128).view(2, r, n)
    w0, w1 = (float(big[a].abs().square().sum()) for a in (0, 1))
    v = big[1, 0]
    out = torch.empty(4 + 2 * n, dtype=torch.float64, device="cuda")
    eps = torch.empty(1, dtype=torch.float64, device="cuda")
    for _ in range(3):
        out.zero_()
        plan.measure_async(st, out)
        plan.dissipation_async(st, eps)
        got = out.cpu().numpy()
        ps = float(v.abs().square().sum())
        # complex64 squares are rounded to FP32 before they are summed: 2^-24 each at worst
        rel = 2e-7 if prec == "c64" else 1e-13
        np.testing.assert_allclose(got[:4], [ps, w1, w0 + w1, float(bn)], rtol=rel)
        # xhat is v over the root of the returned p_success
        np.testing.assert_allclose(got[4::2] + 1j * got[5::2], (v / got[0] ** 0.5).cpu().numpy(), rtol=1e-13, atol=1e-15)
        info = plan.info
        u = torch.empty(n + 2, dtype=torch.float64, device="cuda")
        u[0], u[-1] = 0.5, -0.25
        u[1:-1] = bn * v.real / (info["C"] * info["lambda_ub"])
        assert float(eps) == pytest.approx(0.3 * (n + 1) * float((u[1:] - u[:-1]).square().sum()), rel=1e-12)
    plan.close()
