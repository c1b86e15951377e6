"""Complex128 plans of 2^12 points with one clock qubit apply their two gate products (faster there than the
eigenbasis form), with the whole uncompute the eigenbasis form: each against the explicit choice."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("full", [False, True])
def test_route(full):
    import torch
    import paper_2307_00391_gb300 as hhl
    n_s, n_c = 12, 1
    diag, off = hhl.laplacian(1 << n_s)
    gen = torch.Generator(device="cuda").manual_seed(1)
    psi = torch.view_as_complex(torch.randn((2 << (n_s + n_c), 2), dtype=torch.float64, device="cuda", generator=gen))
    psi /= psi.abs().square().sum().sqrt()
    out = []
    for gemm in ("auto", "simt"):
        plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision="c128", gemm=gemm, full_uncompute=full)
        st = psi.clone()
        plan.apply_circuit(st)
        out.append(st)
        plan.close()
    if full:
        # products of 4096 terms: as for the smaller sizes, 1e-15 a term of an amplitude of at most 1 each
        assert (out[0] - out[1]).abs().max().item() <= 1e-11
    else:
        assert torch.equal(out[0], out[1])
