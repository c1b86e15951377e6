"""Chains of tcgen05 products whose operands the products leave for one another, against the same
products one at a time (each gathering its own rows): bit for bit, on random states, for products
of few tiles (stream-K, operands written by the fix-up pass) and of many (written by the GEMM's
epilogue), both directions, and with a state at a 16-byte but not 32-byte boundary."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_s,n_c,shift", [(7, 8, 0), (8, 9, 0), (7, 12, 0), (10, 11, 0), (9, 10, 2)])
def test_chain_equals_single_products(n_s, n_c, shift):
    import torch
    import paper_2307_00391_gb300 as hhl
    diag, off = hhl.laplacian(1 << n_s)
    size = 2 << (n_s + n_c)
    gen = torch.Generator(device="cuda").manual_seed(n_s * 100 + n_c)
    psi = torch.view_as_complex(torch.randn((size, 2), device="cuda", generator=gen)) * (0.5 / size) ** 0.5
    out = []
    for full in (False, True):     # the uncompute of both halves alternates between them: no chain
        plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision="c64", gemm="tcgen05", full_uncompute=full)
        buf = torch.empty(size + shift, dtype=torch.complex64, device="cuda")
        st = buf[shift:]
        st.copy_(psi)
        plan.apply_stage("uncompute_u", st)
        plan.status()
        out.append(st[size // 2:].clone())
        plan.close()
    assert torch.equal(out[0], out[1])
    # forward then adjoint on the same half returns the state (split FP16: 22 bits, 2 n_c products)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision="c64", gemm="tcgen05")
    st = psi.clone()
    plan.apply_stage("qpe_u", st)
    swapped = torch.cat([st[size // 2:], st[:size // 2]])
    plan.apply_stage("uncompute_u", swapped)
    plan.status()
    err = (swapped[size // 2:] - psi[:size // 2]).abs().max() / psi.abs().max()
    assert float(err) <= 2 * n_c * 4e-6


def test_out_of_range_amplitudes_are_reported():
    """An amplitude of magnitude >= 2 in any row of a later product reaches its operand through the
    chain and is reported, as a gather would."""
    import torch
    import paper_2307_00391_gb300 as hhl
    n_s, n_c = 7, 8
    diag, off = hhl.laplacian(1 << n_s)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision="c64", gemm="tcgen05")
    for row in (1 << 7, 1 << 3):       # rows that only one product touches
        st = torch.zeros(2 << (n_s + n_c), dtype=torch.complex64, device="cuda")
        st[(row << n_s) + 5] = 2.5
        plan.apply_stage("qpe_u", st)
        with pytest.raises(hhl.HHLError) as e:
            plan.status()
        assert e.value.status == 7
