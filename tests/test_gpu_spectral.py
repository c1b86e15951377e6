"""Complex128 dense plans in the eigenbasis of A (the library's choice of product) against the same
circuit with gate products (``gemm="simt"``), at the edges of the kernels' ranges: one and two
clock bits, registers shorter and longer than a block, both uncompute modes, a non-Toeplitz and an
indefinite (signed clock) A.

Tolerance: both sides are FP64 throughout. A product of N <= 512 terms and 13 transform stages
each round to about 1e-15 of an amplitude of at most 1, and 2 n_c <= 26 products accumulate on the
gate side: 1e-12 absolute leaves an order of magnitude."""
import math

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


def _system(hhl, kind, n):
    if kind == "toeplitz":
        diag, off = hhl.laplacian(n)
        return dict(diag=diag, off=off)
    rng = np.random.default_rng(n)
    q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    lam = rng.uniform(1.0, 9.0, n)
    if kind == "signed":
        lam[::2] *= -1.0
    a = q @ np.diag(lam) @ q.T
    return dict(dense=0.5 * (a + a.T), signed_clock=kind == "signed")


CASES = [("toeplitz", 1, 1), ("toeplitz", 1, 13), ("toeplitz", 2, 2), ("toeplitz", 4, 6), ("toeplitz", 5, 7),
         ("toeplitz", 9, 3), ("toeplitz", 8, 8), ("toeplitz", 3, 12), ("dense", 4, 5), ("dense", 7, 9),
         ("signed", 5, 6), ("signed", 2, 10)]


@pytest.mark.parametrize("kind,n_s,n_c", CASES)
@pytest.mark.parametrize("full", [False, True])
def test_circuit_equals_the_gate_products(hhl, kind, n_s, n_c, full):
    import torch
    sysm = _system(hhl, kind, 1 << n_s)
    gen = torch.Generator(device="cuda").manual_seed(100 * n_s + n_c)
    psi = torch.view_as_complex(torch.randn((2 << (n_s + n_c), 2), dtype=torch.float64, device="cuda", generator=gen))
    psi /= psi.abs().square().sum().sqrt()
    out = []
    for gemm in ("auto", "simt"):
        plan = hhl.HHLPlan(n_s, n_c, precision="c128", gemm=gemm, full_uncompute=full, **sysm)
        st = psi.clone()
        plan.apply_circuit(st)
        out.append(st)
        plan.close()
    assert (out[0] - out[1]).abs().max().item() <= 1e-12


@pytest.mark.parametrize("kind,n_s,n_c", CASES)
def test_postselected_solve_equals_the_gate_products(hhl, kind, n_s, n_c):
    import torch
    n = 1 << n_s
    sysm = _system(hhl, kind, n)
    rng = np.random.default_rng(7)
    b = torch.tensor(rng.random(n) + 1j * rng.standard_normal(n), device="cuda")
    got = []
    for gemm in ("auto", "simt"):
        plan = hhl.HHLPlan(n_s, n_c, precision="c128", gemm=gemm, walls=(0.25, 1.0), nu=0.05, **sysm)
        st = plan.new_state()
        out = torch.empty(4 + 2 * n, dtype=torch.float64, device="cuda")
        eps = torch.empty(1, dtype=torch.float64, device="cuda")
        plan.solve_postselected(b, st, out, eps)
        v = st.view(2, 1 << n_c, n)[1, 0].clone()
        got.append((out.cpu().numpy(), float(eps), v.cpu().numpy(), plan.dissipation(st)))
        plan.close()
    (o1, e1, v1, d1), (o2, e2, v2, d2) = got
    assert np.abs(v1 - v2).max() <= 1e-12
    np.testing.assert_allclose(o1[:4], o2[:4], rtol=1e-11, atol=1e-13)
    # xhat = v / |v|: entry-wise the bound on v over |v|, twice
    np.testing.assert_allclose(o1[4:], o2[4:], atol=2e-12 * (1 + math.sqrt(n)) / math.sqrt(o2[0]))
    assert e1 == pytest.approx(e2, rel=1e-9) and d1 == pytest.approx(e1, rel=1e-12) and d2 == pytest.approx(e2, rel=1e-12)


def test_zero_right_hand_side_is_singular(hhl):
    import torch
    diag, off = hhl.laplacian(8)
    plan = hhl.HHLPlan(3, 4, diag=diag, off=off, precision="c128")
    st = plan.new_state()
    out = torch.empty(20, dtype=torch.float64, device="cuda")
    plan.solve_postselected(torch.zeros(8, dtype=torch.complex128, device="cuda"), st, out)
    assert np.array_equal(out.cpu().numpy(), np.zeros(20))
    with pytest.raises(hhl.HHLError) as e:
        plan.dissipation(st)
    assert e.value.status == 3
