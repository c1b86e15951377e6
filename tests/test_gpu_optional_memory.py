"""Plans without the memory they can do without (HHL_FAULT=optional withholds it): complex128 plans then
run their gate products, tcgen05 chains gather every operand; creation succeeds and the results are the
same, bit for bit, as those of the forms they fall back to."""
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


def _solve(hhl, n_s, n_c, precision, gemm):
    import torch
    n = 1 << n_s
    diag, off = hhl.laplacian(n)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision=precision, gemm=gemm, walls=(0.0, 1.0))
    b = torch.tensor(np.random.default_rng(n_c).standard_normal(n) + 0j, device="cuda")
    st, st2 = plan.new_state(), plan.new_state()
    plan.prepare_rhs(b, st)
    plan.apply_circuit(st)
    out = torch.empty(4 + 2 * n, dtype=torch.float64, device="cuda")
    plan.solve_postselected(b, st2, out)
    plan.status()
    info = plan.info
    plan.close()
    return st, st2.view(2, 1 << n_c, n)[1, 0].clone(), out[4:].clone(), info["table_bytes"] + info["workspace_bytes"]


@pytest.mark.parametrize("n_s,n_c,precision,gemm,same_as",
                         [(4, 6, "c128", "auto", "simt"), (6, 4, "c128", "auto", "simt"),
                          (7, 8, "c64", "tcgen05", "tcgen05"), (8, 10, "c64", "tcgen05", "tcgen05")])
def test_results_without_it(hhl, monkeypatch, n_s, n_c, precision, gemm, same_as):
    import torch
    want = _solve(hhl, n_s, n_c, precision, same_as)
    full = _solve(hhl, n_s, n_c, precision, gemm)
    monkeypatch.setenv("HHL_FAULT", "optional")
    got = _solve(hhl, n_s, n_c, precision, gemm)
    assert got[3] < full[3]                                # withheld
    for g, w in zip(got[:3], want[:3]):
        assert torch.equal(g, w)
