"""One-block batch solves (n_s, n_c <= 7) against the single-plan postselected solve, whose launches
they replace operation for operation: the same FP32 states, so the FP64 read-outs agree to
FP64 rounding (only the order of the FP64 sums differs: 1e-12 relative leaves three orders)."""
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


SIZES = [(1, 1), (1, 7), (2, 2), (2, 5), (3, 6), (4, 3), (4, 7), (5, 4), (5, 6), (6, 1), (6, 6), (7, 2), (7, 5), (7, 7)]


def _problems(hhl, sizes):
    rng = np.random.default_rng(3)
    probs, bs = [], []
    for i, (n_s, n_c) in enumerate(sizes):
        n = 1 << n_s
        diag, off = hhl.laplacian(n)
        probs.append(dict(n_sys_qubits=n_s, n_clock=n_c, diag=diag + rng.uniform(0.0, 1.0), off=off, nu=0.07,
                          walls=(0.1, 0.4 * (i % 3)), t0_rule="user", t0=float(rng.uniform(2.0, 40.0))))
        bs.append(rng.standard_normal(n) + 1j * rng.standard_normal(n))
    return probs, bs


def _plan_solve(hhl, pr, b):
    import torch
    n = 1 << pr["n_sys_qubits"]
    plan = hhl.HHLPlan(pr["n_sys_qubits"], pr["n_clock"], diag=pr["diag"], off=pr["off"], precision="c64", gemm="simt",
                       nu=pr["nu"], walls=pr["walls"], t0_rule="user", t0=pr["t0"])
    out = torch.empty(4 + 2 * n, dtype=torch.float64, device="cuda")
    eps = torch.empty(1, dtype=torch.float64, device="cuda")
    plan.solve_postselected(torch.tensor(b, device="cuda"), plan.new_state(), out, eps)
    res = out.cpu().numpy(), float(eps)
    plan.close()
    return res


def test_every_size_matches_the_plan_path(hhl):
    import torch
    probs, bs = _problems(hhl, SIZES)
    batch = hhl.HHLBatch(probs)
    b = torch.tensor(batch.pack_rhs(bs), device="cuda")
    out = torch.full((batch.info["out_doubles"],), float("nan"), dtype=torch.float64, device="cuda")
    eps = torch.full((batch.count,), float("nan"), dtype=torch.float64, device="cuda")
    batch.run(b, out, eps)
    assert 1 <= batch.info["graph_launches"] <= 4
    got, got_eps = out.cpu().numpy(), eps.cpu().numpy()
    for inst, pr, bv, e in zip(batch.instances, probs, bs, got_eps):
        ref, ref_eps = _plan_solve(hhl, pr, bv)
        blk = got[inst["out_offset"]:inst["out_offset"] + 4 + 2 * inst["N"]]
        np.testing.assert_allclose(blk, ref, rtol=1e-12, atol=1e-14, err_msg=str((inst["n_s"], inst["n_c"])))
        assert e == pytest.approx(ref_eps, rel=1e-12)
    # the host-array call and a launch-by-launch run on the retained right-hand sides
    h_out, h_eps = batch.run_host(batch.pack_rhs(bs))
    assert np.array_equal(h_out, got) and np.array_equal(h_eps, got_eps)
    batch.run_eager()
    batch.status()
    batch.close()


def test_mixed_with_larger_instances(hhl):
    """One-block solves beside instances that the graph runs (n_c > 7 or N > 128)."""
    import torch
    probs, bs = _problems(hhl, [(4, 6), (4, 8), (8, 5), (6, 9), (7, 7), (2, 4)])
    batch = hhl.HHLBatch(probs, streams=2)
    b = torch.tensor(batch.pack_rhs(bs), device="cuda")
    out = torch.empty(batch.info["out_doubles"], dtype=torch.float64, device="cuda")
    eps = torch.empty(batch.count, dtype=torch.float64, device="cuda")
    for _ in range(2):
        out.fill_(float("nan"))
        batch.run(b, out, eps)
    got = out.cpu().numpy()
    assert np.isfinite(got).all() and np.isfinite(eps.cpu().numpy()).all()
    for i in (0, 4, 5):
        ref, ref_eps = _plan_solve(hhl, probs[i], bs[i])
        inst = batch.instances[i]
        np.testing.assert_allclose(got[inst["out_offset"]:inst["out_offset"] + 4 + 2 * inst["N"]], ref, rtol=1e-12, atol=1e-14)
        assert float(eps[i]) == pytest.approx(ref_eps, rel=1e-12)
    batch.close()


@pytest.mark.parametrize("form", ["offset", "overlap"])
def test_caller_arrays_of_any_alignment_and_overlap(hhl, form):
    """Right-hand sides at an odd multiple of 8 bytes, and results laid over them: as with arrays of
    their own, bit for bit (one path copies the inputs first, the other reads them in place)."""
    import torch
    probs, bs = _problems(hhl, SIZES)
    batch = hhl.HHLBatch(probs)
    n_b, n_out = batch.info["b_doubles"], batch.info["out_doubles"]
    pool = torch.zeros(max(n_b, n_out) + 1, dtype=torch.float64, device="cuda")
    b = pool[1:1 + n_b] if form == "offset" else pool[:n_b]
    out = torch.empty(n_out, dtype=torch.float64, device="cuda") if form == "offset" else pool[:n_out]
    eps = torch.empty(batch.count, dtype=torch.float64, device="cuda")
    b.copy_(torch.tensor(batch.pack_rhs(bs)))
    batch.run(b, out, eps)
    ref, ref_eps = batch.run_host(batch.pack_rhs(bs))
    assert np.array_equal(out.cpu().numpy(), ref) and np.array_equal(eps.cpu().numpy(), ref_eps)
    batch.close()
