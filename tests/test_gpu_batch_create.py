"""Batch creation: the tables that the worker streams read have reached the device when they start, so
every creation of the same batch gives the same read-outs (the weights up to the order of their FP64
block sums, everything else bit for bit) while other copies from pageable memory are under way."""
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


# one-block solves, graph instances on the CUDA cores and on the tensor cores; all of one kind, and mixed
@pytest.mark.parametrize("sizes", [[(8, 4), (9, 3), (8, 8), (10, 7)], [(3, 5), (8, 4), (6, 6), (9, 8), (2, 2), (8, 6)]])
def test_creations_agree(hhl, sizes):
    import torch
    rng = np.random.default_rng(5)
    probs, bs = [], []
    for n_s, n_c in sizes:
        diag, off = hhl.laplacian(1 << n_s)
        probs.append(dict(n_sys_qubits=n_s, n_clock=n_c, diag=diag, off=off, t0_rule="user", t0=9.0, walls=(0.0, 1.0)))
        bs.append(rng.standard_normal(1 << n_s))
    big = torch.zeros(1 << 24, dtype=torch.float64)              # 128 MiB, pageable
    dst = torch.empty(1 << 24, dtype=torch.float64, device="cuda")
    ref = None
    for _ in range(12):
        dst.copy_(big)
        batch = hhl.HHLBatch(probs, streams=4)
        b = torch.tensor(batch.pack_rhs(bs), device="cuda")
        out = torch.full((batch.info["out_doubles"],), float("nan"), dtype=torch.float64, device="cuda")
        eps = torch.full((batch.count,), float("nan"), dtype=torch.float64, device="cuda")
        batch.run(b, out, eps)
        got = out.cpu().numpy(), eps.cpu().numpy()
        ref = got if ref is None else ref
        np.testing.assert_allclose(got[0], ref[0], rtol=1e-13, atol=1e-16)
        assert np.array_equal(got[1], ref[1])
        batch.close()
