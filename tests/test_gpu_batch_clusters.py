"""One-block batch solves shared by clusters of 8, 4 and 2 blocks (fewer instances than SMs) against the same
instances one block each and against the single-plan solve: the same FP32 states, so the FP64 read-outs
agree to FP64 rounding (only the order of the FP64 sums differs: 1e-12 relative leaves three orders)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# 16 columns a block at least: N = 128 shares an instance among 8, 64 among 4, 32 among 2, 16 not at all
SIZES = [(7, 7), (7, 1), (6, 6), (5, 7), (4, 5), (7, 4), (1, 1), (6, 2), (5, 3)]


def _run(hhl, probs, bs, **kw):
    import torch
    batch = hhl.HHLBatch(probs, **kw)
    b = torch.tensor(batch.pack_rhs(bs), device="cuda")
    out = torch.full((batch.info["out_doubles"],), float("nan"), dtype=torch.float64, device="cuda")
    eps = torch.full((batch.count,), float("nan"), dtype=torch.float64, device="cuda")
    for _ in range(2):
        batch.run(b, out, eps)
    got = [out.cpu().numpy()[i["out_offset"]:i["out_offset"] + 4 + 2 * i["N"]] for i in batch.instances]
    got_eps = eps.cpu().numpy()
    batch.close()
    return got, got_eps


@pytest.mark.parametrize("count", [1, 2, 9, 18, 36, 72, 76, 77, 160])
@pytest.mark.parametrize("beside", [False, True])
def test_every_cluster_size(count, beside):
    import torch
    import paper_2307_00391_gb300 as hhl
    from tests.test_gpu_batch_small import _plan_solve, _problems
    assert torch.cuda.is_available()
    hhl.load()
    probs, bs = _problems(hhl, SIZES)
    ref = [_plan_solve(hhl, pr, b) for pr, b in zip(probs, bs)]
    order = [i % len(SIZES) for i in range(count)]
    probs, bs = [probs[i] for i in order], [bs[i] for i in order]
    if beside:  # two instances that the graph runs
        more, more_b = _problems(hhl, [(8, 4), (5, 8)])
        probs, bs = probs + more, bs + more_b
    got, eps = _run(hhl, probs, bs, streams=2)
    for q, i in enumerate(order):
        np.testing.assert_allclose(got[q], ref[i][0], rtol=1e-12, atol=1e-14, err_msg=str(SIZES[i]))
        assert eps[q] == pytest.approx(ref[i][1], rel=1e-12)
    assert all(np.isfinite(g).all() for g in got) and np.isfinite(eps).all()
