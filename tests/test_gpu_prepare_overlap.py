"""Preparation with the right-hand side inside the state it prepares: b is read whole before any of the
state is stored, so the result is that of a separate copy of b, bit for bit."""
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


# states of many blocks, up to the 4 MiB that one launch takes, and a larger one
@pytest.mark.parametrize("n_s,n_c", [(3, 7), (6, 6), (8, 8), (8, 9), (10, 8)])
@pytest.mark.parametrize("precision", ["c64", "c128"])
@pytest.mark.parametrize("where", ["first", "postselected", "last", "before", "after"])
def test_rhs_inside_the_state(hhl, n_s, n_c, precision, where):
    import torch
    n, half = 1 << n_s, 1 << (n_s + n_c)
    diag, off = hhl.laplacian(n)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision=precision)
    b = np.random.default_rng(n_s).standard_normal((n, 2)).view(np.complex128)[:, 0]
    amp = 8 if precision == "c64" else 16
    pad = 16 * n                                                       # bytes either side of the state
    buf = torch.zeros(2 * half * amp + 2 * pad, dtype=torch.uint8, device="cuda")
    at = {"first": pad, "postselected": pad + half * amp, "last": pad + 2 * half * amp - 16 * n,
          "before": pad - 8 * n, "after": pad + 2 * half * amp - 8 * n}[where]
    state = buf[pad:pad + 2 * half * amp].view(torch.complex64 if precision == "c64" else torch.complex128)
    b_in = buf[at:at + 16 * n].view(torch.complex128)
    want, got = plan.new_state(), [torch.empty(4 + 2 * n, dtype=torch.float64, device="cuda") for _ in range(2)]
    b_dev = torch.tensor(b, device="cuda")
    plan.prepare_rhs(b_dev, want)
    plan.measure_async(want, got[0])
    for _ in range(8):
        b_in.copy_(b_dev)
        plan.prepare_rhs(b_in, state)
        plan.measure_async(state, got[1])
        assert torch.equal(state, want)
        assert torch.equal(got[0], got[1])                             # |b| among them
    plan.close()
