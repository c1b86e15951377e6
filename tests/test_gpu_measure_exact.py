"""The sums over a state (norm, P(anc = 1), P(success)) are FP64 across threads and blocks: exact where
every partial sum is.

Amplitudes k 2^-26 and, a few, k 2^-14 with integers k < 2^12, at most one nonzero amplitude to a
16-byte unit and at most one unit to a thread: their squares are exact in FP32 (24 bits) and
multiples of 2^-52, and every sum stays below 1, so FP64 adds them exactly in any order. The 48 bits of a
double-float value below 1 do not hold such sums. No tolerance is needed."""
from fractions import Fraction

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


@pytest.mark.parametrize("n_s,n_c", [(4, 6), (10, 2), (11, 2)])   # one launch, its largest N, two launches
@pytest.mark.parametrize("precision", ["c64", "c128"])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_sums_are_exact(hhl, n_s, n_c, precision, seed):
    import torch
    n, half = 1 << n_s, 1 << (n_s + n_c)
    rng = np.random.default_rng(seed)
    k = rng.integers(1, 4096, 2 * half)
    if precision == "c64":
        k[1::2] = 0
    amp = k * 2.0 ** -26
    for lo, hi in ((0, half), (half, half + n), (half + n, 2 * half)):
        big = lo + 2 * rng.choice((hi - lo) // 2, 3, replace=False)
        amp[big] = k[big] * 2.0 ** -14
    sq = [Fraction(float(a)) ** 2 for a in amp]
    w0, ps = sum(sq[:half]), sum(sq[half:half + n])
    w1 = ps + sum(sq[half + n:])
    assert w0 + w1 < 1 and (2 ** 52 * (w0 + w1)).denominator == 1
    diag, off = hhl.laplacian(n)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision=precision)
    state = plan.new_state()
    out = torch.empty(4 + 2 * n, dtype=torch.float64, device="cuda")
    plan.prepare_rhs(torch.ones(n, dtype=torch.complex128, device="cuda"), state)
    for turn in (1.0, 1j):                                          # real and imaginary parts
        state.copy_(torch.tensor(amp * turn, device="cuda"))
        plan.measure_async(state, out)
        assert out[:3].tolist() == [float(ps), float(w1), float(w0 + w1)]
    plan.close()
