"""The split clock passes whose twiddles come from a table per tile, on random states, against
FFTs in FP64: every split of the clock bits into high and low passes (4-7 bits each)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# relative 2-norm: two transforms of up to 13 stages, about 1.5 roundings a stage and amplitude, plus
# the factors' and the scalings' own; FP32 2^-24, double-float about 2^-44
TOL = {"c64": 45 * 2.0 ** -24, "c128": 45 * 2.0 ** -44}


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("n_c", [8, 9, 10, 11, 12, 13])
def test_clock_block_with_twiddle_tables(monkeypatch, prec, full, n_c):
    import torch
    import paper_2307_00391_gb300 as hhl
    monkeypatch.setenv("HHL_FFT_SPLIT", "1")
    monkeypatch.setenv("HHL_CLOCK_CLUSTER", "0")
    monkeypatch.setenv("HHL_GROUP", "0")
    n_s, rows = 5 + n_c % 3, 1 << n_c
    n = 1 << n_s
    diag, off = hhl.laplacian(n)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision=prec, gemm="simt", full_uncompute=full)
    rng = np.random.default_rng(n_c)
    x = rng.standard_normal((rows, n)) + 1j * rng.standard_normal((rows, n))
    x = x.astype(np.complex64 if prec == "c64" else np.complex128)
    st = plan.new_state()
    host = np.zeros((2, rows, n), dtype=x.dtype)
    host[0] = x
    st.copy_(torch.from_numpy(host).view(st.dtype).reshape(st.shape))
    plan.apply_stage("clock_block", st)
    got = st.cpu().numpy().reshape(2, rows, n)
    y = np.fft.fft(x.astype(np.complex128), axis=0, norm="ortho")  # the inverse QFT
    s = np.zeros(rows)
    s[1:] = 1.0 / np.arange(1, rows)  # T0 fills the clock range: sin(theta_y / 2) = 1 / y
    c = np.sqrt(1.0 - s * s)
    one = np.fft.ifft(y * s[:, None], axis=0, norm="ortho")
    zero = y * c[:, None]
    if full:
        zero = np.fft.ifft(zero, axis=0, norm="ortho")
    for a, r in ((got[0], zero), (got[1], one)):
        assert np.linalg.norm(a - r) <= TOL[prec] * np.linalg.norm(r)
    plan.close()
