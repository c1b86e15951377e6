"""The tiled whole-register QFT (complex64, from 2^20 amplitudes in all) against torch's FP64 FFT: every
pass width (4 to 9 bits and two passes above the chunk), several states, both directions, and
either side of the size where the tiled form starts.

Tolerance: n radix-2 stages each round an amplitude by about 2^-24 of the state's rms, their twiddles
(products of at most five rounded factors) by a few 2^-24 more: 1e-6 of the rms in the 2-norm,
1e-5 for the largest deviation."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,states", [(16, 8), (16, 16), (17, 8), (18, 4), (19, 2), (20, 1), (20, 4), (21, 1), (22, 1),
                                      (23, 2), (25, 1)])
@pytest.mark.parametrize("direction", [0, 1])
def test_against_fft(n, states, direction):
    import torch
    import paper_2307_00391_gb300 as hhl
    size = 1 << n
    gen = torch.Generator(device="cuda").manual_seed(n * 10 + states)
    z = torch.view_as_complex(torch.randn((states * size, 2), device="cuda", generator=gen)) * math.sqrt(0.5 / size)
    i = torch.arange(size, device="cuda")
    rev = torch.zeros_like(i)
    for b in range(n):
        rev |= ((i >> b) & 1) << (n - 1 - b)
    ref = z.to(torch.complex128).view(states, size)
    ref = torch.fft.ifft(ref, dim=1, norm="ortho")[:, rev] if direction == 0 else torch.fft.fft(ref[:, rev], dim=1, norm="ortho")
    hhl.qft_whole(z, n, states, direction)
    d = (z.view(states, size) - ref).abs()
    rms = float(ref.abs().square().mean().sqrt())
    assert float(d.square().mean().sqrt()) <= 1e-6 * rms
    assert float(d.max()) <= 1e-5 * rms
