"""Launch profiles name the kernels that ran: the tiled whole-register QFT and the passes of smaller ones."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,names", [(20, {"k_qft_low", "k_qft_pass"}), (18, {"k_lowbits_transform", "k_whole_pass"})])
def test_names(n, names):
    import torch
    import paper_2307_00391_gb300 as hhl
    s = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    hhl.qft_whole(s, n, 1, 0)
    hhl.profile_reset()
    hhl.profile_enable(True)
    hhl.qft_whole(s, n, 1, 0)
    hhl.qft_whole(s, n, 1, 1)
    torch.cuda.synchronize()
    hhl.profile_enable(False)
    assert set(hhl.profile_read()) == names
