"""The status word of a bounds-checked library (PCBP_CHECKED=1): every decode clears it, whatever
the workspace held and however few frames the batch has."""
import pytest

from conftest import gpu_device
from test_gpu_checked import status_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [8, 64, 128, 1024])
@pytest.mark.parametrize("B", [1, 40, 9000])
def test_status_word_is_cleared(pcbp, N, B):
    import torch

    if not pcbp.build_checked():
        pytest.skip("not a bounds-checked build (PCBP_CHECKED=1)")
    dev = gpu_device()
    code = pcbp.pc_construct(N, N // 2)
    dec = pcbp.Decoder(code, pcbp.sched(mode=0, stop_kind=1), 3, dev)
    dec.workspace.fill_(0x5A)
    dec(torch.randn((B, N), device=dev))
    torch.cuda.synchronize()
    assert status_of(dec) == 0
