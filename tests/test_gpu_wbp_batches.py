"""The FP32 weighted-BP kernels over batches: one frame, fewer frames than SMs, several frames per
slot.  Frames are independent, so logits and dLoss/dllr of a batch are bit for bit those of its
frames decoded one by one; a frame adds one term to each weight gradient, so the batch's is a sum
of the single-frame gradients in some order, which for B terms in FP32 is off by at most
(B - 1) 2^-24 times the sum of the magnitudes (and the reference sum here is in FP64)."""
import numpy as np
import pytest

from conftest import gpu_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 2, 5])
@pytest.mark.parametrize("N,B", [(16, 1), (16, 333), (128, 5), (128, 2100), (256, 700), (1024, 3), (1024, 310), (1024, 2100)])
def test_batch_is_the_sum_of_its_frames(pcbp, N, B, T):
    import torch

    dev = gpu_device()
    n = N.bit_length() - 1
    code = pcbp.pc_construct(N, N // 2)
    gen = torch.Generator(device=dev).manual_seed(N + B + T)
    llr = torch.randn((B, N), generator=gen, device=dev) * 2.0 + 1.0
    w = 0.9 + 0.1 * torch.randn((T, n, N // 2, 4), generator=gen, device=dev)
    glogits = torch.randn((B, code.K), generator=gen, device=dev)

    def both(rows, shift):
        """logits, dLoss/dw into a buffer `shift` floats past a 16-byte boundary, dLoss/dllr"""
        b = rows.stop - rows.start
        x = llr[rows].contiguous()
        logits = torch.empty((b, code.K), device=dev)
        ckpt = torch.empty(pcbp.wbp_ckpt_count(code, T, b), device=dev)
        ws = torch.empty(pcbp.wbp_workspace_size(code, T, b, 4), dtype=torch.uint8, device=dev)
        pcbp.wbp_forward(code, x, w, T, logits, ckpt, ws)
        gw = torch.zeros(w.numel() + 4, device=dev)[shift:shift + w.numel()].view(w.shape)
        gllr = torch.full_like(x, float("nan"))
        pcbp.wbp_backward(code, x, w, T, ckpt, glogits[rows].contiguous(), gw, gllr, ws)
        return logits, gw, gllr

    logits, gw, gllr = both(slice(0, B), 0)
    total = torch.zeros(w.shape, dtype=torch.float64, device=dev)
    size = torch.zeros_like(total)
    for f in range(0, B, 1 if B <= 400 else 8):
        rows = slice(f, min(B, f + (1 if B <= 400 else 8)))
        l1, w1, g1 = both(rows, 0)
        assert torch.equal(logits[rows], l1) and torch.equal(gllr[rows], g1), rows
        total += w1
        size += w1.abs()
    if B <= 400:                                     # else a row of `size` is a group of frames
        bound = B * 2.0 ** -24 * size
        assert bool(((gw.double() - total).abs() <= bound).all())
    # a gradient buffer on a 4-byte boundary takes scalar reductions
    l3, w3, g3 = both(slice(0, B), 1)
    assert torch.equal(l3, logits) and torch.equal(g3, gllr)
    if B <= 400:
        assert bool(((w3.double() - total).abs() <= bound).all())
    assert np.isfinite(gw.cpu().numpy()).all()
