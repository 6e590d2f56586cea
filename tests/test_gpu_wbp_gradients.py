"""dLoss/dw of FP32 weighted BP over batches of many frames a slot, among them the batches of N = 1024
that take a launch per iteration.  A frame adds one term to each weight's gradient, so the batch's is
the sum of the single-frame gradients in some order, off by at most (B - 1) 2^-24 times the sum of
their magnitudes; both sums are formed here in FP64 from the frames run one by one."""
import pytest

from conftest import gpu_device

pytestmark = pytest.mark.gpu


# frames per SM (N = 1024 holds one frame a CTA; 12 a slot is where the launches change)
@pytest.mark.parametrize("N,per_sm,T", [(64, 60, 2), (128, 40, 2), (256, 30, 3), (512, 25, 3), (1024, 11.9, 2),
                                        (1024, 12.1, 2), (1024, 12.1, 4), (1024, 15.3, 3)])
def test_weight_gradient_is_the_sum_over_frames(pcbp, N, per_sm, T):
    import torch

    dev = gpu_device()
    n = N.bit_length() - 1
    B = int(per_sm * torch.cuda.get_device_properties(dev).multi_processor_count)
    code = pcbp.pc_construct(N, N // 2)
    gen = torch.Generator(device=dev).manual_seed(N + B + T)
    llr = torch.randn((B, N), generator=gen, device=dev) * 2.0 + 1.0
    w = 0.9 + 0.1 * torch.randn((T, n, N // 2, 4), generator=gen, device=dev)
    glogits = torch.randn((B, code.K), generator=gen, device=dev)
    ws = torch.empty(pcbp.wbp_workspace_size(code, T, B, 4), dtype=torch.uint8, device=dev)
    ckpt = torch.empty(pcbp.wbp_ckpt_count(code, T, B), device=dev)
    logits = torch.empty((B, code.K), device=dev)

    def gradient(first, count, gw):
        rows = slice(first, first + count)
        x, g = llr[rows], glogits[rows]
        pcbp.wbp_forward(code, x, w, T, logits[:count], ckpt, ws)
        pcbp.wbp_backward(code, x, w, T, ckpt, g, gw, None, ws)
        return gw

    total = torch.zeros(w.shape, dtype=torch.float64, device=dev)
    size = torch.zeros_like(total)
    one = torch.empty_like(w)
    for f in range(B):
        gradient(f, 1, one.zero_())
        total += one
        size += one.abs()
    assert bool((size > 0).any(dim=(1, 2, 3)).all())          # every iteration has a gradient
    bound = B * 2.0 ** -24 * size
    # a gradient buffer on a 16-byte boundary takes vector reductions, one past it scalar ones
    for shift in (0, 1):
        gw = torch.zeros(w.numel() + 4, device=dev)[shift:shift + w.numel()].view(w.shape)
        gradient(0, B, gw)
        assert bool(((gw.double() - total).abs() <= bound).all()), shift
        gradient(0, B, gw)                                      # added to what the buffer holds
        assert bool(((gw.double() - 2 * total).abs() <= 4 * bound).all()), shift
