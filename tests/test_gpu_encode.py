"""pc_encode against the oracle's encoder: every length, payload rows of odd lengths (each row then
starts at another alignment), CRCs of 0 to 32 bits, batches around the kernel's tile of 8 warps x
(32 * 32 / N) frames, and buffers that start off a 16-byte boundary."""
import numpy as np
import pytest

from paper_1911_08868_gb300 import inputs

from conftest import gpu_device

pytestmark = pytest.mark.gpu

CRCS = [(0, 0), (1, 0x3), (8, 0x9B), (24, 0x1B2B117), (32, 0x104C11DB7)]


@pytest.mark.parametrize("N", [8, 16, 32, 64, 128, 256, 512, 1024, 2048])
def test_encode_equals_oracle(pcbp, oracle, N):
    import torch

    dev = gpu_device()
    tile = max(8, 8 * 1024 // N) if N >= 32 else 256
    for K in sorted({1, N // 4 + 1, N // 2, N - 1, N}):
        _, fr = oracle.construct(N, K)
        for r, poly in CRCS:
            if r >= K:
                continue
            code = pcbp.pc_construct(N, K, r, poly)
            for B, off in ((1, 0), (tile - 1, 3), (tile + 1, 0), (2 * tile + 5, 13)):
                pay = inputs.payload_numpy(N + K + B, B, K - r) | np.uint8(0x54)   # only bit 0 counts
                store = torch.full((off + B * (K - r) + 64,), 255, dtype=torch.uint8, device=dev)
                d_pay = store[off:off + B * (K - r)].view(B, K - r)
                d_pay.copy_(torch.from_numpy(pay))
                out = torch.full((off + B * N + 64,), 7, dtype=torch.uint8, device=dev)
                d_x = out[off:off + B * N].view(B, N)
                pcbp.pc_encode(code, d_pay, d_x)
                torch.cuda.synchronize()
                want = oracle.encode_frames(np.ascontiguousarray(pay & 1), fr, r, poly)
                assert np.array_equal(d_x.cpu().numpy(), want), (K, r, B, off)
                rest = torch.cat((out[:off], out[off + B * N:]))
                assert bool((rest == 7).all()), (K, r, B, off)
