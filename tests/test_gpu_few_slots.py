"""Batches of a mixed sweep that ask for few frames per CTA below N = 128, where an SM then holds several
CTAs of the register-resident kernel: the outputs are those of bp_decode, alone and beside batches of
long codes, whose CTAs take the whole of an SM's tensor memory."""
import pytest

from conftest import gpu_device

pytestmark = pytest.mark.gpu


def batch(pcbp, dev, N, B, slots, fkind=0, mode=1):
    import torch

    n = N.bit_length() - 1
    code = pcbp.pc_construct(N, N // 2)
    gen = torch.Generator(device=dev).manual_seed(N + B)
    llr = torch.randn((B, N), generator=gen, device=dev) * 1.5 + 0.5
    kw = dict(P_range=n, P_level=n - 1, N_min=2, T0=2) if mode == 1 else dict(it_reset_full=2, q_max=0)
    s = pcbp.sched(mode=mode, stop_kind=2, fkind=fkind, seed=N, frame_base=3, **kw)
    return (code, s, 25, llr, slots)


def same_as_bp_decode(pcbp, dev, parts):
    import torch

    got = [[t.clone() for t in ts] for ts in pcbp.MixedDecoder(parts, dev)()]
    for i, (code, s, it, llr, _) in enumerate(parts):
        want = pcbp.Decoder(code, s, it, dev)(llr)
        for w, g in zip(want, got):
            assert torch.equal(w, g[i]), (code.N, i)


@pytest.mark.parametrize("slots", [1, 2, 3, 5, 8, 12, 13, 23])
@pytest.mark.parametrize("N", [8, 16, 32, 64])
def test_outputs(pcbp, N, slots):
    import torch

    dev = gpu_device()
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    for B in (1, sms * slots - 1, sms * slots + 1, 30 * sms * slots + 7):
        for fkind, mode in ((0, 1), (1, 2)):
            same_as_bp_decode(pcbp, dev, [batch(pcbp, dev, N, B, slots, fkind, mode)])


def test_beside_long_codes(pcbp):
    dev = gpu_device()
    sizes = [(64, 9000, 1), (1024, 900, 0), (16, 9000, 1), (8, 9001, 2), (2048, 400, 0), (32, 9000, 3), (256, 3000, 1),
             (64, 700, 2), (512, 1500, 0), (8, 20000, 1)]
    same_as_bp_decode(pcbp, dev, [batch(pcbp, dev, *x) for x in sizes])
    same_as_bp_decode(pcbp, dev, [batch(pcbp, dev, *x) for x in sizes[::-1]])
