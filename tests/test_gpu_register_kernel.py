"""The register-resident decoder kernel (bp_decode's, below every other choice) against the
shared-memory stage-grouped kernel (PCBP_DECODER=grouped): every length it is built for, batches
of one frame, of fewer frames than SMs, and of several frames per slot, and schedules whose
events begin and end at every stage and cover subgraphs of every size.  Scaled min-sum and exact
box-plus evaluate the same operations in the same order in both kernels, so bits, iteration
counts and CRC flags are equal."""
import numpy as np
import pytest

from paper_1911_08868_gb300 import inputs

from conftest import gpu_device

pytestmark = pytest.mark.gpu

SCHEDS = {
    "plain": (dict(mode=0, stop_kind=1), 20),
    "no-iterations": (dict(mode=0, stop_kind=1), 0),
    "no-stop": (dict(mode=0, stop_kind=0), 3),
    "any-range": (dict(mode=1, P_range=99, P_level=99, N_min=1, T0=1, stop_kind=1, stop_from=3), 45),
    "any-range-crc-g": (dict(mode=1, P_range=99, P_level=99, N_min=2, D=3, T0=1, stop_kind=3), 40),
    "small-range-g": (dict(mode=1, P_range=2, P_level=99, N_min=1, T0=2, stop_kind=2), 30),
    "fp": (dict(mode=2, it_reset_full=3, q_max=6, stop_kind=1, alpha=1.0), 40),
    "fp-unlimited-crc-g": (dict(mode=2, it_reset_full=2, q_max=0, stop_kind=3), 20),
    "boxplus": (dict(mode=1, P_range=99, P_level=99, N_min=1, T0=1, stop_kind=1, fkind=1), 20),
}


@pytest.mark.parametrize("sched", SCHEDS, ids=str)
@pytest.mark.parametrize("N", [8, 16, 32, 64, 128, 256, 512, 1024, 2048])
def test_register_kernel_equals_grouped_kernel(pcbp, monkeypatch, N, sched):
    import torch

    dev = gpu_device()
    n = N.bit_length() - 1
    kw, max_iters = SCHEDS[sched]
    kw = {k: {"P_range": n, "P_level": n - 1}[k] if v == 99 else v for k, v in kw.items()}
    codes = [(N // 2, 8, 0x9B) if N > 16 else (N // 2, 0, 0), (N - 1, 0, 0), (N // 4 + 1, 0, 0)]
    if N >= 64:
        codes.append((N // 2 + 3, 24, 0x1B2B117))
    for K, r, poly in codes:
        code = pcbp.pc_construct(N, K, r, poly)
        for B in (1, 37, 2500):
            gen = torch.Generator(device=dev).manual_seed(N + B)
            x = torch.empty((B, N), dtype=torch.uint8, device=dev)
            pcbp.pc_encode(code, inputs.payload_torch(gen, B, K - r, dev), x)
            llr = inputs.bpsk_awgn_llr_torch(x, gen, inputs.sigma2_of(1.5, K, r, N)).contiguous()
            if B > 1:                       # ties and zeros of either sign
                llr[::3] = torch.round(llr[::3])
                llr[5] = 0.0
                llr[6] = -0.0
            s = pcbp.sched(**{"seed": N + B, "frame_base": 17, **kw})
            out = []
            for env in ("", "grouped"):
                monkeypatch.setenv("PCBP_DECODER", env)
                dec = pcbp.Decoder(code, s, max_iters, dev)
                out.append([t.cpu().numpy() for t in dec(llr)])
            for a, b in zip(*out):
                assert np.array_equal(a, b), (K, r, B)


@pytest.mark.parametrize("N,slots", [(64, 24), (256, 16), (512, 8), (2048, 2)])
def test_batches_around_one_frame_per_slot(pcbp, monkeypatch, N, slots):
    """A batch with a slot for every frame runs without a frame counter (whatever the workspace
    holds), one frame more with it."""
    import torch

    dev = gpu_device()
    full = slots * torch.cuda.get_device_properties(dev).multi_processor_count
    code = pcbp.pc_construct(N, N // 2, 8, 0x9B)
    gen = torch.Generator(device=dev).manual_seed(N)
    llr = torch.randn((full + 1, N), generator=gen, device=dev) * 3.0 + 2.0
    s = pcbp.sched(mode=0, stop_kind=1, stop_from=1)
    monkeypatch.setenv("PCBP_DECODER", "grouped")
    want = [t.cpu().numpy() for t in pcbp.Decoder(code, s, 8, dev)(llr)]
    monkeypatch.setenv("PCBP_DECODER", "")
    for B in (full - 1, full, full + 1):
        dec = pcbp.Decoder(code, s, 8, dev)
        dec.workspace.fill_(0x5A)
        for a, b in zip(dec(llr[:B]), want):
            assert np.array_equal(a.cpu().numpy(), b[:B]), B
