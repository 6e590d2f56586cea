"""The messages that bp_decode_posterior returns, by kernel: scaled min-sum runs the register-resident
kernel (bp_decode's) unless PCBP_DECODER keeps to an older one, and both kernels evaluate the same
operations in the same order, so L(n+1), R(1) and the outputs are equal bit for bit, on events that
begin and end at every stage and on frames that stop at any iteration."""
import numpy as np
import pytest

from conftest import gpu_device
from test_gpu_parity import POLY24, POLY8, assert_bitwise_equal, frames
from test_gpu_posterior import gpu_posterior

pytestmark = pytest.mark.gpu

SCHEDS = {
    "any-range": dict(mode=1, P_range=99, P_level=99, N_min=1, T0=1, stop_kind=0),
    "any-range-crc": dict(mode=1, P_range=99, P_level=99, N_min=2, T0=2, stop_kind=1),
    "fp-crc": dict(mode=2, it_reset_full=2, q_max=0, stop_kind=1, stop_from=3),
    "plain-crc": dict(mode=0, stop_kind=1),
    "boxplus": dict(mode=1, P_range=99, P_level=99, N_min=1, T0=1, stop_kind=1, fkind=1, alpha=1.0),
}


@pytest.mark.parametrize("sched", SCHEDS, ids=str)
@pytest.mark.parametrize("N", [128, 256, 512, 1024, 2048])
def test_messages_are_the_same_in_every_kernel(pcbp, oracle, monkeypatch, N, sched):
    import torch

    n = N.bit_length() - 1
    r, poly = (8, POLY8) if N <= 256 else (24, POLY24)
    K, B = N // 2, 400
    _, _, _, llr = frames(oracle, N, K, r, poly, B, 2.5, seed=N + 7)
    kw = {k: {"P_range": n, "P_level": n - 1}[k] if v == 99 else v for k, v in SCHEDS[sched].items()}
    s = pcbp.sched(seed=N, frame_base=5, **kw)
    code = pcbp.pc_construct(N, K, r, poly)
    for max_iters in (1, 2, 7, 16):
        got = {}
        for env in ("", "tmem", "grouped"):
            monkeypatch.setenv("PCBP_DECODER", env)
            got[env] = gpu_posterior(pcbp, code, llr, s, max_iters)
        for env in ("tmem", "grouped"):
            for a, b in zip(got[""][:3], got[env][:3]):
                assert np.array_equal(a, b), (env, max_iters)
            assert_bitwise_equal(got[""][3], got[env][3], f"messages, {env}, {max_iters} iterations")
        monkeypatch.setenv("PCBP_DECODER", "")
        dec = pcbp.Decoder(code, s, max_iters, gpu_device())
        bits, iters, ok = dec(torch.from_numpy(llr).to(gpu_device()))
        assert np.array_equal(pcbp.unpack_bits(bits, K).cpu().numpy(), got[""][0])
        assert np.array_equal(iters.cpu().numpy(), got[""][1]) and np.array_equal(ok.cpu().numpy(), got[""][2])
