"""The status word of a bounds-checked library (PCBP_CHECKED=1): every decode clears it, whatever
the workspace held and however few frames the batch has; such a library decodes with the kernels of
a normal one, and those that its default choice leaves out are checked as well."""
import numpy as np
import pytest

from conftest import gpu_device
from test_gpu_checked import EXTRA, status_of
from test_gpu_parity import DECODE_CASES, KERNEL_CASES, POLY8, POLY24, frames

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


@pytest.mark.parametrize("N,slots", [(64, 24), (128, 24), (256, 16), (512, 8), (1024, 4), (2048, 2)])
def test_min_sum_runs_the_register_resident_kernel(pcbp, monkeypatch, N, slots):
    """On a checked build too: the frames a CTA holds are that kernel's."""
    monkeypatch.delenv("PCBP_DECODER", raising=False)
    assert pcbp.bp_slot_limit(pcbp.pc_construct(N, N // 2), 0, 0) == slots


SHORT = [
    (8, 4, 0, 0, 1.5, dict(mode=1, P_range=3, P_level=2, N_min=1, T0=1), 40, 300),
    (16, 8, 0, 0, 1.5, dict(mode=2, it_reset_full=2, q_max=0, stop_kind=3), 30, 300),
    (32, 16, 0, 0, 1.5, dict(mode=1, P_range=5, P_level=4, N_min=1, T0=1, fkind=1), 40, 6000),
    (64, 40, 8, POLY8, 1.5, dict(mode=1, P_range=6, P_level=5, N_min=1, T0=1, stop_kind=2), 40, 6000),
    (2048, 2048, 24, POLY24, 6.0, dict(mode=1, P_range=11, P_level=10, N_min=1, T0=1, stop_kind=3), 20, 400),
]
TMEM = [c for c in DECODE_CASES + KERNEL_CASES + EXTRA if c[0] >= 128]


@pytest.mark.parametrize("decoder,case", [("", c) for c in SHORT] + [("tmem", c) for c in TMEM],
                         ids=lambda v: v if isinstance(v, str) else f"N{v[0]}-mode{v[5]['mode']}-s{v[5].get('stop_kind', 1)}")
def test_no_access_out_of_range(pcbp, oracle, monkeypatch, decoder, case):
    """Lengths below 64, every position an information bit, and the tensor-memory kernel for scaled min-sum."""
    import torch

    if not pcbp.build_checked():
        pytest.skip("not a bounds-checked build (PCBP_CHECKED=1)")
    dev = gpu_device()
    monkeypatch.setenv("PCBP_DECODER", decoder)
    N, K, r, poly, ebn0, kw, max_iters, B = case
    _, _, _, llr = frames(oracle, N, K, r, poly, B, ebn0, seed=N * 3 + kw["mode"])
    s = pcbp.sched(**{"seed": 41, "stop_kind": 1, **kw})
    dec = pcbp.Decoder(pcbp.pc_construct(N, K, r, poly), s, max_iters, dev)
    dec(torch.from_numpy(np.ascontiguousarray(llr)).to(dev))
    torch.cuda.synchronize()
    assert status_of(dec) == 0, f"out-of-range access classes {status_of(dec):#x}"
