"""Every way to choose a decoder kernel gives the outputs of the others: PCBP_DECODER unset (for
scaled min-sum the register-resident kernel, for exact box-plus from N = 128 on the tensor-memory
kernel), =tmem (the tensor-memory kernel for either f) and =grouped (the shared-memory kernel)."""
import numpy as np
import pytest

from conftest import gpu_device
from test_gpu_checked import EXTRA
from test_gpu_parity import KERNEL_CASES, frames, gpu_decode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", KERNEL_CASES + EXTRA,
                         ids=lambda c: f"N{c[0]}-mode{c[5]['mode']}-f{c[5].get('fkind', 0)}-s{c[5].get('stop_kind', 1)}")
def test_every_choice_gives_the_same_outputs(pcbp, oracle, monkeypatch, case):
    N, K, r, poly, ebn0, kw, max_iters, B = case
    _, _, _, llr = frames(oracle, N, K, r, poly, B, ebn0, seed=N * 17 + kw["mode"])
    s = pcbp.sched(**{"seed": 555, "stop_kind": 1, **kw})
    code = pcbp.pc_construct(N, K, r, poly)
    out = {}
    for env in (None, "tmem", "grouped"):
        if env is None:
            monkeypatch.delenv("PCBP_DECODER", raising=False)
        else:
            monkeypatch.setenv("PCBP_DECODER", env)
        out[env] = gpu_decode(pcbp, code, llr, s, max_iters)[:3]
    for env in ("tmem", "grouped"):
        for a, b in zip(out[None], out[env]):
            assert np.array_equal(a, b), env


@pytest.mark.parametrize("N", [32, 64, 128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("fkind", [0, 1])
def test_slot_limit_without_a_thread_count(pcbp, N, fkind):
    """threads_per_frame 0: the limit of the kernel bp_decode runs, which a batch asking for more is
    clamped to."""
    import torch

    dev = gpu_device()
    n = N.bit_length() - 1
    code = pcbp.pc_construct(N, N // 2, 8, 0x9B)
    s = pcbp.sched(mode=1, P_range=n, P_level=n - 1, N_min=2, T0=2, stop_kind=1, fkind=fkind, seed=N)
    lim = pcbp.bp_slot_limit(code, 0, fkind)
    B = 2 * lim * torch.cuda.get_device_properties(dev).multi_processor_count + 5
    gen = torch.Generator(device=dev).manual_seed(N)
    llr = torch.randn((B, N), generator=gen, device=dev) * 2.0 + 1.0
    outs = []
    for slots in (0, 1, lim, lim + 5):
        md = pcbp.MixedDecoder([(code, s, 12, llr, slots, 0)], dev)
        outs.append([t[0].clone() for t in md()])
    for other in outs[1:]:
        for a, b in zip(outs[0], other):
            assert torch.equal(a, b)
    with pytest.raises(pcbp.PcError) as e:
        pcbp.bp_slot_limit(code, 96, fkind)
    assert e.value.status == pcbp.PC_EUNSUPPORTED
