"""N = 8, 16 and 32 in the register-resident kernel, where a frame has fewer threads than a warp has
lanes and several lanes stand for each thread: hundreds of switches per frame, so a label map that
one of them read after another had replaced it would move messages to wrong places.  Outputs equal
those of the shared-memory kernel, which has one lane a thread."""
import numpy as np
import pytest

from conftest import gpu_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fkind", [0, 1])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("N", [8, 16, 32])
def test_many_switches(pcbp, monkeypatch, N, mode, fkind):
    import torch

    dev = gpu_device()
    n = N.bit_length() - 1
    code = pcbp.pc_construct(N, N // 2)
    gen = torch.Generator(device=dev).manual_seed(N)
    llr = torch.randn((4000, N), generator=gen, device=dev) * 1.5
    kw = dict(mode=1, P_range=n, P_level=n - 1, N_min=1, T0=1) if mode == 1 else dict(mode=2, it_reset_full=1, q_max=0)
    for iters in (301, 302):
        s = pcbp.sched(stop_kind=0, fkind=fkind, seed=N, **kw)
        out = []
        for env in ("", "grouped"):
            monkeypatch.setenv("PCBP_DECODER", env)
            out.append([t.cpu().numpy() for t in pcbp.Decoder(code, s, iters, dev)(llr)])
        for a, b in zip(*out):
            assert np.array_equal(a, b)
