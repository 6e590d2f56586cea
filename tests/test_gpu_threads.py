"""Host threads that call the library at the same time, each with its own stream and buffers: a
launch depends on nothing that another thread's launch of the same kernel sets (a batch of few
frames takes less shared memory than one that fills the slots)."""
import ctypes as C
import threading

import pytest

from conftest import gpu_device

pytestmark = pytest.mark.gpu

CALLS = 6000


def run_threads(calls):
    """Each call (a closure returning a status) CALLS times in its own thread; the statuses seen."""
    seen, start = set(), threading.Barrier(len(calls))

    def loop(call):
        start.wait()
        for _ in range(CALLS):
            seen.add(call())

    threads = [threading.Thread(target=loop, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return seen


def streams(dev, count):
    import torch

    torch.cuda.synchronize()
    return [torch.cuda.Stream(dev) for _ in range(count)]


@pytest.mark.parametrize("N", [1024, 2048])
def test_decoding_batches_of_different_sizes(pcbp, N):
    import torch

    dev = gpu_device()
    code = pcbp.pc_construct(N, N // 2, 24, 0x1B2B117)
    s = pcbp.sched(mode=0, stop_kind=1)
    full = pcbp.bp_slot_limit(code) * torch.cuda.get_device_properties(dev).multi_processor_count
    sizes = (1, full, 1, full)
    decs = [pcbp.Decoder(code, s, 1, dev) for _ in sizes]
    llrs = [torch.randn((B, N), device=dev) * 2.0 + 3.0 for B in sizes]
    sts = streams(dev, len(sizes))
    for d, x in zip(decs, llrs):
        d(x)                                    # makes the outputs
    lib, calls = pcbp._lib, []
    for d, x, st in zip(decs, llrs, sts):
        args = (C.byref(code), x.data_ptr(), C.byref(s), 1, x.shape[0], d.bits.data_ptr(), d.iters.data_ptr(),
                d.crc_ok.data_ptr(), d.workspace.data_ptr(), st.cuda_stream)
        calls.append(lambda a=args: lib.bp_decode(*a))
    assert run_threads(calls) == {pcbp.PC_OK}
    torch.cuda.synchronize()


def test_weighted_bp_batches_of_different_sizes(pcbp):
    import torch

    dev = gpu_device()
    N, T = 256, 1
    code = pcbp.pc_construct(N, N // 2)
    w = torch.ones((T, 8, N // 2, 4), device=dev)
    lib, calls, keep = pcbp._lib, [], []
    sizes = (1, 2000, 1, 2000)
    for B, st in zip(sizes, streams(dev, len(sizes))):
        x, out = torch.randn((B, N), device=dev), torch.empty((B, code.K), device=dev)
        ws = torch.empty(pcbp.wbp_workspace_size(code, T, B, 4), dtype=torch.uint8, device=dev)
        keep.append((x, out, ws, st))
        args = (C.byref(code), x.data_ptr(), w.data_ptr(), T, B, out.data_ptr(), None, ws.data_ptr(), st.cuda_stream)
        calls.append(lambda a=args: lib.wbp_forward(*a))
    torch.cuda.synchronize()
    assert run_threads(calls) == {pcbp.PC_OK}
    torch.cuda.synchronize()
