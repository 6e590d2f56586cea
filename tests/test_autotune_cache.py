"""The autotuner's cache on the CPU (device calls replaced): a shape tuned with PCBP_DECODER set to one
kernel is not taken in a process that decodes with another."""
import pytest
import torch

from paper_1911_08868_gb300 import autotune


@pytest.fixture
def tuner(pcbp, monkeypatch, tmp_path):
    """tune(env) -> (result, shapes timed), on a clock by which more slots are faster."""
    timed = []

    class Mixed:
        def __init__(self, parts, dev):
            timed.append(parts[0][4:6])

        def __call__(self):
            pass

    class Event:
        def __init__(self, enable_timing):
            pass

        def record(self):
            pass

        def elapsed_time(self, other):
            return 1.0 / timed[-1][0]

    monkeypatch.setenv("PCBP_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda dev: "device")
    monkeypatch.setattr(torch.cuda, "synchronize", lambda: None)
    monkeypatch.setattr(torch.cuda, "Event", Event)
    monkeypatch.setattr(pcbp, "MixedDecoder", Mixed)
    monkeypatch.setattr(pcbp, "bp_slot_limit", lambda code, tpf, fkind: 2 if autotune.os.environ.get("PCBP_DECODER") == "grouped" else 16)
    monkeypatch.setattr(autotune, "_synthetic", lambda pcbp, inputs, dev, N, K, r, poly, *a, **k: (pcbp.pc_construct(N, K, r, poly), None))

    def tune(env):
        if env is None:
            monkeypatch.delenv("PCBP_DECODER", raising=False)
        else:
            monkeypatch.setenv("PCBP_DECODER", env)
        timed.clear()
        got = autotune.tune_launch([256], lambda n: pcbp.sched(mode=0))
        return got[256], len(timed)

    return tune


def test_a_shape_belongs_to_the_kernel_it_was_tuned_with(tuner):
    grouped, count = tuner("grouped")
    assert grouped["slots"] == 2 and count > 0
    assert tuner("grouped") == (grouped, 0)             # from the cache
    best, count = tuner(None)
    assert best["slots"] == 16 and count > 0            # tuned afresh
    assert tuner(None) == (best, 0)
    assert tuner("")[1] == 0                            # the same choice
    assert tuner("tmem")[1] > 0
    assert tuner("grouped") == (grouped, 0)
