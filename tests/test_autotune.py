"""The tile autotuner leaves plans alone whose passes run on the resident kernel:
they have no stages, so nothing is timed and no stage size picked by chance is set
or handed on to a streaming plan of the same shapes."""
import json

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_05940_gb300 import autotune


class _Plan:
    """Records what the tuner does; the 80 KB stage is the fastest."""

    def __init__(self, resident):
        self.is_resident, self.stage, self.configured = resident, 65536, []

    def resident(self):
        return dict(forward=self.is_resident, checkpointed=self.is_resident)

    def configure(self, stage_bytes=0, ring_stages=0):
        self.configured.append(stage_bytes)
        self.stage = stage_bytes

    def tiles(self):
        return dict(stage_bytes=self.stage)

    def set_profiling(self, enable=True):
        pass

    def reset_stats(self):
        pass

    def kernel_stats(self, which):
        return 2, 1.0 if self.stage == 80 * 1024 else 2.0, 0.0


class _Sim:
    device = "cuda:0"

    def __init__(self, resident):
        self.plan, self.runs = _Plan(resident), 0
        self.prepared = [dict(kind="plate", omega2=np.ones(96), H=np.zeros((24, 1, 1)))]

    def simulate(self, steps, K=None):
        self.runs += 1


@pytest.fixture
def tune(tmp_path, monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d=None: "device")
    monkeypatch.setattr(torch.cuda, "synchronize", lambda: None)
    path = tmp_path / "tune.json"
    return lambda sim, **kw: (autotune.tune(sim, cache_path=str(path), **kw),
                              json.loads(path.read_text()))


@pytest.mark.parametrize("force", [False, True])
def test_resident_plans_are_left_alone(tune, force):
    sim = _Sim(True)
    res, _ = tune(sim, force=force)
    assert sim.runs == 0 and sim.plan.configured == []
    assert res["stage_bytes"] == 65536 and not res["cached"] and res["us_per_step"] is None
    again, _ = tune(sim)
    assert again["cached"] and again["stage_bytes"] == 65536 and sim.plan.configured == []


def test_entries_of_the_other_kind_do_not_count(tune):
    tune(_Sim(True))
    streaming = _Sim(False)
    res, cache = tune(streaming)
    assert not res["cached"] and res["stage_bytes"] == 80 * 1024 == streaming.plan.stage
    assert list(cache.values())[0]["stage_bytes"] == 80 * 1024
    fresh = _Sim(False)
    assert tune(fresh)[0]["cached"] and fresh.plan.stage == 80 * 1024
    resident = _Sim(True)
    assert not tune(resident)[0]["cached"] and resident.plan.configured == []


@pytest.mark.gpu
def test_plan_says_which_kernel_takes_it():
    if not torch.cuda.is_available():  # pragma: no cover
        pytest.skip("needs a CUDA device")
    from paper_2505_05940_gb300 import modal, workloads as W
    from test_gpu_parity import oracle_instance, to_plan
    wl = W.tiny_random(1, "plate", 40, 10, steps=64)
    dense = W.tiny_random(2, "plate", 48, 6, steps=64)
    p = to_plan(oracle_instance(wl.instances[0], wl.fs, 64), wl.fs)
    q = to_plan(oracle_instance(dense.instances[0], wl.fs, 64), wl.fs, "dense")
    for plan, flags, want in ((p, 0, (True, True)), (p, 16, (False, False)), (q, 0, (True, False))):
        r = modal.Simulator([plan], debug_flags=flags).plan.resident()
        assert (r["forward"], r["checkpointed"]) == want
