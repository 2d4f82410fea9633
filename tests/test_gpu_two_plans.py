"""Two plans at work on two streams: grouped plates (whose CTAs take the whole
tensor memory of an SM and wait for one another) beside resident plates (whose
clusters hold a part of it through their time loop).  Neither may wait for the
other's columns: both report success and give the bits they give alone."""
import copy

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2505_05940_gb300 import modal, workloads as W

from test_gpu_grouped import _group, _plans
from test_gpu_parity import oracle_instance, to_plan


def _grouped(fs, steps, sizes, plates):
    base = W.tiny_random(310, "plate", *sizes[0], steps=steps).instances[0]
    base.F0 = 300.0
    insts = []
    for n, m in sizes:
        x = copy.deepcopy(base)
        x.n_phi, x.n_psi = n, m
        insts.append(x)
    dicts = _plans(_group(insts, fs, steps), fs, 1)
    out = []
    for i in range(plates):
        d = dict(dicts[i % len(dicts)])
        d["kappa"] = np.asarray(d["kappa"]) * (0.5 + i / plates)
        out.append(d)
    return out


def _resident(fs, steps, n, m, plates):
    wl = W.tiny_random(100 + n, "plate", n, m, steps=steps)
    wl.instances[0].F0 = 200.0
    oi = oracle_instance(wl.instances[0], fs, steps)
    return [dict(to_plan(oi, fs), kappa=oi.kappa * (0.5 + i / plates)) for i in range(plates)]


@pytest.mark.parametrize("n,m,plates", [(20, 12, 120), (100, 30, 16)])
def test_grouped_and_resident_plates_together(n, m, plates):
    fs, steps = 44100.0, 800
    sims = [modal.Simulator(_grouped(fs, steps, ((40, 8), (24, 4)), 16)),
            modal.Simulator(_resident(fs, steps, n, m, plates))]
    alone = [s.simulate(steps)["audio"].clone() for s in sims]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for order in ((0, 1), (1, 0)):
        got = {}
        for i in order * 3:
            with torch.cuda.stream(streams[i]):
                got.setdefault(i, []).append(sims[i].simulate(steps, want_status=True))
        torch.cuda.synchronize()
        for i in order:
            for r in got[i]:
                assert (r["status"].cpu().numpy() == 0).all(), (i, r["status"])
                assert torch.equal(r["audio"], alone[i]), i
