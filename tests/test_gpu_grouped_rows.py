"""Grouped plates at the sizes where the kernel's epilogue changes shape: the
states of a thread's rows in tensor memory (four blocks of tiles x plates
columns fit) and in shared memory (five tiles of 32 plates), class positions that
are no multiple of four, plates shorter than the group's, one plate alone.
Every plate against the per-instance FP32 path within the grouped path's
tolerance, 1e-5 relative L2."""
import copy

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2505_05940_gb300 import workloads as W

from test_gpu_grouped import _group, _plans, _run
from test_gpu_parity import TOL, rel


@pytest.mark.parametrize("sizes,plates", [
    (((488, 3), (401, 2), (129, 3)), 17),      # five tiles, 32 columns: shared memory
    (((488, 3), (401, 2), (129, 3)), 16),      # five tiles, 16 columns
    (((130, 5), (33, 4), (7, 2), (1, 1)), 32), (((41, 3),), 1)])
def test_epilogue_shapes(sizes, plates):
    fs, steps = 44100.0, 60
    base = W.tiny_random(300 + plates, "plate", *sizes[0], steps=steps).instances[0]
    base.F0 = 300.0
    insts = []
    for n, m in sizes:
        x = copy.deepcopy(base)
        x.n_phi, x.n_psi = n, m
        insts.append(x)
    dicts = _plans(_group(insts, fs, steps), fs, 1)
    plans = []
    for i in range(plates):
        d = dict(dicts[i % len(dicts)])
        d["kappa"] = np.asarray(d["kappa"]) * (0.5 + i / plates)
        plans.append(d)
    audio, qend, status, sim = _run(plans, steps)
    assert (status == 0).all(), status
    assert sim.plan.kernel_stats(5)[0] == 1
    alone = [{k: v for k, v in d.items() if k != "geom_group"} for d in plans]
    audio1, qend1, status1, _ = _run(alone, steps)
    assert (status1 == 0).all(), status1
    for i in range(plates):
        assert rel(qend[i], qend1[i]) <= TOL, i
        assert np.linalg.norm(audio[i] - audio1[i]) <= TOL * max(np.linalg.norm(audio1[i]), 1e-30) + 1e-7 * np.abs(
            np.asarray(plans[i]["c"]) * qend1[i]).sum(), i
