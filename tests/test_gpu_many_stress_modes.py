"""Small plates with more than 128 stress modes: the forward pass runs with the
coupling rows on the SMs (launch class 6) at every number of warps a CTA takes,
and one beyond it streams.  Audio and state against the FP64 oracle, 1e-5 relative
L2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle
from paper_2505_05940_gb300 import modal, workloads as W

from test_gpu_parity import TOL, oracle_instance, rel, to_plan


def _plate(n, m, steps):
    """Random entries within the class pattern of every stress mode."""
    wl = W.tiny_random(100 + n, "plate", n, 8, steps=steps)
    wl.instances[0].F0 = 200.0
    oi = oracle_instance(wl.instances[0], wl.fs, steps)
    fc = 2 * ((oi.labels[:, 0] + 1) % 2) + (oi.labels[:, 1] + 1) % 2
    pairs = np.unique(fc[:, None] ^ fc[None, :])
    kc = pairs[np.arange(m) % len(pairs)]
    R = np.random.default_rng([n, m]).standard_normal((m, n, n)) * np.abs(oi.H).max() / np.sqrt(m / 8)
    R = (R + R.transpose(0, 2, 1)) * ((fc[:, None] ^ fc[None, :])[None] == kc[:, None, None])
    oi.H = R.astype(np.float32).astype(np.float64)
    oi.M, oi.kappa = m, np.resize(oi.kappa, m)
    return oi, wl.fs


@pytest.mark.parametrize("sizes,resident", [
    (((32, 129),), True), (((30, 200),), True), (((5, 256),), True), (((1, 144),), True),
    (((24, 160), (20, 4), (32, 240)), True), (((30, 257),), False), (((33, 160),), False),
    (((32, 200), (40, 10)), False)])
def test_many_stress_modes(sizes, resident):
    steps = 300
    cases = [_plate(n, m, steps) for n, m in sizes]
    sim = modal.Simulator([to_plan(oi, fs) for oi, fs in cases])
    sim.plan.set_profiling(True)
    r = sim.simulate(steps, want_state=True, want_status=True)
    torch.cuda.synchronize()
    assert sim.plan.kernel_stats(6)[0] == resident == sim.plan.resident()["forward"]
    assert (r["status"].cpu().numpy() == 0).all()
    q = r["q_end"].cpu().numpy()
    for i, (oi, _) in enumerate(cases):
        ref = oracle.forward(oi, steps=steps)
        a = sim.plan.mode_offset[i]
        assert rel(r["audio"][i].cpu().numpy(), ref["y"]) <= TOL, i
        assert rel(q[a:a + oi.N], ref["qN"]) <= TOL, i
