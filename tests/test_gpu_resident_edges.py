"""Resident plates spread over more CTAs than they have modes: a CTA holds at most
eight stress modes, so a plate of more than 8 N of them has CTAs that own no
mode and receive no part of the force.  Every pass against the streaming kernel
(gradients digit for digit) and the FP64 oracle, with the FP32 path's
tolerances: 1e-5 relative L2 on audio and state, 1e-4 on gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle
from paper_2505_05940_gb300 import modal, workloads as W

from test_gpu_parity import GTOL, TOL, oracle_instance, rel, to_plan


def _plate(n, m, steps):
    """A plate whose stress modes all couple: random entries within the class
    pattern (the quadrature's H^k of so few modes are zero but for a handful)."""
    wl = W.tiny_random(100 + n, "plate", n, m, steps=steps)
    wl.instances[0].F0 = 200.0
    oi = oracle_instance(wl.instances[0], wl.fs, steps)
    fc = 2 * ((oi.labels[:, 0] + 1) % 2) + (oi.labels[:, 1] + 1) % 2
    pairs = np.unique(fc[:, None] ^ fc[None, :])
    kc = pairs[np.arange(m) % len(pairs)]
    R = np.random.default_rng([n, m]).standard_normal((m, n, n)) * np.abs(oi.H).max()
    R = (R + R.transpose(0, 2, 1)) * ((fc[:, None] ^ fc[None, :])[None] == kc[:, None, None])
    oi.H = R.astype(np.float32).astype(np.float64)
    return oi, wl.fs


@pytest.mark.parametrize("n,m,layout", [
    (1, 9, "classes"), (1, 16, "classes"), (1, 40, "classes"), (2, 33, "classes"), (3, 25, "dense"),
    (4, 40, "classes"), (4, 40, "dense"), (5, 120, "classes")])
def test_more_ctas_than_modes(n, m, layout):
    steps, K = 300, 128
    oi, fs = _plate(n, m, steps)
    assert m > 8 * n
    ybar = np.random.default_rng(n).normal(size=steps)
    yb = torch.tensor(ybar[None], dtype=torch.float32, device="cuda")
    grads = []
    for flags in (0, 16):          # 16: the streaming kernel
        sim = modal.Simulator([to_plan(oi, fs, layout)], debug_flags=flags)
        sim.plan.set_profiling(True)
        fwd = sim.simulate(steps, want_state=True, want_status=True)
        assert sim.plan.kernel_stats(6)[0] == (flags == 0)
        r = sim.simulate(steps, K=K)
        g = sim.grad(steps, yb, K, r["ckpt"], want_status=True)
        torch.cuda.synchronize()
        assert int(fwd["status"][0]) == 0 and int(g["status"][0]) == 0
        grads.append(g)
        if flags == 0:
            q = fwd["q_end"].cpu().numpy()
            audio = fwd["audio"][0].cpu().numpy()
    for k in grads[0]:
        assert torch.equal(grads[0][k], grads[1][k]), k
    ref = oracle.forward(oi, steps=steps)
    assert rel(audio, ref["y"]) <= TOL
    assert rel(q, ref["qN"]) <= TOL
    adj = oracle.adjoint(oi, ybar)
    dw2, dgm = oracle.coefficient_grads(oi, adj, 1.0 / fs)
    for name, want in (("d_omega2", dw2), ("d_gamma", dgm), ("d_b", adj["db"]), ("d_c", adj["dc"]),
                       ("d_q0", adj["dq0"]), ("d_qm1", adj["dqm1"])):
        e = rel(grads[0][name].cpu().numpy()[:len(want)], want)
        assert e <= GTOL, (name, e)
