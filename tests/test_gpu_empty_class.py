"""Plates whose modes leave a symmetry class empty (three modes or so, or a narrow
plate before its first doubly odd mode): a stress mode that couples the empty
class to another has no rows there, so u^k = H^k q is zero on the other's columns.
The streaming plate kernel, alone and split, and the default path against the FP64
oracle, with the FP32 path's tolerances: 1e-5 relative L2 on audio and state,
1e-4 on gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle
from paper_2505_05940_gb300 import modal, workloads as W

from test_gpu_parity import GTOL, TOL, oracle_instance, rel, to_plan


def _plate(classes, m, steps):
    """A plate with the given number of modes per class; every stress class that
    joins two of them has modes, with random entries within the class pattern."""
    n = sum(classes)
    wl = W.tiny_random(400 + n, "plate", n, m, steps=steps)
    wl.instances[0].F0 = 200.0
    oi = oracle_instance(wl.instances[0], wl.fs, steps)
    fc = np.repeat(np.arange(4), classes)[np.random.default_rng(n).permutation(n)]
    pairs = np.unique(fc[:, None] ^ fc[None, :])
    kc = pairs[np.arange(m) % len(pairs)]
    R = np.random.default_rng([n, m]).standard_normal((m, n, n)) * np.abs(oi.H).max()
    R = (R + R.transpose(0, 2, 1)) * ((fc[:, None] ^ fc[None, :])[None] == kc[:, None, None])
    oi.H = R.astype(np.float32).astype(np.float64)
    d = to_plan(oi, wl.fs, "dense")
    d["phi_class"], d["psi_class"] = fc.astype(np.int32), kc.astype(np.int32)
    return oi, d, wl.fs


@pytest.mark.parametrize("classes", [(1, 1, 1, 0), (2, 0, 1, 1), (9, 1, 0, 5), (0, 12, 20, 3), (7, 0, 0, 6)])
@pytest.mark.parametrize("opts", [dict(debug_flags=16), dict(force_split=2), dict()])
def test_empty_class(classes, opts):
    steps, K, m = 300, 128, 8
    oi, d, fs = _plate(classes, m, steps)
    sim = modal.Simulator([d], **opts)
    r = sim.simulate(steps, want_state=True, want_status=True)
    ref = oracle.forward(oi, steps=steps)
    torch.cuda.synchronize()
    assert int(r["status"][0]) == 0
    assert rel(r["audio"][0].cpu().numpy(), ref["y"]) <= TOL
    assert rel(r["q_end"].cpu().numpy(), ref["qN"]) <= TOL
    ybar = np.random.default_rng(7).normal(size=steps)
    yb = torch.tensor(ybar[None], dtype=torch.float32, device="cuda")
    c = sim.simulate(steps, K=K)
    g = sim.grad(steps, yb, K, c["ckpt"], want_status=True)
    torch.cuda.synchronize()
    assert int(g["status"][0]) == 0
    adj = oracle.adjoint(oi, ybar)
    dw2, dgm = oracle.coefficient_grads(oi, adj, 1.0 / fs)
    for name, want in (("d_omega2", dw2), ("d_gamma", dgm), ("d_b", adj["db"]), ("d_c", adj["dc"]),
                       ("d_q0", adj["dq0"]), ("d_qm1", adj["dqm1"]), ("d_kappa", adj["dkappa"])):
        e = rel(g[name].cpu().numpy()[:len(want)], want)
        assert e <= GTOL, (name, e)
