"""Resident plates (coupling rows in tensor and shared memory, one warp per
stress mode, plates spread over the CTAs of a cluster) against the FP64 oracle
at the sizes where the kernel changes shape: row lengths on both sides of every
variant (16, 24, 32, 40, 48, 56, 64 columns), one mode, one stress mode, more
modes than threads, dense rows over several lanes' rows, checkpoints at a
segment's edge.  Tolerances are those of the FP32 path: 1e-5 relative L2 on
audio and state, 1e-4 on gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle
from paper_2505_05940_gb300 import modal, workloads as W

from test_gpu_parity import GTOL, TOL, classes_of, oracle_instance, rel, run_gpu, to_plan


def _plate(n, m, steps):
    wl = W.tiny_random(100 + n, "plate", n, m, steps=steps)
    wl.instances[0].F0 = 200.0
    return oracle_instance(wl.instances[0], wl.fs, steps), wl.fs


@pytest.mark.parametrize("n,m,layout", [
    (1, 1, "classes"), (5, 1, "classes"), (33, 8, "classes"), (65, 16, "classes"),
    (100, 30, "classes"), (131, 9, "classes"), (160, 21, "classes"), (200, 50, "classes"),
    (224, 13, "classes"), (244, 17, "classes"), (7, 3, "dense"), (24, 5, "dense"),
    (33, 6, "dense"), (56, 3, "dense"), (64, 2, "dense")])
def test_resident_passes_match_the_oracle(n, m, layout):
    steps, K = 400, 128            # three full segments and one of 16 steps
    oi, fs = _plate(n, m, steps)
    ybar = np.random.default_rng(n).normal(size=steps)
    yb = torch.tensor(ybar[None], dtype=torch.float32, device="cuda")
    outs = []
    for flags in (0, 16):          # 16: the streaming kernel
        sim = modal.Simulator([to_plan(oi, fs, layout)], debug_flags=flags)
        sim.plan.set_profiling(True)
        fwd = sim.simulate(steps, want_state=True, want_status=True)
        # the checkpoint-free pass; classes of more than 64 modes stream
        fits = layout == "dense" or np.bincount(classes_of(oi)[0]).max() <= 64
        assert sim.plan.kernel_stats(6)[0] == (flags == 0 and fits)
        r = sim.simulate(steps, K=K)
        g = sim.grad(steps, yb, K, r["ckpt"], want_status=True)
        torch.cuda.synchronize()
        assert int(fwd["status"][0]) == 0 and int(g["status"][0]) == 0
        outs.append((fwd, r, g))
    # passes with checkpoints keep the streaming kernel's order of every sum
    for k in g:
        assert torch.equal(outs[0][2][k], outs[1][2][k]), k
    fwd, r, g = outs[0]
    assert rel(fwd["audio"].cpu().numpy(), r["audio"].cpu().numpy()) <= 1e-6
    ref = oracle.forward(oi, steps=steps)
    assert rel(fwd["audio"][0].cpu().numpy(), ref["y"]) <= TOL
    assert rel(fwd["q_end"].cpu().numpy(), ref["qN"]) <= TOL
    adj = oracle.adjoint(oi, ybar)
    dw2, dgm = oracle.coefficient_grads(oi, adj, 1.0 / fs)
    for name, want in (("d_omega2", dw2), ("d_gamma", dgm), ("d_b", adj["db"]), ("d_c", adj["dc"]),
                       ("d_q0", adj["dq0"]), ("d_qm1", adj["dqm1"]), ("d_kappa", adj["dkappa"])):
        e = rel(g[name].cpu().numpy()[:len(want)], want)
        assert e <= GTOL, (name, e)


@pytest.mark.parametrize("steps", [1, 2, 7, 8, 9, 10, 16, 17, 18, 31, 32, 33])
def test_resident_short_runs(steps):
    """Every length around the groups of 8 and 32 steps: states against the
    oracle; samples against it within 1e-6 of the summed modal terms (the first
    samples cancel almost completely)."""
    oi, fs = _plate(33, 8, 64)
    audio, qend, status, _ = run_gpu([oi], fs, steps)
    assert (status == 0).all()
    ref = oracle.forward(oi, steps=steps)
    assert rel(qend[0], ref["qN"]) <= TOL
    bound = 1e-6 * float(np.sum(np.abs(oi.c * ref["qN"])))
    assert np.abs(audio[0] - ref["y"]).max() <= bound


def test_more_plates_than_clusters():
    """More plates than run at once, of very different sizes (several CTAs and
    one CTA a plate in one launch): every plate as if it were alone."""
    steps = 300
    cases = [_plate(n, m, steps) for n, m in ((100, 30), (48, 12), (20, 4), (9, 2))]
    fs = cases[0][1]
    plans, ref = [], []
    for i in range(180):
        oi = cases[i % 4][0]
        d = to_plan(oi, fs)
        s = 0.5 + (i // 4) / 45.0
        d["kappa"] = oi.kappa * s
        plans.append(d)
    sim = modal.Simulator(plans)
    r = sim.simulate(steps, want_status=True)
    torch.cuda.synchronize()
    assert (r["status"].cpu().numpy() == 0).all()
    for i in (0, 1, 2, 3, 90, 91, 178, 179):
        one = modal.Simulator([plans[i]]).simulate(steps)["audio"]
        assert rel(r["audio"][i].cpu().numpy(), one[0].cpu().numpy()) <= 1e-5, i


@pytest.mark.parametrize("count,n,m", [(20, 150, 37), (32, 150, 37), (24, 200, 50), (48, 130, 32)])
def test_sums_that_span_ctas(count, n, m):
    """Many large plates: the streaming kernel sums more stress modes in a row
    than a CTA holds (parts of the force pass from CTA to CTA) and its rows change
    sides of their two chains (rows with gaps).  Gradients digit for digit."""
    steps, K = 40, 16
    oi, fs = _plate(n, m, steps)
    plans = []
    for i in range(count):
        d = to_plan(oi, fs)
        d["kappa"] = oi.kappa * (0.5 + i / count)
        plans.append(d)
    ybar = np.random.default_rng(n).normal(size=(count, steps))
    yb = torch.tensor(ybar, dtype=torch.float32, device="cuda")
    grads = []
    for flags in (0, 16):          # 16: the streaming kernel
        sim = modal.Simulator(plans, debug_flags=flags)
        r = sim.simulate(steps, K=K)
        g = sim.grad(steps, yb, K, r["ckpt"], want_status=True)
        torch.cuda.synchronize()
        assert (g["status"].cpu().numpy() == 0).all()
        grads.append(g)
    for k in grads[0]:
        assert torch.equal(grads[0][k], grads[1][k]), k
