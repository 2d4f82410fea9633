"""Bounded waits of the resident plate kernel.  One CTA of every plate withholds its
parts of the force (debug flag), so the other CTAs' waits run out: every pass
reports MDX_ERR_TIMEOUT for every plate after the limit that the plan was given,
nothing hangs, and the next plan on the device still matches the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2505_05940_gb300 import modal, workloads as W

from test_gpu_parity import check_parity, oracle_instance, to_plan

WITHHOLD = 32      # debug flag: the second CTA of every plate sends no parts


def _case(n, m, count, steps):
    wl = W.tiny_random(100 + n, "plate", n, m, steps=steps)
    wl.instances[0].F0 = 200.0
    oi = oracle_instance(wl.instances[0], wl.fs, steps)
    plans = [dict(to_plan(oi, wl.fs), kappa=oi.kappa * (0.5 + i / count)) for i in range(count)]
    return oi, wl.fs, plans


@pytest.mark.parametrize("n,m,count", [(100, 30, 1), (33, 16, 3), (150, 37, 20)])
def test_every_pass_reports_the_timeout(n, m, count):
    steps, K = 300, 128
    oi, fs, plans = _case(n, m, count, steps)
    yb = torch.randn(count, steps, device="cuda")
    good = modal.Simulator(plans)
    ckpt = good.simulate(steps, K=K)["ckpt"]
    sim = modal.Simulator(plans, wait_limit=20000, debug_flags=WITHHOLD)
    sim.plan.set_profiling(True)
    fwd = sim.simulate(steps, want_status=True)
    assert sim.plan.kernel_stats(6)[0] == 1
    rec = sim.simulate(steps, K=K, want_status=True)
    g = sim.grad(steps, yb, K, ckpt, want_status=True)
    torch.cuda.synchronize()
    for r in (fwd, rec, g):
        assert (r["status"].cpu().numpy() == 4).all(), r["status"]
    check_parity([oi], fs, steps)


def test_the_limit_is_the_plans():
    """A hundred times the polls take more than ten times as long."""
    steps = 16
    _, _, plans = _case(100, 30, 1, steps)
    ms = []
    for limit in (2000, 200000):
        sim = modal.Simulator(plans, wait_limit=limit, debug_flags=WITHHOLD)
        sim.plan.set_profiling(True)
        r = sim.simulate(steps, want_status=True)
        torch.cuda.synchronize()
        assert int(r["status"][0]) == 4
        ms.append(sim.plan.kernel_stats(6)[1])
    assert ms[1] > 10.0 * ms[0], ms
