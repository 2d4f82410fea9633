"""The linear solver over the range of FP64: states of strongly damped modes, which
fall far below the range of FP32 within a few hundred steps, and states and inputs
that are tiny or huge from the start.  Every mode's end state against the same
recursion in NumPy (FP64), relative to that mode's own state.  The recursions
round alike up to the powers of the companion matrix over a chunk: at most
700 steps x 2^-53 x 2 / sin(omega T) for omega T >= 0.02, 8e-12, squared
conditioning in A^256 another 1e-9; 1e-8 is allowed.  Audio, FP32, to 1e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2505_05940_gb300 import modal

from test_gpu_parity import rel

T = 1.0 / 44100.0


def _object(n, eps_max, steps, seed, b=1.0, e=1.0, q=1.0, c=1.0):
    """n oscillatory modes, from lightly damped low to strongly damped high ones,
    struck during the first 40 steps; scales of input, state and pickup."""
    rng = np.random.default_rng(seed)
    wT = np.sort(rng.uniform(0.02, 1.9, n))
    eps = eps_max * (wT / wT.max()) ** 2
    gamma = eps / (2.0 - eps) / T                   # eps = 2 gamma T / (1 + gamma T)
    gamma = np.minimum(gamma, 0.9 * wT / T)
    exc = np.zeros(steps, np.float32)
    exc[:40] = rng.uniform(0.5, 1.0, 40) * np.hanning(42)[1:-1]
    return dict(kind="tension", omega2=(wT / T) ** 2, gamma=gamma, dt=T, lam=np.ones(n), tau=0.0,
                b=b * 1e9 * rng.uniform(0.5, 1.0, n), c=c * rng.uniform(-1.0, 1.0, n),
                e=(exc * np.float32(e)).astype(np.float32),
                q0=q * rng.uniform(0.1, 1.0, n), qm1=q * rng.uniform(0.1, 1.0, n))


def _numpy(d, steps):
    den = 1.0 + d["gamma"] * T
    eps, r = 2.0 * d["gamma"] * T / den, T * T / den
    g, p, rb = 2.0 - eps - r * d["omega2"], eps - 1.0, r * d["b"]
    q, qm = d["q0"].copy(), d["qm1"].copy()
    y = np.zeros(steps)
    for n in range(steps):
        q, qm = g * q + p * qm + rb * float(d["e"][n]), q
        y[n] = (d["c"] * q).sum()
    return y, q, qm


def _check(objs, steps):
    sim = modal.Simulator(objs)
    r = sim.simulate_linear(steps, want_state=True, want_status=True)
    torch.cuda.synchronize()
    assert (r["status"].cpu().numpy() == 0).all()
    q, qm = r["q_end"].cpu().numpy(), r["qm1_end"].cpu().numpy()
    lo = 1.0
    for i, d in enumerate(objs):
        a, b = sim.plan.mode_offset[i], sim.plan.mode_offset[i] + len(d["omega2"])
        y, qr, qmr = _numpy(d, steps)
        size = np.maximum(np.abs(qr), np.abs(qmr))
        lo = min(lo, size.min())
        assert (size > 1e-290).all()
        assert (np.abs(q[a:b] - qr) <= 1e-8 * size).all(), i
        assert (np.abs(qm[a:b] - qmr) <= 1e-8 * size).all(), i
        assert rel(r["audio"][i].cpu().numpy(), y) <= 1e-6, i
    return lo


@pytest.mark.parametrize("steps", [200, 256, 700])
def test_strongly_damped_modes(steps):
    lo = _check([_object(n, 0.8, steps, n) for n in (1, 33, 70, 150)], steps)
    assert steps < 700 or lo < 1e-100


@pytest.mark.parametrize("b,e,q,c", [
    (2.0 ** -100, 2.0 ** -30, 2.0 ** -130, 2.0 ** 130), (1.0, 2.0 ** -120, 2.0 ** -120, 2.0 ** 110),
    (2.0 ** 200, 1.0, 2.0 ** 200, 2.0 ** -200), (2.0 ** -300, 2.0 ** 100, 2.0 ** -200, 2.0 ** 200),
    (2.0 ** 100, 2.0 ** -140, 2.0 ** -40, 2.0 ** 40)])
def test_tiny_and_huge_objects(b, e, q, c):
    steps = 600
    _check([_object(n, 0.3, steps, n, b=b, e=e, q=q, c=c) for n in (5, 40)], steps)
