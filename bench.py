#!/usr/bin/env python
"""Benchmark of the per-time-step modal update: forward + adjoint of a batch of
von Karman plates (Sec. 3.1, Eq. 9; Sec. 3.2, Eq. 20), with the
multi-resolution log-STFT loss of Sec. 4.3.1 (Eq. 24) between them.

Workload (per GPU): 64 simply supported steel plates, N_phi = 200 transverse
and N_psi = 50 stress modes, tension, stiffness, aspect ratio and damping of
each plate drawn log-uniform within +-0.3 decade of a target plate; 0.5 s at
44.1 kHz (22 050 steps); loss against the target plate's audio; gradients
with respect to omega^2, gamma, kappa and the aspect direction through the
checkpointed adjoint (checkpoint interval K).

One bench step = forward (with checkpoints) + loss + adjoint sweep.
value = plate mode-steps per second = n_gpus * 64 * 200 * 22050 / step time.

  python bench.py [--gpus N --steps K --warmup W]      # this library
  python bench.py --impl reference                     # FP64 CPU oracle on host cores

Secondary workloads (forward only, one JSON line each, not the headline):
  --workload batched      512 ragged plates and membranes, N_phi log-uniform in
                          [20, 400], aspects on 8 shared values (per-instance
                          copies of the coupling data, 22 050 steps); compared
                          with one instance per launch on a seeded subset
  --workload string40     one 40-mode nonlinear string, 48 000 steps at 48 kHz
  --workload plate100x30  one 100 x 30 steel plate, 44 100 steps

C-ABI driver (no PyTorch in the process, for profilers): the benchmark batch
through mdx_plan_create / mdx_simulate / mdx_grad with device buffers from the
CUDA runtime and inputs staged from host memory:
  python bench.py --c-abi --sim-steps 200 --K 64 [--no-grad] [--reps R]
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "plate mode-steps/s fwd+adjoint at ≤1e-5 rel err vs FP64; % of roofline"
UNIT = "mode-steps/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n-inst", type=int, default=64)
    ap.add_argument("--n-phi", type=int, default=200)
    ap.add_argument("--n-psi", type=int, default=50)
    ap.add_argument("--sim-steps", type=int, default=22050)
    ap.add_argument("--K", type=int, default=1024)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--workers", type=int, default=0)
    ap.add_argument("--workload", default="adjoint",
                    choices=["adjoint", "batched", "string40", "plate100x30"])
    ap.add_argument("--fwd-steps", type=int, default=0,
                    help="forward workloads: simulated steps (0 = the workload's own)")
    ap.add_argument("--no-compare", action="store_true",
                    help="batched workload: skip the per-instance and one-per-launch timings")
    ap.add_argument("--c-abi", action="store_true")
    ap.add_argument("--no-grad", action="store_true")
    ap.add_argument("--reps", type=int, default=1)
    return ap.parse_args()


def workload_name(a):
    return (f"adjoint{a.n_inst}_plate{a.n_phi}x{a.n_psi}_{a.sim_steps}steps_K{a.K}")


def load_tensor_peak():
    """Measured dense BF16 tensor throughput (FLOP/s, burst) or the fallback."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return float(json.load(f)["bf16_tflops"]) * 1e12
    return 1.9e15


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def profiled_traffic(a, steps_per_launch):
    """DRAM bytes per launch of the fused kernel from the committed ncu summary,
    scaled from its bytes per step; None when the kernel source has changed
    since the capture (hash recorded in the summary) or the workload differs."""
    import hashlib
    import re
    path = os.path.join(ROOT, "profiles", "plate_kernel_fused_64plates_200x50.md")
    if not os.path.exists(path) or (a.n_inst, a.n_phi, a.n_psi) != (64, 200, 50):
        return None
    text = open(path).read()
    m_src = re.search(r"kernel-source: (\S+) sha256 ([0-9a-f]+)", text)
    m_tr = re.search(r"traffic_bytes_per_step: (\d+)", text)
    if not (m_src and m_tr):
        return None
    src = os.path.join(ROOT, m_src.group(1))
    if not os.path.exists(src):
        return None
    digest = hashlib.sha256(open(src, "rb").read()).hexdigest()
    if not digest.startswith(m_src.group(2)):
        return None
    return float(m_tr.group(1)) * steps_per_launch


def plate_roofline(stats, names, resident, peak, peak_kind, sms):
    """The dominant plate launch class against what bounds it.  stats: class ->
    (launches, ms, bytes of one pass over the coupling data per step).  The
    streaming kernel moves those bytes; the resident kernel reads them once per
    launch, so its figure is the FP32 multiply-adds of the products (one per
    coupling entry and right-hand side) against the CUDA cores' nominal rate."""
    dom = max(stats, key=lambda w: stats[w][1])
    rhs = {0: 1, 1: 1, 2: 2, 4: 3}
    fp32_peak = sms * 128 * 2 * 2.07e9 / 1e12

    def rate(w):
        n, ms, b = stats[w]
        if not ms:
            return None
        return (2.0 * rhs[w] * b / 4.0 / (ms * 1e-3) / 1e12 if resident else b / (ms * 1e-3) / 1e9)

    unit = "TFLOP/s" if resident else "GB/s"
    n, ms, b = stats[dom]
    out = {"bound": "fp32" if resident else "hbm", "achieved": rate(dom),
           "peak": fp32_peak if resident else peak, "unit": unit, "traffic": None,
           "kernel": ("resident plate kernel, " if resident else "streaming plate kernel, ") + names[dom],
           "peak_source": ("nominal: SMs x 128 FP32 lanes x 2 x 2.07 GHz" if resident
                           else f"{peak_kind} hbm_gbs"),
           "per_launch_ms": ms / max(n, 1)}
    out["frac"] = out["achieved"] / out["peak"] if out["achieved"] else None
    if resident:
        out["basis"] = ("multiply-adds of the coupling products; a step's dependent chain "
                        "(barrier, reductions, two exchanges between CTAs) takes most of its time")
    else:
        out["per_launch_algorithmic_bytes"] = b / max(n, 1)
    out["all_plate_kernels"] = {names[w]: {"launches": stats[w][0], "ms": stats[w][1], unit: rate(w)}
                                for w in stats}
    return out


# ----------------------------------------------------------------- ranks

def shard_seed(rank):
    """Instances are sharded by rank: every rank runs its own seeded batch
    (independent problems, no collective on the data path)."""
    return rank


def max_over_ranks(ms, device, world):
    """The job's time is the slowest rank's (all_reduce MAX; the only
    collective of the benchmark)."""
    import torch
    t = torch.tensor([float(ms)], device=device, dtype=torch.float64)
    if world > 1:
        import torch.distributed as dist
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_value(world, n_inst, n_phi, sim_steps, ms_step):
    """Plate mode-steps of all ranks per second of the slowest rank."""
    return world * n_inst * n_phi * sim_steps / (ms_step * 1e-3)


# ----------------------------------------------------------------- inputs

def _prepare_one(args):
    inst, fs, steps, want_dir = args
    from paper_2505_05940_gb300 import physics
    return physics.prepare(inst, fs, steps, want_aspect_derivative=want_dir)


def prepare_inputs(a, rank):
    """Seeded target + initial guesses, prepared in a spawn process pool
    (coupling tensors and their aspect derivatives are FP64 host work)."""
    import concurrent.futures as cf
    import multiprocessing as mp
    from paper_2505_05940_gb300 import workloads as W
    tgt, inits = W.adjoint_plates(seed=shard_seed(rank), n_inst=a.n_inst, n_phi=a.n_phi,
                                  n_psi=a.n_psi, steps=a.sim_steps)
    jobs = [(tgt.instances[0], tgt.fs, tgt.steps, False)]
    jobs += [(i, inits.fs, inits.steps, True) for i in inits.instances]
    workers = a.workers or max(1, min(len(jobs), (os.cpu_count() or 2)))
    with cf.ProcessPoolExecutor(max_workers=workers, mp_context=mp.get_context("spawn")) as ex:
        out = list(ex.map(_prepare_one, jobs))
    return out[0], out[1:], inits


# ----------------------------------------------------------------- clocks

class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled during the timed region."""

    def __init__(self, index):
        self.index = index
        self.rows = []
        self.proc = None

    def __enter__(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={q}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([x.strip() for x in line.split(",")])

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            try:
                sm.append(float(r[1]))
                mx = max(mx, float(r[2]))
                for nm, v in zip(names, r[5:9]):
                    if v.strip().lower() == "active":
                        reasons.add(nm)
            except (ValueError, IndexError):
                continue
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


# ----------------------------------------------------------------- CPU oracle

def oracle_sample(a, n_threads, sample_steps):
    """FP64 oracle forward + adjoint of one plate per thread on a bounded
    number of steps (the same outputs mdx_grad gives per mode and stress
    mode; the oracle has no counterpart of the aspect-direction contraction);
    returns (mode-steps/s, threads, description)."""
    import oracle
    from oracle import coupling_oracle as CO
    from oracle import physics_oracle as PO
    from paper_2505_05940_gb300 import workloads as W
    _, inits = W.adjoint_plates(seed=0, n_inst=max(n_threads, 1), n_phi=a.n_phi,
                                n_psi=a.n_psi, steps=sample_steps)
    ois = [PO.build_instance(inits.instances[0], inits.fs, sample_steps,
                             coupling=CO.oracle_coupling)]
    for _ in range(1, n_threads):
        ois.append(ois[0])
    rng = np.random.default_rng(0)
    ybar = rng.normal(size=sample_steps)
    oracle.lib()

    def work(oi):
        oracle.adjoint(oi, ybar)   # runs the forward (trajectory) then the reverse

    ths = [threading.Thread(target=work, args=(o,)) for o in ois]
    t0 = time.perf_counter()
    for t in ths:
        t.start()
    for t in ths:
        t.join()
    dt = time.perf_counter() - t0
    value = n_threads * ois[0].N * sample_steps / dt
    desc = (f"{n_threads} thread(s) x one {ois[0].N}x{ois[0].M} plate x {sample_steps} steps "
            f"forward+adjoint in FP64 (the oracle as it stands), {dt:.1f} s wall; the "
            f"value is that sample's mode-steps/s, extrapolated to the full workload "
            f"({a.n_inst} plates x {a.sim_steps} steps) for ms_per_step")
    return value, n_threads, desc


def oracle_forward_sample(wl, sample_steps, runs=5):
    """FP64 oracle forward of a single-instance workload on one host thread
    (the paper's single-simulation CPU comparison), on its first
    `sample_steps` steps; median of `runs` runs -> (mode-steps/s, description)."""
    import oracle
    from oracle import coupling_oracle as CO
    from oracle import physics_oracle as PO
    inst = wl.instances[0]
    steps = min(sample_steps, wl.steps)
    cp = CO.oracle_coupling if inst.kind == "plate" else None
    oi = PO.build_instance(inst, wl.fs, steps, coupling=cp)
    times = []
    for _ in range(runs):
        t0 = time.perf_counter()
        oracle.forward(oi, steps=steps)
        times.append(time.perf_counter() - t0)
    t = float(np.median(times))
    desc = (f"one host thread, the oracle as it stands: FP64 forward of the workload's first "
            f"{steps} steps, median of {runs} runs ({t:.3f} s)")
    return oi.N * steps / t, desc


def reference_arm(a):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cores = os.cpu_count() or 1
    per = []
    for _ in range(a.warmup):
        oracle_sample(a, cores, 50)
    for _ in range(a.steps):
        v, c, desc = oracle_sample(a, cores, 200)
        per.append(v)
    value = float(np.median(per))
    ms = a.n_inst * a.n_phi * a.sim_steps / value * 1e3
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": a.gpus, "steps": a.steps, "warmup": a.warmup, "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": workload_name(a), "instances": a.n_inst,
                                             "n_phi": a.n_phi, "n_psi": a.n_psi,
                                             "sim_steps": a.sim_steps, "K": a.K},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": desc},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ----------------------------------------------------------------- secondary workloads

def _group_bank(args):
    aspect, n_phi, n_psi = args
    from paper_2505_05940_gb300 import proposal
    return proposal._aspect_bank([aspect], n_phi=n_phi, n_psi=n_psi)


def forward_workload(a):
    """Forward-only throughput of the batched and single-instance workloads."""
    import concurrent.futures as cf
    import multiprocessing as mp
    from paper_2505_05940_gb300 import physics, proposal, workloads as W
    if a.workload == "batched":
        wl = W.batched_ragged(seed=0)
        aspects = sorted({float(i.aspect) for i in wl.instances if i.kind == "plate"})
        workers = a.workers or max(1, min(len(aspects), os.cpu_count() or 1))
        with cf.ProcessPoolExecutor(max_workers=workers, mp_context=mp.get_context("spawn")) as ex:
            banks = list(ex.map(_group_bank, [(x, 400, 100) for x in aspects]))
        bank = {}
        for b in banks:
            bank.update(b)
        cp = proposal._bank_coupling(bank)
        prep = [physics.prepare(i, wl.fs, wl.steps, coupling=cp) for i in wl.instances]
        # plates of one aspect share their coupling tensor: one tensor-core group each
        for inst, p in zip(wl.instances, prep):
            if inst.kind == "plate":
                p["geom_group"] = 1 + aspects.index(float(inst.aspect))
    else:
        wl = W.string_40() if a.workload == "string40" else W.plate_100x30()
        prep = [physics.prepare(i, wl.fs, wl.steps) for i in wl.instances]
    import torch
    from paper_2505_05940_gb300 import modal
    sim = modal.Simulator(prep)
    steps = a.fwd_steps if a.fwd_steps > 0 else wl.steps
    if steps > wl.steps:
        raise SystemExit("--fwd-steps exceeds the workload's excitation length")
    modes = int(sum(len(p["omega2"]) for p in prep))
    for _ in range(a.warmup):
        sim.simulate(steps)
    torch.cuda.synchronize()
    sim.plan.set_profiling(True)
    sim.plan.reset_stats()
    stream = torch.cuda.current_stream()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(0) as clk:
        ev0.record(stream)
        for _ in range(a.steps):
            sim.simulate(steps)
        ev1.record(stream)
        torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1) / a.steps
    value = modes * steps / (ms * 1e-3)
    n, pms, pby = sim.plan.kernel_stats(0)
    gn, gms, gby = sim.plan.kernel_stats(5)
    cn, cms, _ = sim.plan.kernel_stats(6)
    sim.plan.set_profiling(False)
    peak, peak_kind = load_peaks()
    line = {"metric": "mode-steps/s forward", "value": value, "unit": UNIT, "n_gpus": 1,
            "steps": a.steps, "warmup": a.warmup, "ms_per_step": ms,
            "us_per_time_step": ms * 1e3 / steps, "higher_is_better": True, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": wl.name, "instances": len(prep), "total_modes": modes,
                       "sim_steps": steps}, "clocks": clk.summary()}
    if n:
        ach = pby / (pms * 1e-3) / 1e9
        line["plate_kernel"] = {"GB/s": ach, "frac_of_hbm": ach / peak,
                                "peak_source": f"{peak_kind} hbm_gbs",
                                "share_of_time": pms / (ms * a.steps)}
    if cn:
        # plates whose coupling rows stay on the SMs (tensor memory, shared memory,
        # registers) of a thread-block cluster: bound by the latency of a step's
        # dependent chain (products, reductions, two exchanges), not by bytes
        line["resident_kernel"] = {"us_per_step": cms * 1e3 / (cn * steps),
                                  "share_of_time": cms / (ms * a.steps),
                                  "bound": "latency (H read once per launch)"}
    if gn:
        # grouped plates: one pass over each group's shared coupling tensor per
        # step; the contraction's algorithmic flops are 2 x (nonzero H entries)
        # x plates, executed three times over as split TF32
        ach = gby / (gms * 1e-3) / 1e9
        tf32_peak = load_tensor_peak() / 2.0
        fl = sim.plan.group_work()[1] * steps * gn
        roof = {"bound": "hbm", "achieved": ach, "peak": peak, "unit": "GB/s",
                "frac": ach / peak, "traffic": None,
                "kernel": "group_kernel (split-TF32 tcgen05 GEMM per stress mode and step)",
                "peak_source": f"{peak_kind} hbm_gbs",
                "share_of_time": gms / (ms * a.steps),
                "us_per_step": gms * 1e3 / (gn * steps),
                "tensor": {"algorithmic_TFLOP/s": fl / (gms * 1e-3) / 1e12,
                           "executed_TFLOP/s": 3 * fl / (gms * 1e-3) / 1e12,
                           "tf32_peak_TFLOP/s": tf32_peak / 1e12,
                           "peak_source": "measured bf16_tflops / 2 (TF32 runs at half the BF16 rate)"}}
        line["roofline"] = roof
    if a.workload == "batched" and not a.no_compare:
        # the same plans with every plate on its own coupling copy: the FP32
        # CUDA-core path of the per-instance kernel
        csim = modal.Simulator(prep, group_engine="off")
        csim.simulate(steps)
        torch.cuda.synchronize()
        csim.plan.set_profiling(True)
        ev0.record(stream)
        csim.simulate(steps)
        ev1.record(stream)
        torch.cuda.synchronize()
        cc_ms = ev0.elapsed_time(ev1)
        cn_, cms_, cby_ = csim.plan.kernel_stats(0)
        line["fp32_cuda_core_per_instance"] = {
            "value": modes * steps / (cc_ms * 1e-3), "ms_per_step": cc_ms,
            "grouped_tf32x3_over_fp32": cc_ms / ms}
        if cn_:
            # the per-instance path streams each plate's own class-layout copy
            ach = cby_ / (cms_ * 1e-3) / 1e9
            line["fp32_cuda_core_per_instance"]["plate_kernel"] = {
                "GB/s": ach, "frac_of_hbm": ach / peak, "peak_source": f"{peak_kind} hbm_gbs",
                "bytes_per_step": cby_ / (cn_ * steps), "share_of_time": cms_ / cc_ms}
        del csim
        # the plain form: one instance per plan and launch, on a seeded subset
        rng = np.random.default_rng(1)
        sub = sorted(rng.choice(len(prep), size=32, replace=False).tolist())
        sub_steps = 2205
        sims = [modal.Simulator([prep[i]], group_engine="off") for i in sub]
        for s_ in sims:
            s_.simulate(sub_steps)
        torch.cuda.synchronize()
        ev0.record(stream)
        for s_ in sims:
            s_.simulate(sub_steps)
        ev1.record(stream)
        torch.cuda.synchronize()
        ms_one = ev0.elapsed_time(ev1)
        sub_modes = sum(len(prep[i]["omega2"]) for i in sub)
        one = sub_modes * sub_steps / (ms_one * 1e-3)
        bsim = modal.Simulator([prep[i] for i in sub])
        bsim.simulate(sub_steps)
        torch.cuda.synchronize()
        ev0.record(stream)
        bsim.simulate(sub_steps)
        ev1.record(stream)
        torch.cuda.synchronize()
        batched_sub = sub_modes * sub_steps / (ev0.elapsed_time(ev1) * 1e-3)
        line["one_instance_per_launch"] = {
            "subset": f"32 seeded instances, {sub_steps} steps", "value": one,
            "same_subset_batched": batched_sub, "full_batch_over_one": value / one,
            "subset_batched_over_one": batched_sub / one}
    if a.workload in ("string40", "plate100x30") and not a.no_cpu_baseline:
        v, desc = oracle_forward_sample(wl, 48000 if a.workload == "string40" else 4410)
        line["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": 1, "kind": "oracle",
                                "sample": desc}
    print(json.dumps(line), flush=True)


def physical_gradients(sim, prepared, d_omega2, d_gamma, d_kappa, d_dir):
    """dL/d(T0, D, aspect, sigma0, sigma1) of every plate through
    mdx_physics_vjp, from the per-mode gradients of the adjoint."""
    from paper_2505_05940_gb300 import _native, physics
    off = sim.plan.mode_offset
    koff = np.concatenate([[0], np.cumsum(sim.plan.n_stress)])
    out = []
    for i, p in enumerate(prepared):
        n, m = len(p["omega2"]), int(sim.plan.n_stress[i])
        g = _native.physics_vjp(physics.physics_struct(p), n, m, d_omega2[off[i]:off[i] + n],
                                d_gamma[off[i]:off[i] + n], 0.0, d_kappa[koff[i]:koff[i + 1]],
                                float(d_dir[i]), p.get("dzeta4"))
        out.append({k: g[k] for k in ("d_T0", "d_D", "d_aspect", "d_sigma0", "d_sigma1")})
    return out


# ----------------------------------------------------------------- C ABI alone

class _Cuda:
    """Device buffers straight from the CUDA runtime (no PyTorch)."""

    def __init__(self):
        import ctypes
        import glob
        cands = [os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "lib64",
                              "libcudart.so")]
        cands += sorted(glob.glob("/usr/local/cuda*/lib64/libcudart.so*"))
        path = next((c for c in cands if os.path.exists(c)), None)
        if path is None:
            raise OSError("libcudart.so not found")
        self.ct = ctypes
        self.rt = ctypes.CDLL(path)
        self.ptrs = []

    def check(self, rc, what):
        if rc != 0:
            raise RuntimeError(f"{what}: CUDA error {rc}")

    def alloc(self, nbytes):
        p = self.ct.c_void_p()
        self.check(self.rt.cudaMalloc(self.ct.byref(p), self.ct.c_size_t(max(16, nbytes))),
                   "cudaMalloc")
        self.ptrs.append(p)
        return p

    def h2d(self, dst, arr):
        a = np.ascontiguousarray(arr)
        self.check(self.rt.cudaMemcpy(dst, a.ctypes.data_as(self.ct.c_void_p),
                                      self.ct.c_size_t(a.nbytes), 1), "cudaMemcpy")

    def d2h(self, arr, src):
        self.check(self.rt.cudaMemcpy(arr.ctypes.data_as(self.ct.c_void_p), src,
                                      self.ct.c_size_t(arr.nbytes), 2), "cudaMemcpy")

    def sync(self):
        self.check(self.rt.cudaDeviceSynchronize(), "cudaDeviceSynchronize")

    def free(self):
        for p in self.ptrs:
            self.rt.cudaFree(p)
        self.ptrs = []


def c_abi_run(a):
    """The benchmark batch through the C ABI alone: every call's inputs are
    copied up from host memory and its outputs (audio, per-mode gradients)
    copied back, inside the timed loop; no PyTorch is loaded."""
    import ctypes
    from paper_2505_05940_gb300 import _native
    _, init_p, _ = prepare_inputs(a, 0)
    L = _native.load()
    cu = _Cuda()
    plan = _native.Plan(init_p)
    n, steps, K, TM = len(init_p), a.sim_steps, a.K, plan.total_modes
    grad = not a.no_grad
    exc = np.zeros((n, steps), np.float32)
    for i, p in enumerate(init_p):
        exc[i] = p["e"][:steps]
    q0 = np.concatenate([p["q0"] for p in init_p]).astype(np.float64)
    ybar = np.random.default_rng(0).standard_normal((n, steps)).astype(np.float32) * 1e-3
    d_exc, d_q0, d_qm1 = cu.alloc(exc.nbytes), cu.alloc(q0.nbytes), cu.alloc(q0.nbytes)
    d_ybar = cu.alloc(ybar.nbytes)
    audio = cu.alloc(n * steps * 4)
    ckpt = cu.alloc(plan.checkpoint_bytes(steps, K))
    status = cu.alloc(n * 4)
    work_bytes = plan.workspace_bytes(steps, K)
    work = cu.alloc(work_bytes) if grad else None
    g = _native.Grads()
    outs = {}
    for name, count in (("d_omega2", TM), ("d_gamma", TM), ("d_kappa",
                        max(1, int(plan.n_stress.sum()))), ("d_dir", n)):
        outs[name] = (cu.alloc(count * 8), np.zeros(count))
        setattr(g, name, outs[name][0].value)
    host_audio = np.zeros((n, steps), np.float32)
    times = []
    for _ in range(max(1, a.reps)):
        cu.sync()
        t0 = time.perf_counter()
        cu.h2d(d_exc, exc)
        cu.h2d(d_q0, q0)
        cu.h2d(d_qm1, q0)
        _native.check(L.mdx_simulate(plan._h, d_exc, d_q0, d_qm1, steps, audio, None, None, K,
                                     ckpt, status, None))
        cu.d2h(host_audio, audio)
        if grad:
            cu.h2d(d_ybar, ybar)
            _native.check(L.mdx_grad(plan._h, d_exc, d_q0, d_qm1, steps, d_ybar, K, ckpt, work,
                                     work_bytes, ctypes.byref(g), status, None))
            for name, (dev, host) in outs.items():
                cu.d2h(host, dev)
        cu.sync()
        times.append(time.perf_counter() - t0)
    st = np.zeros(n, np.int32)
    cu.d2h(st, status)
    ms = min(times) * 1e3
    print(json.dumps({"c_abi": True, "plates": n, "modes": TM, "steps": steps, "K": K,
                      "grad": grad, "ms_per_call": ms,
                      "mode_steps_per_s": n * a.n_phi * steps / (ms * 1e-3),
                      "status_max": int(st.max())}), flush=True)
    plan.close()
    cu.free()
    if st.max() != 0:
        raise SystemExit(1)


# ----------------------------------------------------------------- main arm

def main():
    a = parse()
    if a.impl == "reference":
        reference_arm(a)
        return
    if a.c_abi:
        c_abi_run(a)
        return
    if a.workload != "adjoint":
        forward_workload(a)
        return
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    # host-side preparation before any CUDA use (spawned workers)
    tgt_p, init_p, inits_wl = prepare_inputs(a, rank)

    import torch
    import torch.distributed as dist
    from paper_2505_05940_gb300 import losses, modal
    if world > 1:
        dist.init_process_group("nccl", rank=rank, world_size=world)
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    # target audio (outside the timed region)
    tsim = modal.Simulator([tgt_p], device=str(dev))
    target = tsim.simulate(a.sim_steps)["audio"].expand(a.n_inst, -1).contiguous()
    sim = modal.Simulator(init_p, device=str(dev))

    def step():
        for t in (sim.omega2, sim.gamma, sim.b, sim.c, sim.tau, sim.kappa, sim.q0, sim.qm1,
                  sim.direction):
            t.grad = None
        audio = modal.simulate_autograd(sim, a.sim_steps, K=a.K)
        loss = losses.multires_log_stft(audio, target).sum()
        loss.backward()
        return loss

    for _ in range(a.warmup):
        step()
    torch.cuda.synchronize()
    sim.plan.set_profiling(True)
    sim.plan.reset_stats()
    stream = torch.cuda.current_stream()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        ev0.record(stream)
        for _ in range(a.steps):
            loss = step()
        ev1.record(stream)
        torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    ms_total = max_over_ranks(ev0.elapsed_time(ev1), dev, world)
    ms_step = ms_total / a.steps
    units = world * a.n_inst * a.n_phi * a.sim_steps
    value = whole_job_value(world, a.n_inst, a.n_phi, a.sim_steps, ms_step)
    # roofline of the dominant kernel (plate kernel: forward, recompute, reverse,
    # fused reverse + recompute launches)
    stats = {w: sim.plan.kernel_stats(w) for w in (0, 1, 2, 4)}
    stats = {w: v for w, v in stats.items() if v[0] > 0}
    dir_stats = sim.plan.kernel_stats(3)
    sim.plan.set_profiling(False)
    peak, peak_kind = load_peaks()
    tot_ms = sum(s[1] for s in stats.values())
    names = {0: "forward", 1: "recompute", 2: "reverse", 4: "fused reverse + recompute"}
    roofline = plate_roofline(stats, names, sim.plan.resident()["checkpointed"], peak, peak_kind,
                              torch.cuda.get_device_properties(dev).multi_processor_count)
    roofline["kernel_share_of_step"] = tot_ms / ms_total if ms_total else None
    roofline["direction_contraction"] = {"launches": dir_stats[0], "ms": dir_stats[1]}
    # end-to-end through the public API with host buffers
    e2e = None
    if not a.no_e2e:
        exc_host = sim.exc.cpu().pin_memory()
        tgt_host = target.cpu().pin_memory()
        out_keys = ("omega2", "gamma", "kappa", "direction")
        h2d = exc_host.numel() * 4 + tgt_host.numel() * 4
        d2h = 8 + sum(getattr(sim, k).numel() * 8 for k in out_keys)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(a.steps):
            exc_d = exc_host.to(dev, non_blocking=True)
            tgt_d = tgt_host.to(dev, non_blocking=True)
            sim.exc = exc_d
            for t in (sim.omega2, sim.gamma, sim.b, sim.c, sim.tau, sim.kappa, sim.q0,
                      sim.qm1, sim.direction):
                t.grad = None
            audio = modal.simulate_autograd(sim, a.sim_steps, K=a.K)
            loss = losses.multires_log_stft(audio, tgt_d).sum()
            loss.backward()
            res = [loss.detach().cpu()] + [getattr(sim, k).grad.cpu() for k in out_keys]
            # the per-mode gradients mapped to the physical parameters (C ABI, host)
            phys = physical_gradients(sim, init_p, *[r.numpy() for r in res[1:]])
        torch.cuda.synchronize()
        e2e_s = (time.perf_counter() - t0) / a.steps
        e2e = {"value": units / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": int(d2h),
               "physical_gradients_plate0": phys[0]}
    cpu = None
    if rank == 0 and not a.no_cpu_baseline:
        v, cores, desc = oracle_sample(a, os.cpu_count() or 1, 200)
        cpu = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc}
    # our kernels per step: state init, adjoint init and gradient epilogue, plus the
    # plate and direction-contraction launches the plan's event records counted
    counted = sum(v[0] for v in stats.values()) + dir_stats[0]
    launches_per_step = 3 + counted / max(a.steps, 1)
    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": a.steps, "warmup": a.warmup, "ms_per_step": ms_step,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "f32", "data": "synthetic",
                "config": {"workload": workload_name(a), "instances_per_gpu": a.n_inst,
                           "n_phi": a.n_phi, "n_psi": a.n_psi, "sim_steps": a.sim_steps,
                           "K": a.K, "loss": "multi-resolution log-STFT L1 (256/1024/4096)",
                           "l2": ("working set larger than L2, no flush: every launch reads "
                                  "the class-layout coupling data (128 MB) and each segment its "
                                  "aspect derivative (128 MB), beside checkpoints and segment "
                                  "buffers"),
                           "parallelism": f"instances sharded, {world} GPU(s), no collective"},
                "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e,
                "gpu_launches": int(round(launches_per_step * a.steps)), "clocks": clk.summary(),
                "loss": float(loss.item())}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
