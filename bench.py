#!/usr/bin/env python3
"""Throughput of the pooled-chain pCN sampler (4-qubit Pauli tomography, 65536 chains).

One "step" is one pass of the whole hot path over every chain: Philox proposal,
Algorithm 1 assembly, projector contraction, log-likelihood, accept/adapt, pooling
and trajectory store (65536 chain-steps).  Prints one JSON line (rank 0).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
  python bench.py --profile-case [--chains C] [--steps K]     # short run for ncu captures

Under torchrun (N > 1) every rank runs its own 65536 chains with a disjoint global
chain-id range (weak scaling; chains never communicate), timed between barriers and
reported as the max over ranks.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "4-qubit pCN chain-steps/s, mixed vs plain FP32 form, at logL err ≤1e-3"
UNIT = "chain-steps/s"
CONFIG_INDEX = 4
CHAINS = 65536
WORKLOAD = ("config 4: 4-qubit Pauli QST (D=16, 81 bases x 16 outcomes = 1296 projectors, 1000 shots/basis), "
            "Haar pure truth depolarised 0.02, beta0 0.02")

# DRAM bytes per launch of each kernel from one ncu capture (bench.py --profile-case,
# config 4 problem at `chains` chains, one pCN-step launch of the kernel), scaled to a launch
# over the benchmark's chains in proportion to the chains processed.  The capture is only
# used while every source file the kernel is built from is as it was: `sha256` is of their contents,
# one after the other.
CSRC = "paper_2501_17334_gb300/csrc/"
NCU_TRAFFIC = {
    # profiles/propose_kernel_config4.md
    "propose": {"sources": [CSRC + f for f in ("propose.cu", "propose_dev.cuh", "f32x2.cuh", "log_poly.h",
                                               "qst_internal.cuh")],
                "sha256": "31de98d510cfda31f46c6a6d4966086a6de5bf161bdbfa03308315d7b7d01575",
                "chains": 32768, "bytes": 137.366272e6 + 168.434944e6},
    # profiles/project_tc_kernel_config4.md
    "project": {"sources": [CSRC + f for f in ("project_tc.cu", "f32x2.cuh", "log_poly.h", "qst_internal.cuh")],
                "sha256": "3b33ac973a829547b3ce2b71a526f178355cc1bc5e75e93f6b8e04beafa59966",
                "chains": 32768, "bytes": 51.399936e6 + 0.007680e6},
}


def _sha256(paths):
    h = hashlib.sha256()
    for path in paths:
        with open(os.path.join(ROOT, path), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def ncu_traffic(kernel, chains):
    rec = NCU_TRAFFIC.get(kernel)
    if not rec or rec["bytes"] is None or rec["sha256"] != _sha256(rec["sources"]):
        return None
    return rec["bytes"] * chains / rec["chains"]


# ---- algorithmic work per chain-step ------------------------------------------------------

def propose_flops(D):
    """Algorithmic FP32 FLOPs of the proposal and Algorithm 1 per chain-step (FMA = 2): one
    Gram-Schmidt QR of H (8 D^2 (D - 1)), W = (U + I) G (8 D^3), the Hermitian half of W W^dag
    (4 D^2 (D + 1)), the normalisation (D^2) and the pCN update (2 x 4 D^2) -- 83,200 at D = 16.
    The kernel's extra arithmetic for accuracy (the refinement of U, the error-free products,
    the split accumulations) is implementation overhead and is not counted."""
    qr = 8 * D * D * (D - 1)
    w = 8 * D ** 3
    rho = 4 * D * D * (D + 1)
    norm = D * D
    pcn = 2 * 4 * D * D
    return qr + w + rho + norm + pcn


def project_flops(D, KD):
    """Algorithmic FLOPs of the contraction q = vec_h(rho) . P per chain (2 d KD)."""
    return 2 * D * D * KD


def project_issued_flops(D, KD_tc, split=3):
    """bf16 tensor FLOPs issued per chain: rho split into `split` terms, KD padded to KD_tc."""
    return split * 2 * D * D * KD_tc


def propose_bytes(D, tc):
    """HBM bytes per chain-step: read y, write y', write the packed rho (+ its bf16 split), trace."""
    n = 4 * D * D
    return 4 * n + 4 * n + 4 * D * D + (6 * D * D if tc else 0) + 8


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}, \
            "fallback"


class Clocks:
    """Samples nvidia-smi clocks and throttle reasons in the background."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.samples = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                self.samples.append(parts)

    def stop(self):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        if self.thread is not None:
            self.thread.join(timeout=2)

    def summary(self):
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None
        sm = [v for v in (num(s[1]) for s in self.samples) if v is not None]
        mx = [v for v in (num(s[2]) for s in self.samples) if v is not None]
        pw = [v for v in (num(s[3]) for s in self.samples) if v is not None]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for s in self.samples:
            for name, v in zip(names, s[5:9]):
                if v.strip().lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "power_w_max": max(pw) if pw else None, "reasons": sorted(reasons), "samples": len(self.samples)}


def _dist():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def _barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def _max_over_ranks(v, world):
    if world == 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([v], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def time_form(qst, prob, precision, steps, warmup, world, chain_offset):
    """Device-timed steps of one form; inputs (chain state, projectors, counts) resident in HBM.

    The timed region runs the library's default path: one CUDA-graph launch per step (the
    warm-up captures the graph).  A second pass of the same number of steps then runs with
    per-kernel CUDA events recorded on the launching stream around plain launches; it gives
    each kernel's average launch duration (the rooflines and the breakdown) and its own step
    time, which carries the events' and the plain launches' overhead."""
    import torch
    s = qst.Sampler(prob, precision=precision, chain_offsets=[chain_offset])
    s.run_chains(warmup)
    torch.cuda.synchronize()
    launches0 = s.launch_count()
    stream = torch.cuda.current_stream()
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    _barrier(world)
    torch.cuda.synchronize()
    start.record(stream)
    s.run_chains(steps)
    stop.record(stream)
    torch.cuda.synchronize()
    _barrier(world)
    ms = start.elapsed_time(stop)
    launches = s.launch_count() - launches0
    # per-kernel pass
    s.set_profiling(True)
    for k in range(4):
        s.kernel_time(k, reset=True)
    start.record(stream)
    s.run_chains(steps)
    stop.record(stream)
    torch.cuda.synchronize()
    ms_profiled = start.elapsed_time(stop)
    kernel_ms = {qst.KERNEL_NAMES[k]: s.kernel_time(k) for k in range(4)}
    s.set_profiling(False)
    return s, ms, launches, kernel_ms, ms_profiled


def time_handle(qst, probs, precision, steps, warmup, keep=False, **cfg):
    """ms per step of one handle over `probs` (device-timed, steps after warmup); with `keep`
    the sampler is returned too, still open."""
    import torch
    s = qst.Sampler(probs, precision=precision, diag_chains=0, **cfg)
    s.run_chains(warmup)
    stream = torch.cuda.current_stream()
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    start.record(stream)
    s.run_chains(steps)
    stop.record(stream)
    torch.cuda.synchronize()
    ms = start.elapsed_time(stop) / steps
    if keep:
        return ms, s
    s.close()
    return ms


def other_configs(qst, W, oracle):
    """The other workloads, measured briefly (one handle each; chain state resident), each with
    its log L error against the oracle on up to 1024 of its chains' current states (for every
    form of the projection at three qubits; by qubit count for the batch of 64 problems)."""
    out = {}
    precs = {"fp32": qst.PREC_FP32, "bf16x3": qst.PREC_BF16X3, "tf32": qst.PREC_TF32, "tf32x2": qst.PREC_TF32X2,
             "pauli": qst.PREC_PAULI}
    for c, form, steps in [(1, "fp32", 2000), (2, "fp32", 1000), (3, "fp32", 300), (3, "bf16x3", 300),
                           (3, "tf32", 300), (3, "tf32x2", 300), (3, "pauli", 300)]:
        prob = W.config_problem(c)
        ms, s = time_handle(qst, prob, precs[form], steps, 5, keep=True)
        out[f"config{c}_{form}"] = {"chains": prob.num_chains, "qubits": prob.num_qubits, "ms_per_step": ms,
                                    "chain_steps_per_s": prob.num_chains / (ms / 1000.0), "steps": steps}
        # the log L error against the oracle, stated per workload (every form at three qubits)
        out[f"config{c}_{form}"]["logl_err"] = logl_error(qst, oracle, s, prob)
        if form == "fp32":   # the oracle's own throughput on a bounded sample of the same workload
            out[f"config{c}_{form}"]["oracle"] = cpu_baseline(oracle, prob, 3.0, label=f"config {c}", max_steps=2000)
        s.close()
    # 64 problems of 1..5 qubits with uneven chain counts in one handle (one
    # launch per kernel and problem per step, replayed as a CUDA graph), mixed form; the plain
    # FP32 form on the same batch for comparison (few steps: its 5-qubit projections are slow)
    batch = W.heterogeneous_batch(64)
    chains = sum(p.num_chains for p in batch)
    ms_mixed = time_handle(qst, batch, qst.PREC_BF16X3, 20, 3)
    ms_plain = time_handle(qst, batch, qst.PREC_FP32, 3, 1)
    ms_pauli = time_handle(qst, batch, qst.PREC_PAULI, 20, 3)
    # per problem the faster form (timed at creation); the log L error on the chains' states
    # after 1000 steps, with five qubits on the first-order QR (the default) and refined (qr_passes 4)
    ms_auto, s5 = time_handle(qst, batch, qst.PREC_AUTO, 20, 3, keep=True)
    s5.run_chains(1000 - 23)
    err5 = logl_error_batch(qst, oracle, s5, batch, 32, 1000)
    s5.close()
    ms_auto4, s5 = time_handle(qst, batch, qst.PREC_AUTO, 20, 3, keep=True, qr_passes=4)
    s5.run_chains(1000 - 23)
    err5_4 = logl_error_batch(qst, oracle, s5, batch, 32, 1000)
    s5.close()
    # six qubits (D = 64, 46656 projectors): the structured Pauli form is the one that covers it
    p6 = W.six_qubit_problem(num_chains=4096, num_steps=20)
    ms6, s6 = time_handle(qst, p6, qst.PREC_PAULI, 10, 3, keep=True)
    out["six_qubits_pauli"] = {"chains": p6.num_chains, "qubits": 6, "ms_per_step": ms6,
                               "chain_steps_per_s": p6.num_chains / (ms6 / 1000.0), "steps": 10,
                               "logl_err": logl_error(qst, oracle, s6, p6, nsample=8)}
    s6.close()
    out["config5_heterogeneous"] = {
        "problems": len(batch), "chains": chains,
        "qubits_hist": [sum(p.num_qubits == q for p in batch) for q in range(1, 6)],
        "ms_per_step_bf16x3": ms_mixed, "chain_steps_per_s_bf16x3": chains / (ms_mixed / 1000.0),
        "ms_per_step_fp32": ms_plain, "chain_steps_per_s_fp32": chains / (ms_plain / 1000.0),
        "ms_per_step_pauli": ms_pauli, "chain_steps_per_s_pauli": chains / (ms_pauli / 1000.0),
        "ms_per_step_auto": ms_auto, "chain_steps_per_s_auto": chains / (ms_auto / 1000.0),
        "logl_err_auto": err5,
        "ms_per_step_auto_qr4": ms_auto4, "chain_steps_per_s_auto_qr4": chains / (ms_auto4 / 1000.0),
        "logl_err_auto_qr4": err5_4}
    return out


def logl_diffs(qst, oracle, s, prob, nsample=1024, problem=0):
    """|log L_gpu - log L_oracle| on the current states of up to nsample chains of one problem
    of the handle (identical y)."""
    import torch
    st = s.get_state(problem)
    nsample = min(nsample, prob.num_chains)
    idx = np.linspace(0, prob.num_chains - 1, nsample).astype(np.int64)
    y = st["y"][idx]
    _, _, ll = s.evaluate(torch.from_numpy(y).cuda(), problem=problem, want_rho=False, want_p=False)
    torch.cuda.synchronize()
    _, _, ll_ref = oracle.evaluate(prob, y.astype(np.float64), want_rho=False, want_p=False)
    return np.abs(ll.cpu().numpy() - ll_ref)


def _err_summary(d, sample):
    return {"max_abs": float(np.max(d)), "median_abs": float(np.median(d)),
            "frac_le_1e-3": float(np.mean(d <= 1e-3)), "sample": sample}


def logl_error(qst, oracle, s, prob, nsample=1024):
    """|log L_gpu - log L_oracle| on the current states of nsample chains (identical y)."""
    d = logl_diffs(qst, oracle, s, prob, nsample)
    return _err_summary(d, f"{d.size} chains' current states")


def logl_error_batch(qst, oracle, s, probs, per_problem, steps):
    """The same over a batch handle: per_problem chains of every problem, summarised by qubit
    count."""
    by_q = {}
    for i, p in enumerate(probs):
        by_q.setdefault(p.num_qubits, []).append(logl_diffs(qst, oracle, s, p, per_problem, problem=i))
    return {f"{q}_qubits": _err_summary(np.concatenate(v), f"{per_problem} chains of each of {len(v)} problems, "
                                                            f"current states after {steps} steps")
            for q, v in sorted(by_q.items())}


def cpu_baseline(oracle, prob, seconds_target=15.0, label="config 4", max_steps=50):
    """The FP64 oracle (as it stands) on a bounded sample of the workload."""
    nthreads = oracle.num_threads()
    chains = max(16, 16 * nthreads)

    def timed(steps):
        t = time.perf_counter()
        oracle.run(prob, num_chains=chains, num_steps=steps)
        return time.perf_counter() - t

    timed(1)   # warm-up: library, threads, first touch of every buffer
    # the y0 initialisation every run repeats, measured warm and subtracted (never more than
    # half of a run, so that timing noise cannot swamp a short one)
    init = min(timed(0) for _ in range(3))
    per_step = max(timed(1) - init, 1e-6)
    steps = int(max(1, min(max_steps, (seconds_target - init) / per_step)))
    run = timed(steps)
    total = max(run - init, 0.5 * run)
    return {"value": chains * steps / total, "unit": UNIT, "cores": nthreads, "kind": "oracle",
            "sample": f"{label} problem, {chains} chains x {steps} steps (FP64 C oracle, OpenMP over chains); "
                      f"the y0 initialisation time is subtracted"}


def run_reference(args):
    """Reference arm: the FP64 oracle timed on the host cores (rank 0 only)."""
    world, rank, _ = _dist()
    if rank != 0:
        return
    import oracle
    from paper_2501_17334_gb300 import workload as W
    prob = W.config_problem(CONFIG_INDEX)
    oracle.lib()
    nthreads = oracle.num_threads()
    chains = max(16, 8 * nthreads)

    def timed(steps):
        t = time.perf_counter()
        oracle.run(prob, num_chains=chains, num_steps=steps)
        return time.perf_counter() - t

    timed(args.warmup)   # warm-up: library, threads, first touch of every buffer
    # the y0 initialisation every run repeats, measured warm; it is subtracted from the timed run
    # (but never more than half of it, so that a short run's timing noise cannot swamp it)
    init = min(timed(0) for _ in range(3))
    run = timed(args.steps)
    total = max(run - init, 0.5 * run)
    value = chains * args.steps / total
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000 * total / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": WORKLOAD + f"; each step a bounded sample of {chains} chains "
                                              f"(65536 in the GPU arm)", "chains": chains},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": nthreads, "kind": "oracle",
                             "sample": f"{chains} chains x {args.steps} steps of config 4 per timed run"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_profile_case(args):
    """A short run of the headline form (or, with --qubits 5 or 6, the five- or six-qubit problem) for ncu
    captures (no timing)."""
    import torch
    from paper_2501_17334_gb300 import qst, workload as W
    qst.load()
    prec = {"fp32": qst.PREC_FP32, "bf16x3": qst.PREC_BF16X3, "pauli": qst.PREC_PAULI}[args.form]
    # the fixed column-group rule (no autotuner timing pass): a profiler distorts the timings
    # the autotuner compares, and with it the captured kernel's schedule
    if args.qubits == 6:
        prob = W.six_qubit_problem(num_chains=args.chains)
    elif args.qubits == 5:
        prob = W.five_qubit_problem(num_chains=args.chains)
    else:   # the 1- to 4-qubit workloads (4: the headline's)
        prob = W.config_problem(args.qubits, num_chains=args.chains)
    s = qst.Sampler(prob, precision=prec, diag_chains=0, autotune=0, qr_passes=args.qr_passes)
    s.run_chains(args.steps)
    s.synchronize()
    torch.cuda.synchronize()
    print(json.dumps({"profile_case": True, "chains": args.chains, "steps": args.steps, "form": args.form,
                      "qubits": prob.num_qubits, "qr_passes": args.qr_passes}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=400)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--chains", type=int, default=CHAINS)
    ap.add_argument("--form", default="bf16x3", choices=["bf16x3", "fp32", "pauli"])
    ap.add_argument("--profile-case", action="store_true")
    ap.add_argument("--qubits", type=int, default=4, choices=[1, 2, 3, 4, 5, 6], help="profile case: the 1- to 4-qubit "
                    "workloads (4: the headline's), the five- or the six-qubit problem")
    ap.add_argument("--qr-passes", type=int, default=3, choices=[2, 3, 4],
                    help="profile case: the QR setting (4: five qubits refined too)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-plain", action="store_true")
    ap.add_argument("--no-pauli", action="store_true", help="skip the structured Pauli form")
    ap.add_argument("--no-configs", action="store_true", help="skip the brief runs of the other workloads")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
        return
    if args.profile_case:
        run_profile_case(args)
        return

    import torch
    world, rank, local = _dist()
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    from paper_2501_17334_gb300 import qst, workload as W
    qst.load()
    chains = args.chains
    from paper_2501_17334_gb300 import shard
    prob = W.config_problem(CONFIG_INDEX, num_chains=chains)
    offset, _ = shard.chain_range(rank, world, world * chains)   # weak scaling: `chains` per rank
    peaks, peak_src = _peaks()
    D, KD = prob.dim, prob.num_povms * prob.dim

    forms = [("bf16x3", qst.PREC_BF16X3)]
    if not args.no_plain:
        forms.append(("fp32", qst.PREC_FP32))
    if not args.no_pauli:
        forms.append(("pauli", qst.PREC_PAULI))

    clocks = Clocks(local)
    results = {}
    clocks.start()
    time.sleep(0.3)
    for name, prec in forms:
        s, ms, launches, kms, ms_prof = time_form(qst, prob, prec, args.steps, args.warmup, world, offset)
        ms = _max_over_ranks(ms, world)
        results[name] = {"ms": ms, "launches": launches, "kernels": kms, "ms_profiled": ms_prof, "sampler": s}
    clocks.stop()
    head_name = forms[0][0]
    head = results[head_name]
    total_chain_steps = chains * args.steps * world
    value = total_chain_steps / (head["ms"] / 1000.0)

    # rooflines: the dominant kernel of the headline form, and the tensor-core projection
    sm_mhz = peaks.get("sm_max_mhz", 2070.0)
    fp32_peak = 152 * 128 * 2 * sm_mhz * 1e6 / 1e12
    kms = head["kernels"]

    def kernel_avg_s(name):
        ms_, n_ = kms[name]
        return ms_ / 1000.0 / max(n_, 1)

    def roof_propose():
        t = kernel_avg_s("propose")
        ach = propose_flops(D) * chains / t / 1e12
        traffic = ncu_traffic("propose", chains)
        return {"bound": "alu", "achieved": ach, "peak": fp32_peak, "unit": "TFLOP/s", "frac": ach / fp32_peak,
                "traffic": traffic, "kernel": "propose",
                "algorithmic_flops_per_chain_step": propose_flops(D),
                "algorithmic_bytes": propose_bytes(D, True) * chains,
                "hbm_achieved_gbs": propose_bytes(D, True) * chains / t / 1e9,
                "peak_source": "FP32 FFMA: 152 SMs x 128 lanes x 2 FLOP x max SM clock (recipe's unit counts); "
                               "achieved counts the method's FLOPs only (QR, W, W W^dag, normalisation, pCN)"}

    def roof_project():
        t = kernel_avg_s("project")
        ach = project_flops(D, KD) * chains / t / 1e12
        issued = project_issued_flops(D, -(-KD // 128) * 128) * chains / t / 1e12
        peak = peaks.get("bf16_tflops", peaks.get("bf16_tflops_sustained"))
        return {"bound": "tensor", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
                "traffic": ncu_traffic("project", chains), "kernel": "project (tcgen05 BF16x3)",
                "issued_tflops": issued, "issued_frac": issued / peak,
                "peak_source": f"{peak_src} bf16 burst (cuBLAS, a kernel timed by events); achieved = 2 d KD per "
                               f"chain-step (algorithmic, at most 1/3 of peak with three bf16 splits); issued = 3 "
                               f"splits x 2 d KD_tc, the tensor pipe's own work"}

    dom = max(kms, key=lambda k: kms[k][0])
    roof = roof_propose() if dom == "propose" else roof_project()

    import oracle
    err = logl_error(qst, oracle, head["sampler"], prob)
    err["form"] = head_name
    err_plain = None
    if "fp32" in results:
        err_plain = logl_error(qst, oracle, results["fp32"]["sampler"], prob)
    err_pauli = None
    if "pauli" in results:
        err_pauli = logl_error(qst, oracle, results["pauli"]["sampler"], prob)

    # end to end through the C ABI with host buffers: qst_create from host counts and
    # projectors (H2D), run, read the posterior mean back (D2H)
    for r in results.values():
        r["sampler"].close()
    torch.cuda.synchronize()
    _barrier(world)
    t0 = time.perf_counter()
    s = qst.Sampler(prob, precision=forms[0][1], chain_offsets=[offset])
    s.run_chains(args.steps)
    if world > 1:   # the one exchange of the path: merge the raw pooled FP64 sums of all ranks
        psum, npool = s.posterior_sum()
        mean, npool = shard.merge_posterior_sum(psum, npool)
    else:
        mean, npool = s.posterior_mean()
    t1 = time.perf_counter()
    s.close()
    e2e_s = _max_over_ranks(t1 - t0, world)
    h2d = prob.counts.nbytes + prob.povm_re.nbytes + prob.povm_im.nbytes
    e2e = {"value": chains * args.steps * world / e2e_s, "unit": UNIT,
           "h2d_bytes_per_step": h2d / args.steps, "d2h_bytes_per_step": 2 * 8 * D * D / args.steps,
           "includes": "qst_create (validation, packing, upload, y0 init) + run + posterior-mean read-back"
                       + (" + merge over ranks" if world > 1 else "")}

    line = {
        "metric": METRIC, "value": value, "unit": UNIT,
        # the accuracy the metric is quoted at, first so that a truncated log still shows it
        "logl_err_bf16x3": {k: err[k] for k in ("max_abs", "median_abs", "frac_le_1e-3")},
        "logl_err_fp32": None if err_plain is None else {k: err_plain[k] for k in ("max_abs", "median_abs",
                                                                                  "frac_le_1e-3")},
        "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": head["ms"] / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+bf16x3", "data": "synthetic",
        "config": {"workload": WORKLOAD, "chains_per_gpu": chains, "form": head_name,
                   "l2": "chain state 0.6 GB/GPU > 129 MB L2: every step streams it from HBM"},
        "logl_err": err,
        "forms": {n: {"value": total_chain_steps / (r["ms"] / 1000.0), "ms_per_step": r["ms"] / args.steps,
                      "kernel_ms_per_step": {k: v[0] / args.steps for k, v in r["kernels"].items()},
                      "kernel_timing_pass_ms_per_step": r["ms_profiled"] / args.steps}
                  for n, r in results.items()},
        "kernel_timing": "a second pass of the same steps right after the timed one, plain launches with "
                         "per-kernel CUDA events on the launching stream (the timed region itself replays "
                         "one CUDA graph per step)",
        "roofline": roof,
        "roofline_tensor": roof_project(),
        "clocks": clocks.summary(),
        "gpu_launches": head["launches"],
        "e2e": e2e,
    }
    if err_plain is not None:
        line["forms"]["fp32"]["logl_err"] = err_plain
        line["speedup_vs_plain_fp32"] = results["fp32"]["ms"] / head["ms"]
    if err_pauli is not None:
        line["forms"]["pauli"]["logl_err"] = err_pauli
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(oracle, prob)
    if world == 1 and not args.no_configs:
        line["configs"] = other_configs(qst, W, oracle)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
