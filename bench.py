#!/usr/bin/env python
"""PANDA message-passing throughput on one GB300 (and N independent replicas).

One step = one message-passing iteration (Eqs. 2-7: the four Tanimoto
products, the W, P, C updates, the diagonals and h) of the human-sized
network: 1000 TFs x 17000 genes, synthetic priors shaped like the paper's
(motif prior W Bernoulli(0.05), PPI prior P Bernoulli(0.01) with unit
diagonal, C the Pearson correlation of 200 samples from 20 latent factors),
alpha = 0.1.  C alone is 1.16 GB, far larger than L2, so no L2 flush is
needed between iterations.

Prints one JSON line.  ``value`` is iterations/s summed over ranks, timed with
CUDA events on the library's stream with the inputs already in HBM; ``e2e``
is the same metric through the C ABI from pinned host buffers, the
host-to-device copy of the inputs and the read-back of the networks inside
the timed region.  ``--impl reference`` times the FP64 oracle on the host
cores on a bounded sample of the same iteration instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1507_07039_gb300 import synth  # noqa: E402

METRIC = "PANDA iterations/s + TFLOP/s, BF16-split vs FP32, at max|ΔW|≤1e-4 vs FP64"
PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "traffic.json")
FALLBACK = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}
ALPHA = 0.1
GRAPH_ITERS = 8  # iterations per captured graph launch (the library's default)


# ---------------------------------------------------------------------------
# distributed plumbing (N > 1: independent replicas, no data-path collective)
# ---------------------------------------------------------------------------

def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def dist_init(world: int, backend: str = "nccl"):
    if world > 1:
        import torch.distributed as dist
        if not dist.is_initialized():
            os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
            dist.init_process_group(backend)


def barrier(world: int):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int, device=None) -> float:
    """Max of a float over all ranks (the slowest rank sets the job's time)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id: str | None):
        self.gpu_id = gpu_id
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        cmd = ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200"]
        if self.gpu_id is not None:
            cmd += ["-i", self.gpu_id]
        try:
            self.proc = subprocess.Popen(cmd, stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self) -> dict | None:
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def gpu_id_for(device_index: int) -> str | None:
    try:
        import torch
        p = torch.cuda.get_device_properties(device_index)
        return f"{p.pci_domain_id:08X}:{p.pci_bus_id:02X}:{p.pci_device_id:02X}.0"
    except Exception:
        return None


# ---------------------------------------------------------------------------
# workload accounting
# ---------------------------------------------------------------------------

def algorithmic_flops(T: int, G: int) -> float:
    """Flops one iteration must do: W.C (2TG^2), P.W (2T^2 G), and the symmetric
    halves of W'^T.W' (TG^2) and W'.W'^T (T^2 G)."""
    return 3.0 * T * G * G + 3.0 * T * T * G


def kernel_algorithmic_work(name: str, T: int, G: int) -> tuple[float, str]:
    """Algorithmic flops one launch of a kernel does, and the unit."""
    if name in ("k_tc_phase1", "k_f32_phase1"):  # both products of phase 1 in one launch
        return 2.0 * T * G * G + 2.0 * T * T * G, "flop"
    if name in ("k_tc_phase2", "k_f32_phase2"):  # symmetric halves of both similarity products
        return 1.0 * T * G * G + 1.0 * T * T * G, "flop"
    return 0.0, "flop"


def kernel_split_work(name: str, T: int, G: int) -> tuple[float, float]:
    """A tensor-core launch's algorithmic flops split into the gene-sized
    products (W.C, W^T.W) and the TF-sized ones (P.W, W.W^T)."""
    if name in ("k_tc_phase1", "k_f32_phase1"):
        return 2.0 * T * G * G, 2.0 * T * T * G
    if name in ("k_tc_phase2", "k_f32_phase2"):
        return 1.0 * T * G * G, 1.0 * T * T * G
    return 0.0, 0.0


def prec_code(panda, name: str) -> int:
    return {"fp32": panda.PANDA_FP32, "bf16x3": panda.PANDA_BF16X3, "bf16x2": panda.PANDA_BF16X2,
            "fp8mix": panda.PANDA_FP8MIX}[name]


def load_peaks() -> tuple[dict, str]:
    try:
        return json.load(open(PEAKS_FILE)), "measured"
    except (OSError, ValueError):
        return dict(FALLBACK), "fallback"


def traffic_for(kernel: str, workload: str) -> float | None:
    """DRAM bytes per launch from a committed ncu capture, if the kernel's
    source is unchanged since it was taken."""
    try:
        rec = json.load(open(TRAFFIC_FILE))[f"{kernel}@{workload}"]
    except (OSError, ValueError, KeyError):
        return None
    src = os.path.join(ROOT, "paper_1507_07039_gb300", "csrc", rec["source"])
    try:
        sha = hashlib.sha256(open(src, "rb").read()).hexdigest()[:16]
    except OSError:
        return None
    return float(rec["bytes_per_launch"]) if sha == rec["source_sha"] else None


def tensor_peak(peaks: dict, peak_src: str, ck: dict | None, timed_ms: float) -> tuple[float, str]:
    """The BF16 dense peak that applies to a kernel timed inside the bench's
    timed region: the burst figure when that region ran at the maximum SM
    clock and lasted under a second, else the sustained (power-capped) one."""
    burst = peaks.get("bf16_tflops", FALLBACK["bf16_tflops"])
    sustained = peaks.get("bf16_tflops_sustained", FALLBACK["bf16_tflops_sustained"])
    mx = (ck or {}).get("sm_max_mhz") or peaks.get("sm_max_mhz", 2070.0)
    sm = (ck or {}).get("sm_mhz")
    if sm is not None and sm >= 0.97 * mx and timed_ms < 1000.0:
        return burst, (f"bf16 dense burst ({peak_src}): the timed region lasted {timed_ms:.0f} ms "
                       f"at a median {sm:.0f} MHz of {mx:.0f}")
    why = "no clock record" if sm is None else f"median {sm:.0f} MHz, {timed_ms:.0f} ms timed"
    return sustained, f"bf16 dense sustained ({peak_src}; {why})"


def kernel_flops(panda, prec: int, name: str, T: int, G: int) -> tuple[float, float, float]:
    """(useful flops, issued tensor flops, issued flops in BF16-MMA time
    units) of one launch of a tensor-core kernel: FP32 issues six MMAs per
    product (its operands' exact three-way BF16 splits), BF16X3 three, BF16X2
    two; FP8MIX runs the gene-sized products as one E4M3 MMA,
    which takes half the time of a BF16 one, and the TF-sized ones as BF16X3."""
    useful = kernel_algorithmic_work(name, T, G)[0]
    big, small = kernel_split_work(name, T, G)
    if prec == panda.PANDA_FP8MIX:
        return useful, big + 3.0 * small, 0.5 * big + 3.0 * small
    terms = {panda.PANDA_FP32: 6.0, panda.PANDA_BF16X3: 3.0}.get(prec, 2.0)
    return useful, terms * useful, terms * useful


def roofline(panda, prec, kstats, T, G, wl_name, peaks, peak_src, ck, timed_ms, ffma, iters_per_s):
    """The bench line's roofline object: the dominant kernel against the peak
    of its pipe, every product kernel beside it, and the whole iteration.
    ffma: the measured FP32 FMA rate, reported beside the FP32 mode's figures
    (whose products run on the tensor cores)."""
    top = max(kstats, key=lambda k: k[1])
    work, _ = kernel_algorithmic_work(top[0], T, G)
    avg_s = top[1] / top[2] / 1000.0
    hbm = peaks.get("hbm_gbs", FALLBACK["hbm_gbs"])
    bf16, src = tensor_peak(peaks, peak_src, ck, timed_ms)
    fp8 = prec == panda.PANDA_FP8MIX
    peak = 2.0 * bf16 if fp8 else bf16
    if fp8:
        src = "e4m3 dense = 2 x " + src + " (nominal ratio)"
    per_kernel = []
    issued_units_iter = 0.0
    for name, ms_tot, launches in kstats:
        useful, issued, units = kernel_flops(panda, prec, name, T, G)
        if not useful or not launches:
            continue
        t = ms_tot / launches / 1000.0
        traffic = traffic_for(name, wl_name)
        per_kernel.append({
            "kernel": name, "ms_avg": round(1000.0 * t, 5),
            "useful_tflops": useful / t / 1e12, "issued_tensor_tflops": issued / t / 1e12,
            "useful_frac": useful / t / 1e12 / peak,
            # issued MMAs against the BF16 peak (E4M3 MMAs counted at half a BF16 MMA's time)
            "issued_frac": units / t / 1e12 / bf16,
            "traffic": traffic, "hbm_gbs": None if traffic is None else traffic / t / 1e9,
            "hbm_frac": None if traffic is None else traffic / t / 1e9 / hbm})
        issued_units_iter += units
    useful_iter = algorithmic_flops(T, G)
    roof = {"bound": "tensor", "achieved": work / avg_s / 1e12, "peak": peak, "unit": "TFLOP/s",
            "peak_source": src, "kernel": top[0],
            "issued_tensor_tflops": kernel_flops(panda, prec, top[0], T, G)[1] / avg_s / 1e12}
    roof["frac"] = roof["achieved"] / roof["peak"]
    roof["traffic"] = traffic_for(top[0], wl_name)
    roof["kernels"] = per_kernel
    roof["iteration"] = {
        "useful_tflops": useful_iter * iters_per_s / 1e12,
        "useful_frac": useful_iter * iters_per_s / 1e12 / peak,
        "issued_frac": issued_units_iter * iters_per_s / 1e12 / bf16,
        "note": "useful = 3TG^2 + 3T^2G flop per iteration; issued counts every MMA the split issues"}
    roof["hbm_peak_gbs"] = hbm
    if prec == panda.PANDA_FP32:
        roof["ffma_peak_tflops"] = ffma
    return roof


# ---------------------------------------------------------------------------
# CPU baseline: the FP64 oracle on a bounded sample of one iteration
# ---------------------------------------------------------------------------

class OracleSample:
    """Times the oracle on a fraction f of one iteration of the workload: f*T
    rows of W' (Eqs. 2-4), f*T rows of P' and f*G rows of C' (Eq. 5; their
    inputs are the current W standing in for W', the same operation count).
    The diagonals and h (Eqs. 6-7) are O(T^2 + G^2 + TG) and not sampled.
    Seconds per iteration = sampled seconds / f."""

    def __init__(self, W0, P0, C0, threads: int):
        from oracle.oracle import Oracle
        self.orc = Oracle()
        self.orc.set_threads(threads)
        self.threads = threads
        self.W, self.P, self.C = self.orc.normalize(W0, P0, C0)
        self.T, self.G = self.W.shape
        self.cursor = 0

    def run(self, frac: float) -> float:
        """Seconds per full iteration estimated from one sample of size frac."""
        rT, rG = max(1, round(frac * self.T)), max(1, round(frac * self.G))
        rows_t = (self.cursor + np.arange(rT)) % self.T
        rows_g = (self.cursor + np.arange(rG)) % self.G
        self.cursor += rT
        a = float(np.float32(ALPHA))  # the library takes alpha as FP32
        t0 = time.perf_counter()
        self.w_rows = self.orc.w_rows(self.W, self.P, self.C, a, rows_t)
        self.rows = rows_t
        t1 = time.perf_counter()
        self.orc.p_rows(self.W, self.P, a, rows_t)
        t2 = time.perf_counter()
        self.orc.c_rows(self.W, self.C, a, rows_g)
        t3 = time.perf_counter()
        return (t1 - t0) / (rT / self.T) + (t2 - t1) / (rT / self.T) + (t3 - t2) / (rG / self.G)


def cpu_threads() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def accuracy_sample(panda, s, W0, P0, C0, prec, n_rows: int = 100) -> dict:
    """Errors of the first iteration against the FP64 oracle, for the metric's
    gate: rows of W' (the oracle's own Eqs. 2-4 on the rows the CPU sample
    computed), and whole rows of P' and C' with their diagonals (the oracle's
    Eqs. 5-6 given the GPU's W', widened to FP64: W' differs from the oracle's
    by about 1e-5, which moves a P' or C' entry by about 1e-6 of its scale, far
    below the step's own error).  Off-diagonal errors are relative to the row's
    largest entry (at least 1), diagonal errors relative to the entry."""
    with panda.PandaContext(W0, P0, C0, prec=prec) as ctx:
        ctx.step(ALPHA)
        gW, gP, gC = ctx.get()
    orc, a = s.orc, float(np.float32(ALPHA))
    T, G = gW.shape
    errW = float(np.max(np.abs(gW[s.rows].astype(np.float64) - s.w_rows)))
    Wn = gW.astype(np.float64)
    rng = np.random.default_rng(11)
    out = {"W": errW}
    for name, X, gX, rows_of, mult, n in (("P", s.P, gP, orc.p_rows, G, T), ("C", s.C, gC, orc.c_rows, T, G)):
        rows = np.sort(rng.choice(n, min(n_rows, n), replace=False))
        o = rows_of(Wn, X, a, rows)
        eo, ed = 0.0, 0.0
        for q, i in enumerate(rows):
            off = np.arange(n) != i
            scale = max(1.0, float(np.max(np.abs(o[q][off])))) if n > 1 else 1.0
            if n > 1:
                eo = max(eo, float(np.max(np.abs(gX[i][off] - o[q][off]))) / scale)
            d = orc.diag_value(o[q], i, mult, X[i, i], a, 1)
            ed = max(ed, abs(float(gX[i, i]) - d) / max(1.0, abs(d)))
        out[name + "off"], out[name + "diag"] = eo, ed
    return {"max_abs_dW_vs_fp64_oracle": errW, "errors": out, "gate": 1e-4, "within_gate": errW <= 1e-4,
            "iteration": 1, "W_rows": int(len(s.rows)), "P_rows": min(n_rows, T), "C_rows": min(n_rows, G),
            "of": [T, G], "P_C_reference": "oracle Eqs. 5-6 applied to the GPU's W' (FP64-widened)",
            "trajectory_errors": "whole converging runs at T = 1000 are checked by the GPU tests"}


# ---------------------------------------------------------------------------
# the two arms
# ---------------------------------------------------------------------------

def run_reference(args, wl, rank, world):
    if rank != 0:
        return
    W0, P0, C0 = synth.make_inputs(wl)
    threads = cpu_threads()
    s = OracleSample(W0, P0, C0, threads)
    frac = args.ref_frac
    for _ in range(args.warmup):
        s.run(frac)
    t0 = time.perf_counter()
    est = [s.run(frac) for _ in range(args.steps)]
    wall = time.perf_counter() - t0
    sec_per_iter = float(np.median(est))
    value = 1.0 / sec_per_iter
    sample = (f"each step: {max(1, round(frac * wl.T))} rows of W', {max(1, round(frac * wl.T))} rows "
              f"of P', {max(1, round(frac * wl.G))} rows of C' (fraction {frac} of one iteration), "
              f"scaled to a full iteration")
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": "iterations/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * wall / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": wl.name, "T": wl.T, "G": wl.G, "alpha": ALPHA,
                   "step": "sampled fraction of one message-passing iteration", "parallelism": "none"},
        "cpu_baseline": {"value": value, "unit": "iterations/s", "cores": threads, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": "iterations/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


# Under the default diagonal rule the diagonals of P and C grow like e^{2 alpha t}
# (Eq. 6), so with tol = 0 their squared norms leave FP32 after 131-140
# iterations at 1600 x 30000, 141-150 at 1000 x 17000, 191-200 at 64 x 256
# (alpha = 0.1, measured; the method itself stops on h after 12-20).  Longer
# measurements are made of segments of at most SEG iterations, each restarted
# from the Z-scored start state at t = 0.
SEG = 100
# Networks of a set with few TFs and many genes reach that limit first: after
# 66-70 iterations for T ~ 240-300, G ~ 15000-17000 (measured over set64);
# a set's warm-up (SET_WARM: the 25 schedule trials and one captured chunk)
# plus one segment stays within 60.
SET_WARM = 34
SEG_SET = 26


def segments(n: int) -> list[int]:
    out = []
    while n > 0:
        out.append(min(SEG, n))
        n -= out[-1]
    return out


def launched_iterations(steps: int) -> int:
    """Iterations whose kernels the timed graphs launch: whole graphs per
    segment (those past a segment's last iteration return at once)."""
    return sum(-(-n // GRAPH_ITERS) * GRAPH_ITERS for n in segments(steps))


def start_state(panda, torch, ctx, T, G, device):
    """The context's networks at t = 0, kept on the device for restarts."""
    st = [torch.empty(s, dtype=torch.float32, device=device) for s in ((T, G), (T, T), (G, G))]
    panda.panda_get_device(ctx.h, *st)
    torch.cuda.synchronize()
    return st


def time_gpu(panda, torch, W0, P0, C0, prec, steps, warmup, world, local_rank, with_clocks):
    """Device-timed iterations/s of one context (inputs resident in HBM): the
    sum over segments of CUDA-event spans around panda_run, each segment's
    restart and graph capture outside its span."""
    T, G = W0.shape
    ctx = panda.PandaContext(W0, P0, C0, prec=prec, graph_iters=GRAPH_ITERS)
    st = start_state(panda, torch, ctx, T, G, torch.device("cuda", local_rank))
    for k, n in enumerate(segments(warmup)):
        if k:
            panda.panda_set_state_device(ctx.h, *st, 0)
        ctx.run(ALPHA, 0.0, n)
    panda.panda_set_profiling(ctx.h, True)
    stream = torch.cuda.ExternalStream(ctx.stream)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(gpu_id_for(local_rank)) if with_clocks else None
    barrier(world)
    torch.cuda.synchronize()
    if clocks:
        clocks.start()
        time.sleep(0.6)  # let the sampler take its first reading
    ms, acc = 0.0, {}
    for n in segments(steps):
        panda.panda_set_state_device(ctx.h, *st, 0)
        ctx.run(ALPHA, 0.0, 1)  # capture the graphs (one per W buffer parity) outside the timed span
        ctx.run(ALPHA, 0.0, 1)
        panda.panda_set_profiling(ctx.h, True)  # (already on: only clears the per-kernel sums)
        torch.cuda.synchronize()
        e0.record(stream)
        conv, got, h = ctx.run(ALPHA, 0.0, n)
        e1.record(stream)
        e1.synchronize()
        assert got == n, (got, n)
        ms += e0.elapsed_time(e1)
        for i in range(panda.panda_kernel_count(ctx.h)):
            name, kms, launches = panda.panda_kernel_stats(ctx.h, i)
            a = acc.setdefault(name, [0.0, 0])
            a[0] += kms
            a[1] += launches
    torch.cuda.synchronize()
    ck = clocks.stop() if clocks else None
    barrier(world)
    kstats = [(name, a[0], a[1]) for name, a in acc.items()]
    layout = panda.panda_phase1_layout(ctx.h) if prec != panda.PANDA_FP32 else None
    ctx.close()
    return ms, kstats, ck, layout


def run_segments(panda, torch, ctx, steps, T, G, device) -> float:
    """steps iterations, restarted from the start state every SEG iterations.
    Returns the seconds spent on the restarts (the start-state snapshot and
    each panda_set_state_device, timed between device syncs): bench-only work
    that the end-to-end figure leaves out."""
    segs = segments(steps)
    overhead = 0.0
    st = None
    if len(segs) > 1:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        st = start_state(panda, torch, ctx, T, G, device)
        overhead += time.perf_counter() - t0
    for k, n in enumerate(segs):
        if k:
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            panda.panda_set_state_device(ctx.h, *st, 0)
            torch.cuda.synchronize()
            overhead += time.perf_counter() - t0
        ctx.run(ALPHA, 0.0, n)
    return overhead


def time_e2e(panda, torch, W0, P0, C0, prec, steps):
    """Through the C ABI from pinned host buffers: create (H2D + normalise),
    steps iterations, read back W, P, C (D2H)."""
    T, G = W0.shape
    pin = [torch.empty(x.shape, dtype=torch.float32, pin_memory=True).numpy() for x in (W0, P0, C0)]
    for dst, src in zip(pin, (W0, P0, C0)):
        np.copyto(dst, src)
    outs = [torch.empty(x.shape, dtype=torch.float32, pin_memory=True).numpy() for x in (W0, P0, C0)]
    device = torch.device("cuda", torch.cuda.current_device())
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ctx = panda.PandaContext(*pin, prec=prec)
    restarts = run_segments(panda, torch, ctx, steps, T, G, device)
    panda.panda_get_into(ctx.h, *outs)
    t1 = time.perf_counter()
    ctx.close()
    return t1 - t0 - restarts, sum(x.nbytes for x in pin) / steps, sum(x.nbytes for x in outs) / steps


def time_e2e_expression(panda, torch, wl, prec, steps):
    """As time_e2e, starting from the expression data instead of C0: the
    co-regulation prior is computed on the GPU (Sec. II-A), so the host sends
    W0, P0 and the G x N expression matrix."""
    W0, P0, X = synth.make_expression(wl)
    pin = [torch.empty(x.shape, dtype=torch.float32, pin_memory=True).numpy() for x in (W0, P0, X)]
    for dst, src in zip(pin, (W0, P0, X)):
        np.copyto(dst, src)
    T, G = W0.shape
    outs = [torch.empty(s, dtype=torch.float32, pin_memory=True).numpy() for s in ((T, G), (T, T), (G, G))]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ctx = panda.PandaContext.from_expression(*pin, prec=prec)
    t1 = time.perf_counter()
    restarts = run_segments(panda, torch, ctx, steps, T, G, torch.device("cuda", torch.cuda.current_device()))
    panda.panda_get_into(ctx.h, *outs)
    t2 = time.perf_counter()
    ctx.close()
    return t2 - t0 - restarts, t1 - t0, sum(x.nbytes for x in pin) / steps, sum(x.nbytes for x in outs) / steps


def run_ours(args, wl, rank, world, local_rank):
    import torch
    torch.cuda.set_device(local_rank)
    dist_init(world)
    from paper_1507_07039_gb300 import panda
    prec = prec_code(panda, args.prec)
    W0, P0, C0 = synth.make_inputs(wl)
    T, G = wl.T, wl.G

    ms, kstats, ck, layout = time_gpu(panda, torch, W0, P0, C0, prec, args.steps, args.warmup, world,
                                      local_rank, rank == 0)
    ms_max = max_over_ranks(ms, world, torch.device("cuda", local_rank))
    value = world * args.steps / (ms_max / 1000.0)

    # the other precision on the same GPU, for the BF16-split vs FP32 comparison
    other = None
    if args.compare and prec != panda.PANDA_FP32:
        ms32, _, _, _ = time_gpu(panda, torch, W0, P0, C0, panda.PANDA_FP32, max(5, args.steps // 4),
                              args.warmup, world, local_rank, False)
        other = {"fp32_iters_per_s": world * max(5, args.steps // 4) / (max_over_ranks(ms32, world, torch.device("cuda", local_rank)) / 1000.0)}
        if prec == panda.PANDA_BF16X3:  # the lower-precision modes beside it (their errors: tests, notes)
            for name, code in (("bf16x2", panda.PANDA_BF16X2), ("fp8mix", panda.PANDA_FP8MIX)):
                ms2, _, _, _ = time_gpu(panda, torch, W0, P0, C0, code, max(5, args.steps // 2),
                                     args.warmup, world, local_rank, False)
                other[name + "_iters_per_s"] = world * max(5, args.steps // 2) / (
                    max_over_ranks(ms2, world, torch.device("cuda", local_rank)) / 1000.0)

    # dominant kernel and its roofline
    peaks, peak_src = load_peaks()
    tot = sum(k[1] for k in kstats) or 1.0
    kernels = {k[0]: {"launches": k[2], "ms_total": round(k[1], 4),
                      "ms_avg": round(k[1] / k[2], 5) if k[2] else None, "share": round(k[1] / tot, 4)}
               for k in kstats}
    ffma = None
    try:
        ffma = panda.panda_measure_ffma_peak()
    except panda.PandaError:
        pass
    roof = roofline(panda, prec, kstats, T, G, wl.name, peaks, peak_src, ck, ms, ffma,
                    value / world)

    e2e = None
    if args.e2e:
        sec, bi, bo = time_e2e(panda, torch, W0, P0, C0, prec, args.steps)
        sec = max_over_ranks(sec, world, torch.device("cuda", local_rank))
        e2e = {"value": world * args.steps / sec,
               "unit": "iterations/s", "h2d_bytes_per_step": bi, "d2h_bytes_per_step": bo,
               "note": "create from pinned host buffers (H2D + validation + Z-score), the iterations, "
                       "read-back of W, P, C (D2H); per-step bytes = totals / steps; runs of more than "
                       f"{SEG} steps restart from the start state every {SEG} iterations (the diagonals' "
                       "e^(2 alpha t) growth) and leave those restarts out of the time"}
        if wl.n_samples > 0:  # the same from expression data: C0 computed on the GPU (Pearson, Sec. II-A)
            sec2, create2, bi2, bo2 = time_e2e_expression(panda, torch, wl, prec, args.steps)
            sec2 = max_over_ranks(sec2, world, torch.device("cuda", local_rank))
            e2e["from_expression"] = {
                "value": world * args.steps / sec2, "unit": "iterations/s", "h2d_bytes_per_step": bi2,
                "d2h_bytes_per_step": bo2, "create_s": create2,
                "note": "panda_create_from_expression from pinned W0, P0 and the expression matrix "
                        "(%d x %d), the iterations, read-back of W, P, C" % (wl.G, wl.n_samples)}

    cpu = None
    accuracy = None
    if rank == 0 and args.cpu_baseline:
        threads = cpu_threads()
        s = OracleSample(W0, P0, C0, threads)
        t0 = time.perf_counter()
        spi = s.run(args.cpu_frac)
        el = time.perf_counter() - t0
        cpu = {"value": 1.0 / spi, "unit": "iterations/s", "cores": threads, "kind": "oracle",
               "sample": f"fraction {args.cpu_frac} of one iteration ({max(1, round(args.cpu_frac * T))} rows "
                         f"of W' and of P', {max(1, round(args.cpu_frac * G))} rows of C'), "
                         f"{el:.1f} s of CPU time, scaled to a full iteration"}
        accuracy = accuracy_sample(panda, s, W0, P0, C0, prec)

    # each captured graph launches the kernels of all its iterations; those past the run's last
    # iteration return at once, so the launches are whole graphs' worth, the work is `steps`' worth
    launches = launched_iterations(args.steps) * len(kstats)
    launches_with_work = int(sum(k[2] for k in kstats))
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "iterations/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": args.prec.replace("fp32", "f32"),
            "data": "synthetic",
            "config": {"workload": wl.name, "T": T, "G": G, "alpha": ALPHA,
                       "precision": args.prec, "step": "one message-passing iteration (Eqs. 2-7)",
                       "l2": "no flush: inputs larger than L2 (C alone is %.2f GB)" % (4.0 * G * G / 1e9),
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "phase1_launch": layout,
            "useful_tflops": value / world * algorithmic_flops(T, G) / 1e12,
            "roofline": roof,
            "cpu_baseline": cpu,
            "accuracy": accuracy,
            "e2e": e2e,
            "gpu_launches": launches,
            "gpu_launches_with_work": launches_with_work,
            "clocks": ck,
            "kernels": kernels,
            "fp32_ffma_peak_tflops": ffma,
        }
        if other:
            line.update(other)
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_set(args, rank, world, local_rank):
    """A set of 64 networks of uneven size (T ~ U[200, 1000], G ~ U[2000, 17000],
    100 samples from 10 factors each), iterated together by panda_batch_run:
    value = network-iterations/s."""
    import torch
    torch.cuda.set_device(local_rank)
    dist_init(world)
    from paper_1507_07039_gb300 import panda
    prec = prec_code(panda, args.prec)
    wls = synth.set_of_networks(64)
    nets = [synth.make_inputs(w) for w in wls]
    flops = sum(algorithmic_flops(w.T, w.G) for w in wls)
    # warm-up: the schedule trials of the tensor-core set engine (one warm-up iteration, then three
    # per candidate: 22) and one captured chunk of 8, so that neither falls in the timed region
    warm = SET_WARM if prec != panda.PANDA_FP32 else min(args.warmup, SET_WARM)
    # the diagonals' e^{2 alpha t} growth (see SEG): more than SEG_SET timed iterations run as
    # segments, each on a freshly created set with its own warm-up, the creation untimed
    seg_set = min(SEG_SET, 60 - warm)
    segs = []
    left = args.steps
    while left > 0:
        segs.append(min(seg_set, left))
        left -= segs[-1]
    clocks = ClockSampler(gpu_id_for(local_rank)) if rank == 0 else None
    sec, sched = 0.0, None
    for q, n in enumerate(segs):
        with panda.PandaBatch(nets, prec=prec) as b:
            if q == len(segs) - 1:
                del nets
            b.run(ALPHA, 0.0, warm)
            torch.cuda.synchronize()
            if clocks and q == 0:
                clocks.start()
                time.sleep(0.6)
            barrier(world)
            t0 = time.perf_counter()
            conv, iters, _ = b.run(ALPHA, 0.0, n)
            torch.cuda.synchronize()
            sec += time.perf_counter() - t0
            barrier(world)
            sched = b.schedule()
        assert all(i == n for i in iters)
    sec = max_over_ranks(sec, world, torch.device("cuda", local_rank))  # replicas: the slowest rank
    ck = clocks.stop() if clocks else None
    value = world * len(wls) * args.steps / sec  # the whole job: every rank iterates its own copy of the set
    if rank == 0:
        print(json.dumps({
            "metric": "PANDA network-iterations/s over a set of networks", "value": value,
            "unit": "network-iterations/s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1000.0 * sec / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": args.prec.replace("fp32", "f32"), "data": "synthetic",
            "warmup_iterations": warm,
            "config": {"workload": "set64", "networks": len(wls), "T": [w.T for w in wls][:8] + ["..."],
                       "step": "one iteration of every network", "timing": "host clock between device syncs",
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "useful_tflops": flops * args.steps / sec / 1e12, "clocks": ck,
            "schedule": None if sched is None else {
                "phase1": sched["p1_names"][sched["p1"]], "phase2": sched["p2_names"][sched["p2"]],
                "phase1_trial_ms": dict(zip(sched["p1_names"], [round(t, 3) for t in sched["p1_ms"]])),
                "phase2_trial_ms": dict(zip(sched["p2_names"], [round(t, 3) for t in sched["p2_ms"]])),
                "trials": "median of 3 iterations per candidate"}}), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


# The paper's Table I (seconds for the whole message-passing loop, one thread,
# x86_64 MIT SuperCloud, 100 random W per size, P = C = I): context beside the
# replica below, not a target.
PAPER_TABLE1 = {125: (1.05, 0.50, 0.13), 250: (4.65, 0.62, 0.54), 500: (32.73, 2.82, 2.61),
                1000: (241.51, 15.82, 15.06), 2000: (1954.5, 98.59, 95.04)}


def run_table1(args, rank, world, local_rank):
    """Replica of the paper's Table I sweep: N_e = N_a = N, identity P and C,
    random W (density 0.05), the message-passing loop run to h < 1e-3 at
    alpha = 0.1, timed around panda_run only (create excluded, as the paper
    excludes input and output).  Per N: one network alone (host clock around
    the run, device synchronised), a batch of --table-reps such networks run
    together (per-network time = batch time / reps), and the FP64 oracle on
    the host cores, timed on a sampled fraction of one iteration and scaled by
    the iteration count."""
    import torch
    torch.cuda.set_device(local_rank)
    from paper_1507_07039_gb300 import panda
    prec = prec_code(panda, args.prec)
    threads = cpu_threads()
    rows = []
    for n in (125, 250, 500, 1000, 2000):
        nets = [synth.make_inputs(synth.table1(n, r)) for r in range(args.table_reps)]
        W0, P0, C0 = nets[0]
        with panda.PandaContext(W0, P0, C0, prec=prec) as ctx:  # warm the library and the graph
            ctx.run(ALPHA, 0.0, 2)
        with panda.PandaContext(W0, P0, C0, prec=prec) as ctx:
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            conv, iters, _ = ctx.run(ALPHA, 1e-3, 1000)
            torch.cuda.synchronize()
            single = time.perf_counter() - t0
        with panda.PandaBatch(nets, prec=prec) as b:
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            _, it_b, _ = b.run(ALPHA, 1e-3, 1000)
            torch.cuda.synchronize()
            batch = time.perf_counter() - t0
        row = {"N": n, "iterations": int(iters), "converged": bool(conv), "gpu_s": single,
               "gpu_s_per_network_in_set": batch / len(nets), "set_networks": len(nets),
               "set_iterations_mean": float(np.mean(it_b)),
               "paper_s": dict(zip(("C-code", "Octave", "MATLAB"), PAPER_TABLE1[n]))}
        if rank == 0 and args.cpu_baseline:
            frac = min(1.0, 64.0 / n)
            spi = OracleSample(W0, P0, C0, threads).run(frac)
            row["oracle_s"] = spi * iters
            row["oracle_sample"] = f"fraction {frac:.3f} of one iteration, scaled by {iters} iterations"
        rows.append(row)
    if rank == 0:
        print(json.dumps({
            "metric": "PANDA run-time of the message-passing loop (paper Table I replica)",
            "value": rows[-1]["gpu_s"], "unit": "s (N = 2000, one network)", "n_gpus": world, "steps": None,
            "warmup": 1, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": args.prec.replace("fp32", "f32"), "data": "synthetic",
            "config": {"workload": "table1", "alpha": ALPHA, "tol": 1e-3, "P, C": "identity",
                       "W": "Bernoulli(0.05), normalised", "oracle_cores": threads,
                       "paper_hardware": "MIT SuperCloud x86_64, one thread (C-code g++ -O3, Octave 3.8.2, "
                                         "MATLAB R2014a)"},
            "table": rows}), flush=True)


def main(argv=None):
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--prec", choices=["fp32", "bf16x3", "bf16x2", "fp8mix"], default=None)
    ap.add_argument("--workload", default="human1000x17000")
    ap.add_argument("--no-e2e", dest="e2e", action="store_false")
    ap.add_argument("--no-cpu-baseline", dest="cpu_baseline", action="store_false")
    ap.add_argument("--no-compare", dest="compare", action="store_false")
    ap.add_argument("--cpu-frac", type=float, default=0.1)
    ap.add_argument("--ref-frac", type=float, default=0.02)
    ap.add_argument("--table-reps", type=int, default=16, help="networks per size in --workload table1")
    args = ap.parse_args(argv)
    if args.warmup < 3:  # the timing rules want at least 3; the line reports what ran
        print(f"bench.py: --warmup {args.warmup} raised to 3", file=sys.stderr)
        args.warmup = 3
    rank, world, local_rank = dist_env()
    wl = synth.get(args.workload) if args.workload not in ("set64", "table1") else None
    if args.impl == "reference":
        run_reference(args, wl, rank, world)
        return
    if args.prec is None:
        from paper_1507_07039_gb300 import panda
        args.prec = "bf16x3" if panda.tensor_path_available() else "fp32"
    if args.workload == "set64":
        run_set(args, rank, world, local_rank)
        return
    if args.workload == "table1":
        run_table1(args, rank, world, local_rank)
        return
    run_ours(args, wl, rank, world, local_rank)


if __name__ == "__main__":
    main()
