#!/usr/bin/env python
"""Benchmark of the Seed-Q decode-fused GEMV on GB300.

A step is one pass of the hot path over every tensor of the workload at batch
n: the decoder plan is resident, each tensor's compressed stream is in HBM, and
y = W_hat x is computed for all tensors back to back on one stream.  Default
workload: the Llama-2-7B-shaped layer set (q, k, v, o 4096x4096; gate, up
11008x4096; down 4096x11008) at 4.0 bits/weight, batch 1.

Prints one JSON line (rank 0).  --impl reference times the CPU oracle instead.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "decode tokens/s & effective weight GB/s at batch 1; % of roofline"
FLUSH_BYTES = 512 << 20  # > 129 MB L2: written between timed steps


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=None,
                   help="timed steps (default 2000 for the fused GEMV, 5 for the encoder)")
    p.add_argument("--warmup", type=int, default=None)
    p.add_argument("--impl", choices=["ours", "reference"], default="ours")
    p.add_argument("--workload", default="c1")
    p.add_argument("--batch", type=int, default=1)
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--path", choices=["gemv", "encode", "importance", "allocate"], default="gemv",
                   help="gemv: the fused decode + GEMV step (default); encode: the exhaustive "
                        "seed-search encoder")
    p.add_argument("--rung", default="16,3", help="encoder rung S,k")
    p.add_argument("--blocks", type=int, default=4864, help="encoder blocks per step")
    p.add_argument("--model", default="llama2_7b",
                   help="synthetic FP16 checkpoint of the importance path")
    a = p.parse_args()
    if a.steps is None:
        a.steps = {"gemv": 2000, "encode": 5, "importance": 20, "allocate": 5}[a.path]
    if a.warmup is None:
        a.warmup = 10 if a.path == "gemv" else 3
    return a


def load_schedule(name):
    from paper_2609_38477_gb300 import workloads as W

    d = json.load(open(os.path.join(ROOT, "tests", "golden", f"schedule_{name}.json")))
    if d["a_rho_checksum"] != W.a_rho_checksum(W.WORKLOADS[name]):
        raise RuntimeError(f"importance inputs of {name} differ from the stored schedule's")
    return d


def measured_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        return None


# ------------------------------------------------------------------ clocks

class Clocks:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: str):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", self.index, f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
            # nvidia-smi takes a moment to start: wait for its first sample so
            # the samples cover the timed region that follows.
            t0 = time.time()
            while time.time() - t0 < 5.0 and os.path.getsize(self.path) == 0:
                time.sleep(0.02)
        except Exception:
            self.proc = None

    def stop(self):
        if not self.proc:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) < 8:
                continue
            try:
                sm.append(float(f[0]))
                mx.append(float(f[1]))
            except ValueError:
                continue
            for nme, v in zip(names, f[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(nme)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "samples": len(sm),
                "reasons": sorted(reasons)}


def gpu_index(local_rank: int) -> str:
    vis = os.environ.get("CUDA_VISIBLE_DEVICES")
    if vis:
        return vis.split(",")[local_rank].strip()
    return str(local_rank)


# ------------------------------------------------------------- distributed

def dist_init():
    import torch

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    return rank, world, local


def dist_max(v: float) -> float:
    import torch
    import torch.distributed as dist

    if not (dist.is_available() and dist.is_initialized()):
        return v
    dev = "cuda" if torch.cuda.is_available() and dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([v], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_value(world: int, n: int, slowest_ms: float) -> float:
    """Whole-job rate of N independent replicas: every rank runs n tokens per
    step, and the job's step is the slowest rank's."""
    return world * n / (slowest_ms * 1e-3)


def dist_barrier():
    import torch.distributed as dist

    if dist.is_available() and dist.is_initialized():
        dist.barrier()


# ------------------------------------------------------------ algorithmic

def algorithmic_counts(w, gts, sched, n):
    """Per-step algorithmic work: warp-instructions of the issue model
    (per weight: k_b LFSR states, k_b integer MACs, one convert, n FMAs) and
    HBM bytes (payload, plan rows read, x, y); also the mean k_b and the
    blocks at each rung."""
    import numpy as np

    rungs = sched["rungs"]
    J = len(rungs)
    warp_inst, bytes_, ksum, blocks = 0.0, 0, 0, 0
    per_rung = np.zeros(J, np.int64)
    for gt in gts:
        t = gt.spec
        rm = gt.layer.rung_map()
        cnt = np.bincount(rm.ravel(), minlength=J)
        per_rung += cnt[:J]
        for j, (S, k) in enumerate(rungs):
            warp_inst += cnt[j] * 8 * (2 * k + 1 + n) / 32.0
            ksum += int(cnt[j]) * k
        blocks += int(cnt.sum())
        bytes_ += (gt.bits + 7) // 8 + t.R * (8 + 4 * (J - 1)) + 2 * n * t.C + 4 * n * t.R
    hist = {f"{S},{k}": int(c) for (S, k), c in zip(rungs, per_rung)}
    return warp_inst, bytes_, ksum / blocks, hist


def traffic_per_launch(kernel_hash: str, workload: str, batch: int):
    """DRAM bytes of one fused launch from the stored ncu capture, or None when
    the capture is of another kernel source, workload or batch size."""
    path = os.path.join(ROOT, "profiles", "k_gemv_c1_dram_traffic.txt")
    if not os.path.exists(path):
        return None
    kv = {}
    for line in open(path):
        if "=" in line and not line.startswith("#"):
            k, v = line.strip().split("=", 1)
            kv[k.strip()] = v.strip()
    if kv.get("kernel_source_sha256") != kernel_hash:
        return None
    if kv.get("workload") != workload or kv.get("batch") != str(batch):
        return None
    try:
        return float(kv["dram_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


KERNEL_SOURCES = ("gemv.cu", "seedq_internal.cuh", "cp_async.cuh", "f32x2.cuh")


def kernel_source_hash() -> str:
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        h.update(open(os.path.join(ROOT, "paper_2609_38477_gb300", "csrc", f), "rb").read())
    return h.hexdigest()[:16]


# ------------------------------------------------------------- CPU oracle

def oracle_sample(w, sched, n, target_s: float, nthreads: int):
    """Prepare a bounded sample of the workload for the oracle: the first rows
    of every tensor, as many as ~target_s seconds of oracle work allow.
    Returns (run, fraction, description)."""
    sys.path.insert(0, os.path.join(ROOT, "oracle"))
    import oracle as O
    from paper_2609_38477_gb300 import workloads as W

    s = O.Sched([tuple(r) for r in sched["rungs"]], sched["theta"], sched["j_tie"], sched["q"])
    ts = [O.Tensor(t.R, t.C, *W.importance(w, i)) for i, t in enumerate(w.tensors)]
    xs = [W.x_bf16(w, i, n) for i in range(len(w.tensors))]
    # Calibrate on about 2% of the rows of the first tensor (enough rows that
    # the per-call set-up of the oracle does not dominate).
    t0 = ts[0]
    rows0 = max(32, t0.R // 50)
    st, bits = t0.synth_pack_rows(s, sched["tie_count"][0], W.payload_key(w, 0), 0, rows0,
                                  rows0 * t0.C * 6)
    c0 = time.perf_counter()
    t0.decode_gemv_threads(s, sched["tie_count"][0], st, bits, xs[0], nthreads, 0, rows0)
    rate = rows0 * t0.C / max(time.perf_counter() - c0, 1e-6)  # weights / s
    frac = min(1.0, target_s * rate / w.weights)
    jobs = []
    for i, (t, ot) in enumerate(zip(w.tensors, ts)):
        rows = max(1, int(round(frac * t.R)))
        st, bits = ot.synth_pack_rows(s, sched["tie_count"][i], W.payload_key(w, i), 0, rows,
                                      rows * t.C * 6)
        jobs.append((ot, sched["tie_count"][i], st, bits, xs[i], rows))
    sample_w = sum(rows * t.C for (ot, _, _, _, _, rows), t in zip(jobs, w.tensors))
    frac = sample_w / w.weights

    def run():
        used = 0
        for ot, T, st, bits, x, rows in jobs:
            _, used = ot.decode_gemv_threads(s, T, st, bits, x, nthreads, 0, rows)
        return used

    desc = (f"oracle decode (Alg. 2) + fp64 GEMV of the first {frac * 100:.1f}% of rows of every "
            f"tensor ({sample_w / 1e6:.1f} M of {w.weights / 1e6:.1f} M weights), batch {n}; "
            f"tokens/s extrapolated to the full workload")
    return run, frac, desc


def cpu_cores():
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def reference_arm(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from paper_2609_38477_gb300 import workloads as W

    w = W.WORKLOADS[args.workload]
    sched = load_schedule(args.workload)
    n = args.batch
    cores = cpu_cores()
    total_steps = args.steps + args.warmup
    per_step = max(0.02, min(6.0, 150.0 / max(total_steps, 1)))
    run, frac, desc = oracle_sample(w, sched, n, per_step, cores)
    for _ in range(args.warmup):
        run()
    times, used = [], cores
    for _ in range(args.steps):
        t0 = time.perf_counter()
        used = run()
        times.append(time.perf_counter() - t0)
    step = statistics.mean(times) / frac  # full-workload seconds per step
    value = n / step
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "tokens/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": step * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"{w.name}: {w.description}", "batch": n},
        "cpu_baseline": {"value": value, "unit": "tokens/s", "cores": used, "kind": "oracle",
                         "sample": desc},
        "e2e": {"value": value, "unit": "tokens/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------- our arm

def our_arm(args):
    import numpy as np
    import torch

    rank, world, local = dist_init()
    torch.cuda.set_device(local)
    import __graft_entry__ as GE

    GE.build()
    from paper_2609_38477_gb300 import workload_gpu as G
    from paper_2609_38477_gb300 import workloads as W

    w = W.WORKLOADS[args.workload]
    sched = load_schedule(args.workload)
    n = args.batch
    gts = G.prepare_workload(w, sched, max_batch=n)
    # All activations of a step in one device buffer and all outputs in one
    # (views per tensor), so a step's inputs and results move in one copy each.
    xcat = torch.cat([G.x_device(w, i, n).reshape(-1) for i in range(len(w.tensors))])
    ycat = torch.empty(sum(n * t.R for t in w.tensors), dtype=torch.float32, device="cuda")
    xs, ys, ox, oy = [], [], 0, 0
    for t in w.tensors:
        xs.append(xcat[ox:ox + n * t.C].view(n, t.C))
        ys.append(ycat[oy:oy + n * t.R].view(n, t.R))
        ox += n * t.C
        oy += n * t.R
    flush = torch.empty(FLUSH_BYTES, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream()
    h = stream.cuda_stream
    from paper_2609_38477_gb300 import seedq as Q

    layers = [gt.layer for gt in gts]
    # The whole step in one launch: up to 8 tensors through seedq_gemm_multi
    # (descriptors in the parameter block), larger models through a layer set
    # over every tensor (descriptors in device memory; x and y of all tensors
    # in one buffer each, the layout of xcat / ycat above).
    lset = None
    if len(layers) > 8:
        lset = Q.LayerSet(layers)
        assert [int(v) for v in lset.col_offsets[1:]] == list(np.cumsum([t.C for t in w.tensors]))

    def step():
        if lset is None:
            Q.gemm_multi(layers, xs, n, ys, h)
        else:
            lset.gemm(xcat, n, ycat, h)

    for _ in range(max(args.warmup, 3)):
        flush.zero_()
        step()
    torch.cuda.synchronize()

    # Timed steps: device time of each step (CUDA events on the launching stream).
    clocks = Clocks(gpu_index(local))
    dist_barrier()
    torch.cuda.synchronize()
    clocks.start()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    for a, b in ev:
        flush.zero_()
        a.record(stream)
        step()
        b.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    dist_barrier()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    # Per-tensor calls, for a per-tensor view of the same kernel (not the step).
    per_call = [[] for _ in gts]
    for _ in range(min(args.steps, 50)):
        flush.zero_()
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(len(gts) + 1)]
        evs[0].record(stream)
        for i, (gt, x, y) in enumerate(zip(gts, xs, ys)):
            Q.gemm_multi([gt.layer], [x], n, [y], h)
            evs[i + 1].record(stream)
        torch.cuda.synchronize()
        for i in range(len(gts)):
            per_call[i].append(evs[i].elapsed_time(evs[i + 1]))

    # End to end through the C ABI with host buffers: every step copies its
    # activations in from pinned host memory and its outputs back (one copy
    # each way), then waits for them on the host.
    xh = xcat.cpu().pin_memory()
    yh = torch.empty(ycat.shape, dtype=torch.float32).pin_memory()
    h2d = xcat.numel() * 2
    d2h = ycat.numel() * 4
    e2e_ms = []
    for _ in range(args.steps):
        flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        xcat.copy_(xh, non_blocking=True)
        step()
        yh.copy_(ycat, non_blocking=True)
        b.record(stream)
        b.synchronize()
        e2e_ms.append(a.elapsed_time(b))

    mean_step = dist_max(statistics.mean(step_ms))
    mean_e2e = dist_max(statistics.mean(e2e_ms))
    warp_inst, alg_bytes, mean_k, rung_hist = algorithmic_counts(w, gts, sched, n)
    call_ms = [statistics.mean(v) for v in per_call]
    kern_ms = statistics.mean(step_ms)  # the step is the fused launches themselves
    props = torch.cuda.get_device_properties(local)
    sms = props.multi_processor_count
    peaks = measured_peaks()
    sm_max = (peaks or {}).get("sm_max_mhz") or (clk or {}).get("sm_max_mhz") or 2070.0
    issue_peak = 4 * sms * sm_max * 1e6 / 1e9  # Gwarp-inst/s
    hbm_peak = (peaks or {}).get("hbm_gbs") or 6800.0
    achieved_issue = warp_inst / (kern_ms * 1e-3) / 1e9
    achieved_hbm = alg_bytes / (kern_ms * 1e-3) / 1e9
    stream_bytes = sum((gt.bits + 7) // 8 for gt in gts)
    value = replica_value(world, n, mean_step)

    line = {
        "metric": METRIC, "value": value, "unit": "tokens/s", "n_gpus": world,
        "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": mean_step,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "fp32", "data": "synthetic",
        "config": {
            "workload": f"{w.name}: {w.description}", "batch": n,
            "bits_per_weight": sched["mean_bits_per_weight"], "weights": w.weights,
            "stream_bytes": stream_bytes, "mean_k": round(mean_k, 4),
            "blocks_per_rung": rung_hist,
            "l2": f"flushed between timed steps ({FLUSH_BYTES >> 20} MiB write)",
            "parallelism": "replicas" if world > 1 else "single GPU",
        },
        "weight_equiv_gbs": 2 * w.weights / (mean_step * 1e-3) / 1e9,
        "compressed_gbs": stream_bytes / (mean_step * 1e-3) / 1e9,
        "clocks": clk,
        "e2e": {"value": world * n / (mean_e2e * 1e-3), "unit": "tokens/s",
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
        "gpu_launches": args.steps * 2,  # x permutation + fused kernel per step
        "roofline": {
            "bound": "alu", "achieved": achieved_issue, "peak": issue_peak,
            "unit": "Gwarp-inst/s", "frac": achieved_issue / issue_peak,
            "traffic": traffic_per_launch(kernel_source_hash(), w.name, n),
            "kernel": "k_gemv over all tensors of the step in one launch (with its x-permutation pre-kernel)",
            "peak_basis": f"4 warp-inst/clk/SM x {sms} SMs x {sm_max:.0f} MHz",
            "hbm": {"achieved_gbs": achieved_hbm, "peak_gbs": hbm_peak,
                    "frac": achieved_hbm / hbm_peak,
                    "peak_basis": "MEASURED_PEAKS.json hbm_gbs (measured)" if peaks else "fallback"},
            "per_tensor_call_us": {gt.spec.name: round(m * 1e3, 2) for gt, m in zip(gts, call_ms)},
        },
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cores = cpu_cores()
        run, frac, desc = oracle_sample(w, sched, n, 10.0, cores)
        t0 = time.perf_counter()
        used, reps = run(), 1
        while time.perf_counter() - t0 < 10.0 and reps < 50:  # at least ~10 s of CPU work
            used = run()
            reps += 1
        el = (time.perf_counter() - t0) / reps
        line["cpu_baseline"] = {"value": n / (el / frac), "unit": "tokens/s", "cores": used,
                                "kind": "oracle", "sample": desc + f"; {reps} repetitions"}
        # The same oracle on one host thread (a smaller row sample, ~5 s).
        run1, frac1, desc1 = oracle_sample(w, sched, n, 5.0, 1)
        t0 = time.perf_counter()
        run1()
        el1 = time.perf_counter() - t0
        line["cpu_baseline"]["single_thread"] = {"value": n / (el1 / frac1), "unit": "tokens/s",
                                                 "cores": 1, "sample": desc1}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if lset is not None:
        lset.release()
    for gt in gts:
        gt.layer.release()


# ------------------------------------------------------------ encoder path

ENC_METRIC = "encoder blocks/s (exhaustive seed search, Sec. 3.1)"


def encode_inputs(S, k, nblocks):
    """Synthetic weight blocks, w ~ N(0, 0.02^2), seeded; the encoder's work does
    not depend on the values beyond the rare singular seed."""
    import numpy as np
    from paper_2609_38477_gb300 import workloads as W

    w = 0.02 * W.normal(W.derive_key(5, 17, S, k), nblocks * 8)
    return np.ascontiguousarray(w.astype(np.float32).reshape(nblocks, 8))


def encode_flops_per_seed(k):
    """fp64 operations of one seed's fit as the exhaustive kernels perform them
    (the smallest calls; the others are screened): the right-hand side (8 products and 8 sums per coefficient), the elimination
    and back substitution (one division, product and difference per entry
    touched), two exponent probes (one product per mantissa), the mantissas,
    and the error (a product by the exponent, a difference, a square and a
    sum per weight)."""
    rhs = 16 * k
    elim = sum((k - 1 - c) * (1 + 2 * (k - 1 - c) + 2) for c in range(k))
    back = sum(1 + 2 * (k - 1 - r) for r in range(k))
    return rhs + elim + back + 3 * k + 4 * 8


def encode_oracle_sample(S, k, w, target_s, nthreads):
    sys.path.insert(0, os.path.join(ROOT, "oracle"))
    import concurrent.futures as cf

    import oracle as O

    taps = O.find_taps(S)
    t0 = time.perf_counter()
    O.encode_block(S, k, taps, w[0].astype("float64"))
    per = max(time.perf_counter() - t0, 1e-6)
    n = int(max(nthreads, min(len(w), target_s * nthreads / per)))
    n = min(n, len(w))

    def run():
        with cf.ThreadPoolExecutor(nthreads) as ex:
            list(ex.map(lambda b: O.encode_block(S, k, taps, w[b].astype("float64")), range(n)))
        return n

    return run, n


def encode_reference(args):
    if int(os.environ.get("RANK", "0")) != 0:
        return
    S, k = (int(v) for v in args.rung.split(","))
    w = encode_inputs(S, k, args.blocks)
    cores = cpu_cores()
    run, n = encode_oracle_sample(S, k, w, max(0.2, min(6.0, 60.0 / max(args.steps + args.warmup, 1))),
                                  cores)
    for _ in range(args.warmup):
        run()
    times = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        run()
        times.append(time.perf_counter() - t0)
    value = n / statistics.mean(times)
    desc = f"oracle seed search of {n} of the {args.blocks} blocks on {cores} host threads"
    print(json.dumps({
        "impl": "reference", "metric": ENC_METRIC, "value": value, "unit": "blocks/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": statistics.mean(times) * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"exhaustive seed search at rung ({S},{k}), {args.blocks} blocks"},
        "cpu_baseline": {"value": value, "unit": "blocks/s", "cores": cores, "kind": "oracle",
                         "sample": desc},
        "e2e": {"value": value, "unit": "blocks/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def fp64_peak_tflops(Q, stream) -> float:
    """fp64 FMA throughput of this device, measured: the best of five timed
    launches of the library's FMA-chain probe (2 flops per FMA)."""
    import torch

    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    Q.fp64_fma_probe(1000, 4, out, stream.cuda_stream)
    best = 0.0
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        fmas = Q.fp64_fma_probe(20000, 4, out, stream.cuda_stream)
        b.record(stream)
        b.synchronize()
        best = max(best, 2 * fmas / (a.elapsed_time(b) * 1e-3) / 1e12)
    return best


def encode_arm(args):
    import numpy as np
    import torch

    rank, world, local = dist_init()
    torch.cuda.set_device(local)
    import __graft_entry__ as GE

    GE.build()
    from paper_2609_38477_gb300 import seedq as Q

    S, k = (int(v) for v in args.rung.split(","))
    nb = args.blocks
    w = encode_inputs(S, k, nb)
    wd = torch.from_numpy(w).cuda()
    seed = torch.empty(nb, dtype=torch.int32, device="cuda")
    E = torch.empty(nb, dtype=torch.int8, device="cuda")
    t = torch.empty(nb * 6, dtype=torch.int8, device="cuda")
    err = torch.empty(nb, dtype=torch.float64, device="cuda")
    flush = torch.empty(FLUSH_BYTES, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream()
    h = stream.cuda_stream

    def step():
        Q.encode_blocks(S, k, wd, nb, seed, E, t, err, h)

    for _ in range(max(args.warmup, 3)):
        flush.zero_()
        step()
    torch.cuda.synchronize()
    clocks = Clocks(gpu_index(local))
    dist_barrier()
    torch.cuda.synchronize()
    clocks.start()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    for a, b in ev:
        flush.zero_()
        a.record(stream)
        step()
        b.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    dist_barrier()
    step_ms = dist_max(statistics.mean(a.elapsed_time(b) for a, b in ev))

    # End to end through the C ABI: weights copied in, fields copied out.
    wh = torch.from_numpy(w).pin_memory()
    outs = [torch.empty(x.shape, dtype=x.dtype).pin_memory() for x in (seed, E, t, err)]
    e2e = []
    for _ in range(args.steps):
        flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        wd.copy_(wh, non_blocking=True)
        step()
        for o, x in zip(outs, (seed, E, t, err)):
            o.copy_(x, non_blocking=True)
        b.record(stream)
        b.synchronize()
        e2e.append(a.elapsed_time(b))
    e2e_ms = dist_max(statistics.mean(e2e))

    nseeds = (1 << S) - 1
    screened = S > 8 or k > 3 or nb > 2048  # the library's rule
    # Screened search: every (block, seed) pair's products of depth 8 with the
    # seed's k (span) or 8 - k (complement) vectors, on the tensor cores.
    per_seed = 16 * (k if k <= 3 else 8 - k) if screened else encode_flops_per_seed(k)
    flops = per_seed * nseeds * nb
    achieved = flops / (step_ms * 1e-3) / 1e12
    pk = measured_peaks()
    peak = (pk["bf16_tflops"] if pk else 1900.0) if screened else fp64_peak_tflops(Q, stream)
    line = {
        "metric": ENC_METRIC, "value": world * nb / (step_ms * 1e-3), "unit": "blocks/s",
        "n_gpus": world, "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": step_ms,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": f"exhaustive seed search at rung ({S},{k}): {nb} blocks of "
                               f"w ~ N(0, 0.02^2), {nseeds} seeds each",
                   "l2": f"flushed between timed steps ({FLUSH_BYTES >> 20} MiB write)"},
        "seeds_per_s": world * nb * nseeds / (step_ms * 1e-3),
        "clocks": clk,
        "e2e": {"value": world * nb / (e2e_ms * 1e-3), "unit": "blocks/s",
                "h2d_bytes_per_step": w.nbytes,
                "d2h_bytes_per_step": sum(x.numel() * x.element_size() for x in (seed, E, t, err))},
        "gpu_launches": args.steps * (3 if screened else 1),
        "roofline": {"bound": "tensor" if screened else "alu", "achieved": achieved, "peak": peak,
                     "unit": "TFLOP/s", "frac": achieved / peak, "traffic": None,
                     "kernel": "k_screen" if screened else "k_encode_list",
                     "peak_basis": ("MEASURED_PEAKS.json bf16_tflops (measured)" if pk else "fallback")
                     if screened else
                     "measured: fp64 FMA loop (seedq_fp64_fma_probe, 8 independent "
                     "chains per thread, best of 5 launches, CUDA events); nominal 1.25",
                     "flops_per_seed": per_seed},
    }
    if rank == 0 and not args.no_cpu_baseline:
        run, n = encode_oracle_sample(S, k, w, 10.0, cpu_cores())
        t0 = time.perf_counter()
        run()
        dt = time.perf_counter() - t0
        line["cpu_baseline"] = {"value": n / dt, "unit": "blocks/s", "cores": cpu_cores(),
                                "kind": "oracle",
                                "sample": f"oracle seed search of {n} of the {nb} blocks, "
                                          f"one block per host thread at a time"}
    if rank == 0:
        print(json.dumps(line), flush=True)


# ------------------------------------------------------- importance path

IMP_METRIC = "data-free importance + outlier statistics of an FP16 checkpoint: GB/s of weights"


def importance_launches(spec) -> int:
    """Kernels one seedq_importance call launches (gains, head pass and its
    finishing step, six or seven per layer, rho normalization, ratios)."""
    per_layer = 6 + (1 if spec.n_heads > spec.n_kv_heads else 0)
    return (2 * spec.n_layers + 1) + 2 + spec.n_layers * per_layer + 2


def importance_oracle_sample(spec, nthreads):
    """The oracle's work for one layer of the checkpoint (Eq. gamma / prop row
    sums, the backward proxy's column sums, the outlier statistics of its seven
    matrices), timed, and scaled to the whole model by weight count.  Returns
    (seconds for the whole model, description)."""
    import numpy as np

    sys.path.insert(0, os.path.join(ROOT, "oracle"))
    import importance as I

    from paper_2609_38477_gb300 import workloads as W

    l = spec.n_layers - 1
    mats = {k: W.synth_weight_rows(spec, l, k, 0, spec.shape(k)[0]) for k in W.MODEL_KINDS}
    a_attn = I.a_from_gain(W.synth_gain(spec, l, "attn"))
    a_mlp = I.a_from_gain(W.synth_gain(spec, l, "mlp"))
    G = np.ones(spec.d_model)
    t0 = time.perf_counter()
    I.a_o(mats["v"], a_attn, spec.n_heads, spec.n_kv_heads)
    I.a_down(mats["gate"], mats["up"], a_mlp)
    Gh = I.sq_cols(mats["down"], G)
    I.sq_cols(mats["gate"], Gh)
    I.sq_cols(mats["up"], Gh)
    Ga = I.sq_cols(mats["o"], G)
    n_rep = spec.n_heads // spec.n_kv_heads
    I.sq_cols(mats["v"], Ga.reshape(spec.n_kv_heads, n_rep, spec.head_dim).sum(axis=1).ravel())
    for k in W.MODEL_KINDS:
        I.dynamic_range(mats[k])
    dt = time.perf_counter() - t0
    layer_w = sum(m.size for m in mats.values())
    desc = (f"oracle (numpy fp64, {nthreads} host threads available) on layer {l} of the "
            f"checkpoint ({layer_w / 1e6:.0f} M of {spec.weights / 1e6:.0f} M weights: row and "
            f"column sums of squares, full-sort column medians), scaled by weight count")
    return dt * spec.weights / layer_w, desc


def importance_reference(args):
    if int(os.environ.get("RANK", "0")) != 0:
        return
    from paper_2609_38477_gb300 import workloads as W

    spec = W.MODELS[args.model]
    cores = cpu_cores()
    times, desc = [], ""
    for _ in range(max(1, min(args.steps, 2))):  # each sample is ~10-20 s of host work
        t, desc = importance_oracle_sample(spec, cores)
        times.append(t)
    value = spec.weights * 2 / statistics.mean(times) / 1e9
    print(json.dumps({
        "impl": "reference", "metric": IMP_METRIC, "value": value, "unit": "GB/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": 0,
        "ms_per_step": statistics.mean(times) * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": spec.description},
        "cpu_baseline": {"value": value, "unit": "GB/s", "cores": cores, "kind": "oracle",
                         "sample": desc},
        "e2e": {"value": value, "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def importance_arm(args):
    import torch

    rank, world, local = dist_init()
    torch.cuda.set_device(local)
    import __graft_entry__ as GE

    GE.build()
    from paper_2609_38477_gb300 import workload_gpu as G
    from paper_2609_38477_gb300 import workloads as W

    spec = W.MODELS[args.model]
    gm = G.synth_model_device(spec)
    out = G.importance_buffers(spec, with_stats=False)
    stream = torch.cuda.current_stream()
    wbytes = spec.weights * 2

    def step():
        return G.run_importance(gm, out, 4, stream)

    for _ in range(max(args.warmup, 3)):
        outliers = step()
    torch.cuda.synchronize()
    clocks = Clocks(gpu_index(local))
    dist_barrier()
    torch.cuda.synchronize()
    clocks.start()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    # The checkpoint (13.5 GB for the Llama-2-7B shape) is far larger than L2,
    # so no flush is needed between passes.  Each pass ends with a host sync
    # (the outlier selection reads the candidates on the host).
    for a, b in ev:
        a.record(stream)
        step()
        b.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    dist_barrier()
    step_ms = dist_max(statistics.mean(a.elapsed_time(b) for a, b in ev))

    # End to end: every weight and gain copied in from pinned host memory, the
    # tables copied out.
    dev = [t for y in gm.layers for t in y.values()] + [gm.final_norm, gm.lm_head]
    host = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True) for t in dev]
    for h, t in zip(host, dev):
        h.copy_(t)
    outs = {k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True) for k, v in out.items()}
    e2e = []
    for _ in range(max(1, min(args.steps, 3))):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for h, t in zip(host, dev):
            t.copy_(h, non_blocking=True)
        step()
        for k, v in out.items():
            outs[k].copy_(v, non_blocking=True)
        b.record(stream)
        b.synchronize()
        e2e.append(a.elapsed_time(b))
    e2e_ms = dist_max(statistics.mean(e2e))
    h2d = sum(t.numel() * t.element_size() for t in dev)
    d2h = sum(v.numel() * v.element_size() for v in out.values())

    pk = measured_peaks()
    peak = pk["hbm_gbs"] if pk else 6800.0
    achieved = wbytes / (step_ms * 1e-3) / 1e9
    line = {
        "metric": IMP_METRIC, "value": world * achieved, "unit": "GB/s",
        "n_gpus": world, "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": step_ms,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "fp32/fp64",
        "data": "synthetic",
        "config": {"workload": spec.description, "weights": spec.weights,
                   "l2": "inputs far larger than L2 (whole checkpoint read once per pass)",
                   "outliers": [list(o) for o in outliers]},
        "clocks": clk,
        "e2e": {"value": world * wbytes / (e2e_ms * 1e-3) / 1e9, "unit": "GB/s",
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
        "gpu_launches": args.steps * importance_launches(spec),
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": None,
                     "kernel": "the whole pass (column passes over every matrix plus the "
                               "finishing kernels), algorithmic bytes = the FP16 weights once",
                     "peak_basis": "MEASURED_PEAKS.json hbm_gbs (measured)" if pk else
                                   "fallback 6800 GB/s"},
    }
    if rank == 0 and not args.no_cpu_baseline:
        t, desc = importance_oracle_sample(spec, cpu_cores())
        line["cpu_baseline"] = {"value": wbytes / t / 1e9, "unit": "GB/s", "cores": cpu_cores(),
                                "kind": "oracle", "sample": desc}
    if rank == 0:
        print(json.dumps(line), flush=True)


# --------------------------------------------------------- allocator path

ALLOC_METRIC = "Alg. 1 allocation over a model's tensors (floor, multiplier bisection, tie pass)"


def allocate_inputs(name):
    from paper_2609_38477_gb300 import workloads as W

    w = W.WORKLOADS[name]
    d = load_schedule(name)
    factors = []
    for i, t in enumerate(w.tensors):
        a, rho = W.importance(w, i)
        factors.append((t.R, t.C, a, rho))
    return w, d, factors


def allocate_oracle(name, w, d):
    sys.path.insert(0, os.path.join(ROOT, "oracle"))
    import oracle as O
    from paper_2609_38477_gb300 import workloads as W

    ts = [O.Tensor(t.R, t.C, *W.importance(w, i)) for i, t in enumerate(w.tensors)]
    t0 = time.perf_counter()
    O.allocate(ts, [tuple(r) for r in d["rungs"]], d["slopes"], d["rbar"], d["floor_f"])
    return time.perf_counter() - t0


def allocate_reference(args):
    if int(os.environ.get("RANK", "0")) != 0:
        return
    w, d, _ = allocate_inputs(args.workload)
    times = [allocate_oracle(args.workload, w, d) for _ in range(max(1, min(args.steps, 3)))]
    value = 1.0 / statistics.mean(times)
    print(json.dumps({
        "impl": "reference", "metric": ALLOC_METRIC, "value": value, "unit": "allocations/s",
        "n_gpus": args.gpus, "steps": len(times), "warmup": 0,
        "ms_per_step": statistics.mean(times) * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"{w.name}: {w.description}", "tensors": len(w.tensors)},
        "cpu_baseline": {"value": value, "unit": "allocations/s", "cores": 1, "kind": "oracle",
                         "sample": "the oracle's allocator (C, one thread) on the whole tensor set"},
        "e2e": {"value": value, "unit": "allocations/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }), flush=True)


def allocate_arm(args):
    import torch

    rank, world, local = dist_init()
    torch.cuda.set_device(local)
    import __graft_entry__ as GE

    GE.build()
    from paper_2609_38477_gb300 import seedq as Q

    w, d, factors = allocate_inputs(args.workload)
    rungs = [tuple(r) for r in d["rungs"]]

    def step():
        return Q.allocate(factors, rungs, d["slopes"], d["rbar"], d["floor_f"])

    for _ in range(max(args.warmup, 3)):
        got = step()
    assert list(got[0]) == d["theta"] and [int(x) for x in got[3]] == d["tie_count"]
    # The searches' rounds are launches that each wait for the last one: time of
    # such a launch with next to nothing in it, back to back in a graph.
    one = torch.zeros(8, dtype=torch.int16, device="cuda")
    chain = 200
    Q.synth_fp16(0, 0, 1, 1, 0, one)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(chain):
            Q.synth_fp16(0, 0, 1, 1, 0, one)
    rt = float("inf")
    for _ in range(10):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ev[0].record()
        graph.replay()
        ev[1].record()
        ev[1].synchronize()
        rt = min(rt, ev[0].elapsed_time(ev[1]) * 1e-3 / chain)
    clocks = Clocks(gpu_index(local))
    dist_barrier()
    clocks.start()
    times = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        step()
        times.append(time.perf_counter() - t0)
    clk = clocks.stop()
    step_s = dist_max(statistics.mean(times))
    # Launches: two rankings, the factors, two searches in rounds of up to 31
    # points (as many as keep a round near 2^16 row searches), group and tail.
    rows, probes = sum(R if rho is not None else 1 for R, C, a, rho in factors), 31
    while probes > 1 and rows * probes > 1 << 16:
        probes //= 2
    per_round = (probes + 1).bit_length() - 1
    rounds = 2 * ((63 + per_round - 1) // per_round + 1)
    launches = 3 + rounds + 2
    line = {
        "metric": ALLOC_METRIC, "value": world / step_s, "unit": "allocations/s",
        "n_gpus": world, "steps": args.steps, "warmup": max(args.warmup, 3),
        "ms_per_step": step_s * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"{w.name}: {w.description}", "tensors": len(w.tensors),
                   "timing": "host wall clock around the synchronous call (it includes the "
                             "factor upload and kernels and the searches' dependent rounds)"},
        "clocks": clk,
        "e2e": {"value": world / step_s, "unit": "allocations/s",
                "h2d_bytes_per_step": sum(4 * (C + (R if rho is not None else 0))
                                          for R, C, a, rho in factors),
                "d2h_bytes_per_step": 8 * (2 * len(factors) + 47)},
        "gpu_launches": args.steps * launches,
        "roofline": {"bound": "latency", "achieved": rounds / step_s, "peak": 1.0 / rt,
                     "unit": "dependent rounds/s", "frac": rt * rounds / step_s,
                     "traffic": None, "kernel": "k_alloc_round (several points a launch)",
                     "peak_basis": "measured back-to-back dependent launches of a one-element kernel "
                                   f"({rt * 1e6:.2f} us each)"},
    }
    if rank == 0 and not args.no_cpu_baseline:
        t = allocate_oracle(args.workload, w, d)
        line["cpu_baseline"] = {"value": 1.0 / t, "unit": "allocations/s", "cores": 1,
                                "kind": "oracle",
                                "sample": "the oracle's allocator (C, one thread) on the whole set"}
    if rank == 0:
        print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.path == "allocate":
        if args.impl == "reference":
            allocate_reference(args)
        else:
            allocate_arm(args)
        return
    if args.path == "importance":
        if args.impl == "reference":
            importance_reference(args)
        else:
            importance_arm(args)
        return
    if args.path == "encode":
        if args.impl == "reference":
            encode_reference(args)
        else:
            encode_arm(args)
    elif args.impl == "reference":
        reference_arm(args)
    else:
        our_arm(args)


if __name__ == "__main__":
    main()
