#!/usr/bin/env python3
"""Throughput of the CSR-weight training step on one GB300 (or N replicas).

Workload: the AlexNet-sized classifier head (FC 9216 -> 4096 -> 4096 -> 1000,
ReLU, softmax cross-entropy) with CSR weights at 5% / 5% / 15% density,
batch 256, on synthetic half-normal 9216-dim features and uniform labels
(seed 0): one full training step of the l1-proximal phase = forward SpMM x3,
loss, dense weight gradients (tcgen05 TF32), transposed SpMM x2, bias SGD,
prox update + CSR re-compaction x3 (and the transposed pattern of the two
layers whose input gradient is needed).

The prox phase runs each layer's bias and weight update (but the first
layer's) on a second stream, concurrently with the transposed products that
carry dL/dX down the network (--overlap off: one stream).

Timing: W eager warm-up steps, then the step is captured in a CUDA graph and
K replays are timed one by one with CUDA events on the replay stream. Before
every step (outside the timed region) the biases are restored and a 256 MB
buffer is written to flush the 126 MB L2. Every step starts from the initial
CSR weights (the prox step writes the second buffer), so each timed step does
the same work. `value` = samples of all ranks / max over ranks of the summed
step times.

Also reported: `e2e` (the same step with the batch copied from pinned host
memory and the loss read back inside the timed region; the library's input
pipeline copies batch i+1 on a copy stream into one of two device slots while
step i runs, and a graph per slot reads it in place), `roofline` of the
dominant kernel (timed with CUDA events in an instrumented eager step),
`cpu_baseline` (the CPU oracle on a row sample of the same step) and the SM
clocks sampled during the timed region.

`--impl reference` times the CPU oracle instead (rank 0 only).
"""

from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "sparse train-step samples/sec at 1 GB300; SpMM/SDDMM/prox HBM GB/s vs peak"
UNIT = "samples/s"
SIZES = (9216, 4096, 4096, 1000)
DENSITIES = (0.05, 0.05, 0.15)
BATCH = 256
WORKLOAD = "fc_head 9216-4096-4096-1000 CSR 5/5/15%, batch 256, prox-SGD step (eta 0.01, lambda 1e-4)"


def parse_args():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=300)
    p.add_argument("--warmup", type=int, default=5)
    p.add_argument("--impl", choices=["ours", "reference"], default="ours")
    p.add_argument("--precision", choices=["tf32", "fp32"], default="tf32")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--prox-path", choices=["fused", "unfused"], default="fused",
                   help="fused: weight gradient and prox update in one tensor-core pass (G not written)")
    p.add_argument("--profile-ops", action="store_true", help="print the per-operation breakdown to stderr")
    p.add_argument("--overlap", choices=["on", "off"], default="on",
                   help="run each layer's bias and weight update (but the first layer's) on a second stream, "
                        "concurrently with the transposed products")
    p.add_argument("--record-traffic", metavar="CSV",
                   help="write profiles/traffic.json from an ncu CSV of this bench (dram__bytes_read.sum, "
                        "dram__bytes_write.sum, gpu__time_duration.sum; --steps 1 --warmup 1) and exit")
    p.add_argument("--clocks-csv", default=None,
                   help="where nvidia-smi writes its clock samples (default: a file in the system temp dir)")
    p.add_argument("--no-kernels", action="store_true",
                   help="skip the per-kernel HBM measurements on the 4096 x 4096 and 4096 x 9216 layers")
    p.add_argument("--optimizer", choices=["sgd", "rmsprop", "adam"], default="sgd",
                   help="proximal method of the prox phase: SGD, Prox-RMSProp (Algorithm 1) or Prox-ADAM "
                        "(Algorithm 2); the adaptive ones take the unfused gradient + prox calls")
    return p.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


# ---------------------------------------------------------------------------
# CPU oracle on a row sample of the step (cpu_baseline and --impl reference)
# ---------------------------------------------------------------------------

class OracleSample:
    """Every operation of the step is separable over the output rows of each
    layer (forward rows, gradient rows, prox rows, the partial W^T dY of those
    rows). A sample runs every operation on 1/F of each layer's rows, with the
    true layer inputs precomputed once; its time times F estimates one full
    step."""

    def __init__(self, cfg, fraction_denominator: int):
        import numpy as np

        import oracle as O
        self.O, self.np = O, np
        self.F = int(fraction_denominator)
        self.cfg = cfg
        self.eta, self.lam = cfg["eta"], cfg["lambda"]
        ws = [O.csr_from_dense(w) for w in cfg["W"]]
        net = O.Net([{"kind": "fc", "relu": i < 2} for i in range(3)],
                    [{"W": w, "b": b.copy()} for w, b in zip(ws, cfg["b"])])
        logits, cache = O.net_forward(net, cfg["X"], BATCH)
        _, dz = O.softmax_xent(logits, cfg["labels"])
        grads = O.net_backward(net, cache, dz, "debias")   # deltas only (cheap phase)
        self.layers = []
        for li in range(3):
            w = ws[li]
            rows = np.arange(0, w.rows, self.F)
            sub = self._rows(w, rows)
            self.layers.append({"W": sub, "x": cache[li]["x"].astype(np.float32),
                                "delta": grads[li]["delta"][rows].astype(np.float32),
                                "b": cfg["b"][li][rows].copy(), "relu": li < 2, "dx": li > 0})
        self.logits = logits.astype(np.float32)

    def _rows(self, w, rows):
        O, np = self.O, self.np
        rp = w.row_ptr.astype(np.int64)
        idx = np.concatenate([np.arange(rp[r], rp[r + 1]) for r in rows]) if len(rows) else np.zeros(0, np.int64)
        lens = rp[rows + 1] - rp[rows]
        new_rp = np.zeros(len(rows) + 1, np.int64)
        new_rp[1:] = np.cumsum(lens)
        return O.CSR(len(rows), w.cols, new_rp.astype(np.int32), w.col_idx[idx], w.val[idx])

    def step(self):
        """Run one sample; return (measured seconds of the sample, estimated
        seconds of one full step = the row-separable part x F + the loss)."""
        O, np = self.O, self.np
        t0 = time.perf_counter()
        for L in self.layers:
            pre = O.spmm_fwd(L["W"], L["x"]) + L["b"][:, None]
            if L["relu"]:
                pre = O.relu(pre)
        t_rows = time.perf_counter() - t0
        t1 = time.perf_counter()
        O.softmax_xent(self.logits, self.cfg["labels"])     # the loss is computed once per step
        t_once = time.perf_counter() - t1
        t2 = time.perf_counter()
        for L in self.layers:
            G = O.weight_grad_dense(L["delta"], L["x"]).astype(np.float32)
            if L["dx"]:
                O.spmm_bwd_t(L["W"], L["delta"])
            new = O.prox_update_compact(L["W"], G, self.eta, self.lam)
            if L["dx"]:
                O.csr_transpose(new)
            L["delta"].sum(axis=1)
        t_rows += time.perf_counter() - t2
        return t_rows + t_once, t_rows * self.F + t_once

    def describe(self) -> str:
        return (f"CPU oracle (numpy, float64 sums) on every operation of one step restricted to 1/{self.F} "
                f"of each layer's output rows (forward, loss, weight gradient, W^T dY, prox + compaction, "
                f"transposed pattern); the row-separable time x {self.F} + the loss once")


def workload_config(world: int, precision: str = "tf32", prox_path: str = "fused", optimizer: str = "sgd",
                    overlap: str = "on") -> dict:
    """The `config` of both arms' lines: the workload and its settings."""
    return {"workload": WORKLOAD, "global_batch": BATCH * world, "per_gpu_batch": BATCH,
            "layers": list(SIZES), "densities": list(DENSITIES),
            "weight_grad": "tf32 tcgen05" if precision == "tf32" else "fp32 as bf16x3 tcgen05",
            "prox_path": prox_path if optimizer == "sgd" else "unfused", "optimizer": optimizer,
            "backward_streams": 2 if overlap == "on" else 1,
            "l2": "flushed between steps (256 MB write, outside the timed region)",
            "parallelism": f"replicas x{world}" if world > 1 else "single GPU"}


def cpu_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def timed_samples(samp, count: int):
    """`count` oracle samples; returns their (measured s, estimated full-step s)
    pairs and the threads they kept busy on average (process CPU time over
    wall time: the row loops are single-threaded Python, numpy's BLAS may add
    threads to the weight gradients)."""
    w0, c0 = time.perf_counter(), time.process_time()
    runs = [samp.step() for _ in range(count)]
    wall, cpu = time.perf_counter() - w0, time.process_time() - c0
    return runs, max(1, round(cpu / wall)) if wall > 0 else 1, round(cpu, 3)


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    from paper_1905_07931_gb300 import synth
    cfg = synth.fc_head(seed=0)
    samp = OracleSample(cfg, fraction_denominator=8)
    for _ in range(args.warmup):
        samp.step()
    runs, cores_used, cpu_s = timed_samples(samp, args.steps)
    measured = sum(r[0] for r in runs)          # seconds the timed steps took (1/8-row samples)
    estimated = sum(r[1] for r in runs)         # the same steps scaled to whole steps
    # each timed step is one 1/8-row sample of the workload's step: it counts
    # as the samples of the batch it covers in full-step time
    value = args.steps * BATCH / estimated
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * measured / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": workload_config(world),
        "cpu_baseline": {"kind": "oracle", "value": value, "unit": UNIT, "cores": cores_used,
                         "cores_available": cpu_cores(), "cpu_s": cpu_s,
                         "sample": samp.describe() + f"; each step is one sample, {args.steps} timed",
                         "measured_s": round(measured, 3), "scale_factor": samp.F,
                         "estimated_full_step_ms": round(1e3 * estimated / args.steps, 1)},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ---------------------------------------------------------------------------
# Clock sampling during the timed region
# ---------------------------------------------------------------------------

class ClockSampler:
    QUERY = ("timestamp,index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int, path=None):
        import tempfile
        self.gpu = gpu_index
        self.proc = None
        self.path = path or os.path.join(tempfile.gettempdir(), f"csrtrain_clocks_gpu{gpu_index}_{os.getpid()}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self, region=None):
        """Median SM clock and the throttle reasons seen; with region = (t0, t1)
        (time.time() seconds of the timed region) only the samples taken in it
        count, if there are any (a region shorter than the 50 ms sampling
        period may hold none: then every sample of the run counts)."""
        if self.proc is None:
            return None
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.fh.close()
        import datetime
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) < 10:
                    continue
                try:
                    ts = datetime.datetime.strptime(parts[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
                except ValueError:
                    ts = None
                try:
                    rows.append((ts, float(parts[2]), float(parts[3]),
                                 {nm for nm, v in zip(names, parts[6:10]) if v.lower().startswith("active")}))
                except ValueError:
                    continue
        if not rows:
            return None
        inside = [r for r in rows if region and r[0] is not None and region[0] - 0.05 <= r[0] <= region[1] + 0.05]
        use = inside or rows
        reasons = set().union(*(r[3] for r in use))
        return {"sm_mhz": statistics.median(r[1] for r in use), "sm_max_mhz": max(r[2] for r in use),
                "reasons": sorted(reasons), "samples": len(use), "samples_in_timed_region": len(inside)}


# ---------------------------------------------------------------------------
# Roofline bookkeeping
# ---------------------------------------------------------------------------

def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


def measure_tf32_tflops(torch) -> float:
    """cuBLAS TF32 GEMM rate on this GPU, measured like the bf16 entry of
    MEASURED_PEAKS.json: float32 8192^3 with TF32 tensor cores allowed, best of
    10 timed with CUDA events (2*N^3 flops each)."""
    n = 8192
    prev = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = True
    try:
        a = torch.randn(n, n, device="cuda")
        b = torch.randn(n, n, device="cuda")
        c = torch.empty(n, n, device="cuda")
        for _ in range(3):
            torch.matmul(a, b, out=c)
        best = float("inf")
        for _ in range(10):
            st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            st.record()
            torch.matmul(a, b, out=c)
            en.record()
            torch.cuda.synchronize()
            best = min(best, st.elapsed_time(en))
        del a, b, c
        return 2.0 * n ** 3 / (best / 1e3) / 1e12
    finally:
        torch.backends.cuda.matmul.allow_tf32 = prev


def source_digest(files) -> str:
    """First 16 hex digits of the sha256 over the named csrc files, in order."""
    h = hashlib.sha256()
    for name in files:
        with open(os.path.join(ROOT, "paper_1905_07931_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def recorded_traffic(op_label: str):
    """DRAM bytes (read + write) of one call of the op, summed over its kernels,
    from the committed ncu record, if it was taken on the current source of
    the files those kernels live in (else None)."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            rec = json.load(f).get(op_label)
        if not rec:
            return None
        return rec["dram_bytes_per_call"] if source_digest(rec["sources"]) == rec["sha256_16"] else None
    except Exception:
        return None


def op_bytes(name, info):
    """Algorithmic HBM bytes (each operand touched once) of one call."""
    if "M" not in info:
        return None
    M, K, n = info["M"], info["K"], info.get("n", 0)
    nnz, nnz_out = info.get("nnz", 0), info.get("nnz_out", 0)
    if name == "spmm_fwd":
        return 8 * nnz + 4 * (M + 1) + 4 * n * (K + M)
    if name == "spmm_fwd_bias_act":
        return 8 * nnz + 4 * (M + 1) + 4 * n * (K + M) + 4 * M
    if name == "spmm_bwd_t":
        return 8 * nnz + 4 * (K + 1) + 4 * n * (K + M)
    if name == "spmm_bwd_t_relu":
        return 8 * nnz + 4 * (K + 1) + 4 * n * (2 * K + M)
    if name == "weight_grad_dense":
        return 4 * M * K + 4 * n * (M + K)
    if name == "weight_grad_sddmm":
        return 12 * nnz + 4 * (M + 1) + 4 * n * (K + M)
    if name == "weight_grad_prox_update":
        b = 4 * n * (M + K) + 8 * nnz + 4 * (M + 1) + 8 * nnz_out + 4 * (M + 1)
        if info.get("transposed"):
            b += 8 * nnz_out + 4 * (M + 1) + 12 * nnz_out + 4 * (K + 1)
        return b
    if name in ("prox_update_compact", "prox_rmsprop_update_compact", "prox_adam_update_compact"):
        b = 4 * M * K + 8 * nnz + 4 * (M + 1) + 8 * nnz_out + 4 * (M + 1)
        if info.get("transposed"):
            b += 8 * nnz_out + 4 * (M + 1) + 12 * nnz_out + 4 * (K + 1)
        # the dense moments, read and written: v (RMSProp), m and v (Adam)
        b += {"prox_rmsprop_update_compact": 8, "prox_adam_update_compact": 16}.get(name, 0) * M * K
        return b
    return None


# Kernels of one weight_grad_prox_update call: it starts with fp_oldbits_kernel
# and runs on through these (the transposed copy included when built).
FUSED_OP_KERNELS = ("fp_oldbits_kernel", "gemm_prox_tc_kernel", "fp_rowscan_kernel", "scan_clamped_kernel",
                    "fp_rows_cols_scan_kernel", "fp_two_scans_kernel", "scan_single_block_kernel",
                    "trb_count_kernel", "tr_colscan_kernel", "trb_write_kernel")
FUSED_OP_SOURCES = ["fused_prox.cu", "compact.cu", "tc_common.cuh", "common.cuh"]
# the ncu command whose CSV record_traffic reads: the ops' kernels only
TRAFFIC_NCU = ("ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum --clock-control none "
               "-k regex:'fp_oldbits|gemm_prox|fp_rowscan|fp_rows_cols|fp_two_scans|scan_clamped|scan_single|trb_|"
               "tr_colscan|spmm_merge|spmm_tc' "
               "-c 80 --csv --log-file bench_dram.csv")


def record_traffic(csv_path: str, out_path: str) -> dict:
    """profiles/traffic.json from an ncu CSV of `bench.py --steps 1 --warmup 1`:
    per fused gradient + prox call of the second eager step (the instrumented
    one), the DRAM bytes and serialised time summed over its kernels. The
    step's calls run layer 2, layer 1, layer 0."""
    import csv
    launches = {}
    with open(csv_path) as f:
        rows = [r for r in csv.reader(f)]
    hdr = next(i for i, r in enumerate(rows) if r and r[0] == "ID")
    cols = rows[hdr]
    for r in rows[hdr + 1:]:
        if len(r) != len(cols):
            continue
        d = dict(zip(cols, r))
        k = launches.setdefault(int(d["ID"]), {"name": d["Kernel Name"]})
        try:
            k[d["Metric Name"]] = float(d["Metric Value"].replace(",", ""))
        except ValueError:
            pass
    seq = [launches[i] for i in sorted(launches)]
    calls, i = [], 0
    while i < len(seq):
        if seq[i]["name"].split("(")[0].split("::")[-1].startswith("fp_oldbits_kernel"):
            j = i + 1
            while j < len(seq) and any(n in seq[j]["name"] for n in FUSED_OP_KERNELS[1:]):
                j += 1
            calls.append(seq[i:j])
            i = j
        else:
            i += 1
    if len(calls) < 6:
        raise SystemExit(f"record-traffic: found {len(calls)} fused calls, need the 3 of two eager steps")
    pending = {}
    rec = {"_about": "DRAM bytes (read + write) of one call of each fused weight-gradient + prox op and each "
                     "sparse product of the classifier-head step, summed over the op's kernels (second eager step "
                     "of the run), from: " + TRAFFIC_NCU + " python bench.py --steps 1 --warmup 1 --no-cpu-baseline "
                     "--no-kernels --overlap off, then python bench.py --record-traffic bench_dram.csv (the counters "
                     "take one pass; only the ops' kernels are captured, the first 80 launches: 4 at start-up, up to 33 "
                     "per step). ncu flushes the caches between kernels, so output lines still dirty in L2 when a "
                     "kernel ends are not counted: an op whose output fits in L2 shows fewer bytes than it writes."}
    # the step's sparse products, in call order: forward layers 0, 1, 2, then
    # the backward products of layers 2 and 1 (second eager step)
    # (a product that may take the tensor cores launches spmm_tc_kernel behind
    # spmm_merge_kernel)
    sp = []
    for k in seq:
        if "spmm_merge_kernel" in k["name"] or "spmm_group_kernel" in k["name"]:
            sp.append([k])
        elif "spmm_tc_kernel" in k["name"] and sp:
            sp[-1].append(k)
    if len(sp) >= 10:
        labels = ["spmm_fwd_bias_act[layer 0]", "spmm_fwd_bias_act[layer 1]", "spmm_fwd_bias_act[layer 2]",
                  "spmm_bwd_t_relu[layer 2]", "spmm_bwd_t_relu[layer 1]"]
        srcs = ["spmm.cu", "spmm_tc.cu", "spmm_tc.cuh", "split_bf16.cuh", "tc_pair.cuh", "common.cuh"]
        for lab, call in zip(labels, sp[5:10]):
            rd = sum(k.get("dram__bytes_read.sum", 0.0) for k in call)
            wr = sum(k.get("dram__bytes_write.sum", 0.0) for k in call)
            us = sum(k.get("gpu__time_duration.sum", 0.0) for k in call) / 1e3
            pending[lab] = {"dram_bytes_per_call": int(rd + wr), "dram_read": int(rd), "dram_write": int(wr),
                            "ncu_us_serialised": round(us, 1),
                            "kernels": [k["name"].split("(")[0].replace("csrt::", "").replace("void ", "")
                                        for k in call],
                            "sources": srcs, "sha256_16": source_digest(srcs)}
    for layer, call in zip((2, 1, 0), calls[3:6]):
        rd = sum(k.get("dram__bytes_read.sum", 0.0) for k in call)
        wr = sum(k.get("dram__bytes_write.sum", 0.0) for k in call)
        us = sum(k.get("gpu__time_duration.sum", 0.0) for k in call) / 1e3
        rec[f"weight_grad_prox_update[layer {layer}]"] = {
            "dram_bytes_per_call": int(rd + wr), "dram_read": int(rd), "dram_write": int(wr),
            "ncu_us_serialised": round(us, 1),
            "kernels": [k["name"].split("(")[0].replace("csrt::", "").replace("void ", "") for k in call],
            "sources": FUSED_OP_SOURCES, "sha256_16": source_digest(FUSED_OP_SOURCES)}
    rec.update(pending)
    with open(out_path, "w") as f:
        json.dump(rec, f, indent=1)
        f.write("\n")
    return rec


# ---------------------------------------------------------------------------
# The sparse kernels on the largest sparse layers (the metric's second half)
# ---------------------------------------------------------------------------

KERNEL_OF_OP = {"spmm_fwd": "spmm_group_kernel", "spmm_bwd_t": "spmm_group_kernel", "sddmm": "sddmm_kernel",
                "prox (lambda=1e-4)": "prox_count_kernel + prox_place_kernel",
                "prox (lambda*)": "prox_count_kernel + prox_place_kernel"}


def measure_kernels(hbm_peak: float, reps: int = 20):
    """SpMM, SpMM^T and SDDMM at n = 1 on the 4096 x 4096 sweep layer at 5%
    and 50% (uniform rows), and the prox step at lambda = 1e-4 (dense output)
    and at the density-preserving lambda* on the same layers (with the
    transposed copy) and on the 4096 x 9216 first layer of the classifier head
    (without it, as the step runs it). Each call timed alone with CUDA events,
    the 256 MB L2 flush written before every launch, median of `reps`;
    algorithmic bytes count each operand once (the sweep's formulas)."""
    from paper_1905_07931_gb300 import sweep
    out = []
    cases = [(4096, 4096, 0.05, {"spmm_fwd", "spmm_bwd_t", "sddmm", "prox"}, [1], True),
             (4096, 4096, 0.50, {"spmm_fwd", "spmm_bwd_t", "sddmm", "prox"}, [1], True),
             (4096, 9216, 0.05, {"prox"}, [1], False)]
    for m, k, d, ops, batches, transposed in cases:
        for r in sweep.run_layer(m, k, d, False, batches, ops, reps, transposed=transposed):
            gbs = r["bytes"] / (r["us"] / 1e6) / 1e9
            out.append({"kernel": KERNEL_OF_OP.get(r["op"], r["op"]), "op": r["op"], "m": m, "k": k,
                        "density": d, "n": r["n"], "transposed_copy": transposed if r["op"].startswith("prox") else None,
                        "nnz": r["nnz"], "nnz_out": r.get("nnz_out"), "algorithmic_bytes": int(r["bytes"]),
                        "us": r["us"], "gbs": round(gbs, 1), "hbm_frac": round(gbs / hbm_peak, 4)})
    return out


# ---------------------------------------------------------------------------
# Multi-rank bookkeeping (replicas: no collective on the data path)
# ---------------------------------------------------------------------------

def max_over_ranks(x: float, world: int, device="cpu") -> float:
    """The largest value of x over all ranks (the slowest rank's timed region)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    if world > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank_per_step: int, steps: int, world: int, max_total_ms: float) -> float:
    """Units processed by all ranks divided by the slowest rank's time."""
    return world * steps * units_per_rank_per_step / (max_total_ms / 1e3)


# ---------------------------------------------------------------------------
# Our arm
# ---------------------------------------------------------------------------

def main():
    args = parse_args()
    if args.record_traffic:
        rec = record_traffic(args.record_traffic, os.path.join(ROOT, "profiles", "traffic.json"))
        print(json.dumps({k: v["dram_bytes_per_call"] for k, v in rec.items() if k != "_about"}))
        return 0
    if args.impl == "reference":
        return run_reference(args)
    rank, world, local_rank = dist_env()
    import numpy as np
    import torch
    import torch.distributed as dist

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA GPU")
    torch.cuda.set_device(local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    from paper_1905_07931_gb300 import csrtrain as C
    from paper_1905_07931_gb300 import synth
    from paper_1905_07931_gb300.train import BatchPrefetcher, SparseNet, mlp_layers

    prec = C.CSRT_PREC_TF32 if args.precision == "tf32" else C.CSRT_PREC_FP32
    cfg = synth.fc_head(seed=0)
    layers = mlp_layers(3)
    net = SparseNet(layers, cfg["W"], cfg["b"], BATCH, (SIZES[0],), precision=prec,
                    fused=args.prox_path == "fused", optimizer=args.optimizer, overlap=args.overlap == "on")
    x_host = torch.from_numpy(cfg["X"]).pin_memory()
    lab_host = torch.from_numpy(cfg["labels"]).pin_memory()
    net.x_in.copy_(x_host)
    net.labels.copy_(lab_host)
    b0 = [L["b"].clone() for L in net.params]
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    eta, lam = cfg["eta"], cfg["lambda"]

    def restore():
        # every step starts from the initial weights, biases and (adaptive
        # methods) zero moments: each timed step is the first step
        for L, b in zip(net.params, b0):
            L["b"].copy_(b)
            L["cur"] = 0
        net.reset_optimizer()

    # warm-up (eager)
    for _ in range(max(args.warmup, 0)):
        restore()
        net.step("prox", eta, lam)
    torch.cuda.synchronize()
    flags, _ = net.status()
    if flags:
        raise SystemExit(f"device status {flags} after warm-up")

    # per-operation breakdown of one eager step (events around every library call)
    restore()
    prof = profile_ops(net, C, torch, eta, lam, flush)
    restore()

    # capture one step in a CUDA graph
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    C.launch_count(reset=True)
    with torch.cuda.stream(s):
        restore()
        with torch.cuda.graph(graph, stream=s):
            net.step("prox", eta, lam)
    launches_per_step = C.launch_count(reset=True)
    torch.cuda.current_stream().wait_stream(s)
    torch.cuda.synchronize()

    stream = torch.cuda.current_stream()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    clocks = ClockSampler(local_rank, args.clocks_csv)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    time.sleep(0.3)
    wall0 = time.perf_counter()
    t_region0 = time.time()
    for i in range(args.steps):
        restore()
        flush.fill_(float(i))
        starts[i].record(stream)
        graph.replay()
        ends[i].record(stream)
    torch.cuda.synchronize()
    wall = time.perf_counter() - wall0
    clk = clocks.stop(region=(t_region0, time.time()))
    if world > 1:
        dist.barrier()
    times_ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    total_max_ms = max_over_ranks(sum(times_ms), world, "cuda")
    value = whole_job_rate(BATCH, args.steps, world, total_max_ms)
    flags, _ = net.status()
    if flags:
        raise SystemExit(f"device status {flags} after the timed steps")

    # end to end: pinned host batch -> device, step, loss -> pinned host. The
    # input pipeline copies batch i+1 on a copy stream into one of two device
    # slots while step i runs (its copy starts after step i's start event, so
    # every copy lies inside a timed step); batch 0 is copied inside step 0.
    # One graph per slot reads the slot's buffers directly (net.set_input).
    pf = BatchPrefetcher(net)
    x_orig, y_orig = net.x_in, net.labels
    slot_graphs = []
    for slot in range(2):
        net.set_input(pf.x[slot], pf.y[slot])
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            restore()
            with torch.cuda.graph(g, stream=s):
                net.step("prox", eta, lam)
        slot_graphs.append(g)
    net.set_input(x_orig, y_orig)
    torch.cuda.current_stream().wait_stream(s)
    torch.cuda.synchronize()
    loss_host = torch.empty(1, dtype=torch.float32).pin_memory()
    e_starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    e_ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    for i in range(args.steps):
        restore()
        flush.fill_(float(i))
        e_starts[i].record(stream)
        if i == 0:
            pf.issue(x_host, lab_host, after=e_starts[0])
        slot = pf.acquire()
        if i + 1 < args.steps:
            pf.issue(x_host, lab_host, after=e_starts[i])
        slot_graphs[slot].replay()
        pf.release(slot)
        loss_host.copy_(net.loss[:1], non_blocking=True)
        e_ends[i].record(stream)
    torch.cuda.synchronize()
    e2e_ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in zip(e_starts, e_ends)), world, "cuda")
    e2e_value = whole_job_rate(BATCH, args.steps, world, e2e_ms)

    # roofline of the dominant kernel
    peaks, peak_kind = measured_peaks()
    dom = max((r for r in prof if op_bytes(r["name"], r["info"]) is not None), key=lambda r: r["ms"])
    bytes_ = op_bytes(dom["name"], dom["info"])
    kernel = dom["kernel"]
    t_s = dom["ms"] / 1e3
    cands = []
    if bytes_ is not None:
        hbm = peaks["hbm_gbs"]
        cands.append({"bound": "hbm", "achieved": round(bytes_ / t_s / 1e9, 1), "peak": hbm, "unit": "GB/s",
                      "frac": round(bytes_ / t_s / 1e9 / hbm, 4),
                      "peak_source": f"{peak_kind} (MEASURED_PEAKS.json hbm_gbs)" if peak_kind == "measured"
                      else "fallback 6.8 TB/s"})
    if dom["name"] in ("spmm_fwd", "spmm_bwd_t", "spmm_fwd_bias_act", "spmm_bwd_t_relu") and dom["info"].get("n"):
        # a product on the FP32 CUDA cores (no tensor cores for the sparse
        # operand): 2*nnz*n flops against the FMA rate measured by the
        # library's probe on this GPU (nominal 152 SMs x 128 lanes x 2 x clock)
        flops = 2.0 * dom["info"]["nnz"] * dom["info"]["n"]
        peak = C.fma_peak_tflops()
        cands.append({"bound": "alu", "achieved": round(flops / t_s / 1e12, 2), "peak": round(peak, 1),
                      "unit": "TFLOP/s", "frac": round(flops / t_s / 1e12 / peak, 4),
                      "peak_source": "measured FP32 FMA rate (library probe, fma_peak_kernel)"})
    if dom["name"] in ("weight_grad_dense", "weight_grad_prox_update") and dom["info"].get("n") \
            and args.precision == "fp32":
        # --precision fp32: each factor as the sum of three bf16 parts, six
        # products of the parts on the tensor cores; algorithmic flops 2MKN
        # against a sixth of the measured bf16 rate
        flops = 2.0 * dom["info"]["M"] * dom["info"]["K"] * dom["info"]["n"]
        peak = peaks["bf16_tflops"] / 6
        cands.append({"bound": "tensor", "achieved": round(flops / t_s / 1e12, 2), "peak": round(peak, 1),
                      "unit": "TFLOP/s", "frac": round(flops / t_s / 1e12 / peak, 4),
                      "peak_source": f"bf16_tflops / 6 ({peak_kind} peaks)"})
    elif dom["name"] in ("weight_grad_dense", "weight_grad_prox_update") and dom["info"].get("n"):
        # a TF32 contraction: its peak is the cuBLAS TF32 rate measured here (the
        # measured bf16 rate x the nominal tf32/bf16 ratio 1.1/2.25 beside it);
        # algorithmic flops 2MKN (the fused op's second pass recomputes them: not counted)
        flops = 2.0 * dom["info"]["M"] * dom["info"]["K"] * dom["info"]["n"]
        peak = measure_tf32_tflops(torch)
        cands.append({"bound": "tensor", "achieved": round(flops / t_s / 1e12, 1), "peak": round(peak, 1),
                      "unit": "TFLOP/s", "frac": round(flops / t_s / 1e12 / peak, 4),
                      "peak_source": "measured cuBLAS TF32 GEMM 8192^3, best of 10 (bf16_tflops x 1.1/2.25 = "
                                     f"{peaks['bf16_tflops'] * 1.1 / 2.25:.1f} from {peak_kind} peaks)"})
    # the binding resource is the one the op uses the larger fraction of
    cands.sort(key=lambda c: -c["frac"])
    roof = dict(cands[0]) if cands else None
    if roof is not None:
        # the committed traffic record is of the default configuration (TF32,
        # fused path, SGD): the sparse products run the same kernels under
        # every option, the gradient + prox ops do not
        same_kernels = dom["name"] in ("spmm_fwd", "spmm_bwd_t", "spmm_fwd_bias_act", "spmm_bwd_t_relu") or (
            args.precision == "tf32" and args.prox_path == "fused" and args.optimizer == "sgd")
        if args.precision == "fp32" and dom["name"] == "weight_grad_prox_update":
            kernel = ("split_rows_kernel + gemm_split_kernel + prox_count_kernel + prox_place_kernel "
                      "(the op's unfused route at FP32)")
        roof.update({"traffic": recorded_traffic(dom["label"]) if same_kernels else None, "kernel": kernel,
                     "op": dom["label"],
                     "algorithmic_bytes": int(bytes_) if bytes_ else None, "launch_ms": round(dom["ms"], 4)})
        if len(cands) > 1:
            roof["other"] = {k: cands[1][k] for k in ("bound", "achieved", "peak", "unit", "frac")}

    # the largest sparse product of the step against its own roofs: FP32 FMA
    # (measured with the library's probe), HBM (algorithmic bytes), and the
    # rate at which its stored entries gather rows of the dense operand (L2)
    spmm_names = ("spmm_fwd", "spmm_bwd_t", "spmm_fwd_bias_act", "spmm_bwd_t_relu")
    sp = max((r for r in prof if r["name"] in spmm_names and r["info"].get("n")), key=lambda r: r["ms"],
             default=None)
    spmm_roof = None
    if sp is not None:
        t_sp = sp["ms"] / 1e3
        fl = 2.0 * sp["info"]["nnz"] * sp["info"]["n"]
        fma_peak = C.fma_peak_tflops()
        b_sp = op_bytes(sp["name"], sp["info"])
        spmm_roof = {"op": sp["label"], "kernel": sp["kernel"], "launch_ms": round(sp["ms"], 4),
                     "fp32_tflops": round(fl / t_sp / 1e12, 2), "fma_peak_tflops": round(fma_peak, 1),
                     "fma_frac": round(fl / t_sp / 1e12 / fma_peak, 4),
                     "hbm_gbs": round(b_sp / t_sp / 1e9, 1), "hbm_frac": round(b_sp / t_sp / 1e9 / peaks["hbm_gbs"], 4),
                     "gather_tbs": round(4.0 * sp["info"]["nnz"] * sp["info"]["n"] / t_sp / 1e12, 2),
                     "note": "gather = 4*nnz*n bytes of dense-operand rows read per call (from L2)"}

    line = {
        "metric": METRIC, "value": round(value, 1), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(total_max_ms / args.steps, 4), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": dict(workload_config(world, args.precision, args.prox_path, args.optimizer, args.overlap),
                       step_ops=[r["label"] for r in prof]),
        "e2e": {"value": round(e2e_value, 1), "unit": UNIT,
                "h2d_bytes_per_step": int(x_host.numel() * 4 + lab_host.numel() * 4), "d2h_bytes_per_step": 4},
        "gpu_launches": int(launches_per_step * args.steps),
        "roofline": roof,
        "spmm_roofline": spmm_roof,
        "clocks": clk,
        "wall_s_timed_region": round(wall, 3),
    }
    if rank == 0 and not args.no_kernels:
        line["kernels"] = measure_kernels(peaks["hbm_gbs"])
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        samp = OracleSample(cfg, fraction_denominator=4)
        samp.step()
        runs, cores_used, cpu_s = timed_samples(samp, 5)
        est = [r[1] for r in runs]
        v = BATCH / (sum(est) / len(est))
        line["cpu_baseline"] = {"value": round(v, 3), "unit": UNIT, "cores": cores_used,
                                "cores_available": cpu_cores(), "cpu_s": cpu_s, "kind": "oracle",
                                "sample": samp.describe() + ", mean of 5 samples after one untimed",
                                "measured_s": round(sum(r[0] for r in runs), 3), "samples": len(runs),
                                "scale_factor": samp.F,
                                "estimated_full_step_ms": round(1e3 * sum(est) / len(est), 1)}
    if args.profile_ops and rank == 0:
        for r in prof:
            b = op_bytes(r["name"], r["info"])
            gbs = f"{b / (r['ms'] / 1e3) / 1e9:8.1f} GB/s" if b else ""
            print(f"{r['label']:<36s} {r['ms'] * 1e3:9.1f} us {gbs}", file=sys.stderr)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def profile_ops(net, C, torch, eta, lam, flush):
    """Run one eager step with CUDA events around every library call on the
    launching stream; return [{label, name, kernel, ms, info}] in call order."""
    stream = torch.cuda.current_stream()
    records = []
    wrapped = {}
    names = ["spmm_fwd", "spmm_bwd_t", "spmm_fwd_bias_act", "spmm_bwd_t_relu", "weight_grad_dense",
             "weight_grad_sddmm", "prox_update_compact", "prox_rmsprop_update_compact", "prox_adam_update_compact",
             "weight_grad_prox_update", "debias_update", "bias_act_fwd", "relu_bwd", "bias_grad_sgd", "softmax_xent"]
    kernel_of = {"spmm_fwd": "spmm_merge_kernel", "spmm_bwd_t": "spmm_merge_kernel",  # and spmm_tc_kernel, dense layers
                 "spmm_fwd_bias_act": "spmm_merge_kernel", "spmm_bwd_t_relu": "spmm_merge_kernel",
                 "weight_grad_dense": "gemm_tf32_tc_persistent_kernel", "weight_grad_sddmm": "sddmm_wide_kernel",
                 "prox_update_compact": "prox_count_kernel", "prox_rmsprop_update_compact": "prox_rows_kernel",
                 "prox_adam_update_compact": "prox_rows_kernel", "weight_grad_prox_update": "gemm_prox_tc_kernel",
                 "debias_update": "debias_kernel"}
    layer_of = {}
    for i, L in enumerate(net.params):
        for W in L["W"]:
            layer_of[id(W)] = i
    for nm in names:
        orig = getattr(C, nm)
        wrapped[nm] = orig

        def make(nm, orig):
            def fn(*a, **k):
                st = torch.cuda.Event(enable_timing=True)
                en = torch.cuda.Event(enable_timing=True)
                st.record(stream)
                orig(*a, **k)
                en.record(stream)
                info = {}
                W = a[0] if a and isinstance(a[0], C.CSR) else None
                li = layer_of.get(id(W)) if W is not None else None
                out_arg = {"prox_update_compact": 4, "prox_rmsprop_update_compact": 7, "prox_adam_update_compact": 10}
                if nm in ("spmm_fwd", "spmm_bwd_t", "spmm_fwd_bias_act", "spmm_bwd_t_relu", "weight_grad_sddmm",
                          "weight_grad_prox_update", "debias_update") or nm in out_arg:
                    info = {"M": W.rows, "K": W.cols, "W": W}
                    if nm in ("spmm_fwd", "spmm_bwd_t", "spmm_fwd_bias_act", "spmm_bwd_t_relu", "weight_grad_sddmm"):
                        info["n"] = a[1].shape[1] if a[1].dim() == 2 else 0
                    if nm in out_arg:
                        info["W_out"] = a[out_arg[nm]]
                        info["transposed"] = a[out_arg[nm]].transposed
                    if nm == "weight_grad_prox_update":
                        info["n"] = a[1].shape[1]
                        info["W_out"] = a[5]
                        info["transposed"] = a[5].transposed
                elif nm == "weight_grad_dense":
                    dy, x = a[0], a[1]
                    info = {"M": dy.shape[0], "K": x.shape[0], "n": dy.shape[1]}
                    li = next((i for i, L in enumerate(net.params) if L["W"][0].rows == dy.shape[0]
                               and L["W"][0].cols == x.shape[0]), None)
                records.append({"name": nm, "st": st, "en": en, "info": info, "layer": li})
            return fn
        setattr(C, nm, make(nm, orig))
    overlap = net.overlap
    net.overlap = False   # one stream: every call's events bracket that call alone
    try:
        flush.fill_(1.0)
        torch.cuda.synchronize()
        # keep the GPU busy while the host enqueues the step, so that no
        # call's events enclose host-side launch latency
        torch.cuda._sleep(20_000_000)
        net.step("prox", eta, lam)
        torch.cuda.synchronize()
    finally:
        net.overlap = overlap
        for nm, orig in wrapped.items():
            setattr(C, nm, orig)
    out = []
    for r in records:
        info = r["info"]
        if "W" in info:
            info["nnz"] = info["W"].nnz()
            del info["W"]
        if "W_out" in info:
            info["nnz_out"] = info["W_out"].nnz()
            del info["W_out"]
        lab = r["name"] + (f"[layer {r['layer']}]" if r["layer"] is not None else "")
        out.append({"label": lab, "name": r["name"], "kernel": kernel_of.get(r["name"], r["name"]),
                    "ms": r["st"].elapsed_time(r["en"]), "info": info})
    return out


if __name__ == "__main__":
    sys.exit(main())
