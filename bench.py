#!/usr/bin/env python
"""Throughput of the Hilbert-forest path on one GB300 (or N replicas).

One step = the whole path on one synthetic batch: hf_build (range, quantize,
per-tree keys and sort), hf_knn_graph (window distances + top-k merge over all
trees) and hf_search (a batch of queries located and answered in every tree).

Default workload: the full-size kNN-graph configuration, n = 3,000,000 points,
d = 384, float32 unit vectors from a 1,000-component anisotropic Gaussian
mixture with Zipf(1.1) weights, T trees, b = 8, window w, k = 15; plus 10,000
mixture queries with N(0, 0.05^2) noise. The paper measured on GOOAQ
(3M x 384); these seeded synthetic inputs stand in for it.

The default form is the tensor mode: window distances as BF16 Gram tiles on
the tensor cores (tcgen05) keeping k + 1 candidates per point, then an exact
float32 re-rank; `--mode plain` runs the all-float32 window kernel instead
(one plain step is also timed beside the default, for comparison).

Prints one JSON line (rank 0). `value` = points / s of the device-resident
step; `e2e` = the same through the C ABI with pinned host buffers (copies in
the timed region); `roofline` for the dominant kernel (the Gram kernel in
tensor mode, the window kernel in plain mode); `cpu_baseline` = the CPU oracle
on a bounded sample (and the tiny configuration in full). Blocks measured
after the timed region: `plain_f32`, `learned` (per-point budgets), `sketch`
(the paper's second stage), `batched` (64 independent sets, CUDA graph,
autotuner) and `tiny` (20,000 x 16). `--workload c3` runs the large search
workload instead (23M x 384, T = 160, 10k queries) and prints its own line.

--impl reference times the CPU oracle itself (the only reference this
project has: the paper ships no code) on a bounded sample per step.
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

METRIC = "kNN-graph points/s at recall@k>=0.8; Hilbert-sort Mkeys/s; % HBM/TC roofline"
MODES = {"plain": 0, "tensor": 1, "fp8": 2}

# DRAM traffic of the dominant kernels from one ncu capture of a 1M-point
# launch (bytes per point, scaled by n here) and the source file it was taken
# on; a figure is dropped (null) once its source differs.
WINDOW_TRAFFIC = {"bytes_per_point": 2065, "source_sha": "4a28b09c422b9770", "file": "window.cu"}   # w = 32, pair_kernel + merge_kernel
GRAM_TRAFFIC = {"bytes_per_point": 1139, "source_sha": "23ffe7e70668a4e5", "file": "gram.cu", "w": 1024}

# GB300: 152 SMs x 128 FP32 lanes; one pair-coordinate update of the exact-
# difference distance is FADD + FFMA = 2 issue slots = 3 flops.
SMS, FP32_LANES, MAX_SM_MHZ = 152, 128, 2070.0


def args():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=5)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--n", type=int, default=3_000_000)
    p.add_argument("--d", type=int, default=384)
    # T = 64 trees and w = 1024 on each side: of the (T, w) cells whose
    # recall@15 reaches 0.81 in the recall sweep (0.819 here), the one whose
    # BF16-form step measured fastest (the configured T = 32, w = 32 reaches
    # 0.28). The plain form cannot run w > 704: it is compared at its own
    # cheapest cell of the sweep above 0.81 with w <= 704, T = 96, w = 640
    # (0.817; its pair work grows with T w).
    p.add_argument("--T", type=int, default=64)
    p.add_argument("--w", type=int, default=1024)
    p.add_argument("--plain-T", type=int, default=96)
    p.add_argument("--plain-w", type=int, default=640)
    p.add_argument("--k", type=int, default=15)
    p.add_argument("--bits", type=int, default=8)
    p.add_argument("--nq", type=int, default=10_000)
    p.add_argument("--components", type=int, default=1000)
    p.add_argument("--recall-sample", type=int, default=2000)
    p.add_argument("--e2e-steps", type=int, default=2)
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--cpu-sample", type=int, default=4000, help="points per oracle process")
    p.add_argument("--mode", default="tensor", choices=["plain", "tensor", "fp8"])
    p.add_argument("--search-w", type=int, default=32, help="window of the query search (positions [p-w, p+w))")
    p.add_argument("--plain-steps", type=int, default=1, help="plain-mode steps timed beside tensor mode")
    p.add_argument("--tensor-slack", type=int, default=-1)
    p.add_argument("--no-learned", action="store_true", help="skip the learned per-point budget form")
    p.add_argument("--label-sample", type=int, default=200_000, help="points of the label sample")
    p.add_argument("--label-forests", type=int, default=5, help="forests (seeds) over the label sample")
    p.add_argument("--train-steps", type=int, default=3000)
    p.add_argument("--no-sketch", action="store_true", help="skip the sketch-form comparison")
    p.add_argument("--no-batched", action="store_true", help="skip the batched form (64 independent sets)")
    p.add_argument("--no-tiny", action="store_true", help="skip the tiny configuration (20,000 x 16)")
    p.add_argument("--batched-sets", type=int, default=64)
    p.add_argument("--batched-recall", type=float, default=0.8, help="autotuner recall target per d group")
    p.add_argument("--batched-steps", type=int, default=3)
    p.add_argument("--sketch-bits", type=int, default=384)
    p.add_argument("--sketch-graph", default="80,48,60",
                   help="T,w,k2 of the sketch-form graph (the paper's first Table 2 row: 80 sorts, k1 = 96, k2 = 60)")
    p.add_argument("--sketch-search", default="128,300,2",
                   help="w,k2,h of the sketch-form search over the main forest")
    p.add_argument("--workload", default="graph", choices=["graph", "c3"],
                   help="graph: the kNN-graph step (default); c3: the large search workload (23M x 384, T = 160, "
                        "w = 50, k = 30, 10k queries), one JSON line of its own")
    p.add_argument("--c3-n", type=int, default=23_000_000)
    p.add_argument("--c3-w", default="50,200,710",
                   help="query windows of the c3 workload (the first is the configured one; the others trace "
                        "recall against time, 710 being Table 1's k1 = 1420 around each position)")
    p.add_argument("--recall-sweep", default="",
                   help="comma-separated T list x w list, e.g. '8,16,32,64,128,256:16,32,64,128,256': "
                        "print the plain method's recall@k over that (T, w) grid and exit")
    return p.parse_args()


def dist_env():
    r = int(os.environ.get("RANK", "0"))
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    lr = int(os.environ.get("LOCAL_RANK", "0"))
    return r, ws, lr


def workload_name(a):
    return (f"kNN graph + search: n={a.n} d={a.d} mixture({a.components}) T={a.T} b={a.bits} "
            f"w={a.w} k={a.k}; {a.nq} queries (w={a.search_w})")


class ClockSampler:
    """nvidia-smi samples (every 200 ms) during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.rows, self.proc, self.gpu = [], None, gpu_index

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.th = threading.Thread(target=self._read, daemon=True)
            self.th.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([c.strip() for c in line.split(",")])

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            try:
                sm.append(float(r[0]))
                mx.append(float(r[1]))
            except (ValueError, IndexError):
                continue
            for nm, v in zip(names, r[4:8]):
                if v.strip().lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def max_over_ranks(v, dist, dev):
    """The slowest rank's figure (every rank gets it); v itself with one rank.
    The data path has no collective: ranks are independent replicas."""
    if not dist:
        return v
    import torch
    t = torch.tensor([v], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(ws, n, ms_step):
    """Whole-job points/s: every rank processes its own n points per step."""
    return ws * n / (ms_step * 1e-3)


def make_inputs(a, rank):
    import synthdata as S
    x = S.gaussian_mixture(a.n, a.d, n_components=a.components, seed=S.SEED_DATA + 1000 * rank)
    q = S.mixture_queries(a.nq, a.d, n_components=a.components, data_seed=S.SEED_DATA + 1000 * rank,
                          seed=S.SEED_QUERIES)
    return x, q


def exact_knn_gpu(xd, rows_d, k, exclude=None, chunk=None):
    """Ground truth for the recall figure: float32 inner-product screen on the
    GPU (torch matmul, TF32 off), keep k + 16, re-score in float64 on the host
    with exact coordinate differences, order by (distance, index)."""
    import torch
    torch.backends.cuda.matmul.allow_tf32 = False
    nrm = (xd * xd).sum(1)
    out = []
    keep = k + 16
    if chunk is None:  # the distance block stays near 1 GB
        chunk = max(1, min(512, (1 << 28) // xd.shape[0]))
    for s in range(0, rows_d.shape[0], chunk):
        q = rows_d[s:s + chunk]
        g = nrm[None, :] + (q * q).sum(1)[:, None] - 2.0 * (q @ xd.T)
        if exclude is not None:
            g[torch.arange(q.shape[0], device=q.device), exclude[s:s + chunk]] = float("inf")
        cand = torch.topk(g, keep, dim=1, largest=False).indices
        for r in range(q.shape[0]):
            c = cand[r]
            diff = (xd[c].double() - q[r].double()[None, :])
            dd = (diff * diff).sum(1).cpu().numpy()
            cc = c.cpu().numpy()
            o = np.lexsort((cc, dd))[:k]
            out.append(cc[o])
    return np.array(out)


def dist_error(xd, rows_t, idx, dist):
    """Largest relative error of returned float32 distances against float64
    recomputations (exact coordinate differences) over the given rows."""
    ok = idx >= 0
    j = idx.clamp(min=0).long()
    diff = xd[j].double() - xd[rows_t].double()[:, None, :]
    true = (diff * diff).sum(-1)
    err = ((dist.double() - true).abs() / true.clamp(min=1e-30))[ok]
    return float(err.max().item()) if err.numel() else 0.0


def recall(found, exact):
    k = exact.shape[1]
    return float(np.mean([len(set(a[a >= 0].tolist()) & set(b.tolist())) / k for a, b in zip(found, exact)]))


def run_ours(a):
    import torch
    import paper_2508_21682_gb300 as hf

    rank, ws, lr = dist_env()
    torch.cuda.set_device(lr)
    dist = None
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", lr))
    import __graft_entry__ as g
    g.build()
    dev = torch.device("cuda", lr)
    x, q = make_inputs(a, rank)
    xd = torch.from_numpy(x).to(dev)
    qd = torch.from_numpy(q).to(dev)
    n, d, k, w, T = a.n, a.d, a.k, a.w, a.T
    gi = torch.empty((n, k), dtype=torch.int32, device=dev)
    gd = torch.empty((n, k), dtype=torch.float32, device=dev)
    si = torch.empty((a.nq, k), dtype=torch.int32, device=dev)
    sd = torch.empty((a.nq, k), dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)

    def step(tim=None, T=T, w=w):
        G = hf.build(xd, T=T, bits=a.bits, seed=3)
        if a.mode != "plain":
            G.set_option("mode", MODES[a.mode])
            G.set_option("tensor_slack", a.tensor_slack)
        G.knn_graph(k, w, gi, gd)
        G.search(qd, k, a.search_w, si, sd)
        if tim is not None:
            tim.append(G.timings())
        G.close()

    for _ in range(a.warmup):
        step()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(a.steps)]
    phases = []
    l0 = hf.launch_count()
    with ClockSampler(lr) as clk:
        for e0, e1 in evs:
            e0.record(stream)
            step(phases)
            e1.record(stream)
        torch.cuda.synchronize()
    launches = hf.launch_count() - l0
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    ms = [e0.elapsed_time(e1) for e0, e1 in evs]
    ms_step = max_over_ranks(sum(ms) / len(ms), dist, dev)

    ph = {kk: statistics.mean(p[kk] for p in phases) for kk in phases[0]}
    # per Gram launch: the library's CUDA events around each band launch (the
    # row gathers run on a second stream, overlapping the previous band)
    launch_ms = (ph["gram"] if ph.get("gram", 0.0) > 0 else ph["window_merge"] - ph.get("gather", 0.0)) / T
    if a.mode != "plain":
        roof = gram_roofline(a, launch_ms, ph.get("gather", 0.0) / T)
    else:
        roof = window_roofline(a, launch_ms)

    # end to end through the C ABI with pinned host buffers, right after the
    # timed region (the same device state as the timed steps)
    xh = torch.from_numpy(x).pin_memory()
    qh = torch.from_numpy(q).pin_memory()
    gih = torch.empty((n, k), dtype=torch.int32).pin_memory()
    gdh = torch.empty((n, k), dtype=torch.float32).pin_memory()
    sih = torch.empty((a.nq, k), dtype=torch.int32).pin_memory()
    sdh = torch.empty((a.nq, k), dtype=torch.float32).pin_memory()
    e2e_ms, e2e_calls = [], []
    for i in range(a.e2e_steps + 1 if a.e2e_steps > 0 else 0):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        G = hf.build(xh, T=T, bits=a.bits, seed=3)
        t1 = time.perf_counter()
        if a.mode != "plain":
            G.set_option("mode", MODES[a.mode])
            G.set_option("tensor_slack", a.tensor_slack)
        G.knn_graph(k, w, gih, gdh)
        t2 = time.perf_counter()
        G.search(qh, k, a.search_w, sih, sdh)
        t3 = time.perf_counter()
        G.close()
        torch.cuda.synchronize()
        t4 = time.perf_counter()
        if i:  # first one is a warm-up
            e2e_ms.append((t4 - t0) * 1e3)
            # each call returns only after its stream has drained, so these
            # wall-clock spans are the calls' own
            e2e_calls.append({"build": (t1 - t0) * 1e3, "graph": (t2 - t1) * 1e3, "search": (t3 - t2) * 1e3,
                              "close": (t4 - t3) * 1e3})
    e2e_step = max_over_ranks(statistics.mean(e2e_ms) if e2e_ms else float("nan"), dist, dev)

    # plain float32 mode beside it (outside the timed region)
    plain = None
    if a.mode != "plain" and a.plain_steps > 0:
        saved = a.mode
        a.mode = "plain"
        pT, pw = a.plain_T, a.plain_w
        step(T=pT, w=pw)
        torch.cuda.synchronize()
        pe = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(a.plain_steps)]
        for e0, e1 in pe:
            e0.record(stream)
            step(T=pT, w=pw)
            e1.record(stream)
        torch.cuda.synchronize()
        a.mode = saved
        pms = statistics.mean(e0.elapsed_time(e1) for e0, e1 in pe)
        plain = {"ms_per_step": pms, "value": n / (pms * 1e-3), "unit": "points/s", "T": pT, "w": pw}
        gi_plain = gi.cpu().numpy()

    # recall on a seeded sample (outside the timed region)
    rng = np.random.default_rng(4)
    rows = np.sort(rng.choice(n, size=min(a.recall_sample, n), replace=False))
    rows_t = torch.from_numpy(rows).to(dev)
    ex = exact_knn_gpu(xd, xd[rows_t], k, exclude=rows_t)
    if plain is not None:
        plain["recall_at_k"] = recall(gi_plain[rows], ex)
        step()  # the default mode's graph again for its own recall
        torch.cuda.synchronize()
    rec = recall(gi.cpu().numpy()[rows], ex)
    dist_err = dist_error(xd, rows_t, gi[rows_t], gd[rows_t])
    qs = min(500, a.nq)
    exq = exact_knn_gpu(xd, qd[:qs], k)
    rec_q = recall(si[:qs].cpu().numpy(), exq)

    learned = None
    if not a.no_learned and a.mode != "plain":
        learned = learned_form(a, hf, xd, qd, rows, ex, si, sd, stream, dev)
    sketch = None
    if not a.no_sketch:
        sketch = sketch_form(a, hf, xd, qd, rows, ex, exq, qs, dev)
    batched = None
    if not a.no_batched and rank == 0:
        batched = batched_form(a, hf, dev)
    tiny = None
    if not a.no_tiny and rank == 0:
        tiny = tiny_form(a, hf, dev)


    cpu = None
    if rank == 0 and ws == 1 and not a.no_cpu_baseline:
        cpu = cpu_baseline(a)

    if rank == 0:
        clocks = clk.summary()
        hs_ms = ph["keys"] + ph["sort"] + ph["tie_fixup"]
        if int(round(ph.get("graph_form", 0.0))) != MODES[a.mode]:
            raise SystemExit(f"asked for the {a.mode} form, the library ran form {ph.get('graph_form')}")
        line = {
            "metric": METRIC,
            "value": job_value(ws, n, ms_step),
            "unit": "points/s",
            "n_gpus": ws,
            "steps": a.steps,
            "warmup": a.warmup,
            "ms_per_step": ms_step,
            "higher_is_better": True,
            "scaling": "weak",
            "vs_baseline": None,
            "dtype": {"plain": "f32", "tensor": "bf16+f32", "fp8": "e4m3+f32"}[a.mode],
            "data": "synthetic (seeded Gaussian mixture standing in for GOOAQ)",
            "config": {"workload": workload_name(a), "n": n, "d": d, "T": T, "bits": a.bits, "w": w, "k": k,
                       "queries": a.nq, "mode": {"plain": "plain f32", "tensor": "bf16 tcgen05 Gram + f32 re-rank",
                                              "fp8": "e4m3 tcgen05 Gram (scale per vector) + f32 re-rank"}[a.mode],
                       "l2": "inputs larger than L2 (points 4.6 GB per step)",
                       "parallelism": f"replicas x{ws}"},
            "recall_at_k": rec,
            "at_metric_recall": bool(rec >= 0.8),
            "max_rel_dist_err_vs_f64": dist_err,
            "keys_sort_hbm": keys_sort_hbm(a, ph),
            "recall_sample": int(len(rows)),
            "search_recall_at_k": rec_q,
            "hilbert_sort_mkeys_s": n * T / (hs_ms * 1e-3) / 1e6,
            "phase_ms": ph,
            "roofline": roof,
            "plain_f32": plain,
            "learned": learned,
            "sketch": sketch,
            "batched": batched,
            "tiny": tiny,
            "e2e": {"value": job_value(ws, n, e2e_step), "unit": "points/s",
                    "h2d_bytes_per_step": int(x.nbytes + q.nbytes),
                    "d2h_bytes_per_step": int(gih.numel() * 4 + gdh.numel() * 4 + sih.numel() * 4 + sdh.numel() * 4),
                    "ms_per_step": e2e_step,
                    "calls_ms": {c: statistics.mean(r[c] for r in e2e_calls) for c in e2e_calls[0]}
                    if e2e_calls else None},
            "gpu_launches": int(launches),
            "clocks": clocks,
            "cpu_baseline": cpu,
        }
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


def traffic_per_launch(entry, n):
    src = open(os.path.join(ROOT, "paper_2508_21682_gb300", "csrc", entry["file"]), "rb").read()
    if entry["bytes_per_point"] and entry["source_sha"] == hashlib.sha256(src).hexdigest()[:16]:
        return entry["bytes_per_point"] * n
    return None


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return json.load(fh), "of measured"
    except (OSError, ValueError):
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "of fallback"


def keys_sort_hbm(a, ph):
    """Achieved HBM bandwidth of key generation and of the radix sort, from
    the library's phase timings (CUDA events on the launching stream).

    Algorithmic bytes per point and tree: keys read the permuted top bits of
    the point (d / 8 bytes of the bit-sliced top plane when the K-word prefix
    lies in the top bit level, d * L / 8 bytes of planes otherwise) and write
    K 64-bit words. The sort reads the K words for its histograms (8 K bytes),
    makes the passes that its plan keeps (sort_passes of the timings; each reads
    and writes one 64-bit key word and one 32-bit index, 24 bytes), reads the
    first word of the partial order to refine it where passes were left out (8),
    and gathers the words that were not sorted last (4 bytes of index and 16 a
    word: K - 1 words, K where the first one was not sorted by all its digits).
    all_digits is the rate at which the work of all 8 K passes was done, whatever
    the plan left out: no share of the bandwidth."""
    K = min(2, -(-a.d * a.bits // 64))
    L = min(a.bits, -(-64 * K // a.d))
    passes = ph.get("sort_passes") or 8.0 * K
    left_out = passes < 8 * K
    kb = a.n * a.T * (a.d * L / 8 + 8 * K)
    words = K - 1 + (1 if passes < 8 else 0)
    sb = a.n * a.T * (8 * K + 24 * passes + (8 if left_out else 0) + (4 + 16 * words if words else 0))
    peaks, src = measured_peaks()
    peak = float(peaks["hbm_gbs"])
    out = {"peak": peak, "unit": "GB/s", "peak_note": f"hbm_gbs {src} (MEASURED_PEAKS.json)"}
    for name, b, ms in (("keys", kb, ph["keys"]), ("sort", sb, ph["sort"])):
        ach = b / (ms * 1e-3) / 1e9 if ms > 0 else None
        out[name] = {"bytes": b, "ms": ms, "achieved": ach, "frac": ach / peak if ach else None}
    out["sort"]["passes_per_tree"] = passes
    out["sort"]["all_digits"] = a.n * a.T * 8 * K * 24 / (ph["sort"] * 1e-3) / 1e9 if ph["sort"] > 0 else None
    return out


def gram_work(a, fp8=False):
    """Algorithmic work of one Gram launch (one tree).

    Flops: every point against its 2w window neighbours (both ends of a pair
    score it, as the rows own their lists), 2 d flops each: n * 2w * 2d,
    without the band's tile waste. Bytes: the operand row (2 ceil64(d), or
    ceil128(d) for FP8), the point's list read and written (2 KP x 8 bytes,
    KP = list slots), its (norm, scale) and id (12 bytes)."""
    row = -(-a.d // 128) * 128 if fp8 else 2 * (-(-a.d // 64) * 64)
    slack = 1 if a.tensor_slack < 0 else a.tensor_slack
    kp = 16 if a.k + slack <= 16 else 32
    flops = 2.0 * a.n * 2 * a.w * a.d
    per_point = row + 2 * kp * 8 + 12
    return flops, per_point


def gram_roofline(a, launch_ms, gather_ms=0.0):
    """Roofline of one Gram launch (one tree) from the library's CUDA-event
    timings: at wide windows the band is a dense contraction, bound by the
    tensor pipe (peak: the measured sustained BF16 rate, as the kernel runs
    back to back for the whole step; the FP8 peak is twice it, the nominal
    ratio); the HBM side (algorithmic bytes over the same time) is given
    beside it. The per-tree row gather is a separate HBM-bound kernel."""
    fp8 = a.mode == "fp8"
    flops, per_point = gram_work(a, fp8)
    bytes_launch = per_point * a.n
    peaks, src = measured_peaks()
    tf_peak = float(peaks.get("bf16_tflops_sustained", peaks.get("bf16_tflops", 1700.0))) * (2.0 if fp8 else 1.0)
    hbm_peak = float(peaks["hbm_gbs"])
    t_ach = flops / (launch_ms * 1e-3) / 1e12
    b_ach = bytes_launch / (launch_ms * 1e-3) / 1e9
    rowb = (-(-a.d // 128) * 128) if fp8 else 2 * (-(-a.d // 64) * 64)
    g_bytes = 2.0 * a.n * rowb + 16.0 * a.n
    out = {"bound": "tensor", "kernel": "gram_band_kernel (A5+A6: tcgen05 Gram band + top-k merge)",
           "achieved": t_ach, "peak": tf_peak, "unit": "TFLOP/s", "frac": t_ach / tf_peak,
           "traffic": traffic_per_launch(GRAM_TRAFFIC, a.n) if a.w == GRAM_TRAFFIC["w"] and not fp8 else None,
           "flops_per_launch": flops, "launch_ms": launch_ms,
           "peak_note": f"bf16_tflops_sustained {src} (MEASURED_PEAKS.json)" + (" x 2 for e4m3" if fp8 else ""),
           "hbm_side": {"achieved": b_ach, "peak": hbm_peak, "unit": "GB/s", "frac": b_ach / hbm_peak,
                        "bytes_per_launch": bytes_launch, "bytes_per_point": per_point}}
    if gather_ms > 0:
        ga = g_bytes / (gather_ms * 1e-3) / 1e9
        out["gather"] = {"kernel": "gather_rows_kernel", "ms": gather_ms, "achieved": ga, "unit": "GB/s",
                         "frac": ga / hbm_peak, "bytes": g_bytes}
    if t_ach / tf_peak < b_ach / hbm_peak:  # narrow windows: the HBM side dominates
        out.update({"bound": "hbm", "achieved": b_ach, "peak": hbm_peak, "unit": "GB/s", "frac": b_ach / hbm_peak,
                    "peak_note": f"hbm_gbs {src} (MEASURED_PEAKS.json)"})
    return out


def window_roofline(a, launch_ms):
    """ALU roofline of one plain window launch: 3 flops per (pair, coordinate)."""
    n, w, d = a.n, a.w, a.d
    pairs = n * w - w * (w + 1) // 2
    flops = 3.0 * d * pairs
    achieved = flops / (launch_ms * 1e-3) / 1e12
    peak = SMS * FP32_LANES * MAX_SM_MHZ * 1e6 * 1.5 / 1e12
    return {"bound": "alu", "kernel": "pair_kernel + merge_kernel (A5+A6, plain f32)",
            "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
            "traffic": traffic_per_launch(WINDOW_TRAFFIC, n) if w == 32 else None, "launch_ms": launch_ms,
            "peak_note": "152 SMs x 128 FP32 lanes x 2070 MHz, 3 flops per FADD+FFMA pair"}


def oracle_sample(a, n_s, T_s, seed_offset=0):
    """Times the CPU oracle on n_s points of the same mixture, T_s trees."""
    import oracle as O
    import synthdata as S
    x = S.gaussian_mixture(n_s, a.d, n_components=a.components, seed=S.SEED_DATA + seed_offset)
    q = S.mixture_queries(max(1, a.nq * n_s // a.n), a.d, n_components=a.components,
                          data_seed=S.SEED_DATA + seed_offset, seed=S.SEED_QUERIES)
    t0 = time.perf_counter()
    F = O.Forest(x, T=T_s, bits=a.bits, seed=3)
    O.knn_graph(F, a.k, a.w)
    O.search(F, q, a.k, a.search_w)
    return time.perf_counter() - t0


def _oracle_worker(args):
    """One single-threaded oracle run (a spawned process of the pool)."""
    a, n_s, T_s, seed_offset = args
    try:
        from threadpoolctl import threadpool_limits
        threadpool_limits(1)
    except Exception:
        pass
    return oracle_sample(a, n_s, T_s, seed_offset=seed_offset)


def host_cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def cpu_model():
    try:
        with open("/proc/cpuinfo") as fh:
            for line in fh:
                if line.lower().startswith(("model name", "cpu model", "hardware")):
                    return line.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return platform.processor() or platform.machine()


def oracle_parallel(a, procs, n_s, T_s, rounds=1):
    """The oracle as it stands, one single-threaded process per core: procs
    independent samples (each its own seeded data) run at once; returns the
    whole-job points/s (points of all samples per second of wall time,
    scaled from T_s to the workload's T trees) and the wall seconds."""
    import multiprocessing as mp
    ctx = mp.get_context("spawn")  # no fork of a process that has touched the GPU
    with ctx.Pool(procs) as pool:
        pool.map(_oracle_worker, [(a, 500, 1, 100 + i) for i in range(procs)])  # imports, warm caches
        walls = []
        for r in range(rounds):
            t0 = time.perf_counter()
            pool.map(_oracle_worker, [(a, n_s, T_s, 1000 * r + i) for i in range(procs)])
            walls.append(time.perf_counter() - t0)
    wall = statistics.mean(walls)
    return procs * n_s / (wall * a.T / T_s), wall


def cpp_oracle_parallel(a, threads, n_s, T_s):
    """The C++ oracle (scalar loops) on `threads` host threads at once, each on
    its own n_s-point sample with T_s trees (graph and pro-rata queries; ctypes
    releases the interpreter lock during the calls). The samples are made
    before the clock starts. Returns whole-job points/s scaled to a.T trees
    and the wall seconds."""
    from concurrent.futures import ThreadPoolExecutor

    import synthdata as S
    from oracle import c_oracle as C
    C.build()
    nq_s = max(1, a.nq * n_s // a.n)
    data = []
    for i in range(threads):
        x = S.gaussian_mixture(n_s, a.d, n_components=a.components, seed=S.SEED_DATA + 100 + i)
        q = S.mixture_queries(nq_s, a.d, n_components=a.components, data_seed=S.SEED_DATA + 100 + i,
                              seed=S.SEED_QUERIES)
        data.append((x, q))

    def run(xq):
        x, q = xq
        F = C.Forest(x, T=T_s, bits=a.bits, seed=3)
        C.knn_graph(F, a.k, a.w)
        C.search(F, q, a.k, a.search_w)

    with ThreadPoolExecutor(threads) as ex:
        t0 = time.perf_counter()
        list(ex.map(run, data))
        wall = time.perf_counter() - t0
    return threads * n_s / (wall * a.T / T_s), wall


def cpu_baseline(a):
    """The oracle on all host cores and on 8 of them (the paper's budget)."""
    n_s, T_s = min(a.cpu_sample, a.n), 1
    cores = host_cores()
    val, wall = oracle_parallel(a, cores, n_s, T_s)
    p8 = min(8, cores)
    val8, wall8 = oracle_parallel(a, p8, n_s, T_s) if p8 != cores else (val, wall)
    # the tiny configuration in full (20,000 x 16, T = 8, w = 16, k = 10),
    # in this process with numpy's own threads
    import synthdata as S
    import oracle as O
    xt = S.unit_gaussian(20_000, 16, seed=S.SEED_DATA)
    t0 = time.perf_counter()
    F = O.Forest(xt, T=8, bits=a.bits, seed=S.SEED_FOREST)
    O.knn_graph(F, 10, 16)
    tiny_s = time.perf_counter() - t0
    # the C++ oracle on the same kind of sample, all cores
    try:
        cval, cwall = cpp_oracle_parallel(a, cores, n_s, T_s)
        cpp = {"value": cval, "unit": "points/s", "threads": cores,
               "sample": f"C++ oracle (scalar loops, float64 distances), one thread per core, each on its own "
                         f"{n_s} points with {T_s} of {a.T} trees, w={a.w}, k={a.k}, queries pro rata; "
                         f"{cwall:.1f} s wall; scaled to {a.T} trees"}
    except Exception as e:  # a host without a C++ compiler still gets the numpy figures
        cpp = {"unavailable": f"{type(e).__name__}: {e}"[:200]}
    return {"value": val, "unit": "points/s", "cores": cores, "kind": "oracle", "cpp": cpp,
            "cpu": cpu_model(), "value_8": val8, "cores_8": p8,
            "tiny_full": {"workload": "20,000 x 16 unit Gaussian, T=8, b=8, w=16, k=10 (build + graph, in full)",
                          "s": tiny_s, "value": 20_000 / tiny_s, "unit": "points/s"},
            "sample": f"numpy oracle (float64), one single-threaded process per core, each on its own {n_s} points "
                      f"of the same mixture with {T_s} of {a.T} trees, w={a.w}, k={a.k}, queries pro rata "
                      f"(w={a.search_w}); {wall:.1f} s wall on {cores} cores, {wall8:.1f} s on {p8}; "
                      f"scaled to {a.T} trees"}


def learned_form(a, hf, xd, qd, rows, ex, si, sd, stream, dev):
    """The learned per-point budget on the same workload, beside the fixed one.

    Labels: a sample of a.label_sample points of the same mixture (its own
    seed), its exact kNN from the full-window tensor graph, a.label_forests
    forests of 64 orders each: every point of every forest gets the cheapest
    (T, w) of the grid {4..64} x {8..128} at which 12 of its 15 neighbours
    are candidates (1M labels for 5 x 200k). The MLP is trained on them on
    the GPU, predicts (log2 w, log2 T) for all n points; one factor 2^s
    scales every prediction (T capped at the forest's T), s the smallest that
    reaches recall@k >= 0.8 on the recall sample (per-point position gaps to
    the exact neighbours over the forest's orders give the recall of any
    budget). The step is then timed as the fixed one: build + graph with
    the per-point budgets + search."""
    import torch
    import synthdata as S
    n, d, k, T = a.n, a.d, a.k, a.T
    t0 = time.perf_counter()
    ns = min(a.label_sample, n)
    xs = torch.from_numpy(S.gaussian_mixture(ns, d, n_components=a.components, seed=S.SEED_DATA + 500)).to(dev)
    E = hf.build(xs, T=1, bits=a.bits, seed=1)
    E.set_option("mode", 1)
    E.set_option("tensor_slack", 17)
    ei, _ = E.knn_graph(k, ns)
    E.close()
    tg, wg = [4, 8, 16, 32, 64], [8, 16, 32, 64, 128]
    ys, last = [], []
    for r in range(a.label_forests):
        Gs = hf.build(xs, T=tg[-1], bits=a.bits, seed=100 + r)
        tgt, cells = Gs.budget_labels(ei, tg, wg, 12)
        ys.append(tgt)
        last.append(float((cells == len(tg) * len(wg) - 1).float().mean().item()))
        Gs.close()
    gen = torch.Generator(device="cpu").manual_seed(5)
    perm = torch.randperm(ns * len(ys), generator=gen).to(dev)
    X = xs.repeat(len(ys), 1)[perm].contiguous()
    Y = torch.cat(ys)[perm].contiguous()
    labels_s = time.perf_counter() - t0
    m = hf.Mlp(d, seed=5)
    loss = m.train(X, Y, batch=1024, steps=a.train_steps, lr=1e-3)
    torch.cuda.synchronize()
    train_s = time.perf_counter() - t0 - labels_s
    pred = m.predict(xd)
    m.close()
    del X, Y, xs
    # recall of any per-point budget on the sample rows, from position gaps
    G = hf.build(xd, T=T, bits=a.bits, seed=3)
    sig = torch.empty(n, dtype=torch.int32, device=dev)
    inv = torch.empty(n, dtype=torch.int64, device=dev)
    ar = torch.arange(n, device=dev)
    rows_t = torch.from_numpy(rows).to(dev)
    ex_t = torch.from_numpy(ex).to(dev)
    gaps = []
    for t in range(T):
        G.order(t, out=sig)
        inv[sig.long()] = ar
        gaps.append((inv[ex_t] - inv[rows_t][:, None]).abs())
    G.close()
    cm = torch.cummin(torch.stack(gaps), dim=0).values  # [T][R][k]
    prow = pred[rows_t].double()

    # two ways to apply the predictions: (w, T) both scaled by 2^s ("both"),
    # or every point on all T orders and the window 2^(log2 w + log2 T + s)
    # (the predicted total need spent on the window alone: "window")
    def budgets(p, shift, how):
        lw, lt = p[:, 0].double(), p[:, 1].double()
        if how == "both":
            w = torch.clamp(torch.round(2.0 ** (lw + shift)), 1, 4096).int()
            t = torch.clamp(torch.round(2.0 ** (lt + shift)), 1, T).int()
        else:
            w = torch.clamp(torch.round(2.0 ** (lw + lt + shift)), 1, 4096).int()
            t = torch.full_like(w, T)
        return w, t

    def est_recall(shift, how):
        w, t = budgets(prow, shift, how)
        g = cm[(t - 1).long(), torch.arange(len(rows), device=dev)]
        return float(((g <= w[:, None].long()).double().mean()).item())

    target = 0.805  # 0.8 plus the tensor form's estimate loss
    best = None
    for how in ("both", "window"):
        lo, hi = -12.0, 12.0
        if est_recall(hi, how) < target:
            continue
        for _ in range(24):
            mid = 0.5 * (lo + hi)
            if est_recall(mid, how) >= target:
                hi = mid
            else:
                lo = mid
        w, t = budgets(pred, hi, how)
        c = float((t.double() * (128.0 + 2.0 * w.double())).mean())
        if best is None or c < best[0]:
            best = (c, how, hi)
    if best is None:
        return {"reached": False, "note": "the capped budgets do not reach the target recall"}
    cost, how, hi = best
    w_pt, t_pt = budgets(pred, hi, how)
    w_pt, t_pt = w_pt.contiguous(), t_pt.contiguous()
    ucost = T * (128.0 + 2.0 * a.w)
    gi = torch.empty((n, k), dtype=torch.int32, device=dev)
    gd = torch.empty((n, k), dtype=torch.float32, device=dev)

    def step():
        Gb = hf.build(xd, T=T, bits=a.bits, seed=3)
        Gb.set_option("mode", MODES[a.mode])
        Gb.set_option("tensor_slack", a.tensor_slack)
        Gb.knn_graph_budget(k, w_pt, t_pt, gi, gd)
        Gb.search(qd, k, a.search_w, si, sd)
        Gb.close()

    step()
    torch.cuda.synchronize()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(3)]
    for e0, e1 in evs:
        e0.record(stream)
        step()
        e1.record(stream)
    torch.cuda.synchronize()
    ms = statistics.mean(e0.elapsed_time(e1) for e0, e1 in evs)
    rec = recall(gi.cpu().numpy()[rows], ex)
    return {"value": n / (ms * 1e-3), "unit": "points/s", "ms_per_step": ms, "recall_at_k": rec,
            "at_metric_recall": bool(rec >= 0.8), "applied_as": how, "shift": hi,
            "mean_w": float(w_pt.double().mean()),
            "mean_T": float(t_pt.double().mean()), "band_cost_vs_fixed": cost / ucost,
            "train": {"labels": ns * len(ys), "label_sample": ns, "forests": len(ys), "steps": a.train_steps,
                      "batch": 1024, "final_loss": loss, "labels_s": labels_s, "train_s": train_s,
                      "labels_at_largest_cell": float(np.mean(last))},
            "model": "MLP d-256-256-2, GELU, BF16 weights/activations, FP32 accumulation (tcgen05), Adam"}


def sketch_form(a, hf, xd, qd, rows, ex, exq, qs, dev):
    """The paper's second stage on this workload, outside the timed region:
    the graph in the sketch form against the BF16 Gram form at the same
    (T, w) budget, and the search in the sketch form against the plain search
    at the main window, each one timed step with its recall@k."""
    import torch
    import synthdata as S

    n, d, k = a.n, a.d, a.k
    Tg, wg, k2g = (int(v) for v in a.sketch_graph.split(","))
    ws, k2s, hs = (int(v) for v in a.sketch_search.split(","))
    R = torch.from_numpy(S.sketch_projection(a.sketch_bits, d)).to(dev)
    gi = torch.empty((n, k), dtype=torch.int32, device=dev)
    gd = torch.empty((n, k), dtype=torch.float32, device=dev)

    def ev():
        e = torch.cuda.Event(enable_timing=True)
        e.record()
        return e

    out = {"bits": a.sketch_bits, "projection": "i.i.d. N(0, 1) rows (sign random projection)"}
    graph = {"T": Tg, "w": wg, "k2": k2g}
    for form, mode in (("sketch", 3), ("tensor", 1)):
        G = hf.build(xd, T=Tg, bits=a.bits, seed=3)
        torch.cuda.synchronize()
        e0 = ev()
        if mode == 3:
            G.set_sketch(R)
            G.set_option("sketch_k2", k2g)
        G.set_option("mode", mode)
        G.knn_graph(k, wg, gi, gd)
        e1 = ev()
        torch.cuda.synchronize()
        ms = G.timings()
        graph[form] = {"ms_per_step": e0.elapsed_time(e1), "build_ms": ms["keys"] + ms["sort"] + ms["tie_fixup"],
                       "window_ms": ms["window_merge"], "rerank_ms": ms["rerank"],
                       "recall_at_k": recall(gi.cpu().numpy()[rows], ex)}
        graph[form]["value"] = n / (graph[form]["ms_per_step"] * 1e-3)
        G.close()
    out["graph"] = graph
    G = hf.build(xd, T=a.T, bits=a.bits, seed=3)
    G.set_sketch(R)
    search = {"T": a.T, "k": k, "queries": a.nq}
    for form, mode, w in (("sketch", 3, ws), ("plain", 0, a.search_w)):
        G.set_option("mode", mode)
        G.set_option("sketch_k2", k2s)
        G.set_option("expand_h", hs)
        G.search(qd, k, w)  # the first sketch search builds the master layout
        torch.cuda.synchronize()
        e0 = ev()
        si, _ = G.search(qd, k, w)
        e1 = ev()
        torch.cuda.synchronize()
        search[form] = {"w": w, "ms": e0.elapsed_time(e1), "queries_per_s": a.nq / (e0.elapsed_time(e1) * 1e-3),
                        "recall_at_k": recall(si[:qs].cpu().numpy(), exq)}
        if mode == 3:
            search[form].update({"k2": k2s, "h": hs})
    out["search"] = search
    G.close()
    return out


def tiny_form(a, hf, dev):
    """The tiny configuration: n = 20,000, d = 16 unit Gaussian rows, T = 8,
    b = 8, w = 16, k = 10. Everything fits in L2, so the figure is absolute
    time (launch- and latency-bound), not a roofline fraction. Plain float32
    form (the configuration's distances) and the BF16 Gram form, each the
    median of 9 steps (build + graph, CUDA events), with recall@10 against
    exact brute force on every tenth point."""
    import torch
    import synthdata as S

    n, d, T, w, k = 20_000, 16, 8, 16, 10
    xd = torch.from_numpy(S.unit_gaussian(n, d, seed=S.SEED_DATA)).to(dev)
    rows = np.arange(0, n, 10)  # every tenth point: 2,000 recall rows
    rows_t = torch.from_numpy(rows).to(dev)
    ex = exact_knn_gpu(xd, xd[rows_t], k, exclude=rows_t)
    gi = torch.empty((n, k), dtype=torch.int32, device=dev)
    gd = torch.empty((n, k), dtype=torch.float32, device=dev)
    st = torch.cuda.current_stream(dev)
    out = {"workload": f"n={n}, d={d} unit Gaussian, T={T}, b={a.bits}, w={w}, k={k}"}
    for form, mode in (("plain", 0), ("tensor", 1)):
        ms = []
        for i in range(10):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(st)
            G = hf.build(xd, T=T, bits=a.bits, seed=S.SEED_FOREST)
            G.set_option("mode", mode)
            G.knn_graph(k, w, gi, gd)
            G.close()
            e1.record(st)
            torch.cuda.synchronize(dev)
            if i:
                ms.append(e0.elapsed_time(e1))
        med = statistics.median(ms)
        out[form] = {"us_per_step": med * 1e3, "value": n / (med * 1e-3), "unit": "points/s",
                     "recall_at_k": recall(gi.cpu().numpy()[rows], ex)}
    return out


def batched_form(a, hf, dev):
    """The batched workload, outside the main timed region: independent sets
    (sizes log-uniform in [1,000, 200,000], d from {64, 128, 384, 768}, 100-
    component mixtures, T = 16, b = 8, k = 10), stacked per dimension into one
    segmented forest each. The autotuner picks each group's window and block
    size for the recall target on a sample; a step is the segmented builds
    plus one CUDA-graph replay of all groups' graphs. Beside it, the same sets
    one at a time (hf_build + hf_knn_graph per set, same windows)."""
    import torch
    import synthdata as S

    T, k = 16, 10
    sets = S.batched_sets(a.batched_sets)
    dims = sorted({x.shape[1] for x in sets})
    groups = []
    for d in dims:
        idx = [i for i, x in enumerate(sets) if x.shape[1] == d]
        off = np.zeros(len(idx) + 1, np.int64)
        off[1:] = np.cumsum([sets[i].shape[0] for i in idx])
        X = torch.from_numpy(np.concatenate([sets[i] for i in idx])).to(dev)
        groups.append({"d": d, "idx": idx, "off": off, "X": X})
    n_total = int(sum(x.shape[0] for x in sets))
    side = torch.cuda.Stream(dev)
    side.wait_stream(torch.cuda.current_stream(dev))
    # autotune per group (one build each)
    for g in groups:
        G = hf.build_segmented(g["X"], g["off"], T=T, bits=a.bits, seed=3)
        g["tune"] = G.autotune(k, a.batched_recall, sample=1024, w_max=704, forms=7)
        G.close()
    for g in groups:
        n = g["X"].shape[0]
        g["oi"] = torch.empty((n, k), dtype=torch.int32, device=dev)
        g["od"] = torch.empty((n, k), dtype=torch.float32, device=dev)

    def ev(st):
        e = torch.cuda.Event(enable_timing=True)
        e.record(st)
        return e

    def batched_step(capture_graph):
        with torch.cuda.stream(side):
            forests = [hf.build_segmented(g["X"], g["off"], T=T, bits=a.bits, seed=3) for g in groups]
            for G, g in zip(forests, groups):
                G.set_option("mode", g["tune"]["form"])
                if g["tune"]["form"]:
                    G.set_option("tensor_slack", g["tune"]["list_slots"] - k)
                G.graph_plan(k, g["tune"]["w"], g["tune"]["threads"], side.cuda_stream)
            graph = None
            if capture_graph:
                graph = hf.CudaGraph(side.cuda_stream)
                with graph:
                    for G, g in zip(forests, groups):
                        G.knn_graph_enqueue(g["oi"], g["od"], side.cuda_stream)
            return forests, graph

    # warm-up (also the capture's first use)
    forests, graph = batched_step(True)
    graph.launch()
    for G in forests:
        G.status(side.cuda_stream)
    l_cap = None
    ms, build_ms, replay_ms = [], [], []
    for _ in range(a.batched_steps):
        for G in forests:
            G.close()
        graph.close()
        torch.cuda.synchronize(dev)
        l0 = hf.launch_count()
        e0 = ev(side)
        forests, graph = batched_step(True)
        e1 = ev(side)
        l1 = hf.launch_count()
        graph.launch()
        e2 = ev(side)
        for G in forests:
            G.status(side.cuda_stream)
        ms.append(e0.elapsed_time(e2))
        build_ms.append(e0.elapsed_time(e1))
        replay_ms.append(e1.elapsed_time(e2))
        l_cap = l1 - l0
    step_ms = statistics.mean(ms)
    # per-set recall on sampled rows (exact rows within each set)
    per_set = [None] * len(sets)
    for G, g in zip(forests, groups):
        gi = g["oi"].cpu().numpy()
        for j, i in enumerate(g["idx"]):
            a0, a1 = int(g["off"][j]), int(g["off"][j + 1])
            rows = np.unique(np.linspace(a0, a1 - 1, num=min(32, a1 - a0)).astype(np.int64))
            ei, _ = G.exact_knn_rows(rows, k)
            hit = sum(len(set(x[x >= 0]) & set(y[y >= 0])) for x, y in zip(gi[rows], ei))
            rt = torch.from_numpy(rows).to(dev)
            per_set[i] = {"n": a1 - a0, "d": g["d"], "recall_at_k": hit / max(1, int((ei >= 0).sum())),
                          "max_rel_dist_err_vs_f64": dist_error(g["X"], rt, g["oi"][rt], g["od"][rt])}
    for G in forests:
        G.close()
    graph.close()
    # the same sets one at a time
    wmap = {g["d"]: g["tune"]["w"] for g in groups}
    fmap = {g["d"]: g["tune"]["form"] for g in groups}
    smap = {g["d"]: g["tune"]["list_slots"] for g in groups}
    xs = [torch.from_numpy(x).to(dev) for x in sets]
    one_ms = []
    l0 = hf.launch_count()
    for i, x in enumerate(xs):
        torch.cuda.synchronize(dev)
        e0 = ev(torch.cuda.current_stream(dev))
        G = hf.build(x, T=T, bits=a.bits, seed=3)
        G.set_option("mode", fmap[x.shape[1]])
        if fmap[x.shape[1]]:
            G.set_option("tensor_slack", smap[x.shape[1]] - k)
        G.knn_graph(k, wmap[x.shape[1]])
        e1 = ev(torch.cuda.current_stream(dev))
        torch.cuda.synchronize(dev)
        one_ms.append(e0.elapsed_time(e1))
        per_set[i]["one_at_a_time_ms"] = one_ms[-1]
        per_set[i]["one_at_a_time_points_per_s"] = x.shape[0] / (one_ms[-1] * 1e-3)
        G.close()
    l_one = hf.launch_count() - l0
    loop_ms = float(sum(one_ms))
    return {
        "workload": f"{len(sets)} independent sets, sizes log-uniform [1000, 200000], d in {{64,128,384,768}}, "
                    f"100-component mixtures, T={T}, b={a.bits}, k={k}",
        "sets": len(sets), "points": n_total,
        "groups": [{"d": g["d"], "sets": len(g["idx"]), "points": int(g["X"].shape[0]), **g["tune"]} for g in groups],
        "ms_per_step": step_ms, "build_ms": statistics.mean(build_ms), "graph_replay_ms": statistics.mean(replay_ms),
        "value": n_total / (step_ms * 1e-3), "unit": "points/s",
        "launches_per_step": int(l_cap), "one_at_a_time": {"ms": loop_ms, "value": n_total / (loop_ms * 1e-3),
                                                           "launches": int(l_one)},
        "speedup_vs_one_at_a_time": loop_ms / step_ms,
        "recall_target": a.batched_recall,
        "recall_at_k_mean": float(np.mean([p["recall_at_k"] for p in per_set])),
        "max_rel_dist_err_vs_f64": float(max(p["max_rel_dist_err_vs_f64"] for p in per_set)),
        "per_set": per_set,
    }


def recall_sweep(a):
    """Recall@k of the plain method over a (T, w) grid from one forest.

    Point e is in point i's window of tree t exactly when their positions
    differ by at most w (and e != i), and the graph's top k of a candidate set
    C holds every true neighbour that C holds (they are the k nearest of all
    points), so recall@k = |E(i) & C(i)| / k with E the exact k nearest. The
    smallest position gap over the first T trees therefore gives recall at
    every (T, w) at once."""
    import torch
    import paper_2508_21682_gb300 as hf
    import __graft_entry__ as g
    g.build()
    ts_s, ws_s = a.recall_sweep.split(":")
    Ts = sorted(int(v) for v in ts_s.split(","))
    Ws = sorted(int(v) for v in ws_s.split(","))
    dev = torch.device("cuda", 0)
    x, _ = make_inputs(a, 0)
    xd = torch.from_numpy(x).to(dev)
    n = a.n
    rng = np.random.default_rng(4)
    rows = np.sort(rng.choice(n, size=min(a.recall_sample, n), replace=False))
    rows_t = torch.from_numpy(rows).to(dev)
    ex = torch.from_numpy(exact_knn_gpu(xd, xd[rows_t], a.k, exclude=rows_t)).to(dev)
    t0 = time.perf_counter()
    G = hf.build(xd, T=Ts[-1], bits=a.bits, seed=3)
    torch.cuda.synchronize()
    build_s = time.perf_counter() - t0
    sig = torch.empty(n, dtype=torch.int32, device=dev)
    inv = torch.empty(n, dtype=torch.int64, device=dev)
    ar = torch.arange(n, device=dev)
    gap = torch.full(ex.shape, n, dtype=torch.int64, device=dev)
    table = {}
    for t in range(Ts[-1]):
        G.order(t, out=sig)
        inv[sig.long()] = ar
        gap = torch.minimum(gap, (inv[ex] - inv[rows_t][:, None]).abs())
        if t + 1 in Ts:
            table[str(t + 1)] = {str(w): float((gap <= w).double().mean()) for w in Ws}
    G.close()
    print(json.dumps({"recall_sweep": table, "k": a.k, "n": n, "d": a.d, "sample": int(len(rows)),
                      "build_s_T%d" % Ts[-1]: build_s, "workload": workload_name(a)}), flush=True)


def run_reference(a):
    rank, ws, lr = dist_env()
    if rank != 0:
        return
    n_s, T_s = min(a.cpu_sample, a.n), 1
    cores = host_cores()
    val, sec = oracle_parallel(a, cores, n_s, T_s, rounds=a.steps)
    line = {
        "impl": "reference",
        "metric": METRIC,
        "value": val,
        "unit": "points/s",
        "n_gpus": ws,
        "steps": a.steps,
        "warmup": a.warmup,
        "ms_per_step": sec * 1e3,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64",
        "data": "synthetic (seeded Gaussian mixture standing in for GOOAQ)",
        "config": {"workload": workload_name(a), "n": a.n, "d": a.d, "T": a.T, "bits": a.bits, "w": a.w,
                   "k": a.k, "queries": a.nq},
        "cpu_baseline": {"value": val, "unit": "points/s", "cores": cores, "kind": "oracle", "cpu": cpu_model(),
                         "sample": f"numpy oracle (float64) per step: one single-threaded process per core, each on "
                                   f"its own {n_s} points with {T_s} of {a.T} trees, queries pro rata; "
                                   f"scaled to {a.T} trees"},
        "e2e": {"value": val, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def run_c3(a):
    """The large search workload: n points (23M by default) x 384 from the
    mixture, T = 160 trees, b = 8, query window w = 50 on each side (about 100
    candidates per tree), k = 30, 10,000 mixture queries. One JSON line:
    queries/s of hf_search (CUDA events, inputs resident), the build's time,
    recall@30 on 500 queries, and the largest relative error of the returned
    float32 distances against float64 on 200 queries."""
    import torch
    import synthdata as S
    import __graft_entry__ as g
    g.build()
    import paper_2508_21682_gb300 as hf

    n, d, T, k, nq = a.c3_n, 384, 160, 30, 10_000
    windows = [int(v) for v in a.c3_w.split(",")]
    w = windows[0]
    dev = torch.device("cuda", 0)
    t0 = time.perf_counter()
    xd = torch.from_numpy(S.gaussian_mixture(n, d, n_components=1000, seed=S.SEED_DATA)).to(dev)
    qd = torch.from_numpy(S.mixture_queries(nq, d, n_components=1000, data_seed=S.SEED_DATA)).to(dev)
    gen_s = time.perf_counter() - t0
    st = torch.cuda.current_stream(dev)

    def ev():
        e = torch.cuda.Event(enable_timing=True)
        e.record(st)
        return e

    torch.cuda.synchronize()
    e0 = ev()
    G = hf.build(xd, T=T, bits=a.bits, seed=3)
    e1 = ev()
    torch.cuda.synchronize()
    build_ms = e0.elapsed_time(e1)
    ph = G.timings()
    ex = exact_knn_gpu(xd, qd[:500], k)
    sweep = []
    for wv in windows:
        si, sd = G.search(qd, k, wv)  # warm-up
        torch.cuda.synchronize()
        reps = max(3, a.steps)
        e0 = ev()
        for _ in range(reps):
            G.search(qd, k, wv, si, sd)
        e1 = ev()
        torch.cuda.synchronize()
        sweep.append({"w": wv, "ms_per_batch": e0.elapsed_time(e1) / reps,
                      "queries_per_s": nq / (e0.elapsed_time(e1) / reps * 1e-3),
                      "recall_at_k": recall(si[:500].cpu().numpy(), ex)})
        if wv == w:
            first = (si.clone(), sd.clone())
    si, sd = first
    ms, rec = sweep[0]["ms_per_batch"], sweep[0]["recall_at_k"]
    gi = si[:200].long()
    diff = xd[gi.clamp(min=0)].double() - qd[:200].double()[:, None, :]
    true = (diff * diff).sum(-1)
    ok = gi >= 0
    err = ((sd[:200].double() - true).abs() / true.clamp(min=1e-30))[ok].max().item()
    free_b, total_b = torch.cuda.mem_get_info(dev)
    G.close()
    print(json.dumps({
        "workload": f"search: n={n}, d={d} float32 mixture (1000 components), T={T}, b={a.bits}, "
                    f"w={w} on each side, k={k}, {nq} mixture queries",
        "metric": "queries/s", "value": nq / (ms * 1e-3), "unit": "queries/s", "ms_per_batch": ms,
        "recall_at_k": rec, "recall_sample": 500, "windows": sweep, "build_ms": build_ms,
        "build_phase_ms": {kk: ph[kk] for kk in ("quantize", "keys", "sort", "tie_fixup")},
        "hilbert_sort_mkeys_s": n * T / ((ph["keys"] + ph["sort"] + ph["tie_fixup"]) * 1e-3) / 1e6,
        "max_rel_dist_err_vs_f64": err, "generation_s": gen_s, "device_bytes_in_use": int(total_b - free_b),
        "storage": "float32 rows (the library reads float32; 35 GB at 23M x 384)",
    }), flush=True)


if __name__ == "__main__":
    A = args()
    if A.impl == "reference":
        run_reference(A)
    elif A.workload == "c3":
        run_c3(A)
    elif A.recall_sweep:
        recall_sweep(A)
    else:
        run_ours(A)
