#!/usr/bin/env python
"""Benchmark of the biased graph-attention hot path on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME] [--impl reference] [--mode step|ring]

One step = one pass of the whole hot path over one seeded synthetic batch:
gt_spd_build -> gt_biased_attn_fwd -> gt_biased_attn_bwd -> gt_biased_attn_fwd_chunked.
The headline metric is forward+backward attention TFLOP/s (14*H*d*sum n_g^2 FLOPs per step
divided by the forward+backward time inside the step, CUDA events); the SPD build GB/s, the
chunked forward and the whole-step time are reported beside it.  With N > 1 (torchrun) every
rank processes its own batch: weak scaling over independent batches, no data-path collective.

`--mode ring` (under torchrun with N > 1, or alone) measures graph-aware context parallelism instead: ONE
graph, query rows and bias rows sharded over the ranks, K/V blocks (and in the backward their dK/dV sums)
passed round the ring with torch.distributed P2P while every rank runs the caller-driven step kernels on
the block it holds; strong scaling, whole-job FLOPs over the max-over-ranks time.

`--impl reference` times the CPU oracle (fp64, host cores) on a bounded row sample of the
same workload and prints the same JSON line with "impl": "reference".
"""
from __future__ import annotations

import argparse
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

from paper_2609_34420_b200 import workloads as wl  # noqa: E402

METRIC = "fwd+bwd biased-attention TFLOP/s"
UNIT = "TFLOP/s"
DEFAULT_WORKLOAD = "powerlaw64k"
ORACLE_SAMPLE_ROWS = 256
FALLBACK_PEAKS = {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0}
# Measured DRAM traffic (dram__bytes_read.sum + dram__bytes_write.sum of one ncu capture) per launch of the
# backward kernel on a 16 384-node graph, divided by N^2: the traffic is dominated by the N^2 bias-index tiles
# and the N^2/128 dQ reductions, so a launch at another size is estimated as this figure times sum n_g^2.
BWD_KERNEL_DRAM_BYTES_PER_N2 = 1037.7e6 / (16384.0 ** 2)
# The same for the forward kernel (16 384 nodes) and for the bit-matrix SPD build (32 768 nodes, search and expansion
# together; its traffic also grows with the number of BFS levels, so the scaled figure is an estimate).
FWD_KERNEL_DRAM_BYTES_PER_N2 = 438.1e6 / (16384.0 ** 2)
SPD_DENSE_DRAM_BYTES_PER_N2 = 2.262e9 / (32768.0 ** 2)


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            return json.load(fh), "measured"
    return dict(FALLBACK_PEAKS), "fallback"


def host_cores() -> int:
    return len(os.sched_getaffinity(0))


# --------------------------------------------------------------------------------------
# CPU oracle arm (also the cpu_baseline of the CUDA arm)
# --------------------------------------------------------------------------------------
def oracle_sample(w: wl.Workload, n_rows: int, seed: int = 123):
    """Time the oracle (BFS rows + fp64 forward + analytic backward) on `n_rows` seeded
    query rows of graph 0 of the workload.  Returns (seconds, flops_equivalent, spd_seconds)."""
    from oracle import attention as oattn
    from oracle import spd as ospd

    rp, ci = w.batch.graph_csr(0)
    n = len(rp) - 1
    t = w.tensors()
    a, b = int(w.batch.cu_seqlens[0]), int(w.batch.cu_seqlens[1])
    f = wl.bf16_bits_to_f64
    q, k, v, do = f(t.q[a:b]), f(t.k[a:b]), f(t.v[a:b]), f(t.dout[a:b])
    bias = t.bias.astype(np.float64)
    rows = np.sort(np.random.default_rng(seed).choice(n, size=min(n_rows, n), replace=False))
    ospd.spd_rows(rp, ci, w.max_dist, rows[:1])                 # build/load the C library outside the timing
    t0 = time.perf_counter()
    spd = ospd.spd_rows(rp, ci, w.max_dist, rows)
    t1 = time.perf_counter()
    oattn.forward_single(q, k, v, spd, bias, rows=rows, compact_spd=True)
    oattn.backward_single(q, k, v, do, spd, bias, rows=rows, compact_spd=True)
    t2 = time.perf_counter()
    flops = 14.0 * w.n_heads * w.head_dim * len(rows) * n
    return t2 - t1, flops, t1 - t0, len(rows), n


def run_reference(args) -> int:
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    w = wl.make_workload(args.workload)
    for _ in range(min(args.warmup, 1)):
        oracle_sample(w, 32)
    times, flops = [], 0.0
    for _ in range(args.steps):
        sec, flops, spd_sec, n_rows, n = oracle_sample(w, ORACLE_SAMPLE_ROWS)
        times.append(sec)
    ms = 1e3 * sum(times) / len(times)
    value = flops / (ms * 1e-3) / 1e12
    sample = f"{n_rows} seeded query rows of {n} (full key range), fp64 forward + analytic backward per step"
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "note": w.note, "n_heads": w.n_heads, "head_dim": w.head_dim,
                   "max_dist": w.max_dist, "n_total": w.batch.n_total},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": host_cores(), "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


# --------------------------------------------------------------------------------------
# clocks
# --------------------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, device_uuid: str):
        self.tmp = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.proc = None
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={device_uuid}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=self.tmp, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.tmp.flush()
        self.tmp.seek(0)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.tmp.read().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for name, val in zip(names, parts[4:8]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        self.tmp.close()
        os.unlink(self.tmp.name)
        busy = [x for x in sm if x > 0]
        return {"sm_mhz": statistics.median(busy) if busy else None, "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# --------------------------------------------------------------------------------------
# CUDA arm
# --------------------------------------------------------------------------------------
def run_cuda(args) -> int:
    import torch

    from paper_2609_34420_b200 import binding as gt
    from paper_2609_34420_b200 import dist_util

    if not torch.cuda.is_available():
        raise SystemExit("bench.py: no CUDA device (the CUDA path has no CPU fallback)")
    rank, local_rank, world = dist_util.env_world()
    dev = torch.device("cuda", local_rank)
    torch.cuda.set_device(dev)
    dist_util.init_process_group("nccl")
    gt.lib()

    w = wl.make_workload(args.workload, seed=dist_util.shard_seed(0, rank))
    b, t = w.batch, w.tensors()
    T, H, d, D = b.n_total, w.n_heads, w.head_dim, w.max_dist
    single = b.n_graphs == 1
    n_chunks = w.n_kv_chunks if single else 1

    def dev_bf16(bits):
        return torch.from_numpy(bits.view(np.int16)).to(dev).view(torch.bfloat16)

    # ---- device-resident inputs ----
    rp = torch.from_numpy(b.row_ptr).to(dev)
    ci = torch.from_numpy(b.col_idx).to(dev)
    batch = gt.Batch(T, b.n_graphs, b.max_seqlen,
                     None if single else torch.from_numpy(b.cu_seqlens).to(dev),
                     None if single else torch.from_numpy(b.spd_offsets).to(dev))
    q, k, v, do = dev_bf16(t.q), dev_bf16(t.k), dev_bf16(t.v), dev_bf16(t.dout)
    bias = torch.from_numpy(t.bias).to(dev)
    spd = torch.empty(b.spd_bytes, dtype=torch.uint8, device=dev)
    out, dq, dk, dv = (torch.empty_like(q) for _ in range(4))
    out_c = torch.empty_like(q)
    lse = torch.empty(H, T, dtype=torch.float32, device=dev)
    lse_c = torch.empty_like(lse)
    dbias = torch.empty_like(bias)
    ws_spd = gt._workspace(gt.gt_spd_build_workspace(batch, ci.numel(), D), dev)
    ws_fwd = gt._workspace(gt.gt_biased_attn_fwd_workspace(batch, H, d), dev)
    ws_bwd = gt._workspace(gt.gt_biased_attn_bwd_workspace(batch, H, d, D), dev)
    ws_chk = gt._workspace(gt.gt_biased_attn_fwd_chunked_workspace(batch, H, d, n_chunks), dev) if single else None

    def ev():
        return torch.cuda.Event(enable_timing=True)

    def step(marks=None):
        if marks is not None:
            marks[0].record()
        gt.gt_spd_build(rp, ci, batch, D, spd, ws_spd)
        if marks is not None:
            marks[1].record()
        gt.gt_biased_attn_fwd(q, k, v, spd, bias, batch, D, out, lse, ws_fwd)
        if marks is not None:
            marks[2].record()
        gt.gt_biased_attn_bwd(q, k, v, out, do, lse, spd, bias, batch, D, dq, dk, dv, dbias, ws_bwd)
        if marks is not None:
            marks[3].record()
        if single:
            gt.gt_biased_attn_fwd_chunked(q, k, v, spd, bias, batch, D, out_c, lse_c, n_chunks, None, ws_chk)
        if marks is not None:
            marks[4].record()

    # spd: one pull kernel where it needs no workspace beyond the header; a larger single graph: order, lists and pull, or beyond
    # 18 944 nodes two item scans, item table and bit-matrix BFS, from 32 768 to 65 536 nodes with the choice of a core (seven kernels),
    # a second form of the BFS and two of the expansion; a larger batch: setup, components, BFS.
    # fwd: (a batch's maps and work list,) main; bwd: prepare, main, finalize; chunked: main (in parts: partial, merge)
    dense_spd = single and b.max_seqlen > 18944           # the library's switch to the bit-matrix build
    spd_kernel = ("spd_pull_kernel" if ws_spd.numel() <= 256 else "spd_dense_kernel" if dense_spd else
                  "spd_large_pull_kernel" if single else "spd_bfs_kernel")
    spd_launches = 1 if spd_kernel == "spd_pull_kernel" else ((14 if 32768 <= b.max_seqlen <= 65536 else 4) if dense_spd else 3)
    kernels_per_step = spd_launches + (1 if single else 2) + 3 + (1 if single else 0)

    for _ in range(max(args.warmup, 0)):
        step()
    torch.cuda.synchronize()
    for wsx in (ws_spd, ws_fwd, ws_bwd) + ((ws_chk,) if single else ()):
        gt.gt_check(wsx)

    # ---- timed region ----
    sampler = ClockSampler("GPU-" + str(torch.cuda.get_device_properties(dev).uuid)) if rank == 0 else None
    marks = [[ev() for _ in range(5)] for _ in range(args.steps)]
    kern_ev = [[ev() for _ in range(args.steps)] for _ in range(2)]       # around the backward's main kernel, recorded by the library
    gt.gt_profile_bwd_kernel_events(kern_ev[0], kern_ev[1])
    e0, e1 = ev(), ev()
    dist_util.barrier(dev)
    torch.cuda.synchronize()
    e0.record()
    for i in range(args.steps):
        step(marks[i])
    e1.record()
    torch.cuda.synchronize()
    dist_util.barrier(dev)
    clocks = sampler.stop() if sampler else None
    for wsx in (ws_spd, ws_fwd, ws_bwd) + ((ws_chk,) if single else ()):
        gt.gt_check(wsx)

    gt.gt_profile_bwd_kernel_events([], [])
    bwd_kernel_ms = float(np.mean([a_.elapsed_time(b_) for a_, b_ in zip(kern_ev[0], kern_ev[1])]))
    total_ms = e0.elapsed_time(e1)
    ph = np.array([[m[j].elapsed_time(m[j + 1]) for j in range(4)] for m in marks])       # [K, 4]
    spd_ms, fwd_ms, bwd_ms, chk_ms = (float(x) for x in ph.mean(axis=0))
    phase_names = ("spd_build", "fwd", "bwd", "fwd_chunked")
    ph_median = {nm: float(x) for nm, x in zip(phase_names, np.median(ph, axis=0))}
    ph_min = {nm: float(x) for nm, x in zip(phase_names, ph.min(axis=0))}
    fb = ph[:, 1] + ph[:, 2]

    # ---- input statistics (outside the timed region): degrees, and the bucket histogram of a row sample of the built matrix ----
    deg = np.diff(b.row_ptr)
    n0 = int(b.cu_seqlens[1])
    ld0 = int(b.spd_ld[0])
    row_idx = torch.arange(0, n0, max(1, n0 // 1024), device=dev)[:1024]          # rows spread over the whole graph
    n_hist_rows = int(row_idx.numel())
    sample = spd[: n0 * ld0].view(n0, ld0)[row_idx][:, :n0]
    hist = torch.bincount(sample.reshape(-1).to(torch.int32), minlength=D + 2)[: D + 2].double()
    hist = (hist / hist.sum()).cpu().numpy()
    graph_stats = {"deg_min": int(deg.min()), "deg_mean": float(deg.mean()), "deg_max": int(deg.max()),
                   "spd_bucket_fractions": {"rows_sampled": n_hist_rows, "of_graph": 0,
                                            "fractions": [round(float(x), 5) for x in hist]}}
    f_fwd, f_bwd = w.attn_flops()
    ms_step, _ = dist_util.aggregate(total_ms / args.steps, 0.0, dev)
    fb_ms, flops_all = dist_util.aggregate(fwd_ms + bwd_ms, f_fwd + f_bwd, dev)
    value = flops_all / (fb_ms * 1e-3) / 1e12
    spd_alg_bytes = float(b.spd_bytes + 4 * (T + 1) + 4 * ci.numel())

    # ---- the chunked backward (a "next" row: the ring-step view of the backward), timed on its own after the step loop ----
    bwd_chunked = None
    if single:
        ws_bc = gt._workspace(gt.gt_biased_attn_bwd_chunked_workspace(batch, H, d, D, n_chunks), dev)
        gt.gt_biased_attn_bwd_chunked(q, k, v, out, do, lse, spd, bias, batch, D, n_chunks, dq, dk, dv, dbias, None, ws_bc)
        torch.cuda.synchronize()
        b0, b1 = ev(), ev()
        n_bc = max(1, min(args.steps, 3))
        b0.record()
        for _ in range(n_bc):
            gt.gt_biased_attn_bwd_chunked(q, k, v, out, do, lse, spd, bias, batch, D, n_chunks, dq, dk, dv, dbias, None, ws_bc)
        b1.record()
        torch.cuda.synchronize()
        gt.gt_check(ws_bc)
        bc_ms = b0.elapsed_time(b1) / n_bc
        bwd_chunked = {"ms": bc_ms, "tflops": f_bwd / (bc_ms * 1e-3) / 1e12, "n_kv_chunks": n_chunks, "runs": n_bc,
                       "note": "outside the timed step; one launch of the backward kernel per key chunk"}
        del ws_bc

    # ---- caller-driven ring steps (a "next" row): 8 ranks x 8 steps, two-part key slices, carried state ----
    fwd_ring = None
    if single and T >= 8192:
        n_ranks, n_super = 8, 1024
        n_reg = T - n_super
        share = (n_reg // n_ranks + 15) // 16 * 16
        shards = [(r * share, min((r + 1) * share, n_reg)) for r in range(n_ranks)]
        o_acc = torch.zeros(T, H, d, dtype=torch.float32, device=dev)
        lse_acc = torch.empty(H, T, dtype=torch.float32, device=dev)
        ws_st = gt._workspace(gt.gt_biased_attn_fwd_step_workspace(batch, H, d), dev)

        def ring():
            o_acc.zero_()
            lse_acc.fill_(float("-inf"))
            for rank, (qa, qb) in enumerate(shards + [(n_reg, T)]):
                for st_ in range(n_ranks):
                    ka, kb = shards[(rank + st_) % n_ranks]
                    gt.gt_biased_attn_fwd_step(q, k, v, spd, bias, batch, D, (qa, qb), (ka, kb),
                                               (n_reg, T) if st_ == 0 else (0, 0), o_acc, lse_acc, None, ws_st)
        ring()
        torch.cuda.synchronize()
        r0, r1 = ev(), ev()
        r0.record()
        ring()
        r1.record()
        torch.cuda.synchronize()
        gt.gt_check(ws_st)
        ring_ms = r0.elapsed_time(r1)
        fwd_ring = {"ms": ring_ms, "tflops": f_fwd / (ring_ms * 1e-3) / 1e12, "ranks": n_ranks, "super_nodes": n_super,
                    "steps": (n_ranks + 1) * n_ranks,
                    "max_abs_vs_forward": float((o_acc - out.float()).abs().max().item()),
                    "note": "outside the timed step; every rank's query shard (and the super nodes' rows) sees all key blocks once"}
        del o_acc, lse_acc, ws_st

    # ---- the backward of the same ring (a "next" row): prepare + 8 x 8 + 8 step calls + finish ----
    bwd_ring = None
    if single and T >= 8192:
        n_ranks, n_super = 8, 1024
        n_reg = T - n_super
        share = (n_reg // n_ranks + 15) // 16 * 16
        shards = [(r * share, min((r + 1) * share, n_reg)) for r in range(n_ranks)]
        accs = [torch.zeros(T, H, d, dtype=torch.float32, device=dev) for _ in range(3)]
        db_acc = torch.zeros(H, D + 2, dtype=torch.float64, device=dev)
        ctx = gt._workspace(gt.gt_biased_attn_bwd_step_context_bytes(batch, H, d), dev)
        dq_r, dk_r, dv_r = (torch.empty_like(q) for _ in range(3))
        dbias_r = torch.empty_like(bias)

        def bwd_ring_pass():
            for a_ in accs:
                a_.zero_()
            db_acc.zero_()
            gt.gt_biased_attn_bwd_step_prepare(out, do, lse, spd, batch, D, ctx)
            for rank, qr in enumerate(shards):
                for st_ in range(n_ranks):
                    gt.gt_biased_attn_bwd_step(q, k, v, do, bias, batch, D, qr, shards[(rank - st_) % n_ranks],
                                               (n_reg, T) if st_ == 0 else (0, 0), accs[0], accs[1], accs[2], db_acc, ctx)
                gt.gt_biased_attn_bwd_step(q, k, v, do, bias, batch, D, (n_reg, T), qr, (n_reg, T) if rank == 0 else (0, 0),
                                           accs[0], accs[1], accs[2], db_acc, ctx)
            gt.gt_biased_attn_bwd_step_finish(accs[0], accs[1], accs[2], db_acc, batch, D, dq_r, dk_r, dv_r, dbias_r)
        bwd_ring_pass()
        torch.cuda.synchronize()
        r0, r1 = ev(), ev()
        r0.record()
        bwd_ring_pass()
        r1.record()
        torch.cuda.synchronize()
        gt.gt_check(ctx)
        ring_ms = r0.elapsed_time(r1)
        gt.gt_biased_attn_bwd(q, k, v, out, do, lse, spd, bias, batch, D, dq, dk, dv, dbias, ws_bwd)
        torch.cuda.synchronize()
        rel = lambda x, y: float(((x.float() - y.float()).norm() / y.float().norm()).item())
        bwd_ring = {"ms": ring_ms, "tflops": f_bwd / (ring_ms * 1e-3) / 1e12, "ranks": n_ranks, "super_nodes": n_super,
                    "steps": n_ranks * n_ranks + n_ranks,
                    "rel_l2_vs_backward": {"dq": rel(dq_r, dq), "dk": rel(dk_r, dk), "dv": rel(dv_r, dv), "dbias": rel(dbias_r, dbias)},
                    "note": "outside the timed step; includes the prepare pass (SPD transpose) and the final conversion"}
        del accs, ctx, dq_r, dk_r, dv_r

    # ---- outside the timed step: the feature-bias variant (four uint8 features per pair) on 8 192 nodes ----
    feature_bias = None
    if rank == 0 and single:
        from paper_2609_34420_b200.profile_case import feature_timings
        ft = feature_timings(8192, 3, 12)
        tf = lambda flops, ms: flops / (ms * 1e-3) / 1e12
        feature_bias = {"n": ft["n"], "distinct_feature_vectors": ft["codes"], "encode_ms": ft["encode_ms"],
                        "fwd_ms": ft["codes_fwd_ms"], "fwd_tflops": tf(ft["fwd_flops"], ft["codes_fwd_ms"]),
                        "bwd_ms": ft["codes_bwd_ms"], "bwd_tflops": tf(ft["bwd_flops"], ft["codes_bwd_ms"]),
                        "fp32_path_fwd_ms": ft["fp32_fwd_ms"], "fp32_path_bwd_ms": ft["fp32_bwd_ms"],
                        "note": "outside the timed step; categorical features as a code matrix through the tensor-core kernels "
                                "(forward with the fp32 output), next to the path that serves any features"}

    # ---- end to end through the C ABI with host buffers (pinned), copies inside the timed region ----
    host_in = {name: x.cpu().pin_memory() for name, x in
               (("q", q), ("k", k), ("v", v), ("do", do), ("bias", bias), ("rp", rp), ("ci", ci))}
    host_out = {name: torch.empty_like(x, device="cpu").pin_memory() for name, x in
                (("out", out), ("lse", lse), ("dq", dq), ("dk", dk), ("dv", dv), ("dbias", dbias))}
    h2d = sum(x.numel() * x.element_size() for x in host_in.values())
    d2h = sum(x.numel() * x.element_size() for x in host_out.values())

    # The copies that the next kernel does not need run on streams of their own: Q, K, V, dO, bias come in while
    # the SPD build (which needs only the CSR) runs, O and LSE go out while the backward runs, and the gradients go
    # out while the next step's SPD build runs (the last step's are waited for before the clock stops).
    main_s = torch.cuda.current_stream(dev)
    copy_s = torch.cuda.Stream(dev)
    out_s = torch.cuda.Stream(dev)
    ev_in, ev_fwd, ev_bwd, ev_grads = (torch.cuda.Event() for _ in range(4))
    ev_grads.record(main_s)

    def e2e_step():
        rp.copy_(host_in["rp"], non_blocking=True)
        ci.copy_(host_in["ci"], non_blocking=True)
        copy_s.wait_stream(main_s)                 # the previous step's kernels have finished with Q, K, V, dO
        with torch.cuda.stream(copy_s):
            q.copy_(host_in["q"], non_blocking=True)
            k.copy_(host_in["k"], non_blocking=True)
            v.copy_(host_in["v"], non_blocking=True)
            do.copy_(host_in["do"], non_blocking=True)
            bias.copy_(host_in["bias"], non_blocking=True)
            ev_in.record(copy_s)
        gt.gt_spd_build(rp, ci, batch, D, spd, ws_spd)
        main_s.wait_event(ev_in)
        main_s.wait_event(ev_grads)                # O, LSE and the gradients of the previous step have left the device
        gt.gt_biased_attn_fwd(q, k, v, spd, bias, batch, D, out, lse, ws_fwd)
        ev_fwd.record(main_s)
        with torch.cuda.stream(out_s):
            out_s.wait_event(ev_fwd)
            host_out["out"].copy_(out, non_blocking=True)
            host_out["lse"].copy_(lse, non_blocking=True)
        gt.gt_biased_attn_bwd(q, k, v, out, do, lse, spd, bias, batch, D, dq, dk, dv, dbias, ws_bwd)
        ev_bwd.record(main_s)
        with torch.cuda.stream(out_s):
            out_s.wait_event(ev_bwd)
            for name, src in (("dq", dq), ("dk", dk), ("dv", dv), ("dbias", dbias)):
                host_out[name].copy_(src, non_blocking=True)
            ev_grads.record(out_s)

    def e2e_drain():
        main_s.wait_stream(copy_s)                 # the run ends when every copy has landed
        main_s.wait_stream(out_s)

    e2e_step()
    e2e_drain()
    torch.cuda.synchronize()
    n_e2e = max(1, min(args.steps, 3))
    dist_util.barrier(dev)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(n_e2e):
        e2e_step()
    e2e_drain()
    e1.record()
    torch.cuda.synchronize()
    dist_util.barrier(dev)
    e2e_ms, e2e_flops = dist_util.aggregate(e0.elapsed_time(e1) / n_e2e, f_fwd + f_bwd, dev)
    e2e_value = e2e_flops / (e2e_ms * 1e-3) / 1e12

    if rank != 0:
        return 0

    peaks, peak_kind = load_peaks()
    bwd_tflops = f_bwd / (bwd_ms * 1e-3) / 1e12
    bwd_kernel_tflops = f_bwd / (bwd_kernel_ms * 1e-3) / 1e12
    peak_tf = float(peaks.get("bf16_tflops_sustained", peaks["bf16_tflops"]))
    sum_n2 = float(b.sum_n2)
    roofline = {
        "kernel": "attn_bwd_kernel", "bound": "tensor", "achieved": bwd_kernel_tflops, "peak": peak_tf, "unit": "TFLOP/s",
        "frac": bwd_kernel_tflops / peak_tf, "peak_kind": f"bf16_tflops_sustained of {peak_kind} (kernel timed inside a long step)",
        "frac_of_burst_peak": bwd_kernel_tflops / float(peaks["bf16_tflops"]),
        "traffic": None if BWD_KERNEL_DRAM_BYTES_PER_N2 is None else BWD_KERNEL_DRAM_BYTES_PER_N2 * sum_n2,
        "flops_per_launch": f_bwd, "ms_per_launch": bwd_kernel_ms,
        "timing": "CUDA events recorded by the library around the kernel's launch inside every timed step (mean over the steps)",
        "ms_per_call": bwd_ms, "frac_of_call": bwd_tflops / peak_tf,
        "call_note": "gt_biased_attn_bwd also runs the preparation (SPD transpose, per-query terms, zero fills) and the final conversion",
    }
    fwd_tflops_ = f_fwd / (fwd_ms * 1e-3) / 1e12
    roofline_fwd = {
        "kernel": "attn_fwd_kernel", "bound": "tensor", "achieved": fwd_tflops_, "peak": peak_tf, "unit": "TFLOP/s",
        "frac": fwd_tflops_ / peak_tf, "peak_kind": f"bf16_tflops_sustained of {peak_kind} (kernel timed inside a long step)",
        "frac_of_burst_peak": fwd_tflops_ / float(peaks["bf16_tflops"]),
        "traffic": FWD_KERNEL_DRAM_BYTES_PER_N2 * sum_n2, "flops_per_launch": f_fwd, "ms_per_launch": fwd_ms,
    }
    roofline_spd = {
        "kernel": spd_kernel, "bound": "hbm", "achieved": spd_alg_bytes / (spd_ms * 1e-3) / 1e9,
        "peak": float(peaks["hbm_gbs"]), "unit": "GB/s",
        "frac": spd_alg_bytes / (spd_ms * 1e-3) / 1e9 / float(peaks["hbm_gbs"]), "peak_kind": f"hbm_gbs of {peak_kind}",
        "bytes_per_launch": spd_alg_bytes, "ms_per_launch": spd_ms,
        "traffic": SPD_DENSE_DRAM_BYTES_PER_N2 * sum_n2 if dense_spd else None,
    }

    cpu_baseline = None
    if world == 1:
        sec, o_flops, spd_sec, n_rows, n0 = oracle_sample(w, ORACLE_SAMPLE_ROWS)
        cpu_baseline = {"value": o_flops / sec / 1e12, "unit": UNIT, "cores": host_cores(), "kind": "oracle",
                        "sample": f"{n_rows} seeded query rows of {n0} (full key range): fp64 forward + analytic backward "
                                  f"in {sec:.2f} s; BFS rows of the same sources in {spd_sec:.3f} s (BLAS steps threaded, "
                                  "elementwise steps single-threaded numpy)"}

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16", "data": "synthetic",
        "config": {"workload": args.workload, "note": w.note, "n_total": T, "n_graphs": b.n_graphs, "n_heads": H,
                   "head_dim": d, "max_dist": D, "n_kv_chunks": n_chunks, "nnz": int(ci.numel()),
                   "graph": graph_stats,
                   "step": "spd_build + fwd + bwd + chunked fwd", "parallelism": f"dp{world} (independent batches)",
                   "l2": "inputs larger than L2: the SPD matrix (%.2f GB) is rebuilt and re-streamed every step" % (b.spd_bytes / 1e9)},
        "phases_ms": {"spd_build": spd_ms, "fwd": fwd_ms, "bwd": bwd_ms, "fwd_chunked": chk_ms if single else None},
        "phases_ms_median": ph_median, "phases_ms_min": ph_min,
        "fwd_bwd_ms": {"mean": float(fb.mean()), "median": float(np.median(fb)), "min": float(fb.min()), "repetitions": int(len(fb)),
                       "note": "rank 0; `value` uses the mean (max over ranks)"},
        "fwd_tflops": f_fwd / (fwd_ms * 1e-3) / 1e12, "bwd_tflops": bwd_tflops,
        "fwd_chunked_tflops": (f_fwd / (chk_ms * 1e-3) / 1e12) if single else None,
        "bwd_chunked": bwd_chunked, "fwd_ring_steps": fwd_ring, "bwd_ring_steps": bwd_ring, "feature_bias": feature_bias,
        "spd_build_gbs": roofline_spd["achieved"],
        "pct_of_bf16_peak": {"burst": 100 * value / world / float(peaks["bf16_tflops"]),
                             "sustained": 100 * value / world / peak_tf, "nominal_2250": 100 * value / world / 2250.0},
        "roofline": roofline, "roofline_fwd": roofline_fwd, "roofline_spd": roofline_spd, "cpu_baseline": cpu_baseline,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
                "ms_per_step": e2e_ms, "steps": n_e2e, "includes": "H2D of Q,K,V,dO,bias,CSR; spd_build+fwd+bwd; D2H of O,LSE,dQ,dK,dV,dBias (on copy streams: input copies overlap the SPD build, O/LSE copies the backward, gradient copies the next step's SPD build; all copies have landed when the clock stops)"},
        "gpu_launches": kernels_per_step * args.steps, "clocks": clocks,
    }
    print(json.dumps(line))
    return 0


# --------------------------------------------------------------------------------------
# Context-parallel ring (one graph over all ranks): forward ring + backward ring per step
# --------------------------------------------------------------------------------------
def run_ring(args) -> int:
    import torch
    import torch.distributed as dist

    from paper_2609_34420_b200 import binding as gt
    from paper_2609_34420_b200 import dist_util, ring

    if not torch.cuda.is_available():
        raise SystemExit("bench.py: no CUDA device (the CUDA path has no CPU fallback)")
    rank, local_rank, world = dist_util.env_world()
    dev = torch.device("cuda", local_rank)
    torch.cuda.set_device(dev)
    dist_util.init_process_group("nccl")
    gt.lib()
    w = wl.make_workload(args.workload)                     # the SAME graph on every rank: it is one sharded problem
    b, t = w.batch, w.tensors()
    if b.n_graphs != 1:
        raise SystemExit("--mode ring needs a single-graph workload")
    T, H, d, D = b.n_total, w.n_heads, w.head_dim, w.max_dist
    n_super = args.super_nodes if args.super_nodes >= 0 else (1024 if T >= 8192 else 16 * (T // 160))
    layout = ring.RingLayout.even(T, n_super, world)
    (a, e), (sa, sb) = layout.shards[rank], layout.super_range
    share = max(y - x for x, y in layout.shards)

    def dev_bf16(bits):
        return torch.from_numpy(bits.view(np.int16)).to(dev).view(torch.bfloat16)

    batch = gt.Batch(T)
    rp, ci = torch.from_numpy(b.row_ptr).to(dev), torch.from_numpy(b.col_idx).to(dev)
    spd = torch.empty(b.spd_bytes, dtype=torch.uint8, device=dev)
    gt.gt_check(gt.gt_spd_build(rp, ci, batch, D, spd))       # a rank reads only the rows of its queries (its bias shard)
    q, k, v, do = dev_bf16(t.q), dev_bf16(t.k), dev_bf16(t.v), dev_bf16(t.dout)
    bias = torch.from_numpy(t.bias).to(dev)
    # what the rank owns: its regular K/V rows and a replica of the super nodes' rows; everything else arrives
    k_full, v_full = torch.zeros_like(k), torch.zeros_like(v)
    k_full[sa:sb], v_full[sa:sb] = k[sa:sb], v[sa:sb]

    def block(x, with_super):
        blk = torch.zeros((share + (n_super if with_super else 0), H, d), dtype=x.dtype, device=dev)
        blk[: e - a] = x[a:e]
        if with_super:
            blk[share:] = x[sa:sb]
        return blk

    fwd_blocks, bwd_blocks = (block(k, True), block(v, True)), (block(k, False), block(v, False))
    o_acc = torch.zeros(T, H, d, dtype=torch.float32, device=dev)
    lse_acc = torch.empty(H, T, dtype=torch.float32, device=dev)
    out = torch.zeros_like(q)
    accs = [torch.zeros(T, H, d, dtype=torch.float32, device=dev) for _ in range(3)]
    db_acc = torch.zeros(H, D + 2, dtype=torch.float64, device=dev)
    ctx = gt._workspace(gt.gt_biased_attn_bwd_step_context_bytes(batch, H, d), dev)
    ws_step = gt._workspace(gt.gt_biased_attn_fwd_step_workspace(batch, H, d), dev)
    dq, dk, dv = (torch.zeros_like(q) for _ in range(3))
    dbias = torch.zeros_like(bias)
    fwd_step = ring.device_step(gt, q, k_full, v_full, spd, bias, batch, D, layout, o_acc, lse_acc, out, ws_step)
    bwd_step = ring.device_bwd_step(gt, q, k_full, v_full, do, bias, batch, D, layout, accs[0], accs[1], accs[2], db_acc, ctx)
    # replicated on every rank until the all-reduce: the super rows of dq, the super keys' dk / dv, dbias
    replicated = [accs[0][sa:sb], accs[1][sa:sb], accs[2][sa:sb], db_acc] if n_super else [db_acc]

    def one_pass():
        o_acc.zero_()
        lse_acc.fill_(float("-inf"))
        for x in accs:
            x.zero_()
        db_acc.zero_()
        dk_own, dv_own = ring.context_parallel_pass(
            layout, fwd_blocks, fwd_step, bwd_blocks, bwd_step, replicated=replicated,
            between=lambda: gt.gt_biased_attn_bwd_step_prepare(None, do, lse_acc, spd, batch, D, ctx, out_f32=o_acc),
            rank=rank, world=world)
        accs[1][a:e].copy_(dk_own[: e - a])                  # the sums of the rank's own keys are home again
        accs[2][a:e].copy_(dv_own[: e - a])
        gt.gt_biased_attn_bwd_step_finish(accs[0], accs[1], accs[2], db_acc, batch, D, dq, dk, dv, dbias)

    for _ in range(max(args.warmup, 1)):
        one_pass()
    torch.cuda.synchronize()
    gt.gt_check(ctx)
    gt.gt_check(ws_step)
    sampler = ClockSampler("GPU-" + str(torch.cuda.get_device_properties(dev).uuid)) if rank == 0 else None
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    dist_util.barrier(dev)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(args.steps):
        one_pass()
    e1.record()
    torch.cuda.synchronize()
    dist_util.barrier(dev)
    clocks = sampler.stop() if sampler else None
    gt.gt_check(ctx)
    gt.gt_check(ws_step)
    f_fwd, f_bwd = w.attn_flops()
    ms, _ = dist_util.aggregate(e0.elapsed_time(e1) / args.steps, 0.0, dev)
    value = (f_fwd + f_bwd) / (ms * 1e-3) / 1e12

    # the rank's rows against the one-shot calls on the whole graph (every rank holds the full inputs here)
    out_ref, dq_ref, dk_ref, dv_ref = (torch.empty_like(q) for _ in range(4))
    lse_ref = torch.empty(H, T, dtype=torch.float32, device=dev)
    dbias_ref = torch.empty_like(bias)
    gt.gt_check(gt.gt_biased_attn_fwd(q, k, v, spd, bias, batch, D, out_ref, lse_ref))
    gt.gt_check(gt.gt_biased_attn_bwd(q, k, v, out_ref, do, lse_ref, spd, bias, batch, D, dq_ref, dk_ref, dv_ref, dbias_ref))
    rows = torch.cat([torch.arange(a, e, device=dev), torch.arange(sa, sb, device=dev)])
    rel = lambda x, y: float(((x.float() - y.float()).norm() / y.float().norm()).item())
    check = {"out": rel(out[rows], out_ref[rows]), "dq": rel(dq[rows], dq_ref[rows]), "dk": rel(dk[rows], dk_ref[rows]),
             "dv": rel(dv[rows], dv_ref[rows]), "dbias": rel(dbias, dbias_ref)}
    worst = torch.tensor([max(check.values())], dtype=torch.float64, device=dev)
    if dist.is_initialized():
        dist.all_reduce(worst, op=dist.ReduceOp.MAX)
    if rank != 0:
        return 0
    peaks, peak_kind = load_peaks()
    blk_bytes = 2 * (share + n_super) * H * d * 2                       # K and V block, bf16
    bwd_bytes = 2 * share * H * d * 2 + 2 * share * H * d * 4           # K, V (bf16) and their dK, dV sums (fp32)
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": max(args.warmup, 1),
        "ms_per_step": ms, "higher_is_better": True, "scaling": "strong", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "mode": "ring",
        "config": {"workload": args.workload, "note": w.note, "n_total": T, "n_heads": H, "head_dim": d, "max_dist": D,
                   "super_nodes": n_super, "parallelism": f"cp{world} (query rows and bias rows sharded, K/V blocks round the ring)",
                   "step": "forward ring + backward ring + all-reduce of the replicated sums + final conversion",
                   "l2": "inputs larger than L2 at the default workload: every rank streams its %.2f GB bias shard per pass" % (b.spd_bytes / world / 1e9)},
        "p2p_bytes_per_rank_per_step": {"forward": (world - 1) * blk_bytes, "backward": (world - 1) * bwd_bytes + (2 * share * H * d * 4 if world > 1 else 0)},
        "pct_of_bf16_peak": {"sustained": 100 * value / world / float(peaks.get("bf16_tflops_sustained", peaks["bf16_tflops"])),
                             "burst": 100 * value / world / float(peaks["bf16_tflops"])},
        "max_rel_l2_vs_one_shot": float(worst.item()), "rel_l2_vs_one_shot_rank0": check,
        "gpu_launches": None, "clocks": clocks,
    }
    print(json.dumps(line))
    return 0


def main() -> int:
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="cuda", choices=["cuda", "reference"])
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD, choices=list(wl.WORKLOAD_NAMES) + ["tiny_er256_sparse"])
    ap.add_argument("--mode", default="step", choices=["step", "ring"])
    ap.add_argument("--super-nodes", type=int, default=-1, help="ring mode: replicated super nodes (default 1024 from 8192 nodes up)")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.mode == "ring":
        return run_ring(args)
    return run_cuda(args)


if __name__ == "__main__":
    sys.exit(main())
