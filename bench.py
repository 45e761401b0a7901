#!/usr/bin/env python
"""Benchmark of the fused SALAD attention call on the Wan-1.3B-shaped layer
(B=1, H=12, d=128, N=32760 tokens of a 21x30x52 latent grid, 128x64 blocks, 3-D
sliding-window mask at 90 % block sparsity), one process per GPU.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

A step is one `salad_fused_fwd` call: the linear-state reduction, the block-sparse softmax
branch, the linear apply and the scaled sum with its single bf16 write.  The static mask is
built once before the timed region (it is a per-model constant); its build time is reported
separately.  `value` is kept-block TFLOP/s over all ranks (4 * valid_q * valid_k * d flops
per kept block, nothing else counted).  With N > 1 every rank runs the full layer on its own
tensors (heads and batch items are independent: no collective on the data path) and the
time is the maximum over ranks: weak scaling.  `--shard heads` splits ONE layer over the ranks
by contiguous head ranges instead (strong scaling, still no collective).  Started as plain
`python bench.py --gpus N` (no launcher in the environment) the script starts the N ranks itself.

`--impl reference` times the CPU oracle, as it stands, on a bounded sample of the same
workload on the host cores (rank 0 only).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import socket
import subprocess
import sys
import threading
import time

import numpy as np
import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2601_16515_b200 import dist_util, workloads as wlmod  # noqa: E402

METRIC = "fused_salad_attn_kept_block_tflops"
UNIT = "TFLOP/s"


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        p = json.load(open(path))
        return {"source": "measured", "bf16_tflops": p["bf16_tflops"],
                "bf16_tflops_sustained": p.get("bf16_tflops_sustained"), "hbm_gbs": p["hbm_gbs"]}
    return {"source": "fallback", "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "hbm_gbs": 6650.0}


def kernel_source_hash():
    """sha256 over the sources of the attention kernel: a DRAM-traffic figure captured under ncu is only
    quoted while the kernel it was captured from is the one that runs."""
    h = hashlib.sha256()
    for name in ("fused_kernel.cuh", "ptx.cuh"):
        h.update(open(os.path.join(ROOT, "paper_2601_16515_b200", "csrc", name), "rb").read())
    return h.hexdigest()[:16]


def captured_traffic(workload):
    """DRAM bytes per launch of the attention kernel from the committed ncu capture of this workload, or
    None when there is none or the kernel has changed since.  Table: lines `workload bytes source-hash`."""
    path = os.path.join(ROOT, "profiles", "dram_traffic.txt")
    if not os.path.exists(path):
        return None, "no capture"
    for line in open(path):
        f = line.split()
        if len(f) >= 3 and not line.startswith("#") and f[0] == workload:
            if f[2] == kernel_source_hash():
                return float(f[1]), "ncu dram__bytes_read.sum + dram__bytes_write.sum of one launch"
            return None, "the kernel source has changed since the ncu capture"
    return None, "no capture of this workload"


def self_launch(args):
    """`python bench.py --gpus N` without a launcher: start N ranks (one per GPU) through torch's launcher
    and pass the command line on.  Returns the exit code."""
    with socket.socket() as sck:
        sck.bind(("127.0.0.1", 0))
        port = sck.getsockname()[1]
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", f"--nproc-per-node={args.gpus}",
           "--master-addr", "127.0.0.1", "--master-port", str(port), os.path.abspath(__file__)] + sys.argv[1:]
    return subprocess.call(cmd)


def kept_block_flops(wl, row_ptr, col_idx, Hm):
    """4 * valid_q * valid_k * d per kept block, summed over mask rows, times batch*heads."""
    N, Bq, Bk, d = wl.N, wl.Bq, wl.Bk, wl.d
    nQb, nKb = wl.nQb, wl.nKb
    vq = np.minimum(Bq, N - np.arange(nQb) * Bq).astype(np.float64)
    vk = np.minimum(Bk, N - np.arange(nKb) * Bk).astype(np.float64)
    rows = np.repeat(np.arange(Hm * nQb), np.diff(row_ptr))
    per_mask = float((4.0 * d * vq[rows % nQb] * vk[col_idx]).sum())
    return per_mask * wl.B * (wl.H // Hm)


class ClockSampler(threading.Thread):
    """Samples SM clock and clock-event reasons through NVML while the timed region runs."""

    def __init__(self, index: int, period_s: float = 0.02):
        super().__init__(daemon=True)
        self.index, self.period, self.samples, self.reasons = index, period_s, [], set()
        self.stop_flag = threading.Event()
        self.max_mhz = None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM)
        except Exception:
            self.nv = None

    def sample(self):
        if self.nv is None:
            return
        nv = self.nv
        try:
            self.samples.append(nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM))
            r = nv.nvmlDeviceGetCurrentClocksEventReasons(self.h)
            names = {"sw_power_cap": 0x4, "hw_slowdown": 0x8, "sw_thermal_slowdown": 0x20,
                     "hw_thermal_slowdown": 0x40, "hw_power_brake": 0x80}
            for n, bit in names.items():
                if r & bit:
                    self.reasons.add(n)
        except Exception:
            pass

    def run(self):
        while not self.stop_flag.is_set():
            self.sample()
            time.sleep(self.period)

    def result(self):
        return {"sm_mhz": float(np.median(self.samples)) if self.samples else None,
                "sm_max_mhz": self.max_mhz, "reasons": sorted(self.reasons), "samples": len(self.samples)}


def physical_gpu_index(local_rank: int) -> int:
    vis = os.environ.get("CUDA_VISIBLE_DEVICES")
    if vis:
        try:
            return int(vis.split(",")[local_rank])
        except Exception:
            return local_rank
    return local_rank


def oracle_sample(wl, steps, warmup, rank, heads=None, rows=None):
    """CPU oracle on a bounded sample: the first `heads` heads of batch item 0 and the first `rows` query
    rows of each (default: 8 heads, every row); those heads' linear states are computed in full inside the
    timed call."""
    from oracle import salad_oracle as orc
    orc.use_all_cores()          # a multi-process launcher sets OMP_NUM_THREADS=1; the other ranks do no CPU work here
    nh = min(wl.H, heads if heads else int(os.environ.get("SALAD_ORACLE_HEADS", "8")))
    nr = wl.N if not rows else max(1, min(wl.N, int(rows)))
    q, k, v = (t.float().numpy() for t in wlmod.make_qkv(wl, heads=list(range(nh))))
    T, Hs, Ws = wl.grid
    rp, ci = orc.mask_build(T, Hs, Ws, wl.Bq, wl.Bk, wl.windows)
    lam, s = wlmod.make_scales(wl)
    sel = (np.arange(nh, dtype=np.int64)[:, None] * wl.N + np.arange(nr, dtype=np.int64)[None, :]).reshape(-1)
    nQb = wl.nQb
    vk = np.minimum(wl.Bk, wl.N - np.arange(wl.nKb) * wl.Bk).astype(np.float64)
    keys_per_qb = np.array([vk[ci[rp[i]:rp[i + 1]]].sum() for i in range(nQb)])
    flops = float((4.0 * wl.d * keys_per_qb[(sel % wl.N) // wl.Bq]).sum())
    times = []
    for it in range(warmup + steps):
        t0 = time.perf_counter()
        orc.salad_fused(q[:1], k[:1], v[:1], wl.Bq, wl.Bk, rp, ci, 1, lam[:nh], s[:1], sel=sel)
        dt = time.perf_counter() - t0
        if it >= warmup:
            times.append(dt)
    sec = float(np.mean(times))
    return {"value": flops / sec / 1e12, "unit": UNIT, "cores": orc.num_threads(), "kind": "oracle",
            "sample": f"{nh} of {wl.B * wl.H} heads, the first {nr} of {wl.N} query rows each (kept-block flops "
                      f"of those rows), those heads' linear states included in the time; "
                      f"{sec:.2f} s per pass"}, sec


def run_reference(args, wl, rank, world):
    """The oracle as the reference arm: exactly --steps timed passes after --warmup untimed ones, each pass a
    sample of the workload sized (from one calibration pass over a single head) so that the whole run takes
    about two to three minutes."""
    if rank != 0:
        return
    steps, warm = max(1, args.steps), max(0, args.warmup)
    _, t_head = oracle_sample(wl, 1, 0, rank, heads=1)                 # calibration: one head, every row
    per_pass_s = min(20.0, 150.0 / (steps + warm))                         # seconds per pass
    if t_head <= per_pass_s:
        heads, rows = max(1, min(8, wl.H, int(per_pass_s / t_head))), None
    else:                                                              # less than a head: a prefix of its rows
        heads, rows = 1, max(wl.Bq, int(wl.N * per_pass_s / t_head) // wl.Bq * wl.Bq)
    base, sec = oracle_sample(wl, steps, warm, rank, heads=heads, rows=rows)
    line = {"impl": "reference", "metric": METRIC, "value": base["value"], "unit": UNIT, "n_gpus": args.gpus,
            "steps": steps, "warmup": warm, "ms_per_step": sec * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": wl.name, "B": wl.B, "H": wl.H, "N": wl.N, "d": wl.d,
                       "blocks": f"{wl.Bq}x{wl.Bk}", "windows": list(wl.windows)},
            "cpu_baseline": base,
            "e2e": {"value": base["value"], "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="salad", choices=["salad", "reference"])
    ap.add_argument("--workload", default="wan1.3b-90", choices=sorted(wlmod.ALL))
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true", help="skip the dense-run and per-branch timings")
    ap.add_argument("--shard", default="replicas", choices=["replicas", "heads"],
                    help="N > 1: every rank its own layer (weak scaling) or one layer split by heads (strong)")
    ap.add_argument("--sustained-seconds", type=float, default=2.0,
                    help="length of the extra back-to-back loop that shows the power-capped behaviour (0: skip)")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "salad" else args.warmup

    if args.gpus > 1 and "WORLD_SIZE" not in os.environ and args.impl == "salad":
        raise SystemExit(self_launch(args))
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    wl = wlmod.ALL[args.workload]

    if args.impl == "reference":
        run_reference(args, wl, rank, world)
        return

    import torch.distributed as dist
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the SALAD path has no CPU implementation")
    torch.cuda.set_device(local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    from paper_2601_16515_b200 import salad

    peaks = load_peaks()
    dev = torch.device("cuda", local_rank)
    T, Hs, Ws = wl.grid
    K, W = args.steps, args.warmup

    # ---------------- inputs (seeded, synthetic; every rank its own replica of the layer, or with
    # --shard heads its contiguous range of the heads of one layer)
    shard_heads = args.shard == "heads" and world > 1
    full_wl = wl
    h0, h1 = dist_util.head_range(wl.H, world, rank) if shard_heads else (0, wl.H)
    if shard_heads:
        if h1 == h0:
            raise SystemExit("--shard heads needs at least one head per rank")
        wl = wlmod.replace(wl, H=h1 - h0)
        if len(wl.windows) == full_wl.H and full_wl.H > 1:           # one window per head: this rank's
            wl = wlmod.replace(wl, windows=wl.windows[h0:h1])
    q_h, k_h, v_h = (t.pin_memory() for t in wlmod.make_qkv(full_wl, heads=list(range(h0, h1))))
    q, k, v = (t.to(dev, non_blocking=True) for t in (q_h, k_h, v_h))
    lam, s = wlmod.make_scales(full_wl)
    lam = lam[h0:h1].copy()
    lam_d, s_d = torch.from_numpy(lam).to(dev), torch.from_numpy(s).to(dev)
    out = torch.empty_like(q)
    out_h = torch.empty(q_h.shape, dtype=q_h.dtype).pin_memory()
    ws = salad.alloc_workspace(wl.B, wl.H, wl.N, wl.d, wl.Bq, wl.Bk, dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)

    # ---------------- static mask, built once (step a1), timed on its own
    if wl.irregular:
        rp_np, ci_np = wlmod.irregular_csr(full_wl)
        rp_np, ci_np = dist_util.slice_head_lists(rp_np, ci_np, wl.nQb, h0, h1)     # this rank's heads
        rp, ci, Hm = torch.from_numpy(rp_np).to(dev), torch.from_numpy(ci_np).to(dev), wl.H
        mask_ms = None
    else:
        salad.salad_mask_build(T, Hs, Ws, wl.Bq, wl.Bk, wl.windows, dev)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rp, ci = salad.salad_mask_build(T, Hs, Ws, wl.Bq, wl.Bk, wl.windows, dev)
        torch.cuda.synchronize()
        mask_ms = (time.perf_counter() - t0) * 1e3
        Hm = len(wl.windows)
        rp_np, ci_np = rp.cpu().numpy(), ci.cpu().numpy()
    flops = kept_block_flops(wl, rp_np, ci_np, Hm)
    nnz_total = int(len(ci_np)) * wl.B * (wl.H // Hm)
    sparsity = 1.0 - len(ci_np) / (Hm * wl.nQb * wl.nKb)

    def step():
        salad.salad_fused_fwd(q, k, v, rp, ci, Hm, lam_d, s_d, Bq=wl.Bq, Bk=wl.Bk, out=out,
                              workspace=ws, status=status)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    # ---------------- main timed region: device-resident inputs
    for _ in range(W):
        step()
    KP = min(K, 20)                   # steps of the per-kernel timing pass
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(KP)]
    for group in evs:
        for e in group:
            e.record()
    t_start, t_stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    sampler = ClockSampler(physical_gpu_index(local_rank))
    sampler.start()
    # Per-kernel durations first: a few steps with the library recording events around its kernel
    # groups.  (An event between two launches keeps the second kernel from being set up while the
    # first drains, so the timed region below runs without them.)
    for i in range(KP):
        salad.salad_set_profile_events(evs[i])
        step()
    salad.salad_set_profile_events(None)
    barrier()
    t_mid = torch.cuda.Event(enable_timing=True)      # after the first calls of the region: before the power cap bites
    K_head = min(K, 30)
    t_start.record()
    for i in range(K):
        step()
        if i + 1 == K_head:
            t_mid.record()
    t_stop.record()
    sampler.sample()
    barrier()
    sampler.stop_flag.set()
    if int(status.item()) != 0:
        raise SystemExit("a kernel reported an expired wait; no number is valid")
    total_ms = t_start.elapsed_time(t_stop)
    head_ms_per_step = t_start.elapsed_time(t_mid) / K_head
    state_ms = float(np.mean([g[0].elapsed_time(g[1]) for g in evs]))
    attn_ms = float(np.mean([g[2].elapsed_time(g[3]) for g in evs]))
    # replicas: every rank did `flops` of work (weak scaling); head shards: the ranks' shares add up to one
    # layer (strong scaling).  Either way the job took the slowest rank's time.
    if shard_heads:
        total_flops = dist_util.sum_over_ranks(flops, dev)
        total_ms_max = dist_util.max_over_ranks(total_ms, dev)
        flops_per_s = total_flops * K / (total_ms_max * 1e-3)
    else:
        flops_per_s, total_ms_max = dist_util.aggregate_throughput(flops * K, total_ms, dev)
    ms_per_step = total_ms_max / K
    value = flops_per_s / 1e12

    # ---------------- end to end: host buffers in, host buffer out, every step.
    # Every step copies its Q, K, V from pinned host memory and its O back.  The copies of neighbouring
    # steps overlap the compute of the current one: two sets of device buffers, one stream each for
    # host->device, compute and device->host, events in between (what a caller with host-resident
    # data would do; the step stays bound by the host->device copy).  The strictly serial figure
    # (copy in, compute, copy out on one stream) is reported beside it.
    def e2e_step():
        q.copy_(q_h, non_blocking=True); k.copy_(k_h, non_blocking=True); v.copy_(v_h, non_blocking=True)
        step()
        out_h.copy_(out, non_blocking=True)

    Ke = max(3, min(K, 20))
    for _ in range(2):
        e2e_step()
    barrier()
    t_start.record()
    for _ in range(Ke):
        e2e_step()
    t_stop.record()
    barrier()
    e2e_serial_ms = dist_util.max_over_ranks(t_start.elapsed_time(t_stop), dev) / Ke

    bufs = [(q, k, v, out), tuple(torch.empty_like(q) for _ in range(4))]
    outs_h = [out_h, torch.empty(q_h.shape, dtype=q_h.dtype).pin_memory()]
    ws2 = [ws, salad.alloc_workspace(wl.B, wl.H, wl.N, wl.d, wl.Bq, wl.Bk, dev)]
    s_in, s_cmp, s_out = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()

    def e2e_pipelined(n_steps):
        ev_in = [None] * n_steps; ev_cmp = [None] * n_steps; ev_out = [None] * n_steps
        for i in range(n_steps):
            qb, kb, vb, ob = bufs[i & 1]
            with torch.cuda.stream(s_in):
                if i >= 2:
                    s_in.wait_event(ev_cmp[i - 2])            # inputs of step i-2 consumed
                qb.copy_(q_h, non_blocking=True); kb.copy_(k_h, non_blocking=True); vb.copy_(v_h, non_blocking=True)
                ev_in[i] = torch.cuda.Event(); ev_in[i].record(s_in)
            with torch.cuda.stream(s_cmp):
                s_cmp.wait_event(ev_in[i])
                if i >= 2:
                    s_cmp.wait_event(ev_out[i - 2])           # output buffer of step i-2 copied out
                salad.salad_fused_fwd(qb, kb, vb, rp, ci, Hm, lam_d, s_d, Bq=wl.Bq, Bk=wl.Bk, out=ob,
                                      workspace=ws2[i & 1], status=status, stream=s_cmp)
                ev_cmp[i] = torch.cuda.Event(); ev_cmp[i].record(s_cmp)
            with torch.cuda.stream(s_out):
                s_out.wait_event(ev_cmp[i])
                outs_h[i & 1].copy_(ob, non_blocking=True)
                ev_out[i] = torch.cuda.Event(); ev_out[i].record(s_out)
        return ev_out[-1]

    e2e_pipelined(2)
    barrier()
    t_start.record()
    for st_ in (s_in, s_cmp, s_out):
        st_.wait_event(t_start)
    last = e2e_pipelined(Ke)
    torch.cuda.current_stream().wait_event(last)
    t_stop.record()
    barrier()
    e2e_ms = dist_util.max_over_ranks(t_start.elapsed_time(t_stop), dev) / Ke
    if int(status.item()) != 0:
        raise SystemExit("a kernel reported an expired wait; no number is valid")
    tensor_bytes = q_h.numel() * q_h.element_size()
    job_flops = dist_util.sum_over_ranks(flops, dev) if shard_heads else flops * world
    e2e = {"value": job_flops / (e2e_ms * 1e-3) / 1e12, "unit": UNIT, "ms_per_step": e2e_ms,
           "h2d_bytes_per_step": 3 * tensor_bytes, "d2h_bytes_per_step": tensor_bytes,
           "how": "copies of neighbouring steps overlap compute (two buffer sets, three streams)",
           "serial_ms_per_step": e2e_serial_ms,
           "serial_value": job_flops / (e2e_serial_ms * 1e-3) / 1e12}
    del bufs, outs_h, ws2

    # ---------------- extras (rank 0): per-branch calls and the 0 %-sparsity run of the same kernel
    extras = {}
    if rank == 0 and not args.no_extras:
        def timed(fn, iters, reps=1):
            """ms per call over `iters` back-to-back calls; the median of `reps` such loops (the short,
            HBM-bound calls are timed three times: one loop of 20 lasts about a millisecond)."""
            for _ in range(2):
                fn()
            torch.cuda.synchronize()
            got = []
            for _ in range(reps):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(iters):
                    fn()
                b.record()
                torch.cuda.synchronize()
                got.append(a.elapsed_time(b) / iters)
            return sorted(got)[len(got) // 2]
        extras["sparse_only_ms"] = timed(lambda: salad.salad_sparse_attn_fwd(
            q, k, v, rp, ci, Hm, Bq=wl.Bq, Bk=wl.Bk, out=out, workspace=ws), 20)
        extras["linear_only_ms"] = timed(lambda: salad.salad_linear_attn_fwd(q, k, v, out=out, workspace=ws), 20, reps=3)
        # the whole linear branch as one call: K, V read (state), Q read and O written (apply)
        lin_bytes = 4 * q_h.numel() * q_h.element_size()
        def hbm_record(kernel, ms, nbytes):
            gbs = nbytes / (ms * 1e-3) / 1e9
            return {"kernel": kernel, "bound": "hbm", "ms": ms, "algorithmic_bytes": nbytes, "achieved": gbs,
                    "unit": "GB/s", "peak": peaks["hbm_gbs"], "peak_source": peaks["source"] + " copy bandwidth",
                    "frac": gbs / peaks["hbm_gbs"], "frac_of_nominal_8tbs": gbs / 8000.0}
        extras["linear_branch"] = hbm_record("salad_linear_attn_fwd: state (+ finalize beyond eight chunks per head) and apply kernels (K, V, Q read, O written)",
                                             extras["linear_only_ms"], lin_bytes)
        drp, dci = wlmod.dense_csr(wl.nQb, wl.nKb, 1)
        drp_d, dci_d = torch.from_numpy(drp).to(dev), torch.from_numpy(dci).to(dev)
        dense_ms = timed(lambda: salad.salad_fused_fwd(q, k, v, drp_d, dci_d, 1, lam_d, s_d, Bq=wl.Bq, Bk=wl.Bk,
                                                       out=out, workspace=ws), 3)
        dense_flops = kept_block_flops(wl, drp, dci, 1)
        extras.update({"dense_ms": dense_ms, "dense_tflops": dense_flops / (dense_ms * 1e-3) / 1e12,
                       "speedup_vs_dense": dense_ms / ms_per_step})
        # linear-state pass: K and V read once (algorithmic bytes), against the HBM copy peak.  Timed as the
        # library's own call for it (state kernel + finalize kernel, launched back to back); in a fused call
        # the short-ring variant of the same kernels shares its SMs with the attention kernel
        # (`roofline.state_kernels_ms`).
        kv_bytes = 2 * tensor_bytes
        lin_state_ms = timed(lambda: salad.salad_linear_state_fwd(k, v, ws), 20, reps=3)
        extras["linear_state"] = hbm_record("salad_linear_state_fwd: salad_linear_state_kernel (+ finalize beyond eight chunks per head; K, V read once)",
                                            lin_state_ms, kv_bytes)
        # the attention call on a workspace that already holds the state (a caller who ran the state pass
        # early, or beside other work, pays this much per layer)
        prep_ms = timed(lambda: salad.salad_fused_prepared_fwd(q, k, v, rp, ci, Hm, lam_d, s_d, ws, Bq=wl.Bq, Bk=wl.Bk,
                                                               out=out), 20)
        extras["fused_prepared"] = {"ms": prep_ms, "tflops": flops / (prep_ms * 1e-3) / 1e12,
                                    "frac_of_measured_bf16_peak": flops / (prep_ms * 1e-3) / 1e12 / peaks["bf16_tflops"]}

        # dynamic-scale producer (Alg. 1 Level 2) on hidden states of the DiT this workload comes from:
        # a CFG pair of [N, D = H*d] token matrices (larger than L2), read once
        xt = torch.randn(2, wl.N, wl.H * wl.d, device=dev, dtype=torch.float32).to(torch.bfloat16)
        w_dyn = torch.randn(wl.H * wl.d, device=dev, dtype=torch.float32) / (wl.H * wl.d) ** 0.5
        s_out = torch.empty(2, device=dev, dtype=torch.float32)
        dyn_ws = torch.empty(salad.DYN_SCALE_WS_BYTES, dtype=torch.uint8, device=dev)
        dyn_ms = timed(lambda: salad.salad_dynamic_scale(xt, w_dyn, 0.0, out=s_out, workspace=dyn_ws), 20, reps=3)
        x_bytes = xt.numel() * 2
        extras["dynamic_scale"] = hbm_record("dynamic_scale_partial_kernel + finalize (X_t read once)", dyn_ms, x_bytes)
        del xt
        # full D x D projection of the linear branch + residual sum (Alg. 1 level 1): a tensor-core GEMM
        Dm = wl.H * wl.d
        w_proj = (torch.randn(Dm, Dm, device=dev) / Dm ** 0.5).to(torch.bfloat16)
        o_l_buf = torch.randn_like(q)
        proj_out = torch.empty_like(q)
        proj_ms = timed(lambda: salad.salad_proj_combine_fwd(out, o_l_buf, w_proj, s_d, out=proj_out), 10)
        proj_flops = 2.0 * wl.B * wl.N * Dm * Dm
        extras["proj_combine"] = {"ms": proj_ms, "tflops": proj_flops / (proj_ms * 1e-3) / 1e12,
                                  "frac_of_measured_bf16_peak": proj_flops / (proj_ms * 1e-3) / 1e12 / peaks["bf16_tflops"]}
        del w_proj, o_l_buf, proj_out
        # temporal-head permutation (App. A.1): one read and one write of a [B,H,N,d] tensor
        flags = [1] * wl.H
        perm_out = torch.empty_like(q)
        perm_ms = timed(lambda: salad.salad_permute_tokens(q, wl.grid, flags, out=perm_out), 20, reps=3)
        extras["permute_tokens"] = hbm_record("permute_tokens_kernel (one read, one write)", perm_ms, 2 * tensor_bytes)
        del perm_out
        # Top-K mask producer (App. A.1 steps 1-2) at this shape, k chosen for the same 90 % sparsity:
        # block means read Q and K once (the HBM-bound part), then scores and selection
        topk = max(1, round(wl.nKb * (1.0 - sparsity)))
        tk_ws = torch.empty(int(salad._lib.salad_topk_workspace_bytes(wl.B, wl.H, wl.N, wl.d, wl.Bq, wl.Bk)),
                            dtype=torch.uint8, device=dev)
        tk_rp = torch.empty(wl.B * wl.H * wl.nQb + 1, dtype=torch.int32, device=dev)
        tk_ci = torch.empty(wl.B * wl.H * wl.nQb * topk, dtype=torch.int32, device=dev)
        tk_ms = timed(lambda: salad.salad_topk_mask_build(q, k, topk, Bq=wl.Bq, Bk=wl.Bk, row_ptr=tk_rp,
                                                          col_idx=tk_ci, workspace=tk_ws), 20)
        extras["topk_mask"] = hbm_record("salad_topk_mask_build (Q, K read once)", tk_ms, 2 * tensor_bytes)
        extras["topk_mask"]["k"] = topk
        tk_fused_ms = timed(lambda: salad.salad_fused_fwd(q, k, v, tk_rp, tk_ci, wl.B * wl.H, lam_d, s_d, Bq=wl.Bq,
                                                          Bk=wl.Bk, out=out, workspace=ws), 10)
        extras["topk_mask"]["fused_on_topk_lists_ms"] = tk_fused_ms

        # the fused call with one d x d Level-1 projection block per head folded into the linear state (Sec. 4.2)
        if Hm <= wl.H:
            blocks = (torch.randn(wl.H, wl.d, wl.d, device=dev) / wl.d ** 0.5).to(torch.bfloat16)
            bp_ms = timed(lambda: salad.salad_fused_proj_fwd(q, k, v, rp, ci, Hm, blocks, s_d, Bq=wl.Bq, Bk=wl.Bk,
                                                             out=out, workspace=ws), 20)
            extras["fused_block_proj"] = {"ms": bp_ms, "tflops": flops / (bp_ms * 1e-3) / 1e12}
            del blocks
        # the paper's own ST-SWA (App. A.1) through the loads: half of the heads take their tokens grouped by
        # spatial position, every head a 1-D window of a tenth of the sequence (90 % sparse); beside it the
        # same work done with permutation passes (Q, K, V forward, O back) around the fused call
        T_, Hs_, Ws_ = wl.grid
        if T_ <= 64 and wl.Bq == 128 and wl.Bk == 64:
            st_flags = [h % 2 for h in range(wl.H)]
            st_rp, st_ci = salad.salad_stswa_mask_build(wl.grid, st_flags, [wl.N // 20] * wl.H, device=dev)
            st_ms = timed(lambda: salad.salad_fused_stswa_fwd(q, k, v, wl.grid, st_flags, st_rp, st_ci, lam_d, s_d,
                                                              out=out), 10)
            pq, pk, pv, po = (torch.empty_like(q) for _ in range(4))

            def passes():
                salad.salad_permute_tokens(q, wl.grid, st_flags, out=pq)
                salad.salad_permute_tokens(k, wl.grid, st_flags, out=pk)
                salad.salad_permute_tokens(v, wl.grid, st_flags, out=pv)
                salad.salad_permute_tokens(po, wl.grid, st_flags, inverse=True, out=out)
            pass_ms = timed(passes, 10)
            extras["fused_stswa"] = {"ms": st_ms, "kept_blocks": int(st_ci.numel()),
                                     "temporal_heads": sum(st_flags), "window_half_width_tokens": wl.N // 20,
                                     "four_permutation_passes_ms": pass_ms}
            del pq, pk, pv, po, st_rp, st_ci

        # rotary variant of the linear branch (Sec. 4.1): the same fused call with the 3-D rotation table of
        # the workload's latent grid (fp16, 8.4 MB at this shape, shared by all heads)
        rope_d = salad.salad_rope3d_table_build(*wl.grid, wl.d, device=dev)
        rope_ms = timed(lambda: salad.salad_fused_rope_fwd(q, k, v, rp, ci, Hm, lam_d, s_d, rope_d, Bq=wl.Bq, Bk=wl.Bk,
                                                           out=out, workspace=ws), 20)
        rope_lin_ms = timed(lambda: salad.salad_linear_attn_rope_fwd(q, k, v, rope_d, out=out, workspace=ws), 20)
        # the plain call timed the same way right beside it (the long timed region may sit at the power cap)
        plain_ms = timed(lambda: salad.salad_fused_fwd(q, k, v, rp, ci, Hm, lam_d, s_d, Bq=wl.Bq, Bk=wl.Bk,
                                                       out=out, workspace=ws), 20)
        extras["rope_linear_branch"] = {"fused_ms": rope_ms, "fused_tflops": flops / (rope_ms * 1e-3) / 1e12,
                                        "plain_call_ms": plain_ms, "extra_ms_over_plain_call": rope_ms - plain_ms,
                                        "linear_only_ms": rope_lin_ms}

    # ---------------- sustained: the same call back to back for seconds, into the power cap (after everything
    # else, so that the short measurements above are taken at the clock a short call sees)
    sustained = None
    if args.sustained_seconds > 0:
        n_sus = max(K, int(args.sustained_seconds * 1.1 / (total_ms / K * 1e-3)))
        sus_sampler = ClockSampler(physical_gpu_index(local_rank))
        barrier()
        sus_sampler.start()
        t_start.record()
        for _ in range(n_sus):
            step()
        t_stop.record()
        sus_sampler.sample()
        barrier()
        sus_sampler.stop_flag.set()
        sus_ms = dist_util.max_over_ranks(t_start.elapsed_time(t_stop), dev)
        sus_tflops = flops / (sus_ms / n_sus * 1e-3) / 1e12           # per GPU
        clk = sus_sampler.result()
        sustained = {"steps": n_sus, "seconds": sus_ms * 1e-3, "ms_per_step": sus_ms / n_sus,
                     "tflops_per_gpu": sus_tflops, "sm_mhz": clk["sm_mhz"], "reasons": clk["reasons"],
                     "peak": peaks.get("bf16_tflops_sustained"),
                     "frac_of_measured_bf16_sustained": (sus_tflops / peaks["bf16_tflops_sustained"]
                                                         if peaks.get("bf16_tflops_sustained") else None),
                     "frac_of_measured_bf16_burst": sus_tflops / peaks["bf16_tflops"]}

    cpu_baseline = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu_baseline, _ = oracle_sample(wl, 1, 0, rank)

    if rank == 0:
        achieved = flops / (attn_ms * 1e-3) / 1e12
        peak = peaks["bf16_tflops"]
        traffic, traffic_source = captured_traffic(full_wl.name if not shard_heads else "")
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K, "warmup": W,
            "ms_per_step": ms_per_step, "ms_per_call": ms_per_step, "higher_is_better": True,
            "scaling": "strong" if shard_heads else "weak",
            "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
            "config": {"workload": wl.name, "B": wl.B, "H": wl.H, "N": wl.N, "d": wl.d, "grid": list(wl.grid),
                       "blocks": f"{wl.Bq}x{wl.Bk}", "windows": [list(w) for w in wl.windows],
                       "block_sparsity": sparsity, "kept_blocks": nnz_total,
                       "kept_block_tflop_per_call": flops / 1e12,
                       "l2": "inputs (Q,K,V,O = %.0f MB) larger than the 126 MB L2; no flush" % (4 * tensor_bytes / 1e6),
                       "parallelism": ("heads" if shard_heads else "replicas") if world > 1 else "single",
                       "heads_of_rank_0": [h0, h1]},
            "pct_of_measured_bf16_peak": 100.0 * value / world / peak,
            "pct_of_nominal_bf16_peak": 100.0 * value / world / 2250.0,
            # the seconds-long loop against the seconds-long GEMM figure (a short region runs at the burst clock
            # and belongs beside the burst peak above)
            "pct_of_measured_bf16_sustained": (100.0 * sustained["frac_of_measured_bf16_sustained"]
                                               if sustained and sustained["frac_of_measured_bf16_sustained"] else None),
            "sustained": sustained,
            "first_steps": {"steps": K_head, "ms_per_step": head_ms_per_step,
                            "value": flops / (head_ms_per_step * 1e-3) / 1e12,
                            "note": "the first calls of the timed region on this rank; a long region runs into the "
                                    "1 kW power cap, which lowers the clock under every kernel"},
            "mask_build_ms": mask_ms,
            "roofline": {"kernel": "salad_fused_kernel<128>", "bound": "tensor", "achieved": achieved, "peak": peak,
                         "unit": "TFLOP/s", "frac": achieved / peak, "peak_source": peaks["source"] + " (burst)",
                         # DRAM bytes of one launch from the committed ncu capture of this workload, quoted only
                         # while the kernel source is the captured one; algorithmic bytes: Q, K, V read, O written once
                         "traffic": traffic, "traffic_source": traffic_source,
                         "algorithmic_bytes": 4 * tensor_bytes,
                         "kernel_ms": attn_ms, "state_kernels_ms": state_ms,
                         "timed_how": "CUDA events around the launch, %d steps directly before the timed region" % KP},
            "cpu_baseline": cpu_baseline,
            "e2e": e2e,
            # per call: linear state (the work order among its CTAs), attention, and a finalize kernel for the state
            # where a head has more chunks than a cluster has CTAs
            "gpu_launches": (3 if torch.cuda.get_device_properties(dev).multi_processor_count // (wl.B * wl.H) > 8 and wl.N > 64 * wl.d else 2) * K,
            "clocks": sampler.result(),
        }
        line.update(extras)
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
