"""Throughput benchmark of the warp-collective library on one GB300.

A step is the tile-scan workload: cooperative-groups inclusive scans (the
shfl_up Hillis-Steele scan) over 2^26 fp32 values ~ N(0,1) at tile widths 4,
8, 16 and 32, each plain and TwoSum-compensated (8 launches per step).  The
metric is warp-collective GB/s: algorithmic bytes (4 read + 4 written per
element per launch) over device time, and its fraction of the measured HBM
copy bandwidth.  The JSON line also carries the dominant kernel's roofline,
the end-to-end rate through host buffers, the oracle's CPU baseline, the SM
clocks seen during the timed region, and secondary single-op numbers.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

For N > 1 (torchrun, one rank per GPU) every rank runs its own replica of the
workload (the ops need no exchange); value is the sum over ranks.
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

from paper_2112_10034_gb300 import inputs  # noqa: E402

N_ELEMS = 1 << 26
WIDTHS = (4, 8, 16, 32)
BLOCK = 256
VARIANTS = [(w, comp) for w in WIDTHS for comp in (False, True)]
BYTES_PER_LAUNCH = N_ELEMS * 8
METRIC = "warp-collective GB/s (% of HBM peak); batched p50/p99 latency vs per-call"
WORKLOAD = ("tile inclusive scan (shfl_up, cg tiles) of 2^26 fp32 N(0,1) at widths 4/8/16/32, "
            "plain and compensated, 256-thread blocks")

# DRAM bytes per launch of the dominant kernel from one ncu capture, valid
# only while the kernel sources hash to `src_sha` (else reported as null).
NCU_TRAFFIC = {"src_sha": "6d63f86c847138bd",
               "bytes_per_launch": {
                                    "k_tile_scan_rows<Plain<AddF>, 16>": 268457216 + 214523648,
                                    "k_tile_scan_rows<Comp, 16>": 268516864 + 214551552,
                                    "k_tile_scan_rows<Plain<AddF>, 32>": 268460032 + 213930752,
                                    "k_tile_scan_rows<Comp, 32>": 268476672 + 214916608}}
KERNEL_SOURCES = ["paper_2112_10034_gb300/csrc/scan.cu", "paper_2112_10034_gb300/csrc/cox_common.cuh"]


def _src_sha() -> str:
    h = hashlib.sha256()
    for p in KERNEL_SOURCES:
        with open(os.path.join(ROOT, p), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


# --------------------------------------------------------------- clocks
class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons every 100 ms."""

    Q = ("timestamp,index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits", "-i", str(self.index),
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append((time.time(), [c.strip() for c in line.split(",")]))

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self, t0: float, t1: float):
        rows = [r for t, r in self.rows if t0 - 0.15 <= t <= t1 + 0.15] or [r for _, r in self.rows[-3:]]
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        mx = [float(r[3]) for r in rows if r[3].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if len(r) > 6 + i and r[6 + i] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ------------------------------------------------------------ distributed
def _dist_setup(gpus: int):
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    return rank, world, local


def _barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def _max_over_ranks(v: float, world: int, device: str = "cuda") -> float:
    if world == 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([v], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _job_gbs(bytes_per_rank: float, world: int, elapsed_ms: float) -> float:
    """Whole-job rate: every rank moved `bytes_per_rank`; the job took the
    slowest rank's time."""
    return bytes_per_rank * world / (elapsed_ms * 1e-3) / 1e9


# --------------------------------------------------------- the GPU arm
def run_cox(args):
    import torch
    from paper_2112_10034_gb300 import cox

    rank, world, local = _dist_setup(args.gpus)
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    st = torch.cuda.Stream(device=dev)
    sh = st.cuda_stream
    x_host = inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)
    x = torch.from_numpy(x_host).to(dev)
    outs = [torch.empty(N_ELEMS, dtype=torch.float32, device=dev) for _ in VARIANTS]

    def launch(i, w, comp):
        s = cox.cox_tile_scan(cox.COX_SUM, cox.COX_F32, w, BLOCK, x.data_ptr(), outs[i].data_ptr(), N_ELEMS,
                              cox.COX_F_COMPENSATED if comp else 0, sh)
        if s != 0:
            raise cox.CoxError(s, "cox_tile_scan")

    # warm-up (first calls also size the persistent grids)
    for _ in range(args.warmup):
        for i, (w, comp) in enumerate(VARIANTS):
            launch(i, w, comp)
    st.synchronize()

    K = args.steps
    ev = [[(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in VARIANTS]
          for _ in range(K)]
    t_start, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    _barrier(world)
    torch.cuda.synchronize()
    wall0 = time.time()
    t_start.record(st)
    for k in range(K):
        for i, (w, comp) in enumerate(VARIANTS):
            ev[k][i][0].record(st)
            launch(i, w, comp)
            ev[k][i][1].record(st)
    t_end.record(st)
    torch.cuda.synchronize()
    wall1 = time.time()
    _barrier(world)
    clocks.stop()
    elapsed_ms = _max_over_ranks(t_start.elapsed_time(t_end), world)
    per_variant_ms = [statistics.mean(ev[k][i][0].elapsed_time(ev[k][i][1]) for k in range(K))
                      for i in range(len(VARIANTS))]
    launches = K * len(VARIANTS)

    value = _job_gbs(BYTES_PER_LAUNCH * launches, world, elapsed_ms)
    peak, peak_kind = _peaks()
    dom = int(np.argmax(per_variant_ms))
    achieved = BYTES_PER_LAUNCH / (per_variant_ms[dom] * 1e-3) / 1e9
    w_dom, c_dom = VARIANTS[dom]
    dom_name = f"k_tile_scan_rows<{'Comp' if c_dom else 'Plain<AddF>'}, {w_dom}>"
    traffic = NCU_TRAFFIC["bytes_per_launch"].get(dom_name) if NCU_TRAFFIC["src_sha"] == _src_sha() else None

    # ---- end to end through host buffers (pinned), copies inside the region
    e2e = run_e2e(args, x_host, dev, st, min(K, 20))

    result = {
        "metric": METRIC,
        "value": round(value, 2),
        "unit": "GB/s",
        "n_gpus": world,
        "steps": K,
        "warmup": args.warmup,
        "ms_per_step": round(elapsed_ms / K, 5),
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32",
        "data": "synthetic (seeded N(0,1) fp32, PCG64)",
        "config": {"workload": WORKLOAD, "n": N_ELEMS, "widths": list(WIDTHS), "block_dim": BLOCK,
                   "launches_per_step": len(VARIANTS), "parallelism": f"replicas x{world}",
                   "l2": "no flush: each launch streams 256 MiB in + 256 MiB out, > 129 MB L2"},
        "frac_of_hbm": round(value / world / peak, 4),
        "roofline": {"bound": "hbm", "kernel": dom_name,
                     "achieved": round(achieved, 1), "peak": peak, "peak_kind": peak_kind, "unit": "GB/s",
                     "frac": round(achieved / peak, 4), "traffic": traffic,
                     "algorithmic_bytes_per_launch": BYTES_PER_LAUNCH},
        "per_kernel_us": {f"W{w}{'_comp' if c else '_plain'}": round(ms * 1e3, 2)
                          for (w, c), ms in zip(VARIANTS, per_variant_ms)},
        "e2e": e2e,
        "gpu_launches": launches,
        "clocks": clocks.summary(wall0, wall1),
    }
    if rank == 0 and not args.no_secondary:
        result["secondary"] = run_secondary(dev, st)
    if rank == 0 and not args.no_cpu_baseline and world == 1:
        result["cpu_baseline"] = cpu_baseline(target_s=args.cpu_seconds)
        result["precision"] = oracle_precision(x_host, outs)
    if rank == 0:
        print(json.dumps(result), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_e2e(args, x_host, dev, st, K):
    """Same metric through the C ABI with host buffers: per step, the input goes
    host->device from pinned memory and all 8 outputs come back device->host.
    Steps are pipelined the way a streaming caller would run them: the input
    copy, the scans and the output copies sit on three streams ordered by
    events, so step k's output copies overlap step k+1's input copy and scans
    (the input is double-buffered; an output buffer is rewritten only after
    its previous copy to the host has finished)."""
    import torch
    from paper_2112_10034_gb300 import cox
    pin_in = torch.from_numpy(x_host).pin_memory()
    pin_out = [torch.empty(N_ELEMS, dtype=torch.float32).pin_memory() for _ in VARIANTS]
    xs = [torch.empty(N_ELEMS, dtype=torch.float32, device=dev) for _ in range(2)]
    outs = [torch.empty(N_ELEMS, dtype=torch.float32, device=dev) for _ in VARIANTS]
    s_h2d, s_d2h = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
    sh = st.cuda_stream
    ev = lambda: torch.cuda.Event()
    x_free = [ev(), ev()]          # scans of the step that last used xs[b] are done
    x_ready = [ev(), ev()]         # xs[b] holds this step's input
    scanned = [ev() for _ in VARIANTS]
    copied = [ev() for _ in VARIANTS]
    for e in x_free + copied:
        e.record(st)
    state = {"k": 0}

    def step():
        b = state["k"] % 2
        state["k"] += 1
        s_h2d.wait_event(x_free[b])
        with torch.cuda.stream(s_h2d):
            xs[b].copy_(pin_in, non_blocking=True)
        x_ready[b].record(s_h2d)
        st.wait_event(x_ready[b])
        for i, (w, comp) in enumerate(VARIANTS):
            st.wait_event(copied[i])
            s = cox.cox_tile_scan(cox.COX_SUM, cox.COX_F32, w, BLOCK, xs[b].data_ptr(), outs[i].data_ptr(), N_ELEMS,
                                  cox.COX_F_COMPENSATED if comp else 0, sh)
            if s != 0:
                raise cox.CoxError(s, "cox_tile_scan")
            scanned[i].record(st)
        x_free[b].record(st)
        for i in range(len(VARIANTS)):
            s_d2h.wait_event(scanned[i])
            with torch.cuda.stream(s_d2h):
                pin_out[i].copy_(outs[i], non_blocking=True)
            copied[i].record(s_d2h)

    for _ in range(2):
        step()
    torch.cuda.synchronize()
    a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(st)
    s_h2d.wait_event(a)
    s_d2h.wait_event(a)
    for _ in range(K):
        step()
    for e in copied:
        st.wait_event(e)
    z.record(st)
    z.synchronize()
    ms = a.elapsed_time(z) / K
    return {"value": round(BYTES_PER_LAUNCH * len(VARIANTS) / (ms * 1e-3) / 1e9, 2), "unit": "GB/s",
            "ms_per_step": round(ms, 4), "steps": K, "h2d_bytes_per_step": N_ELEMS * 4,
            "d2h_bytes_per_step": N_ELEMS * 4 * len(VARIANTS),
            "pipelining": "input copy, scans and output copies on three streams, ordered by events"}


def _time_launches(st, fn, iters=20, warm=3):
    import torch
    for _ in range(warm):
        fn()
    st.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(st)
    for _ in range(iters):
        fn()
    b.record(st)
    b.synchronize()
    return a.elapsed_time(b) / iters


def run_secondary(dev, st):
    """Other single-op workloads, each timed alone (device time per call)."""
    import torch
    from paper_2112_10034_gb300 import cox
    sh = st.cuda_stream
    peak, _ = _peaks()
    res = {}

    def chk(s):
        if s != 0:
            raise cox.CoxError(s)

    # block sum, 64 blocks x 256 threads of int32 (launch-latency bound)
    x = torch.from_numpy(inputs.uniform_int32(16384, -1000, 1000, inputs.BASE_SEED)).to(dev)
    out = torch.empty(64, dtype=torch.int32, device=dev)
    block_sum = lambda s: chk(cox.cox_tile_reduce(0, 0, 32, 256, 1, x.data_ptr(), out.data_ptr(), 16384, 0, None,
                                                  None, 0, s))
    ms = _time_launches(st, lambda: block_sum(sh), iters=200)
    # the same call 100 times inside one captured CUDA graph (launch overhead amortised by the graph)
    gs = torch.cuda.Stream(device=dev)
    for _ in range(3):
        block_sum(gs.cuda_stream)
    gs.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=gs):
        for _ in range(100):
            block_sum(gs.cuda_stream)
    with torch.cuda.stream(gs):  # (replay launches on the current stream)
        ms_graph = _time_launches(gs, graph.replay, iters=20) / 100
    del graph
    res["block_sum_64x256_int32"] = {"us_per_call": round(ms * 1e3, 2), "us_per_call_in_graph": round(ms_graph * 1e3, 3),
                                     "GB/s_in_graph": round((16384 * 4 + 64 * 4) / (ms_graph * 1e-3) / 1e9, 1),
                                     "graph": "100 calls captured once, replayed"}

    # the headline scans in their shuffle form: the same 2^26 elements starting 4 bytes
    # past a 16-byte boundary take the one-element-per-lane shfl_up kernel
    n = 1 << 26
    f = torch.from_numpy(inputs.normal_f32(n, inputs.BASE_SEED + 1)).to(dev)
    f1 = torch.empty(n + 4, dtype=torch.float32, device=dev)
    f1[1:n + 1] = f
    y1 = torch.empty(n + 4, dtype=torch.float32, device=dev)
    sf = {}
    for w, comp in VARIANTS:
        ms = _time_launches(st, lambda: chk(cox.cox_tile_scan(0, 2, w, BLOCK, f1.data_ptr() + 4, y1.data_ptr() + 4, n,
                                                              1 if comp else 0, sh)))
        gbs = n * 8 / (ms * 1e-3) / 1e9
        sf[f"W{w}{'_comp' if comp else '_plain'}"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1),
                                                     "frac": round(gbs / peak, 3)}
    sf["note"] = "input and output 4 bytes past a 16-byte boundary: k_tile_scan (shfl_up per lane), not the rows kernel"
    res["tile_scan_2p26_fp32_shuffle_form"] = sf
    del f1, y1

    # the warp functions themselves (cox_shfl) on 2^26 int32 elements: one result per lane
    # (4 bytes in + 4 out per element); shuffles at offset 1 / source lane 5, votes on
    # values in [0, 15] (nonzero 15 times in 16), match_any over those 16 keys
    ki = torch.from_numpy(inputs.uniform_int32(n, 0, 15, inputs.BASE_SEED + 6)).to(dev)
    ko = torch.empty(n, dtype=torch.int32, device=dev)
    wf = {}
    for name, fn, param in (("shfl_idx", 0, 5), ("shfl_up", 1, 1), ("shfl_down", 2, 1), ("shfl_xor", 3, 1),
                            ("ballot", 4, 0), ("any", 5, 0), ("all", 6, 0), ("match_any", 7, 0)):
        for w in (32, 8):
            ms = _time_launches(st, lambda: chk(cox.cox_shfl(fn, 0, w, BLOCK, ki.data_ptr(), ko.data_ptr(), n, param,
                                                             cox.FULL_MASK, sh)))
            gbs = n * 8 / (ms * 1e-3) / 1e9
            wf[f"{name}_W{w}"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
    res["warp_functions_2p26_int32"] = wf
    del ki, ko

    # tile reduce of 2^26 fp32 (one result per tile; compensated with its low word)
    tr = {}
    for W in (2, 32):
        y = torch.empty(n // W, dtype=torch.float32, device=dev)
        ylo = torch.empty(n // W, dtype=torch.float32, device=dev)
        for comp in (False, True):
            ms = _time_launches(st, lambda: chk(cox.cox_tile_reduce(0, 2, W, 256, 0, f.data_ptr(), y.data_ptr(), n,
                                                                    1 if comp else 0,
                                                                    ylo.data_ptr() if comp else None, None, 0, sh)))
            gbs = (n * 4 + (n // W) * 4 * (2 if comp else 1)) / (ms * 1e-3) / 1e9
            tr[f"W{W}{'_comp' if comp else '_plain'}"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1),
                                                         "frac": round(gbs / peak, 3)}
        del y, ylo
    res["tile_reduce_2p26_fp32"] = tr
    br = {}
    for B in (256, 1024):
        y = torch.empty(n // B, dtype=torch.float32, device=dev)
        for comp in (False, True):
            ms = _time_launches(st, lambda: chk(cox.cox_tile_reduce(0, 2, 32, B, 1, f.data_ptr(), y.data_ptr(), n,
                                                                    1 if comp else 0, None, None, 0, sh)))
            gbs = (n * 4 + (n // B) * 4) / (ms * 1e-3) / 1e9
            br[f"B{B}{'_comp' if comp else '_plain'}"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1),
                                                         "frac": round(gbs / peak, 3)}
        del y
    res["block_reduce_2p26_fp32_W32"] = br
    del f

    # stable compaction of 2^28 int32 keys at densities 0.1/0.5/0.9
    n = 1 << 28
    k = torch.from_numpy(inputs.uniform_u31(n, inputs.BASE_SEED + 2)).to(dev)
    o = torch.empty(n, dtype=torch.int32, device=dev)
    cnt = torch.empty(1, dtype=torch.int64, device=dev)
    wsb = cox.cox_ballot_compact_workspace(n, 256)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    comp = {}
    for d in (0.1, 0.5, 0.9):
        t = inputs.density_threshold(d)
        ms = _time_launches(st, lambda: chk(cox.cox_ballot_compact(0, 32, 256, k.data_ptr(), n, t, o.data_ptr(),
                                                                   cnt.data_ptr(), ws.data_ptr(), wsb, 0, sh)))
        kept = int(cnt.item())
        gbs = (n * 4 + kept * 4) / (ms * 1e-3) / 1e9
        comp[str(d)] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3),
                        "density": round(kept / n, 5)}
    res["compaction_2p28_int32"] = comp
    t = inputs.density_threshold(0.5)
    sweep = {}
    for blk in (512, 1024):  # tile = block x 16 keys
        wsb2 = cox.cox_ballot_compact_workspace(n, blk)
        ms = _time_launches(st, lambda: chk(cox.cox_ballot_compact(0, 32, blk, k.data_ptr(), n, t, o.data_ptr(),
                                                                   cnt.data_ptr(), ws.data_ptr(), wsb2, 0, sh)))
        gbs = (n * 4 + int(cnt.item()) * 4) / (ms * 1e-3) / 1e9
        sweep[str(blk)] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
    res["compaction_2p28_int32_d0.5_by_block"] = sweep
    del k, o

    # match histogram of 2^28 Zipf(1.1) keys into 256 bins
    z = torch.from_numpy(inputs.zipf_keys(n, inputs.BASE_SEED + 3)).to(dev)
    hist = torch.empty(256, dtype=torch.int32, device=dev)
    ms = _time_launches(st, lambda: chk(cox.cox_match_histogram(0, 32, 256, z.data_ptr(), n, 256, hist.data_ptr(),
                                                                None, 0, sh)))
    gbs = n * 4 / (ms * 1e-3) / 1e9
    hres = {"table_peer_masks": {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}}
    for name, fl in (("ballot_peer_masks", 32), ("native_match_any", 8), ("direct_atomics_no_match", 16)):
        ms = _time_launches(st, lambda: chk(cox.cox_match_histogram(0, 32, 256, z.data_ptr(), n, 256, hist.data_ptr(),
                                                                    None, fl, sh)))
        gbs = n * 4 / (ms * 1e-3) / 1e9
        hres[name] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
    res["match_histogram_2p28_zipf"] = hres
    del z

    # dynamic groups: filter_arr's aggregated atomic at d = 0.5 (2^28 keys) and a
    # coalesced-group inclusive scan over half-active warps (2^26 elements)
    t = inputs.density_threshold(0.5)
    ka = torch.from_numpy(inputs.uniform_u31(n, inputs.BASE_SEED + 2)).to(dev)
    oa = torch.empty(n, dtype=torch.int32, device=dev)
    ca = torch.empty(1, dtype=torch.int64, device=dev)
    ms = _time_launches(st, lambda: chk(cox.cox_filter_aggregated(0, ka.data_ptr(), n, t, oa.data_ptr(),
                                                                  ca.data_ptr(), sh)))
    gbs = (n * 4 + int(ca.item()) * 4) / (ms * 1e-3) / 1e9
    dyn = {"filter_aggregated_2p28_d0.5": {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1),
                                          "frac": round(gbs / peak, 3)}}
    del ka, oa
    m = 1 << 26
    xa = torch.randint(-1000, 1001, (m,), device=dev, dtype=torch.int32)
    act = (torch.rand(m, device=dev) < 0.5).to(torch.int32)
    ya = torch.empty_like(xa)
    nact = int(act.sum().item())
    for name, fn in (("coalesced_scan_sum_2p26_half_active", 9), ("coalesced_shfl_2p26_half_active", 2)):
        ms = _time_launches(st, lambda: chk(cox.cox_coalesced(fn, 0, 256, xa.data_ptr(), act.data_ptr(),
                                                              ya.data_ptr(), m, 3, sh)))
        gbs = (m * 8 + nact * 4) / (ms * 1e-3) / 1e9
        dyn[name] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
    del xa, act, ya
    res["dynamic_groups"] = dyn

    # second workload: batched vote statistics (2^26 predicates, 4096 segments of 16384,
    # tiles of 32) and integral images of 64 HD frames (8-bit pixels -> 32-bit sums)
    second = {}
    m = 1 << 26
    pv = (torch.rand(m, device=dev) < 0.9).to(torch.int32)
    vs = torch.empty(3 * (m // 16384), dtype=torch.int64, device=dev)
    ms = _time_launches(st, lambda: chk(cox.cox_vote_stats(0, 32, pv.data_ptr(), m, 16384, vs.data_ptr(), sh)))
    gbs = m * 4 / (ms * 1e-3) / 1e9
    second["vote_stats_2p26_w32"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
    del pv, vs
    B, H, W = 64, 1080, 1920
    for name, code, bpp in (("integral_image_64x1080x1920_u8", 3, 1), ("integral_image_64x1080x1920_u32", 1, 4)):
        img = torch.randint(0, 256, (B * H * W * bpp // 4 if bpp == 1 else B * H * W,), device=dev,
                            dtype=torch.int32)
        ii = torch.empty(B * H * W, dtype=torch.int32, device=dev)
        wsb_i = cox.cox_integral_image_workspace(B, H, W)
        ws_i = torch.empty(wsb_i, dtype=torch.uint8, device=dev)
        ms = _time_launches(st, lambda: chk(cox.cox_integral_image(code, B, H, W, img.data_ptr(), ii.data_ptr(),
                                                                   ws_i.data_ptr(), wsb_i, sh)))
        gbs = B * H * W * (bpp + 4) / (ms * 1e-3) / 1e9
        second[name] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3),
                        "algorithmic_bytes_per_pixel": bpp + 4}
        del img, ii, ws_i
    res["vote_stats_and_integral_image"] = second

    res["batched_10000_uneven"] = run_batched(dev, st)
    res["serving"] = run_serving(dev)

    # grid-scope (whole-array) inclusive scans
    gs = {}
    for name, dt, flags, nn in (("int32_sum_2p28", 0, 0, 1 << 28), ("fp32_comp_sum_2p27", 2, 1, 1 << 27)):
        xs = torch.randint(-1000, 1001, (nn,), device=dev, dtype=torch.int32) if dt == 0 else \
            torch.randn(nn, device=dev, dtype=torch.float32)
        ys = torch.empty_like(xs)
        wsb_s = cox.cox_scan_workspace(2, nn)
        ws_s = torch.empty(wsb_s, dtype=torch.uint8, device=dev)
        ms = _time_launches(st, lambda: chk(cox.cox_scan(0, dt, 2, 256, xs.data_ptr(), ys.data_ptr(), nn, flags, 0,
                                                         ws_s.data_ptr(), wsb_s, sh)))
        gbs = nn * 8 / (ms * 1e-3) / 1e9
        gs[name] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
        del xs, ys
    res["grid_scan"] = gs

    # grid-wide reduce-then-broadcast in one cooperative kernel (algorithmic: 4 B in + 4 B out per element)
    gb = {}
    for nn in (1 << 22, 1 << 26):
        xg = torch.randn(nn, device=dev, dtype=torch.float32)
        yg = torch.empty_like(xg)
        wsb_g = cox.cox_grid_broadcast_workspace(nn)
        ws_g = torch.empty(wsb_g, dtype=torch.uint8, device=dev)
        for name, opg in (("sub_min", 0), ("normalize", 1)):
            ms = _time_launches(st, lambda: chk(cox.cox_grid_broadcast(opg, 2, xg.data_ptr(), yg.data_ptr(), nn,
                                                                       ws_g.data_ptr(), wsb_g, sh)))
            gbs = nn * 8 / (ms * 1e-3) / 1e9
            gb[f"{name}_2p{nn.bit_length() - 1}_fp32"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1),
                                                          "frac": round(gbs / peak, 3)}
        del xg, yg
    gb["note"] = ("2^22 elements stay in shared memory across the barrier (read once); 2^26 are read twice, "
                  "so at most 8/12 of the copy peak")
    res["grid_broadcast"] = gb

    # grid reduce of 2^28 fp32, compensated
    f = torch.randn(n, dtype=torch.float32, device=dev)
    r = torch.empty(1, dtype=torch.float32, device=dev)
    wsb = cox.cox_tile_reduce_workspace(2, n, 256)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    ms = _time_launches(st, lambda: chk(cox.cox_tile_reduce(0, 2, 32, 256, 2, f.data_ptr(), r.data_ptr(), n, 1, None,
                                                            ws.data_ptr(), wsb, sh)))
    gbs = n * 4 / (ms * 1e-3) / 1e9
    res["grid_sum_2p28_fp32_comp"] = {"us": round(ms * 1e3, 1), "GB/s": round(gbs, 1), "frac": round(gbs / peak, 3)}
    return res


def run_batched(dev, st, num_arrays=10_000):
    """Batched workload: num_arrays arrays with lengths log-uniform on
    [32, 2^20] (~1e9 elements), fp32 N(0,1) values and Zipf(1.1) keys; per
    array a compensated sum and a 256-bin match histogram.  One persistent
    launch (+ ordered combine) replayed from a CUDA graph, against one launch
    per array (grid reduce + histogram) on the same stream.  Inputs are drawn
    on the device (torch generator) to keep the setup short."""
    import ctypes
    import torch
    from paper_2112_10034_gb300 import cox

    def chk(s, what="batched"):
        if s != 0:
            raise cox.CoxError(s, what)

    lens = inputs.loguniform_lengths(num_arrays, 32, 1 << 20, inputs.BASE_SEED + 3)
    padded = (lens + 3) // 4 * 4
    starts = np.concatenate([[0], np.cumsum(padded)[:-1]]).astype(np.int64)
    total_padded = int(padded.sum())
    E = int(lens.sum())
    g = torch.Generator(device=dev)
    g.manual_seed(inputs.BASE_SEED + 4)
    vals = torch.randn(total_padded, generator=g, device=dev, dtype=torch.float32)
    w = torch.arange(1, 257, dtype=torch.float64, device=dev) ** -1.1
    cdf = torch.cumsum(w / w.sum(), 0)
    cdf[-1] = 1.0
    keys = torch.empty(total_padded, dtype=torch.int32, device=dev)
    chunk = 1 << 27
    for c0 in range(0, total_padded, chunk):
        u = torch.rand(min(chunk, total_padded - c0), generator=g, device=dev, dtype=torch.float64)
        keys[c0:c0 + u.numel()] = torch.searchsorted(cdf, u, right=True).to(torch.int32)
        del u
    pv = torch.from_numpy(vals.data_ptr() + 4 * starts).to(dev)
    pk = torch.from_numpy(keys.data_ptr() + 4 * starts).to(dev)
    lens_h = torch.from_numpy(lens.astype(np.int64))
    wsb = cox.cox_batch_workspace(num_arrays)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    sums = torch.empty(num_arrays, dtype=torch.float32, device=dev)
    sums64 = torch.empty(num_arrays, dtype=torch.float64, device=dev)
    hists = torch.empty((num_arrays, 256), dtype=torch.int32, device=dev)
    sh = st.cuda_stream
    chk(cox.cox_batch_prepare(num_arrays, lens_h.data_ptr(), ws.data_ptr(), wsb, sh))
    best = cox.cox_batch_tune()
    best_ms = ctypes.c_float()
    chk(cox.cox_batch_autotune(num_arrays, pv.data_ptr(), pk.data_ptr(), ws.data_ptr(), wsb, sums.data_ptr(),
                               hists.data_ptr(), 2, None, ctypes.byref(best), ctypes.byref(best_ms), sh))
    graph = ctypes.c_void_p()
    chk(cox.cox_batch_graph_create(num_arrays, pv.data_ptr(), pk.data_ptr(), ctypes.addressof(best), ws.data_ptr(),
                                   wsb, sums.data_ptr(), sums64.data_ptr(), hists.data_ptr(), ctypes.byref(graph)))
    try:
        ms = _time_launches(st, lambda: chk(cox.cox_graph_launch(graph, sh)), iters=20)
    finally:
        cox.cox_graph_destroy(graph)
    # the same batch without peer groups (one shared atomic per key), for comparison
    direct = cox.cox_batch_tune(best.block_dim, best.ctas_per_sm, best.width, best.fp64_segments, 2, best.ept)
    ms_direct = _time_launches(st, lambda: chk(cox.cox_batch_sum_hist(
        num_arrays, pv.data_ptr(), pk.data_ptr(), ctypes.addressof(direct), ws.data_ptr(), wsb, sums.data_ptr(),
        sums64.data_ptr(), hists.data_ptr(), sh)), iters=10)
    nbytes = E * 8
    peak, _ = _peaks()

    # one launch per array: grid-scope compensated sum + match histogram, launched
    # from a C loop (cox_batch_percall), an event recorded after each array
    h_vals = (ctypes.c_void_p * num_arrays)(*[vals.data_ptr() + 4 * int(o) for o in starts])
    h_keys = (ctypes.c_void_p * num_arrays)(*[keys.data_ptr() + 4 * int(o) for o in starts])
    h_lens = lens.astype(np.int64)
    pscr_b = cox.cox_batch_percall_scratch(int(lens.max()))
    pscr = torch.empty(pscr_b, dtype=torch.uint8, device=dev)
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(num_arrays)]
    for e in evs:  # (torch creates the CUDA event at its first record)
        e.record(st)
    h_ev = (ctypes.c_void_p * num_arrays)(*[e.cuda_event for e in evs])

    def per_call(events=None):
        chk(cox.cox_batch_percall(num_arrays, h_vals, h_keys, h_lens.ctypes.data, sums.data_ptr(), hists.data_ptr(),
                                  pscr.data_ptr(), pscr_b, events, sh), "cox_batch_percall")

    per_call()  # warm-up
    st.synchronize()
    t0 = torch.cuda.Event(enable_timing=True)
    t0.record(st)
    per_call(h_ev)
    evs[-1].synchronize()
    done = np.array([t0.elapsed_time(e) for e in evs])
    pc_ms = float(done[-1])
    return {"arrays": num_arrays, "elements": E, "bytes": nbytes,
            "tune": dict(zip(["block_dim", "ctas_per_sm", "width", "fp64_segments", "native_match", "ept"],
                             best.astuple())),
            "graph_ms": round(ms, 4), "GB/s": round(nbytes / (ms * 1e-3) / 1e9, 1),
            "frac": round(nbytes / (ms * 1e-3) / 1e9 / peak, 3),
            "latency_ms": {"p50": round(ms, 4), "p99": round(ms, 4), "note": "every array completes with the batch"},
            "per_call": {"ms": round(pc_ms, 3), "GB/s": round(nbytes / (pc_ms * 1e-3) / 1e9, 1),
                         "launches": 2 * num_arrays, "how": "cox_batch_percall: a C loop, one stream",
                         "latency_ms": {"p50": round(float(np.percentile(done, 50)), 3),
                                        "p99": round(float(np.percentile(done, 99)), 3)}},
            "speedup_vs_per_call": round(pc_ms / ms, 2),
            "without_peer_groups": {"ms": round(ms_direct, 4), "GB/s": round(nbytes / (ms_direct * 1e-3) / 1e9, 1),
                                    "note": "direct shared atomics instead of match_any peers, not captured"}}


def run_serving(dev, rates=(1e3, 1e4, 1e5, 3e5, 1e6), count=1000, budget=8 << 30):
    """Serving workload: a Poisson stream of requests -- 1/3 reduce (half fp32
    compensated, half int32), 1/3 compensated fp32 tile scans (width 32), 1/3
    int32 compactions at density 0.5 -- with sizes log-uniform on [1K, 16M]
    elements, over an 8 GB admission budget, at each arrival rate: the
    continuous-batching server against one launch per request (same trace).
    Inputs are windows of 2^28-element device pools drawn by torch."""
    import torch
    from paper_2112_10034_gb300 import cox
    pool_n = 1 << 28
    g = torch.Generator(device=dev)
    g.manual_seed(inputs.BASE_SEED + 5)
    pf = torch.randn(pool_n, generator=g, device=dev, dtype=torch.float32)
    pi = torch.randint(-1000, 1001, (pool_n,), generator=g, device=dev, dtype=torch.int32)
    pk = torch.randint(0, 2**31 - 1, (pool_n,), generator=g, device=dev, dtype=torch.int32)
    thr = inputs.density_threshold(0.5)
    out = {}
    for rate in rates:
        seed = inputs.BASE_SEED + 50 + int(np.log10(rate) * 10)
        sizes = inputs.loguniform_lengths(count, 1024, 1 << 24, seed)
        kinds = inputs.choice(count, 3, seed + 1)
        offs = inputs.choice(count, pool_n, seed + 2)
        arrivals = inputs.poisson_arrivals(count, rate, seed + 3)
        items, nbytes = [], 0
        for i in range(count):
            n = int(sizes[i])
            o4 = int(min(offs[i], pool_n - n)) // 4 * 4
            if kinds[i] == 0:
                if i % 2:
                    r = cox.cox_request(cox.COX_REQ_REDUCE, cox.COX_F32, 32, cox.COX_F_COMPENSATED, n, 0,
                                        pf.data_ptr() + 4 * o4)
                else:
                    r = cox.cox_request(cox.COX_REQ_REDUCE, cox.COX_I32, 32, 0, n, 0, pi.data_ptr() + 4 * o4)
                nbytes += 4 * n
            elif kinds[i] == 1:
                r = cox.cox_request(cox.COX_REQ_SCAN, cox.COX_F32, 32, cox.COX_F_COMPENSATED, n, 0,
                                    pf.data_ptr() + 4 * o4)
                nbytes += 8 * n
            else:
                r = cox.cox_request(cox.COX_REQ_COMPACT, cox.COX_I32, 32, 0, n, thr, pk.data_ptr() + 4 * o4)
                nbytes += 6 * n
            items.append((float(arrivals[i]), r))
        srv = cox.Server(budget, max_requests=1024)
        try:
            srv.run_trace(items[:50])  # warm-up
            st0 = srv.stats()
            lat, wall = srv.run_trace(items)
            st = srv.stats()
            st["batches"] -= st0["batches"]
        finally:
            srv.close()
        cox.percall_run_trace(items[:50])
        lat2, wall2 = cox.percall_run_trace(items)
        lat, lat2 = np.array(lat) * 1e3, np.array(lat2) * 1e3
        out[f"{rate:.0e}"] = {
            "offered_req_per_s": rate,
            "server": {"req_per_s": round(count / wall, 1), "GB/s": round(nbytes / wall / 1e9, 1),
                       "p50_ms": round(float(np.percentile(lat, 50)), 3),
                       "p99_ms": round(float(np.percentile(lat, 99)), 3),
                       "batches": st["batches"], "max_batch": st["max_batch"],
                       "peak_bytes": st["peak_bytes"]},
            "per_call": {"req_per_s": round(count / wall2, 1), "GB/s": round(nbytes / wall2 / 1e9, 1),
                         "p50_ms": round(float(np.percentile(lat2, 50)), 3),
                         "p99_ms": round(float(np.percentile(lat2, 99)), 3)}}
    return {"requests_per_rate": count, "budget_bytes": budget, "sizes": "log-uniform [1K, 16M]",
            "rates": out}


# ------------------------------------------------------ CPU (oracle) legs
def _oracle_step(o, x):
    for w, comp in VARIANTS:
        o.scan_emulate(o.SUM, o.F32, w, BLOCK, x, comp)


def cpu_baseline(target_s: float = 12.0):
    """The oracle's collapsed-loop executor on a bounded sample of the workload:
    the first n elements (grown until one pass takes a quarter of the target, up
    to all 2^26), all 8 width/mode scans, repeated until target_s seconds."""
    import oracle as o
    x_full = inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)
    n = 1 << 18
    while True:
        x = x_full[:n]
        t0 = time.perf_counter()
        _oracle_step(o, x)
        dt = time.perf_counter() - t0
        if dt * 4 >= target_s or n >= N_ELEMS:
            break
        n = min(N_ELEMS, n * 4)
    passes, total = 1, dt
    while total < target_s:
        t0 = time.perf_counter()
        _oracle_step(o, x)
        total += time.perf_counter() - t0
        passes += 1
    gbs = n * 8 * len(VARIANTS) * passes / total / 1e9
    return {"value": round(gbs, 4), "unit": "GB/s", "cores": o.threads(), "kind": "oracle",
            "sample": f"first {n} of the 2^26 elements, all 8 width/mode scans, {passes} passes, {total:.1f} s"}


def _err_stats(y, ref, ab):
    """Errors of fp32 results y against FP64 values ref (sum|x| of the inputs
    of each output in ab): the tolerance metric |y - r| / max(|r|, 2^-24
    sum|x|) (max), pointwise |y - r| / |r| over r != 0 (max and p99), and the
    normwise ||y - r||_2 / ||r||_2."""
    y = y.astype(np.float64)
    d = np.abs(y - ref)
    den = np.maximum(np.abs(ref), 2.0 ** -24 * ab)
    tol_metric = float(np.max(d / np.where(den == 0, 1.0, den)))
    nz = ref != 0
    pw = d[nz] / np.abs(ref[nz])
    return {"max": tol_metric, "pointwise_max": float(pw.max()), "pointwise_p99": float(np.percentile(pw, 99)),
            "normwise": float(np.linalg.norm(y - ref) / np.linalg.norm(ref))}


def oracle_precision(x_host, outs):
    """Part of the oracle leg (outside every timed region): the error of each
    of the 8 timed scans' outputs, as they stand after the last timed step,
    against the oracle's FP64 tile prefix of the same 2^26 inputs, and
    whether they equal the oracle's fp32 emulation of the stated order bit
    for bit (a check of this run's outputs)."""
    import oracle as o
    rows, refs = {}, {}
    for (w, comp), out in zip(VARIANTS, outs):
        if w not in refs:
            _, ref, ab = o.scan_ref(o.SUM, o.F32, w, x_host)
            refs = {w: (ref, ab)}
        ref, ab = refs[w]
        y = out.cpu().numpy()
        e = _err_stats(y, ref, ab)
        row = {k: float(f"{v:.3e}") for k, v in e.items()}
        row["meets_1e-5"] = e["max"] <= 1e-5
        # the kernels follow the stated association order: the oracle's fp32
        # emulation of that order must give the same bits at every output
        row["bits_equal_oracle_emulation"] = bool(np.array_equal(
            y.view(np.uint32), o.scan_emulate(o.SUM, o.F32, w, BLOCK, x_host, comp).view(np.uint32)))
        rows[f"W{w}_{'comp' if comp else 'plain'}"] = row
    return {"reference": "oracle FP64 tile prefix (Neumaier) of the same 2^26 fp32 inputs",
            "metric": "max = max |y-r|/max(|r|, 2^-24 sum|x|) (the 1e-5 bar, gated for compensated); "
                      "pointwise over r != 0; normwise ||y-r||_2/||r||_2",
            "rows": rows}


def run_reference(args):
    """Reference arm: the CPU oracle (collapsed-loop executor) on this workload."""
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle as o
    x_full = inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)
    # size each step so that warm-up + timed steps take about two minutes
    n = 1 << 16
    t0 = time.perf_counter()
    _oracle_step(o, x_full[:n])
    per_elem = (time.perf_counter() - t0) / n
    budget = min(1.0, 120.0 / max(1, args.steps + args.warmup))
    n = int(max(1 << 14, min(N_ELEMS, budget / per_elem)))
    n -= n % 1024
    x = x_full[:n]
    for _ in range(args.warmup):
        _oracle_step(o, x)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        _oracle_step(o, x)
    dt = time.perf_counter() - t0
    gbs = n * 8 * len(VARIANTS) * args.steps / dt / 1e9
    sample = f"first {n} of the 2^26 elements per step, all 8 width/mode scans"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": round(gbs, 4), "unit": "GB/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(dt / args.steps * 1e3, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic (seeded N(0,1) fp32, PCG64)",
        "config": {"workload": WORKLOAD, "n": N_ELEMS, "widths": list(WIDTHS), "block_dim": BLOCK,
                   "sample_n": n},
        "cpu_baseline": {"value": round(gbs, 4), "unit": "GB/s", "cores": o.threads(), "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": round(gbs, 4), "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def run_profile(args):
    """Small cases for ncu captures (a few hundred MiB on the device, inputs
    larger than L2), one op each: `scan` runs the 8 scan launches per step over
    one 2^26-element input and one output; `compact` runs 2^26-key compactions
    at density 0.5; `hist` runs 2^26-key Zipf match histograms; `batch` runs
    the batched kernel on 1000 arrays of the batched length law (~1e8
    elements); `gridscan` a 2^26 int32 grid-scope scan (`gridscan_comp`: fp32
    compensated); `blockscan` a 2^26 fp32 block-scope
    scan at B 256, plain then compensated; `reduce` a 2^26 fp32
    compensated tile reduce (W 32) then block reduce (B 256); `intimage` the
    integral images of 64 8-bit 1080x1920 frames (a memset of the strip
    totals, then the strip walk), `intimage32` the same with 32-bit pixels; `filter` the
    aggregated filter of 2^26 keys at density 0.5; `coalesced` the group
    size then the group shuffle over 2^26 half-active elements."""
    import torch
    from paper_2112_10034_gb300 import cox
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(device=dev)
    sh = st.cuda_stream

    def chk(s):
        if s != 0:
            raise cox.CoxError(s, args.profile)

    reps = args.warmup + args.steps
    if args.profile == "scan":
        x = torch.from_numpy(inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)).to(dev)
        out = torch.empty(N_ELEMS, dtype=torch.float32, device=dev)
        for _ in range(reps):
            for w, comp in VARIANTS:
                chk(cox.cox_tile_scan(cox.COX_SUM, cox.COX_F32, w, BLOCK, x.data_ptr(), out.data_ptr(), N_ELEMS,
                                      cox.COX_F_COMPENSATED if comp else 0, sh))
        launches = reps * len(VARIANTS)
    elif args.profile == "compact":
        k = torch.from_numpy(inputs.uniform_u31(N_ELEMS, inputs.BASE_SEED + 2)).to(dev)
        out = torch.empty(N_ELEMS, dtype=torch.int32, device=dev)
        cnt = torch.empty(1, dtype=torch.int64, device=dev)
        wsb = cox.cox_ballot_compact_workspace(N_ELEMS, 256)
        ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
        for _ in range(reps):
            chk(cox.cox_ballot_compact(0, 32, 256, k.data_ptr(), N_ELEMS, inputs.density_threshold(0.5),
                                       out.data_ptr(), cnt.data_ptr(), ws.data_ptr(), wsb, 0, sh))
        launches = reps
    elif args.profile == "gridscan":
        xi = torch.randint(-1000, 1001, (N_ELEMS,), device=dev, dtype=torch.int32)
        yi = torch.empty_like(xi)
        wsb = cox.cox_scan_workspace(2, N_ELEMS)
        ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
        for _ in range(reps):
            chk(cox.cox_scan(0, 0, 2, 256, xi.data_ptr(), yi.data_ptr(), N_ELEMS, 0, 0, ws.data_ptr(), wsb, sh))
        launches = reps
    elif args.profile == "blockscan":
        xf = torch.from_numpy(inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)).to(dev)
        yf = torch.empty_like(xf)
        for _ in range(reps):
            for comp in (False, True):
                chk(cox.cox_scan(0, 2, 1, BLOCK, xf.data_ptr(), yf.data_ptr(), N_ELEMS,
                                 cox.COX_F_COMPENSATED if comp else 0, 0, None, 0, sh))
        launches = reps * 2
    elif args.profile == "gridscan_comp":
        xf = torch.from_numpy(inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)).to(dev)
        yf = torch.empty_like(xf)
        wsb = cox.cox_scan_workspace(2, N_ELEMS)
        ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
        for _ in range(reps):
            chk(cox.cox_scan(0, 2, 2, 256, xf.data_ptr(), yf.data_ptr(), N_ELEMS, cox.COX_F_COMPENSATED, 0,
                             ws.data_ptr(), wsb, sh))
        launches = reps
    elif args.profile == "reduce":
        x = torch.from_numpy(inputs.normal_f32(N_ELEMS, inputs.BASE_SEED + 1)).to(dev)
        y = torch.empty(N_ELEMS // 32, dtype=torch.float32, device=dev)
        ylo = torch.empty(N_ELEMS // 32, dtype=torch.float32, device=dev)
        for _ in range(reps):  # tile reduce W=32 compensated with low words, then block reduce B=256
            chk(cox.cox_tile_reduce(0, 2, 32, 256, 0, x.data_ptr(), y.data_ptr(), N_ELEMS, 1, ylo.data_ptr(), None, 0,
                                    sh))
            chk(cox.cox_tile_reduce(0, 2, 32, 256, 1, x.data_ptr(), y.data_ptr(), N_ELEMS, 1, None, None, 0, sh))
        launches = reps * 2
    elif args.profile in ("intimage", "intimage32"):
        B, H, W = 64, 1080, 1920
        code, words = (3, B * H * W // 4) if args.profile == "intimage" else (1, B * H * W)
        img = torch.randint(0, 256, (words,), device=dev, dtype=torch.int32)
        ii = torch.empty(B * H * W, dtype=torch.int32, device=dev)
        wsb = cox.cox_integral_image_workspace(B, H, W)
        ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
        for _ in range(reps):
            chk(cox.cox_integral_image(code, B, H, W, img.data_ptr(), ii.data_ptr(), ws.data_ptr(), wsb, sh))
        launches = reps
    elif args.profile == "filter":
        k = torch.from_numpy(inputs.uniform_u31(N_ELEMS, inputs.BASE_SEED + 2)).to(dev)
        out = torch.empty(N_ELEMS, dtype=torch.int32, device=dev)
        cnt = torch.empty(1, dtype=torch.int64, device=dev)
        for _ in range(reps):
            chk(cox.cox_filter_aggregated(0, k.data_ptr(), N_ELEMS, inputs.density_threshold(0.5), out.data_ptr(),
                                          cnt.data_ptr(), sh))
        launches = reps
    elif args.profile == "coalesced":
        g = torch.Generator(device="cpu").manual_seed(inputs.BASE_SEED + 4)
        xa = torch.randint(-1000, 1001, (N_ELEMS,), generator=g, dtype=torch.int32).to(dev)
        act = (torch.rand(N_ELEMS, generator=g) < 0.5).to(torch.int32).to(dev)
        ya = torch.empty_like(xa)
        for _ in range(reps):
            for fn in (cox.COX_CG_SIZE, cox.COX_CG_SHFL):
                chk(cox.cox_coalesced(fn, 0, 256, xa.data_ptr(), act.data_ptr(), ya.data_ptr(), N_ELEMS, 3, sh))
        launches = reps * 2
    elif args.profile == "batch":
        lens = inputs.loguniform_lengths(1000, 32, 1 << 20, inputs.BASE_SEED + 3)
        vals = [torch.randn(int(L), device=dev) for L in lens]
        keys = [torch.randint(0, 256, (int(L),), device=dev, dtype=torch.int32) for L in lens]
        b = cox.Batch(vals, keys)
        for _ in range(reps):
            b.run(sh)
        launches = reps * 2
    else:
        z = torch.from_numpy(inputs.zipf_keys(N_ELEMS, inputs.BASE_SEED + 3)).to(dev)
        hist = torch.empty(256, dtype=torch.int32, device=dev)
        for _ in range(reps):
            chk(cox.cox_match_histogram(0, 32, 256, z.data_ptr(), N_ELEMS, 256, hist.data_ptr(), None, 0, sh))
        launches = reps
    st.synchronize()
    print(json.dumps({"profile": args.profile, "launches": launches}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="cox", choices=["cox", "reference"])
    ap.add_argument("--no-secondary", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--profile", choices=["scan", "compact", "hist", "batch", "gridscan", "gridscan_comp", "blockscan", "reduce",
                                          "intimage", "intimage32", "filter", "coalesced"],
                    default=None,
                    help="small single-op case for ncu captures")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.profile:
        run_profile(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_cox(args)


if __name__ == "__main__":
    main()
