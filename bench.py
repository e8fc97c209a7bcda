#!/usr/bin/env python
"""Benchmark of the LBP-WHT linear-backward hot path on B200.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
  python bench.py --profile-layer L [--profile-config C] [--profile-rank R] [--iters N]

One step = Algorithm 1 (project x and g_y, the two low-rank products, expand
g_x) for the four linear layers of a ViT-B block (qkv, proj, fc1, fc2) on one
batch of B=128 images with a 16x16 token grid, WHT order k=8, rank r=8, bf16
data with fp32 accumulation, issued as one lbp_backward_batch call.  The metric
is tokens/s: tokens of the batch (32768 per GPU) divided by the time of one
step.  The timed region holds nothing but those calls; per-layer and per-phase
times, the other configurations, the rank sweeps and the end-to-end figure are
measured in separate legs after it.

Prints ONE JSON line (rank 0).  `--impl reference` times the fp64 CPU oracle on
a bounded sample of the same workload instead.  `--profile-layer` runs one
layer a few times and prints its time: a small fixed workload for profilers.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "LBP-WHT linear backward tokens/s at rank r; % of HBM/tensor roofline"
UNIT = "tokens/s"
CONFIG = 3
RANK = 8
WORKLOAD = ("config3: ViT-B block linears qkv 768->2304, proj 768->768, fc1 768->3072, "
            "fc2 3072->768; B=128, grid 16x16, k=8, r=8 (PREFIX-8 low-pass set), bf16")


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return {"hbm_gbs": float(p["hbm_gbs"]), "bf16_tflops": float(p["bf16_tflops"]),
                "bf16_tflops_sustained": float(p.get("bf16_tflops_sustained", p["bf16_tflops"])),
                "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0,
            "source": "fallback"}


# DRAM traffic per step (sum over the four layers, bytes) of the two kernels, from
# the ncu capture summarised in profiles/ (dram__bytes_read.sum + dram__bytes_write.sum);
# None = not captured for the current kernels.
NCU_TRAFFIC_PER_STEP = {"wht_project_umma_kernel": 822.5e6, "lbp_products_kernel": 285.3e6}


# ------------------------------------------------------------------ clocks ----
_SAMPLER_CODE = r"""
import sys, time
import pynvml as n
n.nvmlInit()
h = n.nvmlDeviceGetHandleByIndex(int(sys.argv[1]))
mx = n.nvmlDeviceGetMaxClockInfo(h, n.NVML_CLOCK_SM)
for _ in range(5):          # the first queries are slow: not inside the timed region
    try:
        n.nvmlDeviceGetClockInfo(h, n.NVML_CLOCK_SM)
    except Exception:
        pass
print("ready", flush=True)
end = time.time() + 120.0
while time.time() < end:
    try:
        mhz = n.nvmlDeviceGetClockInfo(h, n.NVML_CLOCK_SM)
    except Exception:
        continue
    mask = 0
    for name in ("nvmlDeviceGetCurrentClocksEventReasons", "nvmlDeviceGetCurrentClocksThrottleReasons"):
        try:
            mask = getattr(n, name)(h)
            break
        except Exception:
            pass
    print(repr(time.time()), mhz, mask, mx, flush=True)
    time.sleep(0.001)       # every query costs the running kernels time (about 1.5 % of a step when issued back to back)
"""


class ClockSampler:
    """Samples SM clock and throttle reasons through NVML while the timed region
    runs.  The sampling loop lives in a child process (started before the timed
    region, no GPU context of its own): a thread of this process would share the
    interpreter lock with the launching loop and hardly ever run.  If the child
    yields nothing, nvidia-smi is asked once right after the region."""

    REASONS = {0x8: "hw_slowdown", 0x40: "hw_thermal_slowdown", 0x20: "sw_thermal_slowdown",
               0x4: "sw_power_cap"}

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen([sys.executable, "-c", _SAMPLER_CODE, str(self.index)],
                                         stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)
            self.proc.stdout.readline()      # "ready": the child is up and sampling
        except Exception:
            self.proc = None

    def _smi_once(self):
        try:
            out = subprocess.run(["nvidia-smi", "-i", str(self.index),
                                  "--query-gpu=clocks.sm,clocks.max.sm,clocks_event_reasons.active",
                                  "--format=csv,noheader,nounits"], capture_output=True, text=True,
                                 timeout=20).stdout.strip().split(",")
            return float(out[0]), int(float(out[1])), int(out[2].strip(), 16)
        except Exception:
            return None

    def stop(self, t_begin: float, t_end: float):
        """Summary of the samples taken between the two time.time() stamps."""
        rows, err = [], ""
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, err = self.proc.communicate(timeout=10)
            except Exception:
                out, err = "", "sampler did not end"
            for ln in out.splitlines():
                f = ln.split()
                if len(f) == 4:
                    try:
                        rows.append((float(f[0]), int(f[1]), int(f[2]), int(f[3])))
                    except ValueError:
                        pass
        inside = [r for r in rows if t_begin <= r[0] <= t_end]
        how = "NVML from a child process, about once a millisecond"
        if not inside and rows:     # a region shorter than one sampling period: the nearest sample
            mid = 0.5 * (t_begin + t_end)
            inside = [min(rows, key=lambda r: abs(r[0] - mid))]
        if not inside:
            one = self._smi_once()
            if one is not None:
                inside = [(t_end, int(one[0]), one[2], one[1])]
                how = "nvidia-smi once, right after the timed region (the NVML sampler gave nothing: " \
                      + (err.strip().splitlines()[-1][:120] if err and err.strip() else "no output") + ")"
        reasons = set()
        for r in inside:
            for bit, name in self.REASONS.items():
                if r[2] & bit:
                    reasons.add(name)
        med = statistics.median([r[1] for r in inside]) if inside else None
        return {"sm_mhz": med, "sm_max_mhz": inside[0][3] if inside else None,
                "reasons": sorted(reasons), "samples": len(inside), "sampling": how}


# ------------------------------------------------------------- cpu oracle ----
def _oracle_sample(batch: int, repeats: int = 1, threads: int | None = None):
    """Times the fp64 oracle's low-rank route on `batch` images of every layer."""
    import torch
    import synth
    from oracle import lbp_oracle as O

    cases = synth.config_cases(CONFIG)
    bases = O.select_bases(cases[0].k, O.RULE_PREFIX, RANK)
    data = []
    for c in cases:
        x, gy, w = synth.make_layer_inputs(c, batch=batch)
        data.append((c, x.to(torch.float64).numpy(), gy.to(torch.float64).numpy(),
                     w.to(torch.float64).numpy()))

    def run():
        out = []
        for _ in range(repeats):
            t0 = time.perf_counter()
            for c, x, gy, w in data:
                O.backward_lowrank(x, gy, w, c.k, bases)
            out.append(time.perf_counter() - t0)
        return out

    cores = os.cpu_count() or 1
    try:
        from threadpoolctl import threadpool_info, threadpool_limits
        if threads is not None:
            with threadpool_limits(limits=threads):
                times = run()
            cores = threads
        else:
            times = run()
            cores = max([p.get("num_threads", 1) for p in threadpool_info()] or [1])
    except ImportError:
        times = run()
    tokens = batch * cases[0].H * cases[0].W
    return tokens, times, cores


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    steps = max(1, args.steps)
    # bounded sample: about 0.07 s of oracle time per image; keep the whole run near 90 s
    batch = int(max(1, min(16, 90.0 / (steps + args.warmup) / 0.07)))
    tokens, times, cores = _oracle_sample(batch, repeats=args.warmup + steps)
    timed = times[args.warmup:]
    sec = sum(timed) / len(timed)
    value = tokens / sec
    sample = f"first {batch} of 128 images of all four layers, r={RANK}, fp64 numpy oracle"
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": steps, "warmup": args.warmup, "ms_per_step": sec * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "sample": sample},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line))
    return 0


# ------------------------------------------------------- profiler workload ----
def run_profile(args):
    """lbp_backward on one synthetic layer, a few times (for ncu and quick timing)."""
    import torch
    import paper_2309_15275_b200 as lbp
    import synth

    dev = torch.device("cuda:0")
    case = synth.config_cases(args.profile_config)[args.profile_layer]
    x, gy, w = (t.to(dev) for t in synth.make_layer_inputs(case, batch=args.profile_batch))
    k = case.k
    r = k * k if args.profile_fullrank else args.profile_rank
    bases = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, min(r, k * k))
    ws = lbp.alloc_workspace(x, gy, k, r)
    gx = torch.empty_like(x)
    gw = torch.empty((case.Cout, case.Cin), dtype=torch.float32, device=dev)
    beg, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for it in range(args.iters + 1):
        if it == 1:
            beg.record()
        if args.profile_fullrank:
            lbp.lbp_backward_fullrank(x, gy, w, k, g_x=gx, g_W=gw, ws=ws)
        else:
            lbp.lbp_backward(x, gy, w, k, bases, g_x=gx, g_W=gw, ws=ws)
    end.record()
    st = lbp.lbp_poll_status(ws)
    print(f"{case.name} B={x.shape[0]} r={r}: "
          f"{beg.elapsed_time(end) / max(args.iters, 1) * 1e3:.1f} us/call, status {st}")
    return 0 if st == 0 else 1


# ------------------------------------------------------------------- main ----
def _alg_bytes(T, Cin, Cout, es=2):
    """x, g_y, W read once; g_x and the fp32 g_W written once.  The low-rank
    intermediates are not algorithmic."""
    return es * T * (2 * Cin + Cout) + es * Cin * Cout + 4 * Cin * Cout


def _roof_us(peaks, T, Cin, Cout, rows):
    return max(_alg_bytes(T, Cin, Cout) / (peaks["hbm_gbs"] * 1e9),
               4.0 * Cin * Cout * rows / (peaks["bf16_tflops"] * 1e12)) * 1e6


def run_gpu(args):
    import torch
    import torch.distributed as dist
    import paper_2309_15275_b200 as lbp
    import synth
    from paper_2309_15275_b200.dist import GwReducer, allreduce_gw

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise RuntimeError("bench.py needs a CUDA device: the library has no CPU path")
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl", device_id=dev)

    from paper_2309_15275_b200.build import build_library
    if not os.path.exists(lbp.LIB_PATH):
        build_library()

    cases = synth.config_cases(CONFIG)
    k = cases[0].k
    bases = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, RANK)
    peaks = _peaks()
    steps = max(1, args.steps)
    warmup = max(args.warmup, 3)

    # per-rank batch: every rank owns its own seeded batch of B images (weak scaling)
    layers = []
    for c in cases:
        x, gy, w = synth.make_layer_inputs(c, seed=synth.SEED + rank)
        L = {"case": c, "x_h": x.pin_memory(), "gy_h": gy.pin_memory(), "w_h": w.pin_memory()}
        L["x"], L["gy"], L["w"] = x.to(dev), gy.to(dev), w.to(dev)
        L["gx"] = torch.empty_like(L["x"])
        L["gw"] = torch.empty((c.Cout, c.Cin), dtype=torch.float32, device=dev)
        L["ws"] = lbp.alloc_workspace(L["x"], L["gy"], k, RANK)
        L["ws_full"] = lbp.alloc_workspace(L["x"], L["gy"], k, k * k)
        L["gx_h"] = torch.empty_like(L["x_h"]).pin_memory()
        L["gw_h"] = torch.empty((c.Cout, c.Cin), dtype=torch.float32).pin_memory()
        layers.append(L)
    tokens_per_step = cases[0].tokens          # per GPU
    flush_buf = torch.empty(256 << 20, dtype=torch.uint8, device=dev)   # twice the L2

    # Data-parallel exchange (N > 1): the all-reduce of a layer's g_W runs on a side
    # stream as soon as that layer's kernels are done (an event per layer recorded by
    # the batch call), under the kernels of the layers that follow.
    cur = torch.cuda.current_stream()
    reducer = GwReducer(len(layers), dev)

    def step(wss=None, bases_=bases):
        # the four layers are independent problems with their own buffers: one call
        lbp.lbp_backward_batch([L["x"] for L in layers], [L["gy"] for L in layers],
                               [L["w"] for L in layers], k, bases_,
                               g_xs=[L["gx"] for L in layers], g_Ws=[L["gw"] for L in layers],
                               wss=wss if wss is not None else [L["ws"] for L in layers],
                               done_events=reducer.events())
        reducer.reduce([L["gw"] for L in layers])

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    for _ in range(warmup):
        step()
    barrier()

    # ---- timed region: exactly K steps, CUDA events on the launching stream ----
    sampler = ClockSampler(local_rank)
    if rank == 0:
        sampler.start()
    launches0 = lbp.lbp_launch_count()
    t_beg, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    wall0 = time.time()
    t_beg.record()
    for _ in range(steps):
        step()
    t_end.record()
    barrier()
    wall1 = time.time()
    clocks = sampler.stop(wall0, wall1) if rank == 0 else None
    launches = lbp.lbp_launch_count() - launches0
    ms_total = t_beg.elapsed_time(t_end)
    for L in layers:
        st = lbp.lbp_poll_status(L["ws"])
        if st != 0:
            raise RuntimeError(f"device status {st}: {lbp.lbp_status_string(st)}")
    if world > 1:
        t = torch.tensor([ms_total], dtype=torch.float64, device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms_total = float(t.item())
    ms_per_step = ms_total / steps
    value = tokens_per_step * world / (ms_per_step * 1e-3)

    line = None
    if rank == 0:
        line = _report_legs(args, torch, lbp, synth, dev, layers, k, bases, peaks, flush_buf, step,
                            world, steps, warmup, ms_per_step, value, launches, clocks,
                            tokens_per_step)
    barrier()

    # ---- end to end: host buffers, copies inside the timed region ----
    e2e_steps = max(1, min(steps, 3))
    h2d = sum(L[n].numel() * L[n].element_size() for L in layers for n in ("x_h", "gy_h", "w_h"))
    d2h = sum(L[n].numel() * L[n].element_size() for L in layers for n in ("gx_h", "gw_h"))

    # Copies run on two side streams so that the host-to-device copy of the next
    # layer, the kernels of this layer and the device-to-host copy of the previous
    # one overlap (PCIe is full duplex); events order every reuse of a buffer.
    s_in, s_out = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
    for L in layers:
        L["ev_in"], L["ev_done"], L["ev_out"] = (torch.cuda.Event() for _ in range(3))
        L["ev_done"].record(cur)
        L["ev_out"].record(cur)

    def e2e_step():
        for L in layers:
            with torch.cuda.stream(s_in):
                s_in.wait_event(L["ev_done"])          # the previous step's kernels read these buffers
                L["x"].copy_(L["x_h"], non_blocking=True)
                L["gy"].copy_(L["gy_h"], non_blocking=True)
                L["w"].copy_(L["w_h"], non_blocking=True)
                L["ev_in"].record(s_in)
            cur.wait_event(L["ev_in"])
            cur.wait_event(L["ev_out"])                # the previous step's results have left g_x / g_W
            lbp.lbp_backward(L["x"], L["gy"], L["w"], k, bases, g_x=L["gx"], g_W=L["gw"], ws=L["ws"])
            allreduce_gw(L["gw"])
            L["ev_done"].record(cur)
            with torch.cuda.stream(s_out):
                s_out.wait_event(L["ev_done"])
                L["gx_h"].copy_(L["gx"], non_blocking=True)
                L["gw_h"].copy_(L["gw"], non_blocking=True)
                L["ev_out"].record(s_out)

    def e2e_join():
        for L in layers:
            cur.wait_event(L["ev_out"])

    e2e_step()
    e2e_join()
    barrier()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(e2e_steps):
        e2e_step()
    e2e_join()                                         # every result is in host memory
    b.record()
    barrier()
    e2e_ms = a.elapsed_time(b) / e2e_steps
    if world > 1:
        t = torch.tensor([e2e_ms], dtype=torch.float64, device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        e2e_ms = float(t.item())
    e2e_value = tokens_per_step * world / (e2e_ms * 1e-3)

    if rank == 0:
        line["e2e"] = {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d,
                       "d2h_bytes_per_step": d2h, "ms_per_step": e2e_ms, "steps": e2e_steps}
        if world == 1:
            sample = f"first 16 of 128 images of all four layers, r={RANK}, fp64 numpy oracle"
            tok, t_all, cores = _oracle_sample(16, repeats=1)
            tok1, t_one, _ = _oracle_sample(4, repeats=1, threads=1)
            line["cpu_baseline"] = {"value": tok / t_all[0], "unit": UNIT, "cores": cores,
                                    "kind": "oracle", "sample": sample,
                                    "one_thread": {"value": tok1 / t_one[0], "cores": 1,
                                                   "sample": "first 4 of 128 images, same layers"}}
        print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()
    return 0


def _report_legs(args, torch, lbp, synth, dev, layers, k, bases, peaks, flush_buf, step, world,
                 steps, warmup, ms_per_step, value, launches, clocks, tokens_per_step):
    """Everything rank 0 measures outside the timed region, and the JSON line."""
    es = 2

    def timed(fn, iters=10, flush=False, warm=2):
        """Average device time of fn() in us.  With `flush`, a buffer larger than L2
        is written before every call and only the call itself is inside the events."""
        for _ in range(warm):
            fn()
        if not flush:
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(iters):
                fn()
            b.record()
            torch.cuda.synchronize()
            return a.elapsed_time(b) * 1e3 / iters
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(iters)]
        for a, b in evs:
            flush_buf.zero_()
            a.record()
            fn()
            b.record()
        torch.cuda.synchronize()
        return sum(a.elapsed_time(b) for a, b in evs) * 1e3 / iters

    # ---- per layer and per phase: separate calls that carry phase events ----
    nphase = lbp.lbp_phase_count()
    iters = 10
    phase_us = [[0.0] * nphase for _ in layers]
    evs = [[[torch.cuda.Event(enable_timing=True) for _ in range(nphase)] for _ in layers]
           for _ in range(iters)]
    for it_ in evs:
        for l_ in it_:
            for e in l_:
                e.record()          # materialise the handles
    torch.cuda.synchronize()
    for it in range(iters):
        for li, L in enumerate(layers):
            # boundaries used: 0 start, 1 after the projection, 3 after the products kernel
            lbp.lbp_set_phase_events([e if i in (0, 1, 3) else None for i, e in enumerate(evs[it][li])])
            lbp.lbp_backward(L["x"], L["gy"], L["w"], k, bases, g_x=L["gx"], g_W=L["gw"], ws=L["ws"])
    lbp.lbp_set_phase_events(None)
    torch.cuda.synchronize()
    for it in range(iters):
        for li in range(len(layers)):
            phase_us[li][1] += evs[it][li][0].elapsed_time(evs[it][li][1]) * 1e3 / iters
            phase_us[li][3] += evs[it][li][1].elapsed_time(evs[it][li][3]) * 1e3 / iters

    layer_rows = []
    proj_bytes = proj_us = prod_bytes = prod_flops = prod_us = 0.0
    for li, L in enumerate(layers):
        c = L["case"]
        T, rows = c.tokens, c.blocks * RANK
        roof = _roof_us(peaks, T, c.Cin, c.Cout, rows)
        us = phase_us[li][1] + phase_us[li][3]
        layer_rows.append({
            "layer": c.name, "us": round(us, 2), "tokens_per_s": T / (us * 1e-6),
            "roofline_us": round(roof, 2), "roofline_frac": round(roof / us, 4),
            "phase_us": {"project_x_gy": round(phase_us[li][1], 2),
                         "products_expand": round(phase_us[li][3], 2)},
        })
        proj_bytes += es * T * (c.Cin + c.Cout)                # reads x and g_y once
        proj_us += phase_us[li][1]
        prod_bytes += es * c.Cin * c.Cout + es * T * c.Cin + 4 * c.Cin * c.Cout   # W in; g_x, g_W out
        prod_flops += 4.0 * c.Cin * c.Cout * rows
        prod_us += phase_us[li][3]

    # ---- the library's own full-rank mode (Eq. 2), per layer ----
    for li, L in enumerate(layers):
        full_us = timed(lambda: lbp.lbp_backward_fullrank(L["x"], L["gy"], L["w"], k, g_x=L["gx"],
                                                          g_W=L["gw"], ws=L["ws_full"]), iters=5)
        layer_rows[li]["fullrank_us"] = round(full_us, 2)
        layer_rows[li]["speedup_vs_fullrank"] = round(full_us / layer_rows[li]["us"], 3)
    full_step_us = sum(r_["fullrank_us"] for r_ in layer_rows)

    # ---- the ranks of the configuration (r = 2, 4, 8, 16): whole steps ----
    rank_rows = []
    for rr in (2, 4, 8, 16):
        bases_r = lbp.lbp_select_bases(k, lbp.SEL_PREFIX, rr)
        wss = [lbp.alloc_workspace(L["x"], L["gy"], k, rr) for L in layers]
        us = timed(lambda: step(wss, bases_r), iters=10, warm=3)
        roof = sum(_roof_us(peaks, L["case"].tokens, L["case"].Cin, L["case"].Cout,
                            L["case"].blocks * rr) for L in layers)
        rank_rows.append({"r": rr, "us_per_step": round(us, 2),
                          "tokens_per_s": tokens_per_step / (us * 1e-6),
                          "roofline_us": round(roof, 2), "roofline_frac": round(roof / us, 4),
                          "speedup_vs_fullrank": round(full_step_us / us, 3)})
        del wss

    # ---- the same step captured once and replayed as a CUDA graph ----
    graph_row = None
    try:
        cap = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cap):
            lbp.lbp_backward_batch([L["x"] for L in layers], [L["gy"] for L in layers],
                                   [L["w"] for L in layers], k, bases,
                                   g_xs=[L["gx"] for L in layers], g_Ws=[L["gw"] for L in layers],
                                   wss=[L["ws"] for L in layers])
        us = timed(cap.replay, iters=20, warm=3)
        roof = sum(_roof_us(peaks, L["case"].tokens, L["case"].Cin, L["case"].Cout,
                            L["case"].blocks * RANK) for L in layers)
        graph_row = {"us_per_step": round(us, 2), "roofline_frac": round(roof / us, 4),
                     "tokens_per_s": tokens_per_step / (us * 1e-6)}
        del cap
    except Exception as exc:      # reported, never fatal: the headline is the direct call
        graph_row = {"error": str(exc)[:200]}
    torch.cuda.synchronize()

    # ---- LHE profiling pass (Sec. 3.2) on g_y of every layer ----
    lhe_rows = []
    for L in layers:
        gy = L["gy"]
        Bq, Hq, Wq, Cq = gy.shape
        sws = torch.empty(lbp.lbp_spectrum_workspace_bytes(Bq, Hq, Wq, Cq, k, lbp.LBP_BF16),
                          dtype=torch.uint8, device=dev)
        e_out = torch.empty((k, k), dtype=torch.float64, device=dev)
        us = timed(lambda: lbp.lbp_spectrum(gy, k, out=e_out, ws=sws), iters=5)
        nbytes = gy.numel() * gy.element_size()
        lhe_rows.append({"layer": L["case"].name, "us": round(us, 2), "bytes": nbytes,
                         "gbs": round(nbytes / us / 1e3, 1),
                         "frac_of_hbm_peak": round(nbytes / us / 1e3 / peaks["hbm_gbs"], 4)})
        del sws

    # ---- the other configurations: isolated calls, L2 flushed before each ----
    def device_layer(B, H, W, Cin, Cout, x_kind, seed):
        """Synthetic layer drawn on the device (timing legs only; the parity tests
        use the seeded host generator)."""
        g = torch.Generator(device=dev)
        g.manual_seed(seed)
        z = torch.randn((B, H, W, Cin), generator=g, device=dev, dtype=torch.float32)
        if x_kind == "gelu_normal":
            z = torch.nn.functional.gelu(z)
        elif x_kind == "student_t4":
            chi = torch.randn((4, B, H, W, Cin), generator=g, device=dev).square_().mean(0).sqrt_()
            z = z / chi
        x = z.to(torch.bfloat16)
        gy = (0.01 * torch.randn((B, H, W, Cout), generator=g, device=dev)).to(torch.bfloat16)
        w = (Cin ** -0.5 * torch.randn((Cout, Cin), generator=g, device=dev)).to(torch.bfloat16)
        return x, gy, w

    def time_case(c, ranks):
        x, gy, w = device_layer(c.B, c.H, c.W, c.Cin, c.Cout, c.x_dist[0], 1000 + 16 * c.config + c.case_id)
        gx = torch.empty_like(x)
        gw = torch.empty((c.Cout, c.Cin), dtype=torch.float32, device=dev)
        ws_full = lbp.alloc_workspace(x, gy, c.k, c.k * c.k)
        full_us = timed(lambda: lbp.lbp_backward_fullrank(x, gy, w, c.k, g_x=gx, g_W=gw, ws=ws_full),
                        iters=5, flush=True, warm=1)
        del ws_full
        rows_ = []
        for rr in ranks:
            if rr == c.k * c.k:
                rows_.append({"r": rr, "us": round(full_us, 2), "speedup_vs_fullrank": 1.0,
                              "mode": "full rank (Eq. 2)"})
                continue
            b_ = lbp.lbp_select_bases(c.k, lbp.SEL_PREFIX, rr)
            ws = lbp.alloc_workspace(x, gy, c.k, rr)
            us = timed(lambda: lbp.lbp_backward(x, gy, w, c.k, b_, g_x=gx, g_W=gw, ws=ws),
                       iters=5, flush=True, warm=1)
            st = lbp.lbp_poll_status(ws)
            if st != 0:
                raise RuntimeError(f"device status {st} on {c.name} r={rr}")
            roof = _roof_us(peaks, c.tokens, c.Cin, c.Cout, c.blocks * rr)
            rows_.append({"r": rr, "us": round(us, 2), "tokens_per_s": c.tokens / (us * 1e-6),
                          "roofline_us": round(roof, 2), "roofline_frac": round(roof / us, 4),
                          "speedup_vs_fullrank": round(full_us / us, 3)})
            del ws
        return {"layer": c.name, "k": c.k, "fullrank_us": round(full_us, 2), "ranks": rows_}

    other = {}
    if not args.skip_other_configs:
        other["config2"] = [time_case(c, (8,)) for c in synth.config_cases(2)]
        other["config4"] = [time_case(c, (6,)) for c in synth.config_cases(4)]
        sweep = {4: (1, 2, 4, 8, 12, 16), 8: (1, 2, 4, 8, 12, 16, 21, 32, 48, 64),
                 16: (1, 2, 4, 8, 16, 36, 64, 128, 256)}
        c5 = []
        for c in synth.config_cases(5):
            row = time_case(c, sweep[c.k])
            slower = [q["r"] for q in row["ranks"] if q["speedup_vs_fullrank"] < 1.0]
            row["crossover_r"] = min(slower) if slower else None   # first rank slower than Eq. 2
            c5.append(row)
        other["config5_rank_sweep"] = c5
        other["note"] = ("isolated lbp_backward calls, a 256 MB buffer written before each "
                         "(L2 flush); inputs drawn on the device with the configurations' "
                         "shapes and distributions; speed-up against lbp_backward_fullrank "
                         "(exact BP, Eq. 2) on the same layer")

    # ---- roofline of the two kernels of a step ----
    # The timed region runs the batch call only; the per-kernel times come from the
    # phase-event leg above (separate calls, which is what makes a kernel's own
    # duration observable), the same kernels on the same buffers.
    all_us = proj_us + prod_us
    region_s = ms_per_step * 1e-3 * steps
    burst = region_s < 1.0          # short timed region at full clocks: the burst peak applies
    bf16_peak = peaks["bf16_tflops"] if burst else peaks["bf16_tflops_sustained"]
    proj_ach = proj_bytes / (proj_us * 1e-6) / 1e9
    r_proj = {"bound": "hbm", "kernel": "wht_project_umma_kernel", "achieved": round(proj_ach, 1),
              "peak": peaks["hbm_gbs"], "unit": "GB/s", "frac": round(proj_ach / peaks["hbm_gbs"], 4),
              "traffic": NCU_TRAFFIC_PER_STEP["wht_project_umma_kernel"],
              "algorithmic_bytes": int(proj_bytes), "launches_per_step": len(layers),
              "us_per_step": round(proj_us, 2), "peak_source": peaks["source"],
              "share_of_step": round(proj_us / all_us, 4)}
    t_b = prod_bytes / (peaks["hbm_gbs"] * 1e9)
    t_f = prod_flops / (bf16_peak * 1e12)
    if t_f >= t_b:
        ach = prod_flops / (prod_us * 1e-6) / 1e12
        r_prod = {"bound": "tensor", "achieved": round(ach, 1), "peak": bf16_peak, "unit": "TFLOP/s",
                  "frac": round(ach / bf16_peak, 4),
                  "peak_kind": "burst" if burst else "sustained"}
    else:
        ach = prod_bytes / (prod_us * 1e-6) / 1e9
        r_prod = {"bound": "hbm", "achieved": round(ach, 1), "peak": peaks["hbm_gbs"],
                  "unit": "GB/s", "frac": round(ach / peaks["hbm_gbs"], 4)}
    r_prod.update({"kernel": "lbp_products_kernel",
                   "traffic": NCU_TRAFFIC_PER_STEP["lbp_products_kernel"],
                   "algorithmic_bytes": int(prod_bytes), "algorithmic_flops": prod_flops,
                   "launches_per_step": len(layers), "us_per_step": round(prod_us, 2),
                   "peak_source": peaks["source"], "share_of_step": round(prod_us / all_us, 4)})
    roofline, roofline_other = (r_proj, r_prod) if proj_us >= prod_us else (r_prod, r_proj)
    whole_roof_us = sum(r["roofline_us"] for r in layer_rows)
    sm_mhz = clocks.get("sm_mhz") if clocks else None
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": steps,
        "warmup": warmup, "ms_per_step": ms_per_step, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": WORKLOAD, "tokens_per_step_per_gpu": tokens_per_step,
                   "l2": "inputs larger than L2 (>= 150 MB per layer, 1.2 GB per step)",
                   "multi_gpu": "batch sharded per rank; g_W all-reduced (NCCL) on a side stream "
                                "behind the kernels of the following layers when N > 1"},
        "roofline": roofline,
        "roofline_other": roofline_other,
        "path_roofline": {"roofline_us": round(whole_roof_us, 2),
                          "achieved_us": round(ms_per_step * 1e3, 2),
                          "frac": round(whole_roof_us / (ms_per_step * 1e3), 4),
                          "us_times_sm_mhz": (round(ms_per_step * 1e3 * sm_mhz, 1)
                                              if sm_mhz else None),
                          "sum_of_isolated_layer_us": round(sum(r["us"] for r in layer_rows), 2),
                          "note": "sum over the four layers of max(algorithmic bytes / HBM "
                                  "peak, 4 Cin Cout M_hat / bf16 burst peak), of " + peaks["source"] +
                                  " peaks, against the time of a step of the timed region (one "
                                  "lbp_backward_batch call); per-layer, per-phase and per-kernel "
                                  "figures come from a leg of separate lbp_backward calls with "
                                  "phase events, outside the timed region"},
        "layers": layer_rows,
        "rank_sweep": rank_rows,
        "graph_replay": graph_row,
        "lhe_spectrum": lhe_rows,
        "other_configs": other,
        "gpu_launches": int(launches),
        "clocks": clocks,
    }
    return line


def _spawn_ranks(args) -> int:
    """`python bench.py --gpus N` without a launcher: start the N ranks here."""
    import socket
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1",
           f"--nproc-per-node={args.gpus}", "--master-addr", "127.0.0.1", "--master-port", str(port),
           os.path.abspath(__file__), "--gpus", str(args.gpus), "--steps", str(args.steps),
           "--warmup", str(args.warmup), "--impl", args.impl]
    if args.skip_other_configs:
        cmd.append("--skip-other-configs")
    return subprocess.call(cmd)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--skip-other-configs", action="store_true",
                    help="leave out the legs on configurations 2, 4 and 5")
    ap.add_argument("--profile-layer", type=int, default=None,
                    help="run one layer of --profile-config a few times and exit")
    ap.add_argument("--profile-config", type=int, default=3)
    ap.add_argument("--profile-rank", type=int, default=8)
    ap.add_argument("--profile-batch", type=int, default=None)
    ap.add_argument("--profile-fullrank", action="store_true")
    ap.add_argument("--iters", type=int, default=3)
    args = ap.parse_args()
    if args.profile_layer is not None:
        return run_profile(args)
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        return _spawn_ranks(args)
    if args.impl == "reference":
        return run_reference(args)
    return run_gpu(args)


if __name__ == "__main__":
    sys.exit(main())
