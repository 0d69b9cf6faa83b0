"""Benchmark of the PermuQuant quantized-linear hot path on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

One step = one runtime pass of the FLUX-like QKV projection (X bf16 4608 x 3072, W 3072 x 9216):
NVFP4 activation quantize followed by the W4A4 block-scaled GEMM, bf16 out -- the configuration the
headline metric (W4A4 GEMM TFLOP/s including the activation quantize) is quoted on.  The layer is
first calibrated on the device (statistics, Eq. 9 candidates, Eq. 3 errors, Eq. 10, permuted weight
quantization); those offline kernels and the other streaming kernels are timed separately and
reported under "stages" in GB/s.  Everything runs through the C ABI (paper_2605_09503_b200.binding).

`--impl reference` times the CPU oracle (oracle/) on a bounded row sample of the same workload.
With N > 1 every rank runs the same layer on its own token shard (weak scaling, no data-path
collective); times are taken on the device and reduced with MAX over ranks.  Under torchrun the
ranks are the launcher's; a plain `python bench.py --gpus N` starts N ranks itself
(torch.distributed.run on 127.0.0.1) and `n_gpus` in the output is the number of ranks that ran.
"""
import argparse
import json
import os
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

WORKLOAD = "qkv"
METRIC = "w4a4_nvfp4_linear_tflops_incl_act_quant"
NSETS = 4          # buffer sets the timed loop rotates over (each ~137 MB; L2 is 126 MB)
REPEATS = 5        # the headline loop is timed this many times; the median is reported
REPEAT_PAUSE_S = 0.25
XROT = 10          # activation buffers the stand-alone streaming loops rotate over (283 MB)
ORACLE_ROWS_MAX = 2048   # largest row sample of the workload the oracle legs use
FP4_OVER_BF16 = 4.0  # nominal dense tensor ratio (9 vs 2.25 PFLOP/s)
GEMM_DRAM_BYTES_PER_LAUNCH = 53.60e6   # ncu, 23.92 MB read + 29.68 MB written per launch of the bench workload (mean of two launches)
FALLBACK_PEAKS = {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0}


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return {k: float(p[k]) for k in FALLBACK_PEAKS if k in p} | {"source": "measured"}
    return dict(FALLBACK_PEAKS) | {"source": "fallback"}


# ------------------------------------------------------------------------------------ clocks
class ClockSampler:
    """Reads (never sets) SM clock and throttle reasons through NVML while the timed region runs."""

    REASONS = {0x4: "sw_power_cap", 0x8: "hw_slowdown", 0x20: "sw_thermal_slowdown",
               0x40: "hw_thermal_slowdown", 0x80: "hw_power_brake_slowdown"}

    def __init__(self, index):
        self.samples, self.reasons, self.max_mhz = [], set(), None
        self._stop = threading.Event()
        self._thread = None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            try:
                import torch
                uuid = "GPU-" + str(torch.cuda.get_device_properties(index).uuid)
                self.h = pynvml.nvmlDeviceGetHandleByUUID(uuid.encode())
            except Exception:
                self.h = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = int(pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM))
        except Exception:
            self.nv = None

    def sample(self):
        if self.nv is None:
            return
        try:
            self.samples.append(int(self.nv.nvmlDeviceGetClockInfo(self.h, self.nv.NVML_CLOCK_SM)))
            mask = int(self.nv.nvmlDeviceGetCurrentClocksEventReasons(self.h))
            for bit, name in self.REASONS.items():
                if mask & bit:
                    self.reasons.add(name)
        except Exception:
            pass

    def _run(self):
        while not self._stop.is_set():
            self.sample()
            self._stop.wait(0.02)

    def start(self):
        self._stop.clear()
        self._thread = threading.Thread(target=self._run, daemon=True)
        self._thread.start()

    def stop(self):
        self._stop.set()
        if self._thread:
            self._thread.join()

    def summary(self):
        s = sorted(self.samples)
        return {"sm_mhz": (s[len(s) // 2] if s else None), "sm_max_mhz": self.max_mhz,
                "reasons": sorted(self.reasons), "samples": len(s)}


# ------------------------------------------------------------------------------------ oracle arm
def oracle_sample_run(rows):
    """The oracle on `rows` token rows of the workload: NVFP4 quantize of those rows, then the fp64
    dequantized GEMM against the whole quantized weight.  Returns seconds (weight quantization, an
    offline step, is outside the timed part)."""
    import numpy as np
    from oracle import pq_oracle as O
    from paper_2605_09503_b200 import inputs

    cfg = inputs.CONFIGS[WORKLOAD]
    if not hasattr(oracle_sample_run, "cache"):
        w = inputs.bits(inputs.weight(cfg, 0))
        ts_w = O.tensor_scale(O.calib_stats(w)[1])
        wq, sfw = O.quant_nvfp4(w, ts_w)
        x = inputs.bits(inputs.activations(cfg, 0, 1000, rows=ORACLE_ROWS_MAX))
        ts_x = O.tensor_scale(O.calib_stats(x)[1])
        oracle_sample_run.cache = (wq, sfw, ts_w, x, ts_x)
    wq, sfw, ts_w, x, ts_x = oracle_sample_run.cache
    xs = np.ascontiguousarray(x[:rows])
    t0 = time.perf_counter()
    xq, sfx = O.quant_nvfp4(xs, ts_x)
    O.gemm_ref(xq, sfx, ts_x, wq, sfw, ts_w)
    return time.perf_counter() - t0


def oracle_threads():
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def oracle_rows_for(seconds, cap):
    """Rows of the sample that take the oracle about `seconds` on this host (probe, then scale)."""
    oracle_sample_run(8)                                   # builds the cache, warms the library
    per_row = oracle_sample_run(16) / 16.0
    return int(max(8, min(cap, seconds / max(per_row, 1e-6))))


def cpu_baseline(target_s=15.0):
    """Oracle throughput on a row sample sized for roughly `target_s` seconds of CPU work."""
    from paper_2605_09503_b200 import inputs
    cfg = inputs.CONFIGS[WORKLOAD]
    rows = oracle_rows_for(target_s, ORACLE_ROWS_MAX)
    t = oracle_sample_run(rows)
    flops = 2.0 * rows * cfg.N * cfg.K
    return {"value": flops / t / 1e12, "unit": "TFLOP/s", "cores": oracle_threads(), "kind": "oracle",
            "sample": f"{rows} of {cfg.M} token rows x all {cfg.N} outputs, K={cfg.K}: oracle NVFP4 quantize "
                      f"+ fp64 dequantized GEMM, {t:.2f} s"}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from paper_2605_09503_b200 import inputs
    cfg = inputs.CONFIGS[WORKLOAD]
    budget = 150.0 / max(1, args.steps + args.warmup)               # whole run within a few minutes
    rows = oracle_rows_for(budget, ORACLE_ROWS_MAX)
    for _ in range(args.warmup):
        oracle_sample_run(rows)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle_sample_run(rows)
    dt = (time.perf_counter() - t0) / max(1, args.steps)
    value = 2.0 * rows * cfg.N * cfg.K / dt / 1e12
    sample = f"{rows} of {cfg.M} token rows x all {cfg.N} outputs per step"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": "TFLOP/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_name(cfg), "sample": sample},
        "cpu_baseline": {"value": value, "unit": "TFLOP/s", "cores": oracle_threads(), "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": "TFLOP/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def workload_name(cfg):
    return (f"FLUX-like attention QKV projection: X bf16 {cfg.M}x{cfg.K}, W {cfg.K}x{cfg.N}, NVFP4 W4A4, "
            f"group 16, fp32 accumulate, bf16 out")


# ------------------------------------------------------------------------------------ GPU arm
def timed_loop(torch, fn, iters, warmup):
    """Average milliseconds per call of fn(i), CUDA events on the current stream."""
    for i in range(warmup):
        fn(i)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for i in range(iters):
        fn(i)
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / iters


def graph_loop(torch, fn, iters, warmup=3, replays=3):
    """Average milliseconds per call of fn(i) with `iters` calls captured in one CUDA graph: the
    replay keeps the launches back to back, so short kernels are not timed at the host's launch rate."""
    for i in range(warmup):
        fn(i)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i in range(iters):
            fn(i)
    graph.replay()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(replays):
        graph.replay()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / (iters * replays)


def burst_loop(torch, fn, iters, repeats=5, pause_s=0.25):
    """graph_loop in the regime of the headline loop: `iters` calls in one CUDA graph, replayed once per
    repeat after an idle pause and three warm-up calls; median milliseconds per call.  A kernel timed this
    way has not been running long enough for the board's power cap to lower the clock, which is the
    condition the burst peak was measured under."""
    for i in range(3):
        fn(i)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i in range(iters):
            fn(i)
    graph.replay()
    torch.cuda.synchronize()
    times = []
    for _ in range(repeats):
        time.sleep(pause_s)
        for i in range(3):
            fn(i)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / iters)
    return sorted(times)[len(times) // 2]


def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2605_09503_b200 import binding as B
    from paper_2605_09503_b200 import build as lib_build
    from paper_2605_09503_b200 import inputs, pipeline

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: there is no CPU fallback")
    torch.cuda.set_device(local)
    dev = f"cuda:{local}"
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device(dev))
    if not os.path.exists(B.LIB_PATH):
        if local == 0:
            lib_build.build()
        if world > 1:
            dist.barrier()
    B.lib()

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    def max_over_ranks(ms):
        if world == 1:
            return ms
        t = torch.tensor([ms], dtype=torch.float64, device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        return float(t.item())

    peaks = load_peaks()
    cfg = inputs.CONFIGS[WORKLOAD]
    M, K, N = cfg.M, cfg.K, cfg.N
    layer_seed = rank                       # every rank: same shapes, its own token shard

    # ---- offline: calibrate the layer on the device (two calibration batches keep set-up short)
    calib = [inputs.activations(cfg, layer_seed, b).to(dev) for b in range(2)]
    Wt = inputs.weight(cfg, 0).to(dev)
    cal = pipeline.calibrate(calib, Wt)
    torch.cuda.synchronize()
    order = cal.chosen_perm().cpu()

    # ---- runtime buffers: NSETS complete sets so consecutive steps never hit L2-resident data
    xs_host = [inputs.activations(cfg, layer_seed, 1000 + i)[:, order].contiguous() for i in range(XROT)]
    xs = [x.to(dev) for x in xs_host]
    layers = []
    for i in range(NSETS):
        wq, sfw = (cal.wq, cal.sfw) if i == 0 else (cal.wq.clone(), cal.sfw.clone())
        layers.append(pipeline.QuantLinear(wq, sfw, cal.ts_w, cal.ts_x, M))
    ys = [torch.empty(M, N, dtype=torch.bfloat16, device=dev) for _ in range(NSETS)]
    set_bytes = M * K * 2 + M * K // 2 + B.sf_bytes(M, K, 1) + N * K // 2 + B.sf_bytes(N, K, 1) + M * N * 2

    def step(i):
        j = i % NSETS
        layers[j](xs[j], ys[j])

    def gemm_only(i):
        L = layers[i % NSETS]
        B.pq_gemm_w4a4(L.xq, L.sfx, L.ts_x, L.wq, L.sfw, L.ts_w, ys[i % NSETS], L.ws)

    xq_rot = [torch.empty(M, K // 2, dtype=torch.uint8, device=dev) for _ in range(XROT)]
    sfx_rot = [torch.empty(B.sf_bytes(M, K, 1), dtype=torch.uint8, device=dev) for _ in range(XROT)]

    def quant_only(i):
        j = i % XROT
        B.pq_quant_act_nvfp4(xs[j], cal.ts_x, xq_rot[j], sfx_rot[j], B.PQ_SF_TCGEN05)

    # ---- headline: the K-step loop of quantize + GEMM, timed REPEATS times (each repeat: exactly K steps
    # between two events, a barrier and a synchronize on both sides, max over ranks); the value is the
    # median repeat, the spread is reported beside it
    sampler = ClockSampler(local)
    for i in range(max(args.warmup, 3)):
        step(i)
    # The K steps of a repeat go out as ONE CUDA-graph launch (captured here, through the same public call):
    # the timed region then holds exactly the K steps' kernels back to back, as a serving loop would run them,
    # and not the host's start-up latency of the first launch after the synchronize, which weighs on a short
    # loop (K = 20: about 1 us per step).  Very long loops are launched directly.
    step_graph = None
    if args.steps <= 2000:
        torch.cuda.synchronize()
        step_graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(step_graph):
            for i in range(args.steps):
                step(i)
        torch.cuda.synchronize()
    repeats = []
    sampler.start()
    for _ in range(REPEATS):
        # a pause before every repeat: each one then starts from the state the first one starts from (the
        # 1 kW power cap engages some tens of milliseconds into a dense loop), i.e. all repeats are
        # burst-regime numbers like the burst peak they are compared with; the capped regime is measured
        # separately below (linear_incl_quant_sustained, against the sustained peak)
        barrier()
        time.sleep(REPEAT_PAUSE_S)
        for i in range(3):
            step(i)
        barrier()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        if step_graph is not None:
            step_graph.replay()
        else:
            for i in range(args.steps):
                step(i)
        b.record()
        sampler.sample()                   # the queue is still draining here
        barrier()
        repeats.append(max_over_ranks(a.elapsed_time(b) / args.steps))
    sampler.stop()
    ms_step = sorted(repeats)[len(repeats) // 2]
    for L in layers:
        L.check()
    flops = 2.0 * M * N * K
    value = world * flops / (ms_step * 1e-3) / 1e12

    # ---- the two kernels of the step on their own (same launch configuration, same rotation), in the same
    # regime as the headline loop: short graph launches with idle pauses, before the long loop below heats the board
    # (200 launches per graph whatever --steps says, so that the graph's own start-up does not weigh on a
    # 8 us kernel; fewer only in the very short runs profiler captures use)
    iters = 200 if args.steps >= 5 else 20
    ms_gemm = burst_loop(torch, gemm_only, iters, REPEATS, REPEAT_PAUSE_S)
    ms_quant = burst_loop(torch, quant_only, iters, REPEATS, REPEAT_PAUSE_S)

    # ---- the same loop held for about 1.5 s: the 1 kW power cap engages after a few hundred steps and
    # the SM clock settles near 1.6 GHz; this figure goes with the sustained peak, the headline (a few
    # hundred steps unless --steps says otherwise) with the burst peak
    # (about 1.5 s of steps in an ordinary run, about 0.5 s when --steps is small, none under --steps < 5,
    # which is how profiler captures are run)
    sustained_steps = 20000 if args.steps >= 100 else (7000 if args.steps >= 5 else 0)
    ms_sustained = None
    if sustained_steps:
        for i in range(3):
            step(i)
        barrier()
        a2, b2 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a2.record()
        for i in range(sustained_steps):
            step(i)
        b2.record()
        barrier()
        ms_sustained = max_over_ranks(a2.elapsed_time(b2) / sustained_steps)

    # ---- the GEMM again right behind the long loop: the power-capped figure that goes with the sustained peak
    ms_gemm_capped = graph_loop(torch, gemm_only, iters) if sustained_steps else None
    fp4_peak = peaks["bf16_tflops"] * FP4_OVER_BF16
    gemm_tflops = flops / (ms_gemm * 1e-3) / 1e12
    quant_bytes = M * K * 2 + M * K // 2 + M * K // 16
    roofline = {"kernel": "gemm_w4a4_kernel", "bound": "tensor", "achieved": gemm_tflops, "peak": fp4_peak,
                "unit": "TFLOP/s", "frac": gemm_tflops / fp4_peak, "traffic": GEMM_DRAM_BYTES_PER_LAUNCH,
                "traffic_source": "dram__bytes_read.sum + dram__bytes_write.sum of one ncu capture of this kernel on this "
                                  "workload (profiles/gemm_w4a4_kernel_qkv_4608x3072x9216.md); algorithmic bytes 108.8e6",
                "peak_source": f"{peaks['source']} bf16 burst {peaks['bf16_tflops']} TFLOP/s x {FP4_OVER_BF16:g} "
                               f"(nominal fp4:bf16 ratio)",
                "regime": "burst: CUDA-graph launches of a few milliseconds with idle pauses, like the measured peak",
                "after_sustained_loop": None if ms_gemm_capped is None else {
                    "ms_per_launch": ms_gemm_capped, "achieved": flops / (ms_gemm_capped * 1e-3) / 1e12,
                    "frac_of_sustained_peak": flops / (ms_gemm_capped * 1e-3) / 1e12
                                              / (peaks["bf16_tflops_sustained"] * FP4_OVER_BF16)},
                "frac_of_nominal_9000": gemm_tflops / 9000.0,
                "ms_per_launch": ms_gemm, "flops_per_launch": flops}
    quant_gbs = quant_bytes / (ms_quant * 1e-3) / 1e9
    # yardstick for a kernel of this size: a plain device copy moving the same number of bytes (half read, half
    # written), timed the same way; the peak the fractions use is a copy of 4 GB, where launch, ramp and tail vanish
    copy_src = [torch.empty(quant_bytes // 2, dtype=torch.uint8, device=dev) for _ in range(XROT)]
    copy_dst = [torch.empty(quant_bytes // 2, dtype=torch.uint8, device=dev) for _ in range(XROT)]
    ms_copy = burst_loop(torch, lambda i: copy_dst[i % XROT].copy_(copy_src[i % XROT]), iters, REPEATS, REPEAT_PAUSE_S)
    del copy_src, copy_dst
    stages = {"quant_act_nvfp4": {"ms": ms_quant, "GB/s": quant_gbs, "frac_hbm": quant_gbs / peaks["hbm_gbs"],
                                  "frac_hbm_nominal_8000": quant_gbs / 8000.0, "bytes": quant_bytes,
                                  "plain_copy_of_the_same_bytes": {"ms": ms_copy, "GB/s": quant_bytes / ms_copy / 1e6,
                                                                   "frac_hbm": quant_bytes / ms_copy / 1e6 / peaks["hbm_gbs"]}},
              "gemm_w4a4": {"ms": ms_gemm, "TFLOP/s": gemm_tflops},
              "linear_incl_quant": {"ms": ms_step, "TFLOP/s": flops / (ms_step * 1e-3) / 1e12,
                                    "frac_fp4_peak": flops / (ms_step * 1e-3) / 1e12 / fp4_peak},
              "linear_incl_quant_sustained": None if ms_sustained is None else {
                  "ms": ms_sustained, "steps": sustained_steps, "TFLOP/s": flops / (ms_sustained * 1e-3) / 1e12,
                  "frac_fp4_sustained_peak": flops / (ms_sustained * 1e-3) / 1e12
                                             / (peaks["bf16_tflops_sustained"] * FP4_OVER_BF16)}}

    # ---- the step with the quantizer overlapped: independent batches through one layer
    # (pq_linear_w4a4_batched: quantizer of the next batches beside the GEMM of the current one)
    def batched_ms(layer, inputs_, outputs_, n):
        Xs = [inputs_[i % len(inputs_)] for i in range(n)]
        Ys = [outputs_[i % len(outputs_)] for i in range(n)]
        layer.forward_batches(Xs, Ys)                      # creates the extra intermediates, warms up
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        layer.forward_batches(Xs, Ys)
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / n

    nb = max(20, min(args.steps, 200))
    ms_b = batched_ms(layers[0], xs, ys, nb)
    stages["linear_batched_quant_overlapped"] = {
        "ms": ms_b, "TFLOP/s": flops / (ms_b * 1e-3) / 1e12, "frac_fp4_peak": flops / (ms_b * 1e-3) / 1e12 / fp4_peak,
        "batches_per_call": nb, "note": "one weight for all batches (stays in L2); X rotates over 283 MB"}

    # ---- the long-K workload (MLP down-projection, X 4608 x 12288, W 12288 x 3072): the same three numbers
    if rank == 0:
        cfg3 = inputs.CONFIGS["mlp_down"]
        M3, K3, N3 = cfg3.M, cfg3.K, cfg3.N
        x3 = [inputs.activations(cfg3, 0, 1000 + i).to(dev) for i in range(3)]          # 3 x 113 MB
        w3 = inputs.weight(cfg3, 0).to(dev)
        amax3 = torch.stack([x.abs().max() for x in x3]).max().float().reshape(1)
        ts_x3 = (amax3 / 2688.0).contiguous()
        wq3 = torch.empty(N3, K3 // 2, dtype=torch.uint8, device=dev)
        sfw3 = torch.empty(B.sf_bytes(N3, K3, 1), dtype=torch.uint8, device=dev)
        ts_w3 = torch.empty(1, dtype=torch.float32, device=dev)
        B.pq_quant_weight(w3, None, None, wq3, sfw3, B.PQ_SF_TCGEN05, ts_w3, B.workspace(B.OP_QUANT_WEIGHT, N3, K3))
        L3 = pipeline.QuantLinear(wq3, sfw3, ts_w3, ts_x3, M3)
        y3 = [torch.empty(M3, N3, dtype=torch.bfloat16, device=dev) for _ in range(3)]
        f3 = 2.0 * M3 * N3 * K3
        it3 = max(10, min(args.steps, 60))
        L3(x3[0], y3[0])
        ms_g3 = graph_loop(torch, lambda i: B.pq_gemm_w4a4(L3.xq, L3.sfx, L3.ts_x, L3.wq, L3.sfw, L3.ts_w, y3[i % 3], L3.ws), it3)
        ms_q3 = graph_loop(torch, lambda i: B.pq_quant_act_nvfp4(x3[i % 3], ts_x3, L3.xq, L3.sfx, B.PQ_SF_TCGEN05), it3)
        ms_l3 = graph_loop(torch, lambda i: L3(x3[i % 3], y3[i % 3]), it3)
        ms_b3 = batched_ms(L3, x3, y3, it3)
        L3.check()
        qb3 = M3 * K3 * 2 + M3 * K3 // 2 + M3 * K3 // 16
        stages["mlp_down_4608x12288x3072"] = {
            "gemm_alone": {"ms": ms_g3, "TFLOP/s": f3 / ms_g3 / 1e9, "frac_fp4_peak": f3 / ms_g3 / 1e9 / fp4_peak},
            "quant_act_nvfp4": {"ms": ms_q3, "GB/s": qb3 / ms_q3 / 1e6, "frac_hbm": qb3 / ms_q3 / 1e6 / peaks["hbm_gbs"]},
            "linear_serial": {"ms": ms_l3, "TFLOP/s": f3 / ms_l3 / 1e9, "frac_fp4_peak": f3 / ms_l3 / 1e9 / fp4_peak},
            "linear_batched_quant_overlapped": {"ms": ms_b3, "TFLOP/s": f3 / ms_b3 / 1e9,
                                                "frac_fp4_peak": f3 / ms_b3 / 1e9 / fp4_peak}}
        del x3, w3, y3, L3

    # ---- offline / streaming kernels, each against HBM bandwidth (algorithmic bytes), on one
    # calibration batch (M rows) and on the 8 calibration batches of the workload stacked into one
    # call (8 M rows), where launch ramp and tail weigh less
    if rank == 0:
        it = 50 if args.steps >= 5 else 10
        hbm = peaks["hbm_gbs"]

        def stage(name, ms, nbytes, **extra):
            gbs = nbytes / ms / 1e6
            stages[name] = {"ms": ms, "GB/s": gbs, "frac_hbm": gbs / hbm, "frac_hbm_nominal_8000": gbs / 8000.0,
                            "bytes": nbytes, **extra}

        big = [torch.cat(xs[0:8]), torch.cat(xs[2:10])]          # 2 x 226 MB
        for tag, src, rows in (("", xs, M), ("_8batches", big, 8 * M)):
            nsrc = len(src)
            S = torch.zeros(K, dtype=torch.float64, device=dev)
            A = torch.zeros(K, dtype=torch.float32, device=dev)
            ws_stats = B.workspace(B.OP_CALIB_STATS, rows, K)
            stage("calib_stats" + tag, graph_loop(torch, lambda i: B.pq_calib_stats(src[i % nsrc], S, A, ws_stats), it),
                  rows * K * 2)
            ws_err = B.workspace(B.OP_GROUP_ERROR, rows, K, 0, 6)
            e1 = torch.zeros(1, K // 16, dtype=torch.float64, device=dev)
            stage("group_error_nvfp4_P1" + tag,
                  graph_loop(torch, lambda i: B.pq_group_error(src[i % nsrc], pipeline.NVFP4, cal.ts_x, None, e1, ws_err),
                             it), rows * K * 2)
            for bits, group in ((3, 64), (4, 128)):
                eg = torch.zeros(1, K // group, dtype=torch.float64, device=dev)
                stage(f"group_error_int{bits}_g{group}_P1" + tag,
                      graph_loop(torch, lambda i: B.pq_group_error(src[i % nsrc], (B.KIND_INT, bits, group), None, None,
                                                                   eg, ws_err), it), rows * K * 2)
            xq_b = torch.empty(rows, K // 2, dtype=torch.uint8, device=dev)
            sfx_b = torch.empty(B.sf_bytes(rows, K, 1), dtype=torch.uint8, device=dev)
            if tag:
                stage("quant_act_nvfp4" + tag,
                      graph_loop(torch, lambda i: B.pq_quant_act_nvfp4(src[i % nsrc], cal.ts_x, xq_b, sfx_b,
                                                                       B.PQ_SF_TCGEN05), it),
                      rows * K * 2 + rows * K // 2 + rows * K // 16)
            fq = torch.empty(rows, K, dtype=torch.bfloat16, device=dev)
            stage("fakequant_int4_g64" + tag,
                  graph_loop(torch, lambda i: B.pq_fakequant_int(src[i % nsrc], (B.KIND_INT, 4, 64), None, fq), it),
                  rows * K * 4)
            del fq, xq_b, sfx_b
        del big
        # fused producer: adaptive LayerNorm / RMSNorm + reordering + quantizer (reads 2 B, writes 0.5625 B per element)
        av = 0.2 * torch.randn(K, device=dev)
        bv = torch.randn(K, device=dev)
        order = cal.perms[5].contiguous()
        for kind, name in ((B.NORM_ADALN, "norm_quant_adaln"), (B.NORM_RMS, "norm_quant_rms")):
            stage(name, graph_loop(torch, lambda i: B.pq_norm_quant_nvfp4(xs[i % XROT], kind, av, bv, 1e-6, order, cal.ts_x,
                                                                          xq_rot[i % XROT], sfx_rot[i % XROT],
                                                                          B.PQ_SF_TCGEN05), it),
                  quant_bytes, bound="instruction issue / latency (one wave of 16 warps per SM; 16-21 instructions per element)")
            # the same producer when the channels arrive already in output order (reordering absorbed upstream):
            # no gather, a row never leaves the registers
            stage(name + "_preordered",
                  graph_loop(torch, lambda i: B.pq_norm_quant_nvfp4(xs[i % XROT], kind, av, bv, 1e-6, None, cal.ts_x,
                                                                    xq_rot[i % XROT], sfx_rot[i % XROT], B.PQ_SF_TCGEN05), it),
                  quant_bytes, bound="instruction issue (about 15 instructions per element), not the gather")
        # PermuQuant-H producer: Hadamard transform + reordering + quantizer (same bytes as the plain quantizer)
        stage("hadamard_quant", graph_loop(torch, lambda i: B.pq_hadamard_quant_nvfp4(xs[i % XROT], order, cal.ts_x,
                                                                                      xq_rot[i % XROT], sfx_rot[i % XROT],
                                                                                      B.PQ_SF_TCGEN05), it),
              quant_bytes, bound="fp32 additions (20 per element) and shared-memory passes, not HBM")
        ws_err = B.workspace(B.OP_GROUP_ERROR, M, K, 0, 6)
        e6 = torch.zeros(6, K // 16, dtype=torch.float64, device=dev)
        ms = graph_loop(torch, lambda i: B.pq_group_error(xs[i % XROT], pipeline.NVFP4, cal.ts_x, cal.perms, e6, ws_err),
                        max(5, it // 4))
        stages["group_error_nvfp4_P6"] = {"ms": ms, "GB/s_effective": 6 * M * K * 2 / ms / 1e6, "bound": "alu"}
        wq2 = torch.empty_like(cal.wq)
        sfw2 = torch.empty_like(cal.sfw)
        tsw2 = torch.empty(1, dtype=torch.float32, device=dev)
        ws_qw = B.workspace(B.OP_QUANT_WEIGHT, N, K)
        stage("quant_weight", graph_loop(torch, lambda i: B.pq_quant_weight(Wt, cal.perms, cal.select, wq2, sfw2, 1, tsw2,
                                                                            ws_qw), max(5, it // 4)),
              2 * N * K * 2 + N * K // 2 + N * K // 16, note="two reads of W (absmax, then gather + quantize, four rows per block)")

        # output-side calibration error: fp32 reference and bf16 layer output of one batch (6 B per element)
        yrefs = [torch.randn(M, N, device=dev) for _ in range(2)]
        yqs = [(r * 1.01).to(torch.bfloat16) for r in yrefs]
        eo = torch.zeros(N, dtype=torch.float64, device=dev)
        ws_oe = B.workspace(B.OP_OUTPUT_ERROR, M, N)
        stage("output_error", graph_loop(torch, lambda i: B.pq_output_error(yrefs[i % 2], yqs[i % 2], eo, ws_oe), it),
              M * N * 6)
        stage("quant_act_nvfp4_candidate_order",
              graph_loop(torch, lambda i: B.pq_quant_act_nvfp4_perm(xs[i % XROT], order, cal.ts_x, xq_rot[i % XROT],
                                                                    sfx_rot[i % XROT], B.PQ_SF_TCGEN05), it),
              quant_bytes, note="calibration-time gather quantizer: four rows per block share indices and gathers")
        del yrefs, yqs

    # ---- end to end: host tensors in, host tensor out, through the C ABI
    xh = [x.pin_memory() for x in xs_host[:2]]
    yh = [torch.empty(M, N, dtype=torch.bfloat16).pin_memory() for _ in range(2)]
    L0 = layers[0]

    def e2e_step(i):
        B.pq_linear_w4a4_host(xh[i % 2], L0.ts_x, xs[0], L0.xq, L0.sfx, L0.wq, L0.sfw, L0.ts_w, ys[0], yh[i % 2],
                              L0.ws)

    e2e_iters = max(3, min(args.steps, 100))
    for i in range(3):
        e2e_step(i)
    barrier()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for i in range(e2e_iters):
        e2e_step(i)
    b.record()
    barrier()
    ms_e2e = max_over_ranks(a.elapsed_time(b) / e2e_iters)
    # the same with the batches of the loop handed over in one call: uploads, kernels and downloads of
    # neighbouring batches overlap (every batch is still copied in and out inside the timed region)
    xd2 = [xs[0], xs[1]]
    yd2 = [ys[0], ys[1]]
    Xh = [xh[i % 2] for i in range(e2e_iters)]
    Yh = [yh[i % 2] for i in range(e2e_iters)]

    def e2e_pipelined():
        B.pq_linear_w4a4_host_batched(Xh, L0.ts_x, xd2, yd2, L0.xq, L0.sfx, L0.wq, L0.sfw, L0.ts_w, Yh, L0.ws)

    e2e_pipelined()
    barrier()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    e2e_pipelined()
    b.record()
    barrier()
    ms_e2e_pipe = max_over_ranks(a.elapsed_time(b) / e2e_iters)
    L0.check()
    e2e = {"value": world * flops / (ms_e2e_pipe * 1e-3) / 1e12, "unit": "TFLOP/s", "h2d_bytes_per_step": M * K * 2,
           "d2h_bytes_per_step": M * N * 2, "ms_per_step": ms_e2e_pipe, "steps": e2e_iters,
           "call": "pq_linear_w4a4_host_batched (copies of neighbouring batches overlap)",
           "one_batch_per_call": {"value": world * flops / (ms_e2e * 1e-3) / 1e12, "ms_per_step": ms_e2e,
                                  "call": "pq_linear_w4a4_host"}}

    if rank == 0:
        out = {
            "metric": METRIC, "value": value, "unit": "TFLOP/s", "n_gpus": world, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "fp4_e2m1 x ue4m3 block scales, fp32 accumulate", "data": "synthetic",
            "config": {"workload": workload_name(cfg), "tokens_per_gpu": M,
                       "l2": f"timed loop rotates over {NSETS} complete buffer sets ({NSETS * set_bytes / 1e6:.0f} MB "
                             f"> 126 MB L2); stand-alone kernel loops are CUDA-graph replays rotating over {XROT} "
                             f"inputs of 28 MB or 2 of 226 MB",
                       "timing": f"value = median of {REPEATS} repeats of the {args.steps}-step loop"
                                 f"{' (one CUDA-graph launch of the public call per repeat)' if step_graph is not None else ''}, "
                                 f"{REPEAT_PAUSE_S} s idle and 3 "
                                 f"warm-up steps before each (burst regime); stages.linear_incl_quant_sustained holds the "
                                 f"loop for about a second (power-capped regime)",
                       "accepted_permutation": bool(cal.select[1].item())},
            "ms_per_step_repeats": {"n": len(repeats), "min": min(repeats), "median": ms_step, "max": max(repeats)},
            "frac_fp4_peak_incl_quant": value / world / fp4_peak,
            # the targets of the metric, against the nominal figures it names (dense FP4 9000 TFLOP/s, HBM 8000 GB/s)
            # as well as against what a cuBLAS bf16 GEMM x 4 and a plain copy reach on this machine
            "targets": {"linear_incl_quant_frac_of_nominal_fp4_9000": value / world / 9000.0,
                        "linear_incl_quant_frac_of_measured_bf16x4": value / world / fp4_peak,
                        "linear_target": 0.60,
                        "quant_act_frac_of_nominal_hbm_8000": quant_gbs / 8000.0,
                        "quant_act_frac_of_measured_copy": quant_gbs / peaks["hbm_gbs"],
                        "quant_target": 0.75},
            "roofline": roofline, "stages": stages, "e2e": e2e, "gpu_launches": 2 * args.steps * REPEATS,
            "clocks": sampler.summary(),
            "cpu_baseline": cpu_baseline() if world == 1 else None,
        }
        print(json.dumps(out))
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def spawn_ranks(args):
    """`python bench.py --gpus N` without a launcher: re-run this file as N ranks of one node."""
    import socket
    import subprocess
    with socket.socket() as sock:
        sock.bind(("127.0.0.1", 0))
        port = sock.getsockname()[1]
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", f"--nproc-per-node={args.gpus}",
           "--master-addr", "127.0.0.1", "--master-port", str(port), os.path.abspath(__file__),
           "--gpus", str(args.gpus), "--steps", str(args.steps), "--warmup", str(args.warmup), "--impl", args.impl]
    return subprocess.call(cmd)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=500)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    args = ap.parse_args()
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        raise SystemExit(spawn_ranks(args))
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
