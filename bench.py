#!/usr/bin/env python
"""Benchmark of the group-wise int8-quantized Winograd convolution on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--config 5] [--impl reference]

A *step* is one pass of the whole forward path (input transform + group quantization,
int8 tensor-core contraction with per-group dequantization, output transform) over
every layer of one workload configuration, called through the C ABI.  The metric is
direct-convolution-equivalent throughput, 2*N*K*C*H*W*9 operations per layer divided
by the time of the forward call (filter preparation is offline and not timed).  The
headline workload is configuration 5, the largest one (the full UNet conv-layer set).

One JSON line is printed by rank 0 on stdout, short enough to survive where only the end of a program's output is
kept: the throughput and, of the blocks below, the figures themselves.  The whole record goes to stderr as
one JSON line before it (`details`); it carries
  roofline      achieved HBM GB/s of the kernel that takes the most time in a step,
                from CUDA events around the chain prefixes K1, K1+K2, K1+K2+K3
  per_config    the same figures for each of the five configurations (fewer steps)
  contraction   the contraction kernel against the measured rate of the int8 tensor pipe
                (an SMEM-resident tcgen05.mma kind::i8 loop), stand-alone with operands
                warm in L2, and on one large off-configuration shape with groups of 128
  parity        the timed outputs compared with the CPU oracle on sampled tiles
  e2e           the same metric through wfq_conv_forward_host (pinned host buffers,
                host<->device copies inside the timed region)
  cpu_baseline  the CPU oracle timed on this machine's cores on a sample of tiles
  clocks        SM clock and throttle reasons sampled during the timed region

With --gpus N > 1 every rank runs an independent replica of the workload (the path
needs no exchange between GPUs); the value is the aggregate over the ranks.
--impl reference times the CPU oracle instead of the CUDA path.
"""
import argparse
import json
import os
import statistics
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "direct_conv_equivalent_TOPS"
UNIT = "TOPS"
FALLBACK_HBM_GBS = 6650.0
L2_FLUSH_BYTES = 256 << 20
NOMINAL_INT8_TOPS = 4500.0
KERNELS = ["input_transform_quantize", "gemm_dequantize", "output_transform"]
# dram__bytes_read.sum + dram__bytes_write.sum per launch, mean over the launches of one step,
# from one ncu capture of this command (profiles/gemm_dequant_cfg5_dram_traffic.txt).  Keyed by
# (configuration, kernel); anything else has no capture of the current kernels and reports null.
# The written Y stays in the 126 MB L2 for the output transform, so this is below the
# algorithmic bytes.
NCU_TRAFFIC = {(5, "gemm_dequantize"): 39352474}


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=40)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--config", type=int, default=5, help="headline workload configuration 1..5")
    ap.add_argument("--impl", default="wfq", choices=["wfq", "reference"])
    ap.add_argument("--reps", type=int, default=5,
                    help="graph replays per step; the step's time is their median")
    ap.add_argument("--only-layer", type=int, default=None,
                    help="restrict the workload to one layer of the configuration (profiling)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-per-config", action="store_true", help="skip the other configurations")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the tensor-pipe rate, stand-alone contraction, sustained and parity legs")
    ap.add_argument("--no-graph", action="store_true",
                    help="enqueue every step with stream launches instead of replaying a CUDA graph")
    ap.add_argument("--k1-kernel", type=int, default=0, choices=[0, 1, 2],
                    help="input-transform kernel: 0 the library's choice, 1 cp.async, 2 tensor cores "
                         "where they apply (profiling)")
    ap.add_argument("--nhwc", action="store_true",
                    help="hand x over as [N][H][W][C] (the library then uses its NHWC input transforms); the "
                         "default workload is NCHW")
    ap.add_argument("--cpu-seconds", type=float, default=16.0,
                    help="CPU time budget of the oracle baseline")
    return ap.parse_args()


def workload_name(cfg):
    return {1: "cfg1: single 64->64 32x32 F(4,3) layer, fp32 input",
            2: "cfg2: ResNet-18-style stage, four 3x3 layers N=32 C=K=64/128/256/512 "
               "at 56/28/14/7, F(6,3), group 64, fp16 input",
            3: "cfg3: ResNet-34-style sweep, N=64, 12 runs F(4,3)/F(6,3) x groups 32/64/128",
            4: "cfg4: diffusion-UNet block, N=2, C=K=320/640/1280 at 64/32/16, F(4,3), group 64",
            5: "cfg5: UNet conv-layer set at 128/64/32 latent, N=1, F(4,3) and F(6,3), "
               "C,K in {320,640,1280}, group 64, fp16 input, ten layers end to end"}[cfg]


# ---- byte counts the method itself must move (per launch) ----------------------------

def geometry(L):
    n = L.m + 2
    P = n * n
    T = L.N * (-(-L.H // L.m)) * (-(-L.W // L.m))
    G = L.C // L.gs
    return P, T, G


def algorithmic_bytes(L):
    """Bytes each of the three kernels has to read and write once."""
    P, T, G = geometry(L)
    e_in = 2 if L.dtype == "f16" else 4
    k1 = L.N * L.C * L.H * L.W * e_in + P * T * L.C + 4 * P * T * G
    k2 = P * T * L.C + P * L.K * L.C + 4 * P * G * (T + L.K) + 4 * P * T * L.K
    k3 = 4 * P * T * L.K + 4 * L.N * L.K * L.H * L.W
    return {KERNELS[0]: k1, KERNELS[1]: k2, KERNELS[2]: k3}


def gemm_ops(L):
    """Integer operations of the Winograd-domain contraction, 2*P*T*C*K."""
    P, T, _ = geometry(L)
    return 2.0 * P * T * L.C * L.K


def hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured copy bandwidth", d
    return FALLBACK_HBM_GBS, "fallback", {}


# ---- clocks -----------------------------------------------------------------------------

class ClockSampler:
    """Samples SM clock and throttle reasons through NVML while the timed region runs."""

    def __init__(self, index):
        self.samples, self.reasons = [], set()
        self.max_mhz = None
        self._stop = threading.Event()
        self._thread = None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = int(pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM))
        except Exception:
            self.nv = None

    def _loop(self):
        nv = self.nv
        names = {"hw_slowdown": getattr(nv, "nvmlClocksThrottleReasonHwSlowdown", 0x8),
                 "hw_thermal_slowdown": getattr(nv, "nvmlClocksThrottleReasonHwThermalSlowdown", 0x40),
                 "sw_thermal_slowdown": getattr(nv, "nvmlClocksThrottleReasonSwThermalSlowdown", 0x20),
                 "sw_power_cap": getattr(nv, "nvmlClocksThrottleReasonSwPowerCap", 0x4)}
        while not self._stop.is_set():
            try:
                self.samples.append(int(nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM)))
                mask = int(nv.nvmlDeviceGetCurrentClocksThrottleReasons(self.h))
                for k, bit in names.items():
                    if mask & bit:
                        self.reasons.add(k)
            except Exception:
                pass
            self._stop.wait(0.005)

    def start(self):
        if self.nv is not None:
            self._thread = threading.Thread(target=self._loop, daemon=True)
            self._thread.start()

    def stop(self):
        self._stop.set()
        if self._thread is not None:
            self._thread.join()
        med = None
        if self.samples:
            s = sorted(self.samples)
            med = s[len(s) // 2]
        return {"sm_mhz": med, "sm_max_mhz": self.max_mhz, "reasons": sorted(self.reasons),
                "samples": len(self.samples)}


# ---- CPU oracle legs -------------------------------------------------------------------

def oracle_time_sample(layers, tensors, seconds):
    """Times the oracle's forward pipeline on a sample of tiles of every layer.

    Each layer gets an equal share of `seconds`: as many (randomly chosen) tiles as that
    share allows, or, where the whole layer takes less, the whole layer several times.
    Returns (ops, secs, description, threads): direct-equivalent operations covered and
    the CPU seconds they took (filter preparation excluded, as on the GPU side).
    """
    import numpy as np
    from oracle import oracle as orc
    total_ops, total_s, desc = 0.0, 0.0, []
    per_layer = seconds / max(len(layers), 1)
    for L, (x, w, sB, sG) in zip(layers, tensors):
        P, T, G = geometry(L)
        mats = orc.matrices(L.m, sB, sG)
        filt = orc.prepare_filters(w, L.m, L.gs, mats)
        rng = np.random.default_rng(L.seed + 7)

        def run(n):
            tiles = np.sort(rng.choice(T, n, replace=False))
            t0 = time.perf_counter()
            orc.wfq(x, w, L.m, L.gs, sB=sB, sG=sG, tiles=tiles, filters=filt)
            return time.perf_counter() - t0

        n = min(T, 16)
        dt = run(n)
        while n < T and dt < 0.25 * per_layer:            # grow the sample towards the budget
            n = min(T, max(2 * n, int(n * 0.8 * per_layer / max(dt, 1e-6))))
            dt = run(n)
        reps, spent = 1, dt
        while n == T and spent + dt < per_layer:          # a small layer: whole layer, repeated
            spent += run(n)
            reps += 1
        total_ops += L.direct_ops * (n / T) * reps
        total_s += spent
        desc.append(f"{n}/{T}" + (f"x{reps}" if reps > 1 else ""))
    return total_ops, total_s, "tiles per layer " + ",".join(desc), orc.num_threads()


def run_reference(args):
    """The CPU oracle as the reference arm (rank 0 only)."""
    if int(os.environ.get("RANK", "0")) != 0:
        return
    from paper_2412_19867_b200 import workloads as wl
    layers = select_layers(wl, args.config, args.only_layer)
    tensors = [wl.make_tensors(L) for L in layers]
    nsteps = args.steps + args.warmup
    per_step = max(0.5, min(20.0, 90.0 / max(nsteps, 1)))
    ops = secs = 0.0
    sample, cores = "", 0
    for i in range(nsteps):
        o, s, sample, cores = oracle_time_sample(layers, tensors, per_step)
        if i >= args.warmup:
            ops += o
            secs += s
    value = ops / secs / 1e12
    step_ops = sum(L.direct_ops for L in layers)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": step_ops / (value * 1e12) * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": workload_name(args.config),
                       "note": "CPU oracle; each step times a sample of tiles and is scaled "
                               "to the whole workload"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample + " per step"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


# ---- the printed line ------------------------------------------------------------------
LINE_LIMIT = 2500          # characters


def _part(block, keys):
    return None if block is None else {k: block[k] for k in keys if k in block}


def _values(blocks):
    return {name: b_["error"] if "error" in b_ else b_["value"] for name, b_ in (blocks or {}).items() if b_ is not None}


def printed_line(record):
    """The stdout line of a record: every scalar and `config` whole, of the other blocks the figures themselves."""
    line = {k: v for k, v in record.items() if not isinstance(v, (dict, list))}
    line["config"] = record["config"]
    line["clocks"] = record.get("clocks")
    line["e2e"] = _part(record.get("e2e"), ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step", "steps",
                                            "matches_synchronous_result"))
    line["roofline"] = _part(record.get("roofline"), ("bound", "kernel", "achieved", "peak", "unit", "frac", "traffic",
                                                      "launches_per_step", "algorithmic_bytes_per_launch", "us_per_launch"))
    line["parity"] = _part(record.get("parity"), ("ok", "worst_rel_err", "tolerance", "int8_code_mismatch_rate"))
    line["cpu_baseline"] = _part(record.get("cpu_baseline"), ("value", "unit", "cores", "kind"))
    line["us_per_step"] = {name: _part(record.get(name), ("us_per_step",)).get("us_per_step")
                           for name in ("nhwc_input", "layers_on_three_streams", "w4_weights") if record.get(name)}
    line["values"] = dict(_values(record.get("per_config")), **_values(record.get("full_quant")))
    for k in ("us_per_step", "values"):
        if not line[k]:
            del line[k]
    text = json.dumps(line)
    for k in ("values", "us_per_step", "cpu_baseline", "parity", "roofline"):     # least needed first
        if len(text) <= LINE_LIMIT:
            break
        line.pop(k, None)
        text = json.dumps(line)
    return text


# ---- aggregation over replicas ---------------------------------------------------------

def max_over_ranks(value, device=None):
    """The maximum of a per-rank time over all ranks (no-op without a process group)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(value)
    t = torch.tensor([float(value)], dtype=torch.float64, device=device or "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(ops_per_replica, world, ms_per_step):
    """Whole-job throughput in TOPS: every rank runs an independent replica of the
    workload (the path needs no exchange), the job takes as long as its slowest rank."""
    return world * ops_per_replica / (ms_per_step * 1e-3) / 1e12


def select_layers(wl, cfg, only_layer=None):
    layers = wl.config_layers(cfg)
    return layers if only_layer is None else [layers[only_layer]]


# ---- one configuration on the device ---------------------------------------------------

class Workload:
    """The layers of one configuration: plans, device tensors, and the step as a CUDA graph."""

    def __init__(self, cfg, only_layer, dev, stream, flush, use_graph=True, k1_kernel=0, full_quant=None,
                 nhwc=False, streams=1, w_bits=8):
        import torch
        from paper_2412_19867_b200 import binding as b
        from paper_2412_19867_b200 import workloads as wl
        self.torch, self.b, self.dev, self.stream, self.flush = torch, b, dev, stream, flush
        self.cfg = cfg
        self.w_bits = w_bits
        self.layers = select_layers(wl, cfg, only_layer)
        self.tensors = [wl.make_tensors(L) for L in self.layers]
        self.convs, self.xs, self.ys = [], [], []
        for L, (x, w, sB, sG) in zip(self.layers, self.tensors):
            conv = b.Conv(L.N, L.C, L.K, L.H, L.W, L.m, L.gs, L.dtype, dev)
            if w_bits != 8:                 # filter codes in [-7, 7]; activations stay at 8 bits
                conv.set_weight_bits(w_bits)
            conv.prepare(torch.from_numpy(w).to(dev), list(sB), list(sG))
            if k1_kernel:
                b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_INPUT_TRANSFORM_KERNEL, k1_kernel)
            if full_quant is not None:      # (integer input transform, scale of Y: 1 per tile, 2 per row / column)
                b.wfq_plan_set_full_quant(conv.plan, full_quant[0], full_quant[1])
            self.convs.append(conv)
            xd = torch.from_numpy(x).to(dev)
            if nhwc:                        # x handed over as [N][H][W][C]
                conv.set_input_layout("nhwc")
                xd = xd.permute(0, 2, 3, 1).contiguous()
            self.xs.append(xd)
            self.ys.append(torch.empty((L.N, L.K, L.H, L.W), dtype=torch.float32, device=dev))
        self.step_ops = float(sum(L.direct_ops for L in self.layers))
        self.sptr = stream.cuda_stream
        # streams > 1: the layers (independent problems, each with its own plan and workspace) are
        # dealt round-robin onto that many streams forked from and joined to the launching stream
        self.extra = [torch.cuda.Stream(dev) for _ in range(streams - 1)] if streams > 1 else []
        # One step = the forward calls of all layers.  They are captured once into a CUDA
        # graph and replayed (same kernels, same order, one submission per step); stream
        # launches are the fallback and what --no-graph selects.
        self.enqueue(self.sptr)
        torch.cuda.synchronize(dev)
        self.graph, self.launch_mode = None, "stream launches"
        if use_graph:
            try:
                side = torch.cuda.Stream(dev)
                side.wait_stream(stream)
                cand = torch.cuda.CUDAGraph()
                with torch.cuda.graph(cand, stream=side):
                    self.enqueue(side.cuda_stream, side)
                torch.cuda.synchronize(dev)
                self.graph, self.launch_mode = cand, "CUDA graph replay"
            except Exception as exc:   # capture is an optimisation of the submission only
                print(f"bench: graph capture failed ({exc!r}); using stream launches", file=sys.stderr)
                torch.cuda.synchronize(dev)

    def enqueue(self, stream_ptr, main=None):
        if not self.extra:
            for conv, x, y in zip(self.convs, self.xs, self.ys):
                self.b.wfq_conv_forward(conv.plan, x.data_ptr(), y.data_ptr(), stream_ptr)
            return
        main = self.stream if main is None else main
        lanes = [main] + self.extra
        for s in self.extra:
            s.wait_stream(main)
        for i, (conv, x, y) in enumerate(zip(self.convs, self.xs, self.ys)):
            self.b.wfq_conv_forward(conv.plan, x.data_ptr(), y.data_ptr(), lanes[i % len(lanes)].cuda_stream)
        for s in self.extra:
            main.wait_stream(s)

    def step(self):
        if self.graph is not None:
            self.graph.replay()
        else:
            self.enqueue(self.sptr)

    def check(self):
        for conv in self.convs:
            conv.check_status()

    def timed_replays(self, count, flush=True):
        """`count` replays, each in its own event pair (L2 flushed before each); ms each."""
        torch = self.torch
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(count)]
        for e0, e1 in ev:
            if flush:
                self.flush.zero_()
            e0.record(self.stream)
            self.step()
            e1.record(self.stream)
        torch.cuda.synchronize(self.dev)
        return [e0.elapsed_time(e1) for e0, e1 in ev]

    def kernel_split(self, ksteps):
        """Per layer and kernel: ms from differences of the chain prefixes K1, K1+K2,
        K1+K2+K3 (L2 flushed before each prefix, one event pair around each; medians)."""
        torch, b = self.torch, self.b
        acc = [[[], [], []] for _ in self.layers]
        for _ in range(ksteps):
            evs = []
            for conv, x, y in zip(self.convs, self.xs, self.ys):
                per_prefix = []
                for depth in (1, 2, 3):
                    self.flush.zero_()
                    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    e0.record(self.stream)
                    b.wfq_input_transform_quantize(conv.plan, x.data_ptr(), self.sptr)
                    if depth >= 2:
                        b.wfq_gemm_dequantize(conv.plan, self.sptr)
                    if depth >= 3:
                        b.wfq_output_transform(conv.plan, y.data_ptr(), self.sptr)
                    e1.record(self.stream)
                    per_prefix.append((e0, e1))
                evs.append(per_prefix)
            torch.cuda.synchronize(self.dev)
            for li, per_prefix in enumerate(evs):
                t = [a.elapsed_time(z) for a, z in per_prefix]
                acc[li][0].append(t[0])
                acc[li][1].append(t[1] - t[0])
                acc[li][2].append(t[2] - t[1])
        return [[statistics.median(v) for v in layer] for layer in acc]

    def gemm_warm(self, reps=6):
        """The contraction alone, back to back on operands the previous launch left in L2."""
        torch, b = self.torch, self.b
        out = []
        for conv in self.convs:
            b.wfq_gemm_dequantize(conv.plan, self.sptr)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(self.stream)
            for _ in range(reps):
                b.wfq_gemm_dequantize(conv.plan, self.sptr)
            e1.record(self.stream)
            torch.cuda.synchronize(self.dev)
            out.append(e0.elapsed_time(e1) / reps)
        return out

    def summary(self, ms_per_step, kern_ms, peak, world=1):
        """eq-TOPS, per-layer microseconds and per-kernel roofline fractions."""
        abytes = [algorithmic_bytes(L) for L in self.layers]
        nl = len(self.layers)
        tot_ms = [sum(kern_ms[li][k] for li in range(nl)) for k in range(3)]
        tot_bytes = [sum(abytes[li][KERNELS[k]] for li in range(nl)) for k in range(3)]
        kernels = {}
        for k in range(3):
            gbps = tot_bytes[k] / (tot_ms[k] * 1e-3) / 1e9
            kernels[KERNELS[k]] = {"us_per_step": tot_ms[k] * 1e3, "GBps": gbps, "frac_of_hbm": gbps / peak,
                                   "algorithmic_bytes_per_step": tot_bytes[k]}
        g_ops = float(sum(gemm_ops(L) for L in self.layers))
        kernels[KERNELS[1]]["int8_TOPS"] = g_ops / (tot_ms[1] * 1e-3) / 1e12
        rows = []
        for li, L in enumerate(self.layers):
            us = [kern_ms[li][k] * 1e3 for k in range(3)]
            rows.append({"layer": L.name, "us": round(sum(us), 2), "us_k1_k2_k3": [round(u, 2) for u in us],
                         "frac_of_hbm_k1_k2_k3": [round(abytes[li][KERNELS[k]] / (max(us[k], 1e-3) * 1e-6) / 1e9 / peak, 3)
                                                  for k in range(3)],
                         "eq_TOPS": round(L.direct_ops / (sum(us) * 1e-6) / 1e12, 1)})
        return {"workload": workload_name(self.cfg), "layers": nl,
                "value": replica_throughput(self.step_ops, world, ms_per_step), "unit": UNIT,
                "us_per_step": ms_per_step * 1e3, "direct_GOP_per_step": self.step_ops / 1e9,
                "kernels": kernels, "us_per_layer": rows}, tot_ms, tot_bytes

    def parity(self, tiles_per_layer=6, channels=12):
        """The outputs of the last step against the CPU oracle on sampled tiles and output
        channels (the oracle evaluates the pipeline tile by tile): worst error relative to
        max |y| of the layer, and the int8 code mismatch rate of the sampled tiles."""
        import numpy as np
        from oracle import oracle as orc
        b, torch = self.b, self.torch
        worst, worst_layer, mism, ncodes = 0.0, None, 0, 0
        for L, conv, (x, w, sB, sG), y in zip(self.layers, self.convs, self.tensors, self.ys):
            yh = y.cpu().numpy()
            rng = np.random.default_rng(L.seed + 13)
            T = conv.T
            tiles = np.unique(np.concatenate([[0, T - 1], rng.integers(0, T, tiles_per_layer)]))
            ks = np.unique(np.concatenate([[0, L.K - 1], rng.integers(0, L.K, channels)]))
            filters = None
            if self.w_bits != 8:
                filters = orc.prepare_filters(w[ks], L.m, L.gs, orc.matrices(L.m, sB, sG, None), bits=self.w_bits)
            ref = orc.wfq(x, w[ks], L.m, L.gs, sB=sB, sG=sG, tiles=tiles, filters=filters)
            xq = conv.buffer(b.WFQ_BUF_XQ)[:, torch.from_numpy(tiles).to(self.dev)].cpu().numpy()
            mism += int(np.count_nonzero(xq != ref.Xq))
            ncodes += xq.size
            geo = orc.geometry(L.N, L.H, L.W, L.m)
            scale = float(np.max(np.abs(yh)))
            for i, t in enumerate(tiles):
                tw, th, img = t % geo.TW, (t // geo.TW) % geo.TH, t // (geo.TW * geo.TH)
                hh, ww = min(L.m, L.H - th * L.m), min(L.m, L.W - tw * L.m)
                got = yh[img][ks][:, th * L.m:th * L.m + hh, tw * L.m:tw * L.m + ww]
                err = float(np.max(np.abs(got - ref.ytile[i][:, :hh, :ww]))) / scale
                if err > worst:
                    worst, worst_layer = err, L.name
        return {"checked": True, "against": "CPU oracle, sampled tiles and output channels of every layer",
                "worst_rel_err": worst, "worst_layer": worst_layer, "tolerance": 2e-3, "ok": worst <= 2e-3,
                "int8_code_mismatch_rate": mism / max(ncodes, 1), "codes_compared": ncodes}

    def parity_full_quant(self, y_scale, tiles_per_layer=6, channels=12):
        """The fully quantized pipeline's outputs against the oracle's on sampled tiles and
        output channels: relative L2 distance over the sample (a code of Y that flips through
        the fp32 accumulation order of Y moves one tile by a quantization step, so there is
        no element-wise bar) and the mismatch rate of the int8 codes (bit exact by design)."""
        import numpy as np
        from oracle import full_quant as fq
        from oracle import oracle as orc
        b, torch = self.b, self.torch
        num = den = 0.0
        mism = ncodes = 0
        for L, conv, (x, w, sB, sG), y in zip(self.layers, self.convs, self.tensors, self.ys):
            yh = y.cpu().numpy()
            rng = np.random.default_rng(L.seed + 17)
            T = conv.T
            tiles = np.unique(np.concatenate([[0, T - 1], rng.integers(0, T, tiles_per_layer)]))
            ks = np.unique(np.concatenate([[0, L.K - 1], rng.integers(0, L.K, channels)]))
            ref = fq.wfq_full(x, w[ks], L.m, L.gs, sB, sG, tiles=tiles, quant_input=True, quant_output=True,
                              y_scale=y_scale)
            xq = conv.buffer(b.WFQ_BUF_XQ)[:, torch.from_numpy(tiles).to(self.dev)].cpu().numpy()
            mism += int(np.count_nonzero(xq != ref.Xq))
            ncodes += xq.size
            geo = orc.geometry(L.N, L.H, L.W, L.m)
            for i, t in enumerate(tiles):
                tw, th, img = t % geo.TW, (t // geo.TW) % geo.TH, t // (geo.TW * geo.TH)
                hh, ww = min(L.m, L.H - th * L.m), min(L.m, L.W - tw * L.m)
                got = yh[img][ks][:, th * L.m:th * L.m + hh, tw * L.m:tw * L.m + ww]
                want = ref.ytile[i][:, :hh, :ww]
                num += float(np.sum((got - want) ** 2))
                den += float(np.sum(want ** 2))
        rel = (num / max(den, 1e-300)) ** 0.5
        return {"against": "CPU oracle of the fully quantized pipeline, sampled tiles and output channels",
                "rel_l2": rel, "tolerance": 1e-2, "ok": rel <= 1e-2,
                "int8_code_mismatch_rate": mism / max(ncodes, 1), "codes_compared": ncodes}

    def close(self):
        for conv in self.convs:
            conv.check_status()
            conv.close()
        self.graph = None


# ---- the CUDA path ---------------------------------------------------------------------

def run_wfq(args):
    import torch
    import torch.distributed as dist
    from paper_2412_19867_b200 import binding as b
    from paper_2412_19867_b200 import build as wfq_build
    from paper_2412_19867_b200 import workloads as wl

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise RuntimeError("bench.py needs a CUDA device; there is no CPU fallback")
    if rank == 0:
        wfq_build.build()
    if world > 1:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        dist.barrier()
    b.load()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    peak, peak_src, peaks = hbm_peak()
    warmup = max(args.warmup, 3)
    reps = max(args.reps, 1)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize(dev)

    wk = Workload(args.config, args.only_layer, dev, stream, flush, use_graph=not args.no_graph,
                  k1_kernel=args.k1_kernel, nhwc=args.nhwc)
    for _ in range(warmup):
        flush.zero_()
        wk.step()
    barrier()
    wk.check()

    # ---- timed region: K steps; a step's time is the median of `reps` graph replays, each
    # behind its own L2 flush and inside its own event pair ---------------------------------
    sampler = ClockSampler(local)
    barrier()
    sampler.start()
    wall0 = time.perf_counter()
    step_ms, step_spread = [], []
    for _ in range(args.steps):
        t = wk.timed_replays(reps)
        step_ms.append(statistics.median(t))
        step_spread.append((max(t) - min(t)) / max(statistics.median(t), 1e-9))
    barrier()
    wall = time.perf_counter() - wall0
    clocks = sampler.stop()
    total_ms = max_over_ranks(float(sum(step_ms)), dev)
    ms_per_step = total_ms / args.steps
    value = replica_throughput(wk.step_ops, world, ms_per_step)
    timing = {"replays_per_step": reps, "step_time": "median of the replays",
              "ms_per_step_min": min(step_ms), "ms_per_step_max": max(step_ms),
              "ms_per_step_stdev": statistics.pstdev(step_ms),
              "median_spread_within_step": statistics.median(step_spread)}

    # ---- the same steps back to back, no L2 flush (operands may sit in the 126 MB L2) ------
    wsteps = min(max(args.steps, 10), 100)
    wk.step()
    torch.cuda.synchronize(dev)
    w0, w1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    w0.record(stream)
    for _ in range(wsteps):
        wk.step()
    w1.record(stream)
    torch.cuda.synchronize(dev)
    warm_ms = max_over_ranks(w0.elapsed_time(w1) / wsteps, dev)
    warm = {"ms_per_step": warm_ms, "value": replica_throughput(wk.step_ops, world, warm_ms), "unit": UNIT,
            "steps": wsteps, "l2": "not flushed"}

    # ---- per-kernel durations and roofline of the headline workload -----------------------
    ksteps = min(max(args.steps, 10), 40)
    kern_ms = wk.kernel_split(ksteps)
    head, tot_ms, tot_bytes = wk.summary(ms_per_step, kern_ms, peak, world)
    dom = max(range(3), key=lambda k: tot_ms[k])
    achieved = tot_bytes[dom] / (tot_ms[dom] * 1e-3) / 1e9
    nl = len(wk.layers)
    roofline = {"bound": "hbm", "kernel": KERNELS[dom], "achieved": achieved, "peak": peak, "unit": "GB/s",
                "frac": achieved / peak, "traffic": NCU_TRAFFIC.get((args.config, KERNELS[dom])) if args.only_layer is None else None,
                "peak_source": peak_src,
                "launches_per_step": nl, "algorithmic_bytes_per_step": tot_bytes[dom],
                "algorithmic_bytes_per_launch": tot_bytes[dom] / nl,
                "us_per_launch": tot_ms[dom] * 1e3 / nl,
                "note": "traffic: mean DRAM bytes per launch over the launches of one step (ncu, "
                        "profiles/); null where the current kernels have no capture on this workload",
                "all_kernels": head["kernels"]}

    # ---- sustained: the same step replayed for about two seconds -------------------------
    sustained = None
    contraction = None
    parity = None
    if not args.no_extras:
        s_sampler = ClockSampler(local)
        s_sampler.start()
        t_end = time.perf_counter() + 2.0
        s_ms = []
        while time.perf_counter() < t_end:
            s_ms += wk.timed_replays(20)
        s_clocks = s_sampler.stop()
        s_med = statistics.median(s_ms)
        sustained = {"seconds": 2.0, "replays": len(s_ms), "ms_per_step_median": s_med,
                     "value": replica_throughput(wk.step_ops, world, s_med), "unit": UNIT, "clocks": s_clocks}

        # ---- outputs of the timed workload against the oracle (outside every timed region) ---
        if rank == 0:
            flush.zero_()
            wk.step()
            torch.cuda.synchronize(dev)
            parity = wk.parity()

        # ---- the contraction against the rate of the int8 tensor pipe -------------------
        rate = {}
        for n_cols in (64, 128, 256):
            best = 0.0
            for _ in range(3):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                ops = b.wfq_debug_int8_mma_rate(wk.convs[0].plan, n_cols, 20000, stream.cuda_stream)
                e1.record(stream)
                torch.cuda.synchronize(dev)
                best = max(best, ops / (e0.elapsed_time(e1) * 1e-3) / 1e12)
            rate[f"128x{n_cols}x32"] = best
        int8_peak = max(rate.values())
        g_warm = wk.gemm_warm()
        g_ops = [gemm_ops(L) for L in wk.layers]
        warm_tops = sum(g_ops) / (sum(g_warm) * 1e-3) / 1e12
        chain_tops = head["kernels"][KERNELS[1]]["int8_TOPS"]
        # the promotion of a group's int32 sums takes about 2.3 issue slots per accumulator
        # element, an SM issues 128 per clock and the tensor pipe yields 8192/gs elements
        ceil64 = 64.0 / (64.0 * 2.3)
        contraction = {"int8_peak_measured_TOPS": int8_peak, "int8_rate_by_shape_TOPS": rate,
                       "int8_peak_how": "SMEM-resident accumulating tcgen05.mma kind::i8, one CTA per SM, "
                                        "20000 instructions each, best of 3",
                       "int8_nominal_TOPS": NOMINAL_INT8_TOPS,
                       "in_chain": {"int8_TOPS": chain_tops, "frac_of_measured_peak": chain_tops / int8_peak,
                                    "frac_of_nominal": chain_tops / NOMINAL_INT8_TOPS},
                       "stand_alone_l2_warm": {"int8_TOPS": warm_tops, "frac_of_measured_peak": warm_tops / int8_peak,
                                               "us_per_layer": [round(t * 1e3, 2) for t in g_warm]},
                       "promotion_ceiling_frac": {"group_64": ceil64, "group_128": min(1.0, 2 * ceil64),
                                                  "issue_slots_per_accumulator": 2.3}}
        # one large shape outside the configurations: many tiles, groups of 128 channels
        try:
            big = wl.Layer(8, 1024, 256, 112, 112, 4, 128, "f16", "silu_outlier", "kaiming_chan", 6, 0, 0)
            x, w, sB, sG = wl.make_tensors(big)
            conv = b.Conv(big.N, big.C, big.K, big.H, big.W, big.m, big.gs, big.dtype, dev)
            conv.prepare(torch.from_numpy(w).to(dev), list(sB), list(sG))
            xd = torch.from_numpy(x).to(dev)
            b.wfq_input_transform_quantize(conv.plan, xd.data_ptr(), stream.cuda_stream)
            b.wfq_gemm_dequantize(conv.plan, stream.cuda_stream)
            ts = []
            for _ in range(5):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                b.wfq_gemm_dequantize(conv.plan, stream.cuda_stream)
                e1.record(stream)
                torch.cuda.synchronize(dev)
                ts.append(e0.elapsed_time(e1))
            conv.check_status()
            t = statistics.median(ts)
            tops = gemm_ops(big) / (t * 1e-3) / 1e12
            contraction["large_shape_group_128"] = {
                "layer": big.name, "us": t * 1e3, "int8_TOPS": tops, "frac_of_measured_peak": tops / int8_peak,
                "GBps": algorithmic_bytes(big)[KERNELS[1]] / (t * 1e-3) / 1e9,
                "note": "contraction kernel only; operands and Y (231 MB each) exceed L2"}
            conv.close()
            del xd
        except Exception as exc:
            contraction["large_shape_group_128"] = {"error": repr(exc)}

    # ---- end to end through the host-buffer entry point ----------------------------------
    # One step = every layer through wfq_conv_forward_host_async from pinned host buffers (copy in,
    # three kernels, copy out), the layers spread over three streams so that the copy in of one
    # layer overlaps the copy out of another, then a wait for all of them.  `serial` is the same
    # through the synchronous entry point, one layer after the other.
    e2e = None
    if not args.no_e2e:
        xh = [torch.from_numpy(t[0]).pin_memory() for t in wk.tensors]
        yh = [torch.empty(y.shape, dtype=torch.float32).pin_memory() for y in wk.ys]
        esteps = max(3, min(args.steps, 20))
        side = [torch.cuda.Stream(dev) for _ in range(3)]

        def e2e_step():
            for i, (conv, x, y) in enumerate(zip(wk.convs, xh, yh)):
                conv.forward_host_async(x, y, side[i % 3])
            for st in side:
                st.synchronize()

        for conv, x, y in zip(wk.convs, xh, yh):
            conv.forward_host(x, y)
        want = [y.clone() for y in yh]
        e2e_step()
        same = all(torch.equal(a, b_) for a, b_ in zip(want, yh))
        barrier()
        t0 = time.perf_counter()
        for _ in range(esteps):
            e2e_step()
        torch.cuda.synchronize(dev)
        dt = max_over_ranks(time.perf_counter() - t0, dev)
        barrier()
        t0 = time.perf_counter()
        for _ in range(esteps):
            for conv, x, y in zip(wk.convs, xh, yh):
                conv.forward_host(x, y)          # synchronous: copies + kernels + copy back
        torch.cuda.synchronize(dev)
        dts = max_over_ranks(time.perf_counter() - t0, dev)
        # the same with y written and copied out as fp16 (wfq_plan_set_output_dtype): half the bytes out
        for conv in wk.convs:
            conv.set_output_dtype("f16")
        yh16 = [torch.empty(y.shape, dtype=torch.float16).pin_memory() for y in wk.ys]

        def e2e_step16():
            for i, (conv, x, y) in enumerate(zip(wk.convs, xh, yh16)):
                conv.forward_host_async(x, y, side[i % 3])
            for st in side:
                st.synchronize()

        e2e_step16()
        same16 = all(torch.equal(a.to(torch.float16), b_) for a, b_ in zip(want, yh16))
        barrier()
        t0 = time.perf_counter()
        for _ in range(esteps):
            e2e_step16()
        torch.cuda.synchronize(dev)
        dt16 = max_over_ranks(time.perf_counter() - t0, dev)
        for conv in wk.convs:
            conv.set_output_dtype("f32")
        e2e = {"value": replica_throughput(wk.step_ops, world, dt * 1e3 / esteps), "unit": UNIT,
               "h2d_bytes_per_step": int(sum(x.numel() * x.element_size() for x in xh)),
               "d2h_bytes_per_step": int(sum(y.numel() * 4 for y in yh)), "steps": esteps,
               "api": "wfq_conv_forward_host_async per layer on three streams, one wait per step",
               "matches_synchronous_result": bool(same),
               "serial": {"value": replica_throughput(wk.step_ops, world, dts * 1e3 / esteps), "unit": UNIT,
                          "api": "wfq_conv_forward_host per layer"},
               "fp16_output": {"value": replica_throughput(wk.step_ops, world, dt16 * 1e3 / esteps), "unit": UNIT,
                               "d2h_bytes_per_step": int(sum(y.numel() * 2 for y in yh16)),
                               "equals_fp32_result_rounded_once": bool(same16)}}
        del xh, yh, yh16, want

    layers, tensors = wk.layers, wk.tensors
    ys_headline = [y.clone() for y in wk.ys] if (rank == 0 and world == 1 and not args.no_extras) else []
    launch_mode = wk.launch_mode
    wk.close()

    # ---- the other configurations, fewer steps -------------------------------------------
    per_config = None
    if rank == 0 and world == 1 and not args.no_per_config and args.only_layer is None:
        per_config = {f"cfg{args.config}": {k: head[k] for k in head}}
        for cfg in (1, 2, 3, 4, 5):
            if cfg == args.config:
                continue
            try:
                w2 = Workload(cfg, None, dev, stream, flush, use_graph=not args.no_graph)
                for _ in range(3):
                    flush.zero_()
                    w2.step()
                torch.cuda.synchronize(dev)
                ms = [statistics.median(w2.timed_replays(reps)) for _ in range(10)]
                s2, _, _ = w2.summary(statistics.mean(ms), w2.kernel_split(10), peak)
                s2["steps"] = 10
                w2.close()
                per_config[f"cfg{cfg}"] = s2
                del w2
                torch.cuda.empty_cache()
                if cfg in (2, 3, 4) and not args.no_extras:      # the same layers handed over as NHWC
                    w2 = Workload(cfg, None, dev, stream, flush, use_graph=not args.no_graph, nhwc=True)
                    for _ in range(3):
                        flush.zero_()
                        w2.step()
                    torch.cuda.synchronize(dev)
                    ms = [statistics.median(w2.timed_replays(reps)) for _ in range(10)]
                    s2n, _, _ = w2.summary(statistics.mean(ms), w2.kernel_split(10), peak)
                    s2["nhwc_input"] = {"value": s2n["value"], "unit": UNIT, "us_per_step": s2n["us_per_step"],
                                        "input_transform_us_per_step": s2n["kernels"][KERNELS[0]]["us_per_step"]}
                    w2.close()
                    del w2
                    torch.cuda.empty_cache()
            except Exception as exc:
                per_config[f"cfg{cfg}"] = {"error": repr(exc)}

    # ---- the fully quantized transforms (Section 4.1) on the UNet block, reported beside ----
    full_quant = None
    if rank == 0 and world == 1 and not args.no_extras and args.only_layer is None:
        full_quant = {}
        for label, mode, y_scale in (("y_per_tile", 1, "tile"), ("y_per_row_column", 2, "row")):
            try:
                w3 = Workload(4, None, dev, stream, flush, use_graph=not args.no_graph, full_quant=(1, mode))
                for _ in range(3):
                    flush.zero_()
                    w3.step()
                torch.cuda.synchronize(dev)
                ms = [statistics.median(w3.timed_replays(reps)) for _ in range(10)]
                s3, _, _ = w3.summary(statistics.mean(ms), w3.kernel_split(10), peak)
                flush.zero_()
                w3.step()
                torch.cuda.synchronize(dev)
                full_quant[label] = {"workload": s3["workload"], "value": s3["value"], "unit": UNIT,
                                     "us_per_step": s3["us_per_step"], "kernels": s3["kernels"],
                                     "us_per_layer": s3["us_per_layer"], "parity": w3.parity_full_quant(y_scale),
                                     "note": "integer input and output transforms (Eqs. quant-B, quant-y); "
                                             "same contraction kernel"}
                w3.close()
                del w3
                torch.cuda.empty_cache()
            except Exception as exc:
                full_quant[label] = {"error": repr(exc)}

    # ---- the headline workload with NHWC input (TMA-staged input transform), reported beside ----
    nhwc = None
    if rank == 0 and world == 1 and not args.no_extras and args.only_layer is None:
        try:
            w4 = Workload(args.config, None, dev, stream, flush, use_graph=not args.no_graph, nhwc=True)
            for _ in range(3):
                flush.zero_()
                w4.step()
            torch.cuda.synchronize(dev)
            ms = [statistics.median(w4.timed_replays(reps)) for _ in range(10)]
            s4, _, _ = w4.summary(statistics.mean(ms), w4.kernel_split(10), peak)
            # the tensor cores accumulate V in another order than the NCHW kernel's add/fma chains: group
            # scales differ in the last bit, and a code in about a million by one step (which moves its tile
            # by a quantization step: visible in the norm on the F(6,3) layers), so the outputs are compared
            # in norm with each other and, like the headline's, with the oracle on sampled tiles
            dev_rel = max(float(torch.linalg.vector_norm(a.float() - b_.float()) /
                                torch.linalg.vector_norm(b_.float())) for a, b_ in zip(w4.ys, ys_headline))
            nhwc = {"workload": s4["workload"], "value": s4["value"], "unit": UNIT, "us_per_step": s4["us_per_step"],
                    "input_transform_us_per_step": s4["kernels"][KERNELS[0]]["us_per_step"],
                    "kernel": "input_transform_tcn_kernel (TMA box as the MN-major operand of tcgen05.mma kind::f16)",
                    "parity": w4.parity(), "worst_rel_l2_vs_nchw_result": dev_rel}
            w4.close()
            del w4
            torch.cuda.empty_cache()
        except Exception as exc:
            nhwc = {"error": repr(exc)}

    # ---- 4-bit filter codes (W4A8) on the UNet block, reported beside ----
    w4 = None
    if rank == 0 and world == 1 and not args.no_extras and args.only_layer is None:
        try:
            w6 = Workload(4, None, dev, stream, flush, use_graph=not args.no_graph, w_bits=4)
            for _ in range(3):
                flush.zero_()
                w6.step()
            torch.cuda.synchronize(dev)
            ms = statistics.mean(statistics.median(w6.timed_replays(reps)) for _ in range(10))
            flush.zero_()
            w6.step()
            torch.cuda.synchronize(dev)
            w4 = {"workload": "cfg4 with the filters quantized to 4 bits (codes in [-7, 7], one per byte on the "
                              "device; activations at 8 bits)",
                  "value": w6.step_ops / (ms * 1e-3) / 1e12, "unit": UNIT, "us_per_step": ms * 1e3,
                  "parity": w6.parity(),
                  "filter_blob_bytes": int(sum(b.wfq_filters_bytes(c.plan) for c in w6.convs)),
                  "note": "same kernels as with 8-bit filters; the exported filter blob stores two codes per byte"}
            w6.close()
            del w6
            torch.cuda.empty_cache()
        except Exception as exc:
            w4 = {"error": repr(exc)}

    # ---- the headline workload with its layers on three streams, reported beside ----
    concurrent = None
    if rank == 0 and world == 1 and not args.no_extras and args.only_layer is None:
        try:
            w5 = Workload(args.config, None, dev, stream, flush, use_graph=not args.no_graph, streams=3)
            for _ in range(3):
                flush.zero_()
                w5.step()
            torch.cuda.synchronize(dev)
            w5.check()
            ms = statistics.mean(statistics.median(w5.timed_replays(reps)) for _ in range(10))
            same = all(torch.equal(a, b_) for a, b_ in zip(w5.ys, ys_headline))
            concurrent = {"streams": 3, "value": w5.step_ops / (ms * 1e-3) / 1e12, "unit": UNIT,
                          "us_per_step": ms * 1e3, "equals_serial_result": bool(same),
                          "note": "the layers of a step are independent problems: dealt round-robin onto three "
                                  "streams inside the replayed graph, so that one layer's latency-bound input and "
                                  "output transforms overlap another layer's contraction; the headline keeps them "
                                  "in one stream, which is what the per-kernel split needs"}
            w5.close()
            del w5
            torch.cuda.empty_cache()
        except Exception as exc:
            concurrent = {"error": repr(exc)}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        o, s, sample, cores = oracle_time_sample(layers, tensors, args.cpu_seconds)
        cpu = {"value": o / s / 1e12, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": sample + f" ({s:.1f} s of CPU time)"}

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": warmup, "ms_per_step": ms_per_step, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "int8", "data": "synthetic",
                "config": {"workload": workload_name(args.config) +
                           ("" if args.only_layer is None else f" (layer {args.only_layer} only)"),
                           "layers": len(layers), "launch": launch_mode,
                           "l2": "flushed before every replay (256 MiB memset outside the replay's "
                                 "event pair)",
                           "parallelism": "replicas" if world > 1 else "single GPU"},
                "timing": timing, "us_per_layer": head["us_per_layer"], "wall_s_timed_region": wall,
                "warm": warm, "sustained": sustained, "roofline": roofline, "contraction": contraction,
                "parity": parity, "per_config": per_config, "full_quant": full_quant, "nhwc_input": nhwc, "layers_on_three_streams": concurrent, "w4_weights": w4, "cpu_baseline": cpu, "e2e": e2e,
                "gpu_launches": 3 * len(layers) * args.steps * reps, "clocks": clocks}
        print("details " + json.dumps(line), file=sys.stderr, flush=True)
        print(printed_line(line), flush=True)
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_wfq(args)


if __name__ == "__main__":
    main()
