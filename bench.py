"""Benchmark of the Log_bQuant inference hot path on GB300.

Workload (one step): the decode step of a Llama-3.1-8B-shaped model at batch
1 -- all 32 layers x 7 linears (q/o 4096x4096, k/v 1024x4096, gate/up
14336x4096, down 4096x14336), 4-bit Log_b codes with a per-layer base drawn
from U[1.2, 2.0] and a per-tensor range max|W|, Student-t(4)*0.02 weights
with 0.1 % x20 outliers, bf16 activations and outputs.  Linears that read the
same activations share a launch (q/k/v and gate/up through
logq_linear_grouped), so a layer is four launches; each launch asks L2 to
fetch the codes of the next one.  The 128 launches of a step are captured once
in a CUDA graph and replayed; the step's 3.49 GB of codes exceed L2, so no
flush is needed between steps.  The Llama-3.2-1B-shaped step (16 layers, 64
launches) is measured the same way as a second workload.

metric: GEMV HBM GB/s at batch 1, counting the algorithmic bytes of every
linear (packed codes + activations + outputs) per step.  The same run also
measures the other rows of the path -- the skinny GEMM at batch 4 and 16,
quantise (absmax + quantise + pack), the prefill GEMM on Llama-3.1-8B shapes
(2048 tokens) -- each with its own roofline, and times the fp64 oracle on the
host cores.

python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
N > 1 runs N independent replicas (one per GPU, launched by torchrun).
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from paper_2607_01127_gb300 import workloads  # noqa: E402

METRIC = "Log_b 4-bit GEMV HBM GB/s (% of ~8 TB/s) at batch 1; prefill GEMM TFLOP/s"
# decode-step workloads: layer shapes, layer count, seed of the configuration
MODELS = {
    "8b": dict(shapes=workloads.LLAMA_8B_SHAPES, layers=workloads.LLAMA_8B_LAYERS, cfg_seed=3,
               name="llama-3.1-8b decode step: 32 layers x {q,k,v,o,gate,up,down} 4-bit Log_b GEMV, batch 1"),
    "1b": dict(shapes=workloads.LLAMA_1B_SHAPES, layers=workloads.LLAMA_1B_LAYERS, cfg_seed=1,
               name="llama-3.2-1b decode step: 16 layers x {q,k,v,o,gate,up,down} 4-bit Log_b GEMV, batch 1"),
}
HEADLINE = "8b"
WORKLOAD = MODELS[HEADLINE]["name"]
PREFILL_TOKENS = 2048


def peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


def model_layers(model: str = HEADLINE):
    """(layer, proj, N, K, seed) for every linear of the model."""
    spec = MODELS[model]
    out = []
    for layer in range(spec["layers"]):
        for pi, name in enumerate(workloads.PROJ_NAMES):
            N, K = spec["shapes"][name]
            out.append((layer, name, N, K, workloads.layer_seed(spec["cfg_seed"], layer, pi)))
    return out


def linear_bytes(N, K, B=1, bits=4, y_bytes=4):
    """Algorithmic bytes of one linear: packed codes, bf16 activations, outputs."""
    return N * K * bits // 8 + B * K * 2 + B * N * y_bytes


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, smax, reasons = [], 0.0, set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = max(smax, float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm)}


def traffic_for(kernel: str, source: str):
    """DRAM bytes per launch from the committed ncu summary, or None when the
    kernel source changed since those counters were taken."""
    try:
        t = json.load(open(os.path.join(ROOT, "profiles", "traffic.json")))[kernel]
        digest = hashlib.sha256(open(os.path.join(ROOT, source), "rb").read()).hexdigest()[:16]
        return t["bytes_per_launch"] if t.get("source_sha") == digest else None
    except Exception:
        return None


# ----------------------------------------------------------------- oracle ---

def oracle_gemv_sample(rows_per_layer: int = 8, seed: int = 0, model: str = HEADLINE):
    """Inputs of the CPU baseline: the first rows of every linear of the model,
    quantised by the oracle (setup, untimed)."""
    import oracle
    spec = MODELS[model]
    bases = workloads.layer_bases(spec["layers"], spec["cfg_seed"])
    items = []
    for layer, name, N, K, s in model_layers(model):
        w = workloads.weights_np(rows_per_layer, K, s + seed, outliers=True)
        cb = oracle.build_codebook(4, float(bases[layer]), float(np.abs(w).max()))
        packed = oracle.pack(oracle.quantize_log(w, cb), 4)
        x = workloads.activations_np(1, K, s).astype(np.float32)
        items.append((cb, packed, x.astype(np.float64), rows_per_layer, K))
    return items


def oracle_gemv_run(items, threads: int):
    import oracle
    nbytes = 0
    for cb, packed, x, R, K in items:
        bs = np.zeros(R, np.int64)
        ns = np.arange(R, dtype=np.int64)
        oracle.linear_sampled(x, packed, 4, cb, oracle.TABLE_BF16, bs, ns, nthreads=threads)
        nbytes += linear_bytes(R, K, y_bytes=2)      # same per-output bytes as the device step
    return nbytes


def cpu_baseline(seconds: float = 12.0):
    threads = len(os.sched_getaffinity(0))
    items = oracle_gemv_sample()
    oracle_gemv_run(items, threads)
    t0, nbytes, reps = time.perf_counter(), 0, 0
    while time.perf_counter() - t0 < seconds:
        nbytes += oracle_gemv_run(items, threads)
        reps += 1
    dt = time.perf_counter() - t0
    return {"value": round(nbytes / dt / 1e9, 4), "unit": "GB/s", "cores": threads, "kind": "oracle",
            "sample": f"fp64 oracle GEMV over the first 8 rows of all {len(items)} linears of the decode "
                      f"step, {reps} passes in {dt:.1f} s",
            "rates": oracle_rates(threads)}


def oracle_rates(threads: int, seconds: float = 1.5):
    """The oracle's other rates on the host cores, one core and all of them: the
    GEMV sample in GB/s, quantisation (Eq. (1) through fp64 logarithms) in
    weights/s, and the fp64 product of a 2048-token prefill slice in GFLOP/s."""
    import oracle
    from concurrent.futures import ThreadPoolExecutor

    def rate(fn, units):
        fn()
        t0, n = time.perf_counter(), 0
        while time.perf_counter() - t0 < seconds:
            fn()
            n += 1
        return units * n / (time.perf_counter() - t0)

    out = {"cores_all": threads}
    items = oracle_gemv_sample()
    gb = oracle_gemv_run(items, 1)
    out["gemv_gbs_1core"] = round(rate(lambda: oracle_gemv_run(items, 1), gb) / 1e9, 4)
    w = workloads.weights_np(512, 4096, 21, outliers=True)
    cb = oracle.build_codebook(4, 1.5, float(np.abs(w).max()))
    out["quantize_weights_per_s_1core"] = round(rate(lambda: oracle.quantize_log(w, cb), w.size), 1)
    chunks = np.array_split(w, threads)                 # the C call releases the GIL
    with ThreadPoolExecutor(threads) as ex:
        out["quantize_weights_per_s_all"] = round(
            rate(lambda: list(ex.map(lambda c: oracle.quantize_log(c, cb), chunks)), w.size), 1)
    X = workloads.activations_np(16, 4096, 22).astype(np.float64)
    What = oracle.dequant(oracle.quantize_log(w, cb), cb)
    fl = 2.0 * X.shape[0] * What.shape[0] * X.shape[1]
    out["prefill_gflops_1core"] = round(rate(lambda: oracle.linear(X, What, 1), fl) / 1e9, 3)
    out["prefill_gflops_all"] = round(rate(lambda: oracle.linear(X, What, threads), fl) / 1e9, 3)
    out["note"] = ("GEMV: the sample above; quantise: 512 x 4096 Student-t weights, 4-bit; prefill: 16 "
                   "tokens x 512 x 4096 of a 2048-token batch (fp64, the oracle's own loops)")
    return out


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    threads = len(os.sched_getaffinity(0))
    items = oracle_gemv_sample()
    for _ in range(args.warmup):
        oracle_gemv_run(items, threads)
    t0 = time.perf_counter()
    nbytes = 0
    for _ in range(args.steps):
        nbytes += oracle_gemv_run(items, threads)
    dt = time.perf_counter() - t0
    v = nbytes / dt / 1e9
    line = {"impl": "reference", "metric": METRIC, "value": round(v, 4), "unit": "GB/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(dt / args.steps * 1e3, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD + " (oracle: first 8 rows of each linear per step)",
                       "l2": "n/a (host)"},
            "cpu_baseline": {"value": round(v, 4), "unit": "GB/s", "cores": threads, "kind": "oracle",
                             "sample": f"first 8 rows of each of the {len(items)} linears per step"},
            "e2e": {"value": round(v, 4), "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ----------------------------------------------------------------- GPU arm ---

# launch groups of one layer: linears that read the same activations share a launch
GROUPS = (("q", "k", "v"), ("o",), ("gate", "up"), ("down",))


def build_decode_model(logq, torch, dev, model: str = HEADLINE, layers: int | None = None):
    """Quantise every linear of the model into one contiguous code buffer (in
    launch order) and prepare the per-launch groups of the decode step.

    The launches form a chain like a model's decode step: launch 0 reads the
    step's input activation, and every later launch reads the bf16 output of
    the launch before it (q -> o -> gate/up -> down -> the next layer's q/k/v;
    gate's output stands in for the activated MLP input of down).  So each
    launch depends on the previous one and finds its X in L2, as it would
    after the attention / norm / activation kernels of a real model.

    Also counts the weights that lie within one fp32 ulp of a decision
    boundary of their codebook (|w| equal to a boundary, rounded up to fp32,
    or to the float just below it): the only weights whose code could depend
    on how a boundary is rounded."""
    spec = MODELS[model]
    n_layers = spec["layers"] if layers is None else layers
    bases = workloads.layer_bases(spec["layers"], spec["cfg_seed"])
    ws = logq.new_workspace(dev)
    specs = [x for x in model_layers(model) if x[0] < n_layers]
    total = sum(N * K // 2 for _, _, N, K, _ in specs)
    arena = torch.empty(total, dtype=torch.uint8, device=dev)
    lin = {}
    off = 0
    near = 0
    for layer, name, N, K, s in specs:
        W = workloads.weights_torch(N, K, s, outliers=True, device=dev)
        nb = N * K // 2
        codes, cb = logq.logq_quantize(W, 4, float(bases[layer]), codes=arena[off:off + nb], workspace=ws)
        near += boundary_neighbours(torch, W, cb)
        del W
        lin[(layer, name)] = dict(N=N, K=K, codes=codes, cb=cb, off=off, nbytes=nb, seed=s)
        off += nb
    launches = []
    X = workloads.activations_torch(1, spec["shapes"]["q"][1], spec["cfg_seed"], torch.bfloat16, dev)
    for layer in range(n_layers):
        for grp in GROUPS:
            members = [lin[(layer, nm)] for nm in grp]
            K = members[0]["K"]
            assert X.shape[1] == K
            for m in members:
                m["Y"] = torch.empty(1, m["N"], dtype=torch.bfloat16, device=dev)
            launches.append(dict(members=members, K=K, X=X, off=members[0]["off"],
                                 nbytes=sum(m["nbytes"] for m in members)))
            X = members[0]["Y"]                  # the next launch reads this launch's first output
    for i, L in enumerate(launches):          # warm L2 with the next launch's codes
        nxt = launches[(i + 1) % len(launches)]
        L["pf"] = arena[nxt["off"]:nxt["off"] + nxt["nbytes"]]
    stats = {"weights": sum(N * K for _, _, N, K, _ in specs), "boundary_neighbours": int(near)}
    return launches, ws, arena, stats


def boundary_neighbours(torch, W, cb) -> int:
    """Weights of W whose magnitude is a decision boundary of cb (fp32, rounded up)
    or the fp32 value just below one."""
    t = torch.tensor([cb.thresh[j] for j in range(cb.qmax)], dtype=torch.float32, device=W.device)
    cand = torch.cat([t, torch.nextafter(t, torch.zeros_like(t))])
    return int(torch.isin(W.abs(), cand).sum().item())


def linear_bytes_of(launch):
    # the chained step writes bf16 outputs (2 bytes each)
    return sum(linear_bytes(m["N"], m["K"], y_bytes=2) for m in launch["members"])


def time_quantize(logq, torch, dev, reps: int = 2):
    """Quantise the first layer of the model (absmax pass + quantise-and-pack pass)."""
    bases = workloads.layer_bases(MODELS[HEADLINE]["layers"], MODELS[HEADLINE]["cfg_seed"])
    ws = logq.new_workspace(dev)
    shapes = [(layer, N, K, s) for layer, name, N, K, s in model_layers()][:7]  # one layer, all shapes
    Ws = [workloads.weights_torch(N, K, s, outliers=True, device=dev) for _, N, K, s in shapes]
    outs = [torch.empty(N * K // 2, dtype=torch.uint8, device=dev) for _, N, K, _ in shapes]
    nweights = sum(N * K for _, N, K, _ in shapes)
    for W, o, (layer, N, K, s) in zip(Ws, outs, shapes):
        logq.logq_quantize(W, 4, float(bases[layer]), codes=o, workspace=ws)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(reps):
        for W, o, (layer, N, K, s) in zip(Ws, outs, shapes):
            logq.logq_quantize(W, 4, float(bases[layer]), codes=o, workspace=ws)
    dt = (time.perf_counter() - t0) / reps          # logq_quantize synchronises per call
    nbytes = nweights * (4 + 4 + 0.5)
    return {"weights": nweights, "s": dt, "gbs": nbytes / dt / 1e9, "launches_per_pass": 2 * len(shapes),
            "bytes_per_weight": 8.5}


def time_energy(logq, torch, dev, reps: int = 5):
    """Self-calibrating quantisation (Sec. 3.2, Eqs. (3)-(5)) of an 8B gate matrix, eps = 4e-3:
    absmax, the energy selection's three passes over W, then the quantise pass."""
    N, K = workloads.LLAMA_8B_SHAPES["gate"]
    W = workloads.weights_torch(N, K, workloads.layer_seed(4, 0, 4), outliers=True, device=dev)
    ws = logq.new_workspace(dev)
    scratch = torch.empty(logq.logq_energy_scratch_bytes(), dtype=torch.uint8, device=dev)
    codes = torch.empty(N * K // 2, dtype=torch.uint8, device=dev)
    _, cb, wmin = logq.logq_quantize_energy(W, 4, 4e-3, codes=codes, workspace=ws, scratch=scratch)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(reps):
        logq.logq_quantize_energy(W, 4, 4e-3, codes=codes, workspace=ws, scratch=scratch)
    dt = (time.perf_counter() - t0) / reps          # the call synchronises twice
    return {"us": dt * 1e6, "weights": N * K, "wmin": wmin, "base": cb.base, "range": cb.range}


def time_8bit(logq, torch, dev, reps: int = 10):
    """8-bit codes (q_max = 127) on the Llama-3.1-8B gate shape: the batch-1 decode GEMV over
    rotating copies of the codes (more than L2 holds), and the 2048-token prefill GEMM."""
    N, K = workloads.LLAMA_8B_SHAPES["gate"]
    ws = logq.new_workspace(dev)
    W = workloads.weights_torch(N, K, workloads.layer_seed(4, 0, 4), outliers=True, device=dev)
    codes, cb = logq.logq_quantize(W, 8, 1.04, workspace=ws)
    del W
    copies = [codes] + [codes.clone() for _ in range(11)]          # 12 x 58.7 MB
    X = workloads.activations_torch(1, K, 3, torch.bfloat16, dev)
    Y = torch.empty(1, N, dtype=torch.bfloat16, device=dev)
    s = torch.cuda.Stream(dev)
    def launches():
        for c in copies:
            logq.logq_linear(c, cb, X, N, K, y_dtype=torch.bfloat16, Y=Y, workspace=ws)
    with torch.cuda.stream(s):
        launches()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            launches()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()                                     # replays run on the current stream
    for _ in range(reps):
        g.replay()
    e1.record()
    torch.cuda.synchronize()
    t = e0.elapsed_time(e1) * 1e-3 / (reps * len(copies))
    nbytes = linear_bytes(N, K, bits=8, y_bytes=2)
    del copies
    Xp = workloads.activations_torch(PREFILL_TOKENS, K, 4, torch.bfloat16, dev)
    Yp = torch.empty(PREFILL_TOKENS, N, dtype=torch.bfloat16, device=dev)
    logq.logq_linear(codes, cb, Xp, N, K, y_dtype=torch.bfloat16, Y=Yp, workspace=ws)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(3):
        logq.logq_linear(codes, cb, Xp, N, K, y_dtype=torch.bfloat16, Y=Yp, workspace=ws)
    e1.record()
    torch.cuda.synchronize()
    tp = e0.elapsed_time(e1) * 1e-3 / 3
    st, _ = logq.logq_workspace_status(ws)
    assert st == logq.LOGQ_OK
    return {"gemv_us": t * 1e6, "gemv_gbs": nbytes / t / 1e9, "gemv_bytes": nbytes,
            "prefill_us": tp * 1e6, "prefill_tflops": 2.0 * PREFILL_TOKENS * N * K / tp / 1e12}


def time_gptq(logq, torch, dev):
    """GPTQ with the Log_b quantiser on the Llama-3.1-8B q shape (4096 x 4096): Hessian of
    3 K synthetic tokens (neighbouring inputs correlated), the self-calibrated 4-bit codebook;
    the device time of the factor (logq_gptq_factor) and of the quantisation (logq_gptq),
    and the layer loss tr((W - What) H (W - What)^T) against plain rounding with the same
    codebook."""
    import ctypes
    N, K = workloads.LLAMA_8B_SHAPES["q"]
    W = workloads.weights_torch(N, K, workloads.layer_seed(4, 0, 0), outliers=True, device=dev)
    g = torch.Generator(device=dev).manual_seed(MODELS[HEADLINE]["cfg_seed"])
    X = torch.randn(3 * K, K, device=dev, generator=g, dtype=torch.float64)
    X[:, 1:] += 0.5 * X[:, :-1].clone()
    H64 = X.T @ X
    del X
    H = H64.float()
    rtn, cb, _ = logq.logq_quantize_energy(W, 4, 4e-3)
    U = torch.empty(K, K, device=dev)
    dead = torch.empty(K, dtype=torch.uint8, device=dev)
    fscratch = torch.empty(int(logq._lib().logq_gptq_factor_scratch_bytes(K)), dtype=torch.uint8, device=dev)
    codes = torch.empty(N * K // 2, dtype=torch.uint8, device=dev)
    scratch = torch.empty(int(logq._lib().logq_gptq_scratch_bytes(N, K)), dtype=torch.uint8, device=dev)
    def factor():
        logq.gptq_factor(H, 0.01, U=U, dead=dead, scratch=fscratch)
    def run():
        st = logq._lib().logq_gptq(ctypes.c_void_p(W.data_ptr()), N, K, ctypes.c_void_p(U.data_ptr()),
                                   ctypes.c_void_p(dead.data_ptr()), ctypes.byref(cb),
                                   ctypes.c_void_p(codes.data_ptr()), ctypes.c_void_p(scratch.data_ptr()),
                                   scratch.numel(), None)
        assert st == logq.LOGQ_OK
    def timed(fn):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        fn()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1)
    factor()
    run()
    torch.cuda.synchronize()
    factor_ms = timed(factor)
    ms = timed(run)
    lv = torch.tensor(list(cb.level[:16]), dtype=torch.float64, device=dev)
    def loss(c):
        b = c.view(N, K // 2)
        d = W.double() - lv[torch.stack([b & 15, b >> 4], dim=-1).view(N, K).long()]
        return float(((d @ H64) * d).sum())
    upd = sum(2 * N * 128 * (K - j0 - 128) for j0 in range(0, K, 128))
    return {"ms": ms, "factor_ms": factor_ms, "update_tflops": upd / (ms * 1e-3) / 1e12,
            "loss_ratio": loss(codes) / loss(rtn)}


def time_prefill(logq, torch, dev, reps: int = 3):
    """Prefill GEMM at 2048 tokens on one Llama-3.1-8B layer's linears: each shape in a
    launch of its own, and the layer as a model runs it -- q/k/v in one grouped launch
    (they read the same X), o, gate/up in one grouped launch, down."""
    sh = workloads.LLAMA_8B_SHAPES
    T = PREFILL_TOKENS
    groups = {"qkv": ("q", "k", "v"), "gateup": ("gate", "up")}
    # room for split-k partial sums of every launch (k/v alone: too few output tiles)
    wsb = max([logq.logq_linear_workspace_bytes(T, N, K, 4) for N, K in sh.values()] +
              [logq.logq_linear_grouped_workspace_bytes(T, [sh[n][0] for n in g], sh[g[0]][1], 4)
               for g in groups.values()])
    ws = logq.new_workspace(dev, wsb)
    s = torch.cuda.Stream(dev)
    mats = {}
    for pi, name in enumerate(workloads.PROJ_NAMES):
        N, K = sh[name]
        W = workloads.weights_torch(N, K, workloads.layer_seed(4, 0, pi), outliers=True, device=dev)
        codes, cb = logq.logq_quantize(W, 4, 1.5, workspace=ws)
        del W
        mats[name] = (codes, cb, N, K, torch.empty(T, N, dtype=torch.bfloat16, device=dev))
    xs = {K: workloads.activations_torch(T, K, K, torch.bfloat16, dev) for K in {k for _, k in sh.values()}}

    def single(name):
        codes, cb, N, K, Y = mats[name]
        logq.logq_linear(codes, cb, xs[K], N, K, y_dtype=torch.bfloat16, Y=Y, workspace=ws, stream=s)

    def grouped(key):
        names = groups[key]
        K = mats[names[0]][3]
        logq.logq_linear_grouped([(mats[n][0], mats[n][1], mats[n][2], mats[n][4]) for n in names], xs[K], K,
                                 y_dtype=torch.bfloat16, workspace=ws, stream=s)

    def timed(fn):
        # reps back-to-back calls captured in a graph (a split call is two launches:
        # the GEMM and the sum of its k ranges), so host launch gaps stay out
        fn()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            with torch.cuda.graph(g, stream=s):
                for _ in range(reps):
                    fn()
        g.replay()
        torch.cuda.synchronize()
        t = time_replays(torch, g, s, 2) / (2 * reps)
        del g
        return t

    try:
        single("q")
    except logq.LogqError as e:
        if e.status == logq.LOGQ_ERR_UNSUPPORTED:
            return None
        raise
    res, grp = {}, {}
    one_flop, one_t = 0.0, 0.0
    for name in workloads.PROJ_NAMES:
        N, K = sh[name]
        flop = 2.0 * T * N * K
        if name in ("v", "up"):                      # same shapes as k and gate
            t = res["k" if name == "v" else "gate"]["us"] * 1e-6
        else:
            t = timed(lambda: single(name))
            res[name] = {"N": N, "K": K, "us": round(t * 1e6, 2), "tflops": round(flop / t / 1e12, 1)}
        one_flop += flop
        one_t += t
    layer_flop, layer_t = 0.0, 0.0
    for key, names in groups.items():
        t = timed(lambda: grouped(key))
        flop = sum(2.0 * T * sh[n][0] * sh[n][1] for n in names)
        grp[key] = {"N": sum(sh[n][0] for n in names), "K": sh[names[0]][1], "us": round(t * 1e6, 2),
                    "tflops": round(flop / t / 1e12, 1)}
        layer_flop += flop
        layer_t += t
    for name in ("o", "down"):
        layer_flop += 2.0 * T * sh[name][0] * sh[name][1]
        layer_t += res[name]["us"] * 1e-6
    st, _ = logq.logq_workspace_status(ws)
    assert st == logq.LOGQ_OK, "prefill pipeline reported a timeout"
    return {"layers": res, "grouped": grp, "tflops": layer_flop / layer_t / 1e12,
            "tflops_one_launch_per_matrix": one_flop / one_t / 1e12, "layer_us": round(layer_t * 1e6, 1)}


def replica_totals(t_local: float, units_local: float, dist=None, device=None):
    """Whole-job throughput of N independent replicas: every rank processed
    units_local in t_local seconds; the job takes as long as the slowest rank.
    Returns (max time over ranks, total units over ranks)."""
    import torch
    if dist is None or not dist.is_initialized() or dist.get_world_size() == 1:
        return t_local, units_local
    t = torch.tensor([t_local], dtype=torch.float64, device=device)
    u = torch.tensor([units_local], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t.item()), float(u.item())


def step_graph(logq, torch, launches, ws, stream, first_x=None):
    """CUDA graph of one decode step (every launch of the chain, in order)."""
    def run_launch(L, X=None):
        items = [(m["codes"], m["cb"], m["N"], m["Y"]) for m in L["members"]]
        logq.logq_linear_grouped(items, L["X"] if X is None else X, L["K"], y_dtype=torch.bfloat16,
                                 workspace=ws, prefetch=L["pf"], prefetch_bytes=L["pf"].numel(), stream=stream)

    def calls():
        run_launch(launches[0], X=first_x)
        for L in launches[1:]:
            run_launch(L)

    with torch.cuda.stream(stream):
        calls()                                               # warm-up outside capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        with torch.cuda.graph(graph, stream=stream):
            calls()
    return graph


def time_replays(torch, graph, stream, steps: int) -> float:
    """Seconds for `steps` replays, CUDA events on the launching stream."""
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with torch.cuda.stream(stream):
        e0.record(stream)
        for _ in range(steps):
            graph.replay()
        e1.record(stream)
    e1.synchronize()
    return e0.elapsed_time(e1) * 1e-3


def time_decode_1b(logq, torch, dev, steps: int, warmup: int):
    """The Llama-3.2-1B-shaped decode step, measured like the headline step."""
    launches, ws, arena, _ = build_decode_model(logq, torch, dev, "1b")
    stream = torch.cuda.Stream(device=dev)
    graph = step_graph(logq, torch, launches, ws, stream)
    for _ in range(warmup):
        graph.replay()
    torch.cuda.synchronize()
    t = time_replays(torch, graph, stream, steps)
    st, _ = logq.logq_workspace_status(ws)
    assert st == logq.LOGQ_OK
    step_bytes = sum(linear_bytes_of(L) for L in launches)
    del graph, arena
    return {"gbs": step_bytes * steps / t / 1e9, "ms_per_step": t / steps * 1e3, "launches": len(launches),
            "bytes_per_step": step_bytes}


def time_skinny(logq, torch, dev, batches=(1, 4, 16), reps: int = 10):
    """Decode GEMV / skinny GEMM on the Llama-3.1-8B gate shape (14336 x 4096, 4-bit) at
    several batch sizes, over rotating copies of the codes (more than L2 holds)."""
    N, K = workloads.LLAMA_8B_SHAPES["gate"]
    ws = logq.new_workspace(dev, max(logq.logq_linear_workspace_bytes(B, N, K, 4) for B in batches))
    W = workloads.weights_torch(N, K, workloads.layer_seed(3, 0, 4), outliers=True, device=dev)
    codes, cb = logq.logq_quantize(W, 4, 1.5, workspace=ws)
    del W
    copies = [codes] + [codes.clone() for _ in range(11)]          # 12 x 29.4 MB
    s = torch.cuda.Stream(dev)
    out = {}
    for B in batches:
        X = workloads.activations_torch(B, K, 3, torch.bfloat16, dev)
        Y = torch.empty(B, N, dtype=torch.bfloat16, device=dev)

        def launches():
            for c in copies:
                logq.logq_linear(c, cb, X, N, K, y_dtype=torch.bfloat16, Y=Y, workspace=ws, stream=s)
        with torch.cuda.stream(s):
            launches()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            with torch.cuda.graph(g, stream=s):
                launches()
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        t = time_replays(torch, g, s, reps) / (reps * len(copies))
        out[B] = {"us": t * 1e6, "gbs": linear_bytes(N, K, B=B, y_bytes=2) / t / 1e9,
                  "tflops": 2.0 * B * N * K / t / 1e12}
        del g
    st, _ = logq.logq_workspace_status(ws)
    assert st == logq.LOGQ_OK
    return out


def fp32_peak_tflops(sm_mhz: float) -> float:
    """CUDA-core fp32 FMA rate: SMs x 128 lanes x 2 flops x clock."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sms * 128 * 2 * sm_mhz * 1e6 / 1e12


def run_ours(args):
    import torch
    import paper_2607_01127_gb300 as logq

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    launches, ws, arena, stats = build_decode_model(logq, torch, dev)
    step_bytes = sum(linear_bytes_of(L) for L in launches)
    n_linears = sum(len(L["members"]) for L in launches)
    launches_per_step = len(launches)
    stream = torch.cuda.Stream(device=dev)
    graph = step_graph(logq, torch, launches, ws, stream)
    for _ in range(args.warmup):
        graph.replay()
    barrier()
    # one event before the first replay and one after each: the whole region's
    # time (the value) and each step's (median and best)
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    e0, e1 = evs[0], evs[-1]
    with ClockSampler(local) as clocks:
        time.sleep(0.25)
        barrier()
        with torch.cuda.stream(stream):
            e0.record(stream)
            for i in range(args.steps):
                graph.replay()
                evs[i + 1].record(stream)
        barrier()
        time.sleep(0.25)
    per_step = sorted(evs[i].elapsed_time(evs[i + 1]) for i in range(args.steps))
    t, total_bytes = replica_totals(e0.elapsed_time(e1) * 1e-3, step_bytes * args.steps, dist, dev)
    value = total_bytes / t / 1e9
    ms_per_step = t / args.steps * 1e3
    st, _ = logq.logq_workspace_status(ws, stream)
    assert st == logq.LOGQ_OK, "decode step reported a device-side timeout"

    final = launches[-1]["members"][0]["Y"]
    y_device = final.clone()

    # e2e: every step copies its input activation in from pinned host memory
    # and reads its final output back (the chain's intermediate activations stay
    # on the device, as in a model's decode step)
    x0 = launches[0]["X"]
    xh = torch.empty(x0.numel(), dtype=torch.bfloat16, pin_memory=True)
    yh = torch.empty(final.numel(), dtype=torch.bfloat16, pin_memory=True)
    xh.copy_(x0.view(-1).cpu())
    xd = torch.empty_like(x0)
    with torch.cuda.stream(stream):
        xd.copy_(xh.view(1, -1), non_blocking=True)
    g2 = step_graph(logq, torch, launches, ws, stream, first_x=xd)
    h2d, d2h = xh.numel() * 2, yh.numel() * 2
    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            xd.copy_(xh.view(1, -1), non_blocking=True)
            g2.replay()
            yh.copy_(final.view(-1), non_blocking=True)
        barrier()
        f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        for _ in range(args.steps):
            xd.copy_(xh.view(1, -1), non_blocking=True)
            g2.replay()
            yh.copy_(final.view(-1), non_blocking=True)
        f1.record(stream)
    barrier()
    t2, total_bytes2 = replica_totals(f0.elapsed_time(f1) * 1e-3, step_bytes * args.steps, dist, dev)
    e2e_value = total_bytes2 / t2 / 1e9
    # the step is deterministic: the end-to-end output equals the device-resident run
    assert torch.equal(yh.view(1, -1).to(dev), y_device)
    assert bool(torch.isfinite(y_device.float()).all())
    del graph, g2, arena, launches

    pk, pk_kind = peaks()
    gemv_bytes_per_launch = step_bytes / launches_per_step
    achieved = gemv_bytes_per_launch / (t / args.steps / launches_per_step) / 1e9
    tr = traffic_for("gemv_kernel_8b_step", "paper_2607_01127_gb300/csrc/gemv.cu")
    line = {
        "metric": METRIC, "value": round(value, 1), "unit": "GB/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_per_step, 4),
        "step_ms": {"median": round(per_step[len(per_step) // 2], 4), "best": round(per_step[0], 4),
                    "worst": round(per_step[-1], 4), "note": "this rank's steps, one event pair each"},
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "global_batch": 1 * world, "linears_per_step": n_linears,
                   "launches_per_step": launches_per_step,
                   "bytes_per_step": step_bytes, "bits": 4,
                   "l2": f"inputs larger than L2 ({step_bytes / 1e9:.2f} GB of codes per step vs 126 MB L2)",
                   "parallelism": f"replicas x{world}" if world > 1 else "single GPU",
                   "graph": "one CUDA graph per step: per layer qkv | o | gate+up | down launches "
                            "(linears that read the same activations share a launch), chained: each "
                            "launch reads the previous launch's bf16 output; programmatic dependent "
                            "launch, each launch warms L2 with the next launch's codes when they are "
                            "under 4 MiB"},
        "e2e": {"value": round(e2e_value, 1), "unit": "GB/s", "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": d2h},
        "gpu_launches": launches_per_step * args.steps,
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": pk["hbm_gbs"], "unit": "GB/s",
                     "frac": round(achieved / pk["hbm_gbs"], 4), "peak_source": pk_kind,
                     "traffic": tr, "kernel": "gemv_kernel, batch 1, 4-bit (the 128 launches of the 8B step: 8-warp CTAs, two per SM)",
                     "algorithmic_bytes_per_launch": round(gemv_bytes_per_launch, 1),
                     "frac_of_8TBs": round(achieved / 8000.0, 4)},
        "boundary_codes": {"within_1ulp_of_a_boundary": stats["boundary_neighbours"],
                           "weights": stats["weights"],
                           "note": "weights whose |w| is an fp32 decision boundary (rounded up) or the float "
                                   "just below one: the only codes that depend on how a boundary is rounded"},
        "clocks": clocks.summary(),
    }
    if rank == 0:
        try:
            d1 = time_decode_1b(logq, torch, dev, min(args.steps, 200), args.warmup)
            line["decode_1b"] = {"gbs": round(d1["gbs"], 1), "frac": round(d1["gbs"] / pk["hbm_gbs"], 4),
                                 "ms_per_step": round(d1["ms_per_step"], 4), "launches_per_step": d1["launches"],
                                 "bytes_per_step": d1["bytes_per_step"],
                                 "note": MODELS["1b"]["name"] + ", measured like the headline step"}
        except Exception as e:
            line["decode_1b"] = {"error": str(e)[:200]}
        try:
            sk = time_skinny(logq, torch, dev)
            mhz = (line["clocks"] or {}).get("sm_mhz") or 2070.0
            fp32 = fp32_peak_tflops(mhz)
            line["skinny"] = {
                f"B{B}": {"us": round(v["us"], 2), "gbs": round(v["gbs"], 1),
                          "hbm_frac": round(v["gbs"] / pk["hbm_gbs"], 4), "tflops": round(v["tflops"], 2),
                          "path": "decode kernel (lookups, warp-level tensor-core multiply-adds)",
                          "fp32_frac": round(v["tflops"] / fp32, 4)} for B, v in sk.items()}
            line["skinny"]["fp32_peak_tflops"] = round(fp32, 1)
            line["skinny"]["note"] = ("Llama-3.1-8B gate 14336x4096, 4-bit, bf16 in/out, 12 rotating code copies "
                                      "(beyond L2), workspace of logq_linear_workspace_bytes; fp32_frac against "
                                      "SMs x 128 lanes x 2 flops x the median SM clock of the headline run (the "
                                      "CUDA cores' fp32 rate, which the kernel does not use)")
        except Exception as e:
            line["skinny"] = {"error": str(e)[:200]}
    if rank == 0:
        try:
            q = time_quantize(logq, torch, dev)
            line["quantize"] = {"gbs": round(q["gbs"], 1), "unit": "GB/s",
                                "frac": round(q["gbs"] / pk["hbm_gbs"], 4),
                                "weights_per_s": round(q["weights"] / q["s"], 1),
                                "note": "absmax + quantise-and-pack of one layer's 7 linears, "
                                        "8.5 B/weight algorithmic, host sync per call"}
        except Exception as e:  # the headline line must still print
            line["quantize"] = {"error": str(e)[:200]}
        try:
            en = time_energy(logq, torch, dev)
            line["energy_quantize"] = {
                "us_per_call": round(en["us"], 1), "weights": en["weights"],
                "gbs_of_w": round(en["weights"] * 4 / (en["us"] * 1e-6) / 1e9, 1),
                "wmin": en["wmin"], "base": en["base"], "range": en["range"], "eps": 4e-3,
                "note": "Llama-3.1-8B gate 14336x4096: 3 selection passes + quantise, "
                        "host sync twice per call"}
        except Exception as e:
            line["energy_quantize"] = {"error": str(e)[:200]}
        try:
            e8 = time_8bit(logq, torch, dev)
            line["bits8"] = {
                "gemv_us": round(e8["gemv_us"], 2), "gemv_gbs": round(e8["gemv_gbs"], 1),
                "gemv_frac": round(e8["gemv_gbs"] / pk["hbm_gbs"], 4),
                "prefill_tflops": round(e8["prefill_tflops"], 1),
                "prefill_frac": round(e8["prefill_tflops"] / pk["bf16_tflops"], 4),
                "note": "8-bit codes, Llama-3.1-8B gate 14336x4096: batch-1 decode GEMV over 12 rotating "
                        "copies of the codes (0.70 GB, beyond L2), bf16 output; prefill with 2048 tokens"}
        except Exception as e:
            line["bits8"] = {"error": str(e)[:200]}
        try:
            gq = time_gptq(logq, torch, dev)
            line["gptq"] = {"ms": round(gq["ms"], 2), "factor_ms": round(gq["factor_ms"], 1),
                            "update_tflops": round(gq["update_tflops"], 2),
                            "loss_vs_rounding": round(gq["loss_ratio"], 4),
                            "note": "4-bit GPTQ of a Llama-3.1-8B q matrix (4096x4096), Hessian of 12288 synthetic "
                                    "tokens, self-calibrated codebook; ms = logq_gptq (column blocks + fp32 "
                                    "updates), factor_ms = logq_gptq_factor (fp32 Cholesky + triangular inverse, "
                                    "one host sync)"}
        except Exception as e:
            line["gptq"] = {"error": str(e)[:200]}
        try:
            pf = time_prefill(logq, torch, dev)
            if pf is not None:
                line["prefill"] = {"tflops": round(pf["tflops"], 1), "unit": "TFLOP/s",
                                   "peak": pk["bf16_tflops"],
                                   "frac": round(pf["tflops"] / pk["bf16_tflops"], 4),
                                   "layer_us": pf["layer_us"], "grouped": pf["grouped"],
                                   "layers": pf["layers"], "tokens": PREFILL_TOKENS,
                                   "tflops_one_launch_per_matrix": round(pf["tflops_one_launch_per_matrix"], 1),
                                   "note": "tflops: one Llama-3.1-8B layer's linears as a model runs them "
                                           "(q/k/v one grouped launch, o, gate/up one grouped launch, down); "
                                           "layers: each shape in a launch of its own"}
            else:
                line["prefill"] = None
        except Exception as e:
            line["prefill"] = {"error": str(e)[:200]}
        if world == 1 and not args.no_cpu_baseline:
            line["cpu_baseline"] = cpu_baseline()
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()


CASES = ("decode_layers_8b", "decode_step_1b", "skinny_gate_8b", "gemv_gateup_1b", "gemv_gate_8b", "prefill_q_8b",
         "prefill8_q_8b", "prefill_gate_8b_33", "prefill_qkv_8b", "quantize_gate_8b", "energy_gate_8b",
         "gemv3_gate_8b", "gemv8_gate_8b", "gptq_q_8b", "gptq_update_q_8b", "quantize3_gate_8b")


def run_case(name: str):
    """One small workload run twice (for a profiler capture of the second run):
    the gate+up launch of the 1B decode step, the 8B gate GEMV, the 8B q-shaped
    prefill GEMM (2048 tokens, 4 or 8 bits), the gate one at 33 tokens and the grouped q/k/v one,
    the quantisation of an 8B gate matrix, its
    self-calibrating (energy-range) quantisation, the 3- and 8-bit gate GEMVs and 4-bit
    GPTQ of an 8B q matrix (factor and quantisation; or the quantisation alone with a
    fixed upper-triangular factor standing in for U)."""
    import torch
    import paper_2607_01127_gb300 as logq
    dev = torch.device("cuda", 0)
    ws = logq.new_workspace(dev)
    if name == "decode_layers_8b":
        # the first two layers of the 8B decode step (8 chained launches, each
        # warming L2 with the next one's codes), run twice
        launches, ws, arena, _ = build_decode_model(logq, torch, dev, layers=2)
        stream = torch.cuda.Stream(device=dev)
        for _ in range(2):
            step_graph(logq, torch, launches, ws, stream)
        torch.cuda.synchronize()
    elif name == "decode_step_1b":
        # the Llama-3.2-1B decode step (64 chained launches), run twice
        launches, ws, arena, _ = build_decode_model(logq, torch, dev, "1b")
        stream = torch.cuda.Stream(device=dev)
        for _ in range(2):
            step_graph(logq, torch, launches, ws, stream)
        torch.cuda.synchronize()
    elif name == "skinny_gate_8b":
        # the 8B gate at batch 4 and 16, twice each
        N, K = workloads.LLAMA_8B_SHAPES["gate"]
        c = logq.logq_quantize(workloads.weights_torch(N, K, 13, True, dev), 4, 1.5, workspace=ws)
        for B in (4, 16):
            X = workloads.activations_torch(B, K, 1, torch.bfloat16, dev)
            for _ in range(2):
                logq.logq_linear(c[0], c[1], X, N, K, y_dtype=torch.bfloat16, workspace=ws)
    elif name == "gemv_gateup_1b":
        K = 2048
        a = logq.logq_quantize(workloads.weights_torch(8192, K, 11, True, dev), 4, 1.4, workspace=ws)
        b = logq.logq_quantize(workloads.weights_torch(8192, K, 12, True, dev), 4, 1.6, workspace=ws)
        X = workloads.activations_torch(1, K, 1, torch.bfloat16, dev)
        for _ in range(2):
            logq.logq_linear_grouped([(a[0], a[1], 8192, None), (b[0], b[1], 8192, None)], X, K, workspace=ws)
    elif name == "gemv_gate_8b":
        N, K = workloads.LLAMA_8B_SHAPES["gate"]
        c = logq.logq_quantize(workloads.weights_torch(N, K, 13, True, dev), 4, 1.5, workspace=ws)
        X = workloads.activations_torch(1, K, 1, torch.bfloat16, dev)
        for _ in range(2):
            logq.logq_linear(c[0], c[1], X, N, K, workspace=ws)
    elif name in ("prefill_q_8b", "prefill8_q_8b", "prefill_gate_8b_33"):
        N, K = workloads.LLAMA_8B_SHAPES["gate" if "gate" in name else "q"]
        bits, base = (8, 1.04) if "8_q" in name else (4, 1.5)
        c = logq.logq_quantize(workloads.weights_torch(N, K, 14, True, dev), bits, base, workspace=ws)
        X = workloads.activations_torch(33 if name.endswith("_33") else PREFILL_TOKENS, K, 2, torch.bfloat16, dev)
        for _ in range(2):
            logq.logq_linear(c[0], c[1], X, N, K, y_dtype=torch.bfloat16, workspace=ws)
    elif name == "prefill_qkv_8b":
        K = workloads.LLAMA_8B_SHAPES["q"][1]
        items = []
        for i, proj in enumerate(("q", "k", "v")):
            N = workloads.LLAMA_8B_SHAPES[proj][0]
            c = logq.logq_quantize(workloads.weights_torch(N, K, 20 + i, True, dev), 4, 1.5, workspace=ws)
            items.append((c[0], c[1], N, None))
        X = workloads.activations_torch(PREFILL_TOKENS, K, 2, torch.bfloat16, dev)
        for _ in range(2):
            logq.logq_linear_grouped(items, X, K, y_dtype=torch.bfloat16, workspace=ws)
    elif name == "quantize_gate_8b":
        N, K = workloads.LLAMA_8B_SHAPES["gate"]
        W = workloads.weights_torch(N, K, 15, True, dev)
        for _ in range(2):
            logq.logq_quantize(W, 4, 1.5, workspace=ws)
    elif name == "quantize3_gate_8b":
        N, K = workloads.LLAMA_8B_SHAPES["gate"]
        W = workloads.weights_torch(N, K, 15, True, dev)
        for _ in range(2):
            logq.logq_quantize(W, 3, 1.8, workspace=ws)
    elif name in ("gemv3_gate_8b", "gemv8_gate_8b"):
        N, K = workloads.LLAMA_8B_SHAPES["gate"]
        bits, base = (3, 1.8) if name.startswith("gemv3") else (8, 1.04)
        c = logq.logq_quantize(workloads.weights_torch(N, K, 13, True, dev), bits, base, workspace=ws)
        X = workloads.activations_torch(1, K, 1, torch.bfloat16, dev)
        for _ in range(2):
            logq.logq_linear(c[0], c[1], X, N, K, workspace=ws)
    elif name == "energy_gate_8b":
        N, K = workloads.LLAMA_8B_SHAPES["gate"]
        W = workloads.weights_torch(N, K, 15, True, dev)
        for _ in range(2):
            logq.logq_quantize_energy(W, 4, 4e-3, workspace=ws)
    elif name == "gptq_q_8b":
        N, K = workloads.LLAMA_8B_SHAPES["q"]
        W = workloads.weights_torch(N, K, 16, True, dev)
        g = torch.Generator(device=dev).manual_seed(17)
        X = torch.randn(2 * K, K, device=dev, generator=g)
        H = X.T @ X
        del X
        cb = logq.logq_build_codebook(4, 1.5, float(W.abs().max()))
        for _ in range(2):
            logq.logq_gptq(W, H, cb)
    elif name == "gptq_update_q_8b":
        import ctypes
        N, K = workloads.LLAMA_8B_SHAPES["q"]
        W = workloads.weights_torch(N, K, 16, True, dev)
        U = torch.triu(torch.full((K, K), 1e-3, device=dev)) + torch.eye(K, device=dev)
        cb = logq.logq_build_codebook(4, 1.5, float(W.abs().max()))
        codes = torch.empty(N * K // 2, dtype=torch.uint8, device=dev)
        scratch = torch.empty(int(logq._lib().logq_gptq_scratch_bytes(N, K)), dtype=torch.uint8, device=dev)
        for _ in range(2):
            st = logq._lib().logq_gptq(ctypes.c_void_p(W.data_ptr()), N, K, ctypes.c_void_p(U.data_ptr()), None,
                                       ctypes.byref(cb), ctypes.c_void_p(codes.data_ptr()),
                                       ctypes.c_void_p(scratch.data_ptr()), scratch.numel(), None)
            assert st == logq.LOGQ_OK
    torch.cuda.synchronize()
    st, _ = logq.logq_workspace_status(ws)
    assert st == logq.LOGQ_OK
    print("case", name, "ok")


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--case", choices=CASES, help="run one small profiling case and exit")
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.case:
        run_case(args.case)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
