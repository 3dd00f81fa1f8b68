"""Performance cases of the library: what its users run, through the public entry points.

A user of the library quantises a model's linear layers once (logq_quantize, or
logq_quantize_energy / logq_gptq for a calibrated codebook) and then runs the
layers: at small batches while decoding (captured once as a CUDA graph and
replayed for every token, as serving programs do), at hundreds to thousands of
tokens while reading a prompt.  A case names one such call or step:

  linear    one logq_linear call, the smallest unit (latency and launches count)
  decode    the linears of some layers of a Llama-shaped model at a small batch:
            q/k/v and gate/up grouped, one launch after the other, each layer on
            its own normalised input, a captured graph
  prefill   the linears of one layer over a prompt, direct calls
  quantize  logq_quantize of one layer's matrices
  energy    logq_quantize_energy of one matrix
  factor    gptq_factor of one Hessian
  gptq      logq_gptq of one matrix (factor, column loop and compensations)

Weights are Student-t(4) * 0.02 with 0.1 % of the entries 20 times larger, the
heavy-tailed histogram of trained weights; activations are N(0, 1).
"""
from __future__ import annotations

import math

import torch

import paper_2607_01127_gb300 as logq
from paper_2607_01127_gb300 import workloads

SHAPES = {"1b": workloads.LLAMA_1B_SHAPES, "8b": workloads.LLAMA_8B_SHAPES}
GROUPS = (("q", "k", "v"), ("o",), ("gate", "up"), ("down",))
# a group's input within a layer: the layer's normalised input, or the output of a projection before it
# (it stands in for what attention and the activation function make of that output)
SOURCE = {"q": None, "o": "q", "gate": "o", "down": "gate"}
DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
DEVICE = "cuda"


# ------------------------------------------------------------------ cases ---

def listed():
    return [
        # the smallest call: one fp16 token through one 512 x 2048 layer
        dict(name="linear_512x2048_b1_f16", kind="linear", N=512, K=2048, batch=1, bits=4, base=2.7, x="f16", y="f32"),
        # one token of a Llama-3.2-1B-shaped model, all 16 layers: launch-bound decode
        dict(name="decode_1b_b1", kind="decode", model="1b", layers=16, batch=1, bits=4, base=2.7, x="bf16"),
        # one token of a Llama-3.1-8B-shaped model, all 32 layers: the headline decode step
        dict(name="decode_8b_b1", kind="decode", model="8b", layers=32, batch=1, bits=4, base=2.7, x="bf16"),
        # four and sixteen sequences decoding together
        dict(name="decode_8b_b4", kind="decode", model="8b", layers=4, batch=4, bits=4, base=2.7, x="bf16"),
        dict(name="decode_8b_b16", kind="decode", model="8b", layers=4, batch=16, bits=4, base=2.7, x="bf16"),
        # 3-bit weights, fp16 activations
        dict(name="decode_8b_3bit_b1_f16", kind="decode", model="8b", layers=4, batch=1, bits=3, base=8.0, x="f16"),
        # a 2048-token prompt
        dict(name="prefill_8b_2048", kind="prefill", model="8b", tokens=2048, bits=4, base=2.7, x="bf16"),
        # a shorter prompt of an odd length, 8-bit weights
        dict(name="prefill_1b_517_8bit", kind="prefill", model="1b", tokens=517, bits=8, base=1.08, x="bf16"),
        # quantising a model, layer by layer, ranges from the weights
        dict(name="quantize_8b_layer", kind="quantize", model="8b", bits=4, base=2.0, given=False),
        # the self-calibrating quantiser on a layer's largest matrix
        dict(name="energy_8b_gate", kind="energy", N=14336, K=4096, bits=4, eps=4e-3),
        # calibration: the inverse-Hessian factor of a layer's inputs, and a whole GPTQ call
        dict(name="factor_4096", kind="factor", K=4096),
        dict(name="gptq_8b_q", kind="gptq", N=4096, K=4096, bits=4, eps=4e-3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _k(rng, hi):
    """An input width: a multiple of 128, as the layouts require."""
    return 128 * _log_int(rng, 1, hi // 128)


def _base(rng, bits, flat=False):
    """Bases around those the self-calibration derives (flatter ones leave nearly every weight of a heavy-tailed
    matrix 0: the quantiser alone is also run with those)."""
    lo, hi = {3: (5.0, 11.0), 4: (2.0, 3.0), 8: (1.05, 1.1)}[bits]
    if flat:
        lo = {3: 1.25, 4: 1.2, 8: 1.02}[bits]
    return round(rng.uniform(lo, hi), 3)


def draw(rng):
    kind = rng.choice(["linear", "linear", "decode", "decode", "decode", "prefill", "prefill",
                       "quantize", "energy", "factor", "gptq"])
    bits = rng.choice([3, 4, 4, 4, 8])
    if kind == "linear":
        x = rng.choice(["bf16", "f16"])
        return dict(kind=kind, N=_log_int(rng, 1, 16384), K=_k(rng, 14336), batch=_log_int(rng, 1, 64), bits=bits,
                    base=_base(rng, bits), x=x, y=rng.choice(["f32", x]))
    if kind == "decode":
        model = rng.choice(["1b", "8b"])
        return dict(kind=kind, model=model, layers=rng.randint(6, 16) if model == "1b" else rng.randint(2, 8),
                    batch=_log_int(rng, 1, 64), bits=bits, base=_base(rng, bits), x=rng.choice(["bf16", "bf16", "f16"]))
    if kind == "prefill":
        return dict(kind=kind, model=rng.choice(["1b", "8b"]), tokens=_log_int(rng, 65, 2047), bits=bits,
                    base=_base(rng, bits), x=rng.choice(["bf16", "bf16", "f16"]))
    if kind == "quantize":
        return dict(kind=kind, model=rng.choice(["1b", "8b"]), bits=bits, base=_base(rng, bits, flat=True),
                    given=rng.choice([False, False, True]))
    if kind == "energy":
        return dict(kind=kind, N=_log_int(rng, 16, 14336), K=_k(rng, 4096), bits=bits,
                    eps=1e-6 if bits == 8 else 4e-3)
    if kind == "factor":
        return dict(kind=kind, K=_k(rng, 4096))
    return dict(kind=kind, N=_log_int(rng, 64, 4096), K=_k(rng, 4096), bits=rng.choice([4, 4, 8]), eps=4e-3)


# ----------------------------------------------------------------- inputs ---

def _generator(seed, *more):
    g = torch.Generator(device=DEVICE)
    for m in more:
        seed = seed * 1009 + m + 1
    g.manual_seed(seed % (1 << 62))
    return g


def _weights(N, K, seed, *more):
    """fp32 [N, K]: Student-t(4) * 0.02, 0.1 % of the entries 20 times larger.  (The chi-square of 4 degrees of
    freedom is twice a sum of two exponentials.)"""
    g = _generator(seed, 1, *more)
    w = torch.randn(N, K, device=DEVICE, generator=g)
    e = torch.empty(N, K, device=DEVICE)
    chi = torch.empty(N, K, device=DEVICE).exponential_(generator=g).add_(e.exponential_(generator=g)).mul_(0.5)
    w.div_(chi.sqrt_()).mul_(workloads.WEIGHT_SCALE)
    hot = e.uniform_(generator=g) < workloads.OUTLIER_FRACTION
    return torch.where(hot, w * workloads.OUTLIER_FACTOR, w)


def _activations(shape, dtype, seed, *more):
    return torch.randn(shape, device=DEVICE, generator=_generator(seed, 2, *more)).to(dtype)


def _hessian(K, seed):
    """H = X^T X of 3 K calibration tokens, neighbouring inputs correlated, two inputs that never fire."""
    X = torch.randn(3 * K, K, device=DEVICE, generator=_generator(seed, 3))
    X[:, 1:] += 0.5 * X[:, :-1].clone()
    if K >= 256:
        X[:, [K // 5, K - 7]] = 0
    H = X.T @ X
    return (H + H.T) * 0.5


def _layer_base(case, layer):
    """Bases differ a little from layer to layer, as calibrated ones do."""
    return 1.0 + (case["base"] - 1.0) * (1.0 + 0.04 * math.cos(2.4 * layer))


def _layers(case):
    return case.get("layers", 1)


def _quantised(case, seed, ws):
    """Codes and codebooks of every projection, the codes of a step in one buffer in launch order."""
    shapes, bits = SHAPES[case["model"]], case["bits"]
    sizes = [logq.logq_packed_bytes(N, K, bits) for N, K in shapes.values()]
    arena = torch.empty(_layers(case) * sum(sizes), dtype=torch.uint8, device=DEVICE)
    mats, off = {}, 0
    for layer in range(_layers(case)):
        for p, (name, (N, K)) in enumerate(shapes.items()):
            n = logq.logq_packed_bytes(N, K, bits)
            codes, cb = logq.logq_quantize(_weights(N, K, seed, layer, p), bits, _layer_base(case, layer),
                                           codes=arena[off:off + n], workspace=ws)
            mats[layer, name] = (codes, cb, N, K, off, n)
            off += n
    return arena, mats


def _workspace(batch, case):
    """One workspace for every launch of a step."""
    need = [logq.logq_linear_grouped_workspace_bytes(batch, [SHAPES[case["model"]][n][0] for n in grp],
                                                     SHAPES[case["model"]][grp[0]][1], case["bits"])
            for grp in GROUPS]
    return logq.new_workspace(DEVICE, max(need))


def _prepare_decode(case, seed):
    shapes, dtype, B, L = SHAPES[case["model"]], DTYPES[case["x"]], case["batch"], case["layers"]
    ws = _workspace(B, case)
    arena, mats = _quantised(case, seed, ws)
    X = _activations((L, B, shapes["q"][1]), dtype, seed)
    Y = {name: torch.empty(L, B, N, dtype=dtype, device=DEVICE) for name, (N, _) in shapes.items()}
    launches = []
    for layer in range(L):
        for grp in GROUPS:
            first = mats[layer, grp[0]]
            src = SOURCE[grp[0]]
            launches.append(([(*mats[layer, n][:3], Y[n][layer]) for n in grp], first[3],
                             X[layer] if src is None else Y[src][layer],
                             (first[4], sum(mats[layer, n][5] for n in grp))))

    def step():
        for i, (items, K, x, _) in enumerate(launches):
            off, n = launches[(i + 1) % len(launches)][3]     # the next launch's codes, to warm L2 with
            logq.logq_linear_grouped(items, x, K, y_dtype=dtype, workspace=ws, prefetch=arena[off:off + n],
                                     prefetch_bytes=n)

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    return dict(case=case, graph=graph, Y=Y, keep=(arena, mats, X, ws, launches, stream))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "decode":
        return _prepare_decode(case, seed)
    if kind == "prefill":
        ws = _workspace(case["tokens"], case)
        arena, mats = _quantised(case, seed, ws)
        X = _activations((case["tokens"], SHAPES[case["model"]]["q"][1]), DTYPES[case["x"]], seed)
        return dict(case=case, mats=mats, X=X, ws=ws)
    if kind == "linear":
        N, K, B, bits = case["N"], case["K"], case["batch"], case["bits"]
        ws = logq.new_workspace(DEVICE, logq.logq_linear_workspace_bytes(B, N, K, bits))
        codes, cb = logq.logq_quantize(_weights(N, K, seed), bits, case["base"], workspace=ws)
        return dict(case=case, codes=codes, cb=cb, ws=ws, X=_activations((B, K), DTYPES[case["x"]], seed))
    if kind == "quantize":
        W = {name: _weights(N, K, seed, p) for p, (name, (N, K)) in enumerate(SHAPES[case["model"]].items())}
        # a range chosen beforehand clamps the largest weights
        ranges = {n: 0.8 * float(w.abs().max()) if case["given"] else 0.0 for n, w in W.items()}
        return dict(case=case, W=W, ranges=ranges, ws=logq.new_workspace(DEVICE))
    if kind == "energy":
        return dict(case=case, W=_weights(case["N"], case["K"], seed), ws=logq.new_workspace(DEVICE),
                    scratch=torch.empty(logq.logq_energy_scratch_bytes(), dtype=torch.uint8, device=DEVICE))
    if kind == "factor":
        return dict(case=case, H=_hessian(case["K"], seed))
    W = _weights(case["N"], case["K"], seed)
    _, cb, _ = logq.logq_quantize_energy(W, case["bits"], case["eps"])
    return dict(case=case, W=W, H=_hessian(case["K"], seed), cb=cb)


# -------------------------------------------------------------------- run ---

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "decode":
        s["graph"].replay()
        return s["Y"]
    if kind == "linear":
        return logq.logq_linear(s["codes"], s["cb"], s["X"], case["N"], case["K"], y_dtype=DTYPES[case["y"]],
                                workspace=s["ws"])
    if kind == "prefill":
        Y, dtype = {}, DTYPES[case["x"]]
        for grp in GROUPS:
            src = SOURCE[grp[0]]
            x = s["X"] if src is None else Y[src]
            outs = logq.logq_linear_grouped([(*s["mats"][0, n][:3], None) for n in grp], x, s["mats"][0, grp[0]][3],
                                            y_dtype=dtype, workspace=s["ws"])
            Y.update(zip(grp, outs))
        return Y
    if kind == "quantize":
        out = {}
        for name, W in s["W"].items():
            codes, cb = logq.logq_quantize(W, case["bits"], case["base"], s["ranges"][name], workspace=s["ws"])
            out[name] = (codes, cb.range)
        return out
    if kind == "energy":
        codes, cb, wmin = logq.logq_quantize_energy(s["W"], case["bits"], case["eps"], workspace=s["ws"],
                                                    scratch=s["scratch"])
        return codes, cb.range, cb.base, wmin
    if kind == "factor":
        return logq.gptq_factor(s["H"])
    return logq.logq_gptq(s["W"], s["H"], s["cb"])


# ------------------------------------------------------------------- work ---

def work(case):
    kind = case["kind"]
    packed = lambda N, K: N * K * case["bits"] / 8  # noqa: E731
    if kind in ("decode", "prefill"):
        B = case.get("batch", case.get("tokens"))
        shapes = SHAPES[case["model"]]
        nbytes = sum(packed(N, K) + 2 * B * N for N, K in shapes.values())
        nbytes += sum(2 * B * shapes[grp[0]][1] for grp in GROUPS)
        return {"bytes": _layers(case) * nbytes, "flops": _layers(case) * sum(2 * B * N * K for N, K in shapes.values())}
    if kind == "quantize":
        return {"bytes": sum(4 * N * K + packed(N, K) for N, K in SHAPES[case["model"]].values()), "flops": 0}
    K = case["K"]
    if kind == "factor":     # a Cholesky factorisation and a triangular inverse
        return {"bytes": 8 * K * K, "flops": 2 * K ** 3 / 3}
    N = case["N"]
    if kind == "linear":
        B = case["batch"]
        return {"bytes": packed(N, K) + 2 * B * K + (4 if case["y"] == "f32" else 2) * B * N, "flops": 2 * B * N * K}
    if kind == "energy":
        return {"bytes": 4 * N * K + packed(N, K), "flops": 0}
    return {"bytes": 4 * N * K + 4 * K * K + packed(N, K), "flops": 2 * K ** 3 / 3 + N * K * K}


def tolerance(case):
    kind = case["kind"]
    if kind in ("quantize", "energy"):
        return "exact"
    if kind == "gptq":
        # a weight that two summation orders put on different sides of a boundary changes the rest of its row:
        # against 64 bits 5e-5 (4-bit) to 6e-4 (8-bit) of the bytes of large matrices, up to a row of small ones
        return {"rel": 1e-5, "differ": min(0.01, 2.4e-3 + 2.0 / case["N"])}
    if kind == "factor":
        return {"rel": 2e-6}         # 3e-7 to 5.5e-7 off 64 bits
    if kind == "linear":             # fp32 sums; a 16-bit output may round to the neighbour
        return {"rel": {"f32": 2e-6, "bf16": 8e-3, "f16": 1e-3}[case["y"]]}
    # up to four roundings to 16 bits, one after the other: bf16 0.0033 off 64 bits, f16 an eighth of that
    return {"rel": {"bf16": 1.2e-2, "f16": 1.5e-3}[case["x"]]}


# ------------------------------------------------------------------ exact ---

def _dequantised(W, bits, base, dtype):
    """What in fp64: every weight's level (nearest in the logarithm, smaller ones 0), as dtype holds it."""
    qmax = 2 ** (bits - 1) - 1
    a = W.abs().double()
    rng = float(a.max())
    steps = torch.arange(qmax, device=DEVICE, dtype=torch.float64)
    tau = rng * base ** (steps + 0.5 - qmax)
    level = torch.cat([torch.zeros(1, device=DEVICE, dtype=torch.float64), rng * base ** (steps + 1 - qmax)])
    level = level.float().to(dtype).double()
    return torch.copysign(level[torch.bucketize(a, tau, right=True)], W.double())


def _exact_layers(case, seed, X):
    Y = {}
    shapes, dtype = SHAPES[case["model"]], DTYPES[case["x"]]
    for layer in range(_layers(case)):
        at = {}
        for grp in GROUPS:
            src = SOURCE[grp[0]]
            x = X[layer].double() if src is None else at[src]
            for name in grp:
                N, K = shapes[name]
                W = _weights(N, K, seed, layer, list(shapes).index(name))
                at[name] = x @ _dequantised(W, case["bits"], _layer_base(case, layer), dtype).T
        for name, y in at.items():
            Y.setdefault(name, []).append(y)
    return {name: torch.stack(ys) for name, ys in Y.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "decode":
        return _exact_layers(case, seed, _activations((case["layers"], case["batch"], SHAPES[case["model"]]["q"][1]),
                                                      DTYPES[case["x"]], seed))
    if kind == "prefill":
        X = _activations((case["tokens"], SHAPES[case["model"]]["q"][1]), DTYPES[case["x"]], seed)
        return {name: y[0] for name, y in _exact_layers(case, seed, X[None]).items()}
    if kind == "linear":
        W = _weights(case["N"], case["K"], seed)
        X = _activations((case["batch"], case["K"]), DTYPES[case["x"]], seed)
        return X.double() @ _dequantised(W, case["bits"], case["base"], X.dtype).T
    if kind == "quantize":
        out = {}
        for p, (name, (N, K)) in enumerate(SHAPES[case["model"]].items()):
            rng = float(_weights(N, K, seed, p).abs().max())
            out[name] = (None, 0.8 * rng if case["given"] else rng)
        return out
    if kind == "energy":
        a = _weights(case["N"], case["K"], seed).abs().reshape(-1).double().sort().values
        energy = torch.cumsum(a * a, 0)
        wmin = float(a[int(torch.searchsorted(energy, case["eps"] * energy[-1]))])
        wmax = float(a[-1])
        return None, wmax, (wmax / wmin) ** (1.0 / (2 ** (case["bits"] - 1) - 1)), wmin
    if kind == "factor":
        H = _hessian(case["K"], seed).double()
        d = torch.diagonal(H)
        mean = d.mean()
        d[d == 0] = 1.0
        d += 0.01 * mean
        return torch.linalg.cholesky(torch.linalg.inv(H), upper=True), None
    return None          # codes only: whole values
