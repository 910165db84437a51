"""The work that users of this package have it do, as cases that can be timed and compared.

A case names one path through the public entry points of ``paper_2605_08692_b200.binding`` and the
sizes and options of one call:

  layer      one linear on its own: importances from its activations, fit, pack
  trio       attention, gate and down projections of one block in one call, reconstructions included
             (the workload of ``bench.py``)
  block      the seven linears of one decoder block in one call, activations shared as in a model
  act_stats  importances streamed from two chunks of calibration tokens
  dequant    a stored layer expanded to BF16
  prescale   input channels scaled before a fit
  host       one linear from page-locked host buffers and back

Weights are normal (or Student-t with five degrees of freedom) with 1 % of the input channels ten
times larger; activations have log-normal channel scales and 0.5 % massive channels.
"""
import math

import torch

from paper_2605_08692_b200 import binding

MODES = {"int4": binding.INT4, "nvfp4": binding.NVFP4}
INITS = {"grid": binding.INIT_GRID, "quantile": binding.INIT_QUANTILE}


def listed():
    return [
        # A first try on a toy layer, and the smallest linears of small models: launches and latency.
        dict(name="layer_toy_int4", path="layer", N=512, K=512, mode="int4", S=128, dist="normal", T=256, init="grid",
             rounds=10, inner=1),
        # Sizes that divide nothing (a vocabulary-like row count, a width that ends inside a column slab).
        dict(name="layer_ragged_nvfp4", path="layer", N=1531, K=2064, mode="nvfp4", S=16, dist="student5", T=333,
             init="quantile", rounds=20, inner=1),
        # A single 4096 x 4096 linear with the paper's default budget: inner refinement.
        dict(name="layer_inner_nvfp4", path="layer", N=4096, K=4096, mode="nvfp4", S=16, dist="normal", T=8192,
             init="quantile", rounds=3, inner=10),
        # The paper's INT4 variant with selection groups of 16, on a wide down projection.
        dict(name="layer_s16_int4", path="layer", N=4096, K=14336, mode="int4", S=16, dist="normal", T=4096,
             init="quantile", rounds=20, inner=1),
        # The largest linears of 70B-shaped models: memory streaming over many rounds.
        dict(name="layer_70b_nvfp4", path="layer", N=28672, K=8192, mode="nvfp4", S=16, dist="normal", T=32768,
             init="quantile", rounds=30, inner=1),
        # The benchmark's step: three 8B-shaped linears.
        dict(name="trio_8b_nvfp4", path="trio", hidden=4096, kv=1024, inter=14336, mode="nvfp4", S=16, dist="normal",
             T=4096, init="quantile", rounds=20, inner=1),
        # One decoder block of the 8B-shaped and of the 7B-shaped stack: what whole-model quantisation repeats.
        dict(name="block_8b_int4", path="block", hidden=4096, kv=1024, inter=14336, mode="int4", S=128, dist="normal",
             T=16384, init="quantile", rounds=20, inner=1),
        dict(name="block_7b_nvfp4", path="block", hidden=3584, kv=512, inter=18944, mode="nvfp4", S=16, dist="student5",
             T=16384, init="quantile", rounds=20, inner=1),
        # Calibration alone: the widest input of a block, its tokens in two chunks.
        dict(name="act_stats_wide", path="act_stats", K=14336, T=16384),
        # A stored layer read back for use.
        dict(name="dequant_gate_nvfp4", path="dequant", N=14336, K=4096, mode="nvfp4", S=16),
        # AWQ-style scaling of a layer before its fit.
        dict(name="prescale_down", path="prescale", N=4096, K=14336),
        # A caller that keeps weights and activations in host memory.
        dict(name="host_q_nvfp4", path="host", N=4096, K=4096, mode="nvfp4", S=16, dist="normal", T=4096,
             init="quantile", rounds=20, inner=1),
    ]


def _log_int(rng, lo, hi, step=1):
    """A multiple of ``step`` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    path = rng.choice(["layer", "layer", "layer", "trio", "block", "act_stats", "dequant", "prescale", "host"])
    mode = rng.choice(["int4", "nvfp4"])
    g = 128 if mode == "int4" else 16
    S = rng.choice([g, 16])
    if path == "act_stats":
        return dict(path=path, K=_log_int(rng, 256, 28672, 8), T=_log_int(rng, 64, 16384))
    if path == "dequant":
        return dict(path=path, N=_log_int(rng, 64, 16384), K=_log_int(rng, 256, 16384, g), mode=mode, S=S)
    if path == "prescale":
        return dict(path=path, N=_log_int(rng, 64, 16384), K=_log_int(rng, 256, 16384, 8))
    fit = dict(mode=mode, S=S, dist=rng.choice(["normal", "student5"]), init=rng.choice(["quantile", "quantile", "grid"]),
               rounds=rng.randint(5, 30), inner=1)
    if path == "layer":
        if rng.random() < 0.25:
            fit.update(rounds=rng.randint(1, 3), inner=rng.randint(2, 10))
        return dict(path=path, N=_log_int(rng, 128, 16384), K=_log_int(rng, 256, 14336, g), T=_log_int(rng, 64, 16384), **fit)
    if path == "host":
        fit.update(S=g)
        return dict(path=path, N=_log_int(rng, 128, 8192), K=_log_int(rng, 256, 8192, g), T=_log_int(rng, 64, 4096), **fit)
    hidden = _log_int(rng, 512, 4096, 128)
    fit.update(rounds=rng.randint(5, 20))
    return dict(path=path, hidden=hidden, kv=max(128, hidden // rng.choice([1, 4, 8]) // 128 * 128),
                inter=int(hidden * rng.uniform(2.0, 3.5)) // 128 * 128, T=_log_int(rng, 256, 16384), **fit)


def _linears(case):
    """(rows, input channels, name of the activations) of every linear of the case."""
    if case["path"] == "trio":
        H, F = case["hidden"], case["inter"]
        return [(H, H, "attn"), (F, H, "mlp"), (H, F, "down")]
    if case["path"] == "block":
        H, KV, F = case["hidden"], case["kv"], case["inter"]
        return [(H, H, "attn"), (KV, H, "attn"), (KV, H, "attn"), (H, H, "o"), (F, H, "mlp"), (F, H, "mlp"), (H, F, "down")]
    return [(case["N"], case["K"], "x")]


def _weights(N, K, dist, gen):
    w = torch.randn(N, K, device="cuda", generator=gen)
    if dist == "student5":
        chi = torch.zeros_like(w)
        for _ in range(5):
            chi += torch.randn(N, K, device="cuda", generator=gen).square_()
        w /= (chi / 5.0).sqrt_()
    cols = torch.randperm(K, device="cuda", generator=gen)[: max(1, K // 100)]
    w[:, cols] *= 10.0
    return (w * 0.02).to(torch.bfloat16)


def _activations(T, K, gen):
    c = torch.exp(torch.randn(K, device="cuda", generator=gen))
    c[torch.randperm(K, device="cuda", generator=gen)[: max(1, K // 200)]] *= 30.0
    return (torch.randn(T, K, device="cuda", generator=gen) * c).to(torch.bfloat16)


def _outputs(N, K, case):
    """Buffers for the results of one linear (the bit patterns of unsigned 16-bit fields in int16)."""
    mode = MODES[case["mode"]]
    g = binding.group_of(mode)
    out = dict(T01=torch.zeros(2, 16, dtype=torch.float32, device="cuda"),
               T01_bf16=torch.zeros(2, 16, dtype=torch.bfloat16, device="cuda"),
               scales=torch.zeros(N, K // g, dtype=torch.int16 if mode == binding.INT4 else torch.uint8, device="cuda"),
               tensor_scale=torch.ones(1, dtype=torch.float32, device="cuda"),
               codes=torch.zeros(N, K // 2, dtype=torch.uint8, device="cuda"),
               err_out=torch.zeros(2, dtype=torch.float64, device="cuda"))
    if case["S"] != g:
        out["sigma_bits"] = torch.zeros(N, K // (8 * case["S"]), dtype=torch.uint8, device="cuda")
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    path = case["path"]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if path == "act_stats":
        K = case["K"]
        return dict(case=case, X=_activations(case["T"], K, gen), I=torch.zeros(K, dtype=torch.float32, device="cuda"),
                    ws=binding.alloc_workspace(binding.NVFP4, 1, K, case["T"]), status=status)
    if path == "prescale":
        N, K = case["N"], case["K"]
        return dict(case=case, W=_weights(N, K, "normal", gen), a=torch.exp(0.5 * torch.randn(K, device="cuda", generator=gen)),
                    I=torch.exp(2.0 * torch.randn(K, device="cuda", generator=gen)),
                    W_out=torch.zeros(N, K, dtype=torch.bfloat16, device="cuda"),
                    I_out=torch.zeros(K, dtype=torch.float32, device="cuda"), status=status)
    mode = MODES[case["mode"]]
    g = binding.group_of(mode)
    if path == "dequant":
        N, K = case["N"], case["K"]
        out = _outputs(N, K, case)
        out["codes"].random_(0, 256, generator=gen)
        if mode == binding.INT4:         # positive BF16 scales around 0.01, the selection bit in the sign (S = 128)
            s = torch.exp(0.3 * torch.randn(N, K // g, device="cuda", generator=gen)) * 0.01
            if case["S"] == g:
                s *= 1.0 - 2.0 * torch.randint(0, 2, s.shape, device="cuda", generator=gen)
            out["scales"] = s.to(torch.bfloat16).view(torch.int16)
        else:
            out["scales"] = (torch.randint(0x20, 0x7F, (N, K // g), device="cuda", generator=gen)
                             + 128 * torch.randint(0, 2, (N, K // g), device="cuda", generator=gen)).to(torch.uint8)
            out["tensor_scale"].fill_(3e-5)
        if "sigma_bits" in out:
            out["sigma_bits"].random_(0, 256, generator=gen)
        out["T01_bf16"] = torch.sort(3.0 * torch.randn(2, 16, device="cuda", generator=gen), dim=1).values.to(torch.bfloat16)
        return dict(case=case, out=out, What=torch.zeros(N, K, dtype=torch.bfloat16, device="cuda"))
    linears = _linears(case)
    X = {}
    for _, K, x in linears:
        if x not in X:
            X[x] = _activations(case["T"], K, gen)
    layers = []
    for N, K, x in linears:
        d = dict(_outputs(N, K, case), W=_weights(N, K, case["dist"], gen), X=X[x])
        if path == "trio":
            d["What"] = torch.zeros(N, K, dtype=torch.bfloat16, device="cuda")
        if path != "host":
            d["ws"] = binding.alloc_workspace(mode, N, K, case["T"])
        layers.append(d)
    state = dict(case=case, layers=layers, status=status)
    if path == "layer":
        layers[0]["I"] = torch.zeros(case["K"], dtype=torch.float32, device="cuda")
        layers[0]["err_trace"] = torch.zeros(case["rounds"], dtype=torch.float64, device="cuda")
    if path == "host":
        state["host"] = {k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True).copy_(v) for k, v in layers[0].items()}
        state["layers"] = []
        state["ws"] = torch.empty(binding.host_workspace_bytes(mode, case["N"], case["K"], case["T"]), dtype=torch.uint8,
                                  device="cuda")
    return state


_RESULTS = ("T01", "T01_bf16", "scales", "tensor_scale", "codes", "err_out", "sigma_bits", "What", "I", "err_trace")


def _results(d):
    return {k: d[k] for k in _RESULTS if k in d}


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "act_stats":
        X, h = state["X"], case["T"] // 2
        binding.act_stats(X[:h], state["I"], state["ws"], dev_status=state["status"])
        binding.act_stats(X[h:], state["I"], state["ws"], accumulate=True, dev_status=state["status"])
        return state["I"], state["status"]
    if path == "prescale":
        binding.prescale_columns(state["W"], state["a"], state["W_out"], I=state["I"], I_out=state["I_out"],
                                 dev_status=state["status"])
        return state["W_out"], state["I_out"], state["status"]
    mode = MODES[case["mode"]]
    if path == "dequant":
        o = state["out"]
        binding.dequant(o["codes"], o["scales"], o["tensor_scale"], o["T01_bf16"], mode, state["What"], sel_group=case["S"],
                        sigma_bits=o.get("sigma_bits"))
        return state["What"]
    init = INITS[case["init"]]
    if path == "host":
        h = state["host"]
        binding.quantize_layer_host(h["W"], h["X"], mode, n_outer=case["rounds"], init=init, T01_host=h["T01"],
                                    T01_bf16_host=h["T01_bf16"], scales_host=h["scales"], tensor_scale_host=h["tensor_scale"],
                                    codes_host=h["codes"], err_out_host=h["err_out"], ws=state["ws"])
        return _results(h)
    if path == "layer":
        d = state["layers"][0]
        binding.act_stats(d["X"], d["I"], d["ws"], dev_status=state["status"])
        binding.fit_layer(d["W"], mode, I=d["I"], n_outer=case["rounds"], n_inner=case["inner"], init=init, T01=d["T01"],
                          scales=d["scales"], tensor_scale=d["tensor_scale"], ws=d["ws"], err_trace=d["err_trace"],
                          dev_status=state["status"], sel_group=case["S"])
        binding.pack(d["W"], mode, I=d["I"], T01=d["T01"], T01_bf16=d["T01_bf16"], scales=d["scales"],
                     tensor_scale=d["tensor_scale"], codes=d["codes"], ws=d["ws"], err_out=d["err_out"],
                     sel_group=case["S"], sigma_bits=d.get("sigma_bits"))
        return _results(d), state["status"]
    binding.quantize_layers(state["layers"], mode, n_outer=case["rounds"], n_inner=case["inner"], init=init,
                            dev_status=state["status"], sel_group=case["S"])
    return [_results(d) for d in state["layers"]], state["status"]


def work(case):
    path = case["path"]
    if path == "act_stats":
        n = case["T"] * case["K"]
        return {"bytes": 2 * n + 4 * case["K"], "flops": 2 * n}
    if path == "prescale":
        n = case["N"] * case["K"]
        return {"bytes": 4 * n + 12 * case["K"], "flops": n}
    g = 128 if case["mode"] == "int4" else 16
    per_scale = 2 if case["mode"] == "int4" else 1
    stored = 0.5 + per_scale / g + (1 / (8 * case["S"]) if case["S"] != g else 0)      # bytes per weight as stored
    if path == "dequant":
        n = case["N"] * case["K"]
        return {"bytes": (2 + stored) * n + 64, "flops": n}
    n = b = f = 0
    seen = set()
    for N, K, x in _linears(case):
        n += N * K
        if x not in seen:
            seen.add(x)
            b += 2 * case["T"] * K
            f += 2 * case["T"] * K
    b += (2 + stored + (2 if path == "trio" else 0)) * n
    # per weight and assignment pass: normalise, two distances squared and weighted, the two sums of the chosen
    # entry; a further inner iteration needs no second distance; the pack pass is one more assignment
    f += (case["rounds"] * (9 + 5 * (case["inner"] - 1)) + 9) * n
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["path"] in ("dequant", "prescale"):
        return "exact"                       # one product, rounded once
    if case["path"] == "act_stats":
        return {"rel": 1e-6, "max": 4e-6}    # sums given as FP32
    # The tables are stored as BF16 (steps of 2^-8): an entry next to a rounding boundary may fall on either side,
    # and then the few weights next to that entry's midpoints take a neighbouring code.
    return {"rel": 4e-3, "max": 0.5, "differ": 2e-3}
