"""The work a user of this library has it do, as cases that can be timed: decode and prefill calls of a MeteoRA linear,
the seven linears of a decoder layer, the standalone LoRA term, a training step of the gate, and the call on host
buffers.

`listed()` are the fixed cases, `draw()` gives more of the same ranges; `prepare()` makes what a program holds before
the call (weights, activations, workspaces), `run()` is one pass through the public entry points, `work()` the bytes
and operations that pass cannot do without, `tolerance()` how far another correct implementation may be off.
"""
import math

import torch

from paper_2405_13053_b200 import binding as mb
from paper_2405_13053_b200 import decoder_layer as dl

# Projection shapes of the two model sizes the workloads of this repository use (hidden 4096 / MLP 14336 / k,v 1024, and
# hidden 5120 / MLP 13824).
SHAPES = ((4096, 4096), (4096, 1024), (4096, 14336), (14336, 4096), (5120, 5120), (5120, 13824), (13824, 5120))
B_STD = 0.05      # makes the LoRA term about 6 % of y, so that an error in it shows in y's own error
TIE_GAP = 1e-4    # tokens whose pick hangs on less than this between two gate logits are drawn again


def _linear(T, d_in, d_out, N=28, r=8, k=2, dtype="bf16", x="rms", temperature=1.0, kind="linear"):
    return {"kind": kind, "T": T, "d_in": d_in, "d_out": d_out, "N": N, "r": r, "k": k, "dtype": dtype, "x": x,
            "temperature": temperature}


def listed():
    return [
        # One sequence generating: a single token through an attention projection.  Latency and host work count.
        dict(_linear(1, 4096, 4096), name="decode_1"),
        # A full decode batch through the same projection: the shape of the headline benchmark.
        dict(_linear(128, 4096, 4096), name="decode_128"),
        # A large, ragged decode batch through the wide projection of the larger model.
        dict(_linear(200, 5120, 13824, x="normal"), name="decode_200_wide"),
        # 64 sequences, one new token each, through all seven linears of a decoder layer (q/k/v and gate/up grouped).
        {"kind": "layer", "T": 64, "N": 28, "r": 8, "k": 2, "name": "decode_layer_64"},
        # A short prompt through the narrow k / v projection: many small steps, little arithmetic in each.
        dict(_linear(512, 4096, 1024, x="clusters"), name="prefill_512_narrow"),
        # A prompt of ordinary length through the wide projection, skewed routing.
        dict(_linear(2048, 4096, 14336, x="clusters"), name="prefill_2048_wide"),
        # A ragged prompt, adapters of twice the rank, four picks per token, softened gate.
        dict(_linear(1531, 5120, 5120, r=16, k=4, x="normal", temperature=15.0), name="prefill_1531_rank16"),
        # A long prompt through all seven linears of a decoder layer.
        {"kind": "layer", "T": 4096, "N": 28, "r": 8, "k": 2, "name": "prefill_layer_4096"},
        # The small fp32 layer used where results are checked by hand.
        dict(_linear(64, 256, 256, N=4, dtype="f32", x="normal"), name="fp32_64"),
        # The LoRA term alone for a caller that has its own base product: gate, bucketing, shrink and expand.
        dict(_linear(2048, 4096, 4096, x="clusters", kind="delta"), name="delta_2048"),
        # Training the gate: forward, then the gradient of the gate weights for the loss that came back.
        dict(_linear(2048, 4096, 4096, x="clusters", kind="train"), name="train_gate_2048"),
        # Activations in pinned host memory, copied in, through the layer and out again.
        dict(_linear(128, 4096, 4096, kind="host"), name="host_128"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("linear", "linear", "linear", "linear", "linear", "layer", "fp32", "delta", "train", "host"))
    if kind == "layer":
        return {"kind": "layer", "T": _log_int(rng, 1, 4096), "N": rng.choice((8, 28, 28)), "r": 8, "k": rng.choice((1, 2, 2, 4))}
    if kind == "fp32":
        return _linear(_log_int(rng, 1, 512), _log_int(rng, 250, 2048), _log_int(rng, 250, 2048), N=rng.choice((4, 8, 28)),
                       dtype="f32", x="normal")
    d_in, d_out = rng.choice(SHAPES)
    if rng.random() < 0.25:  # other widths, in steps that keep rows 16-byte aligned
        d_in, d_out = 8 * _log_int(rng, 128, 1024), 8 * _log_int(rng, 128, 1024)
    T = _log_int(rng, 1, {"linear": 8192, "delta": 4096, "train": 4096, "host": 512}[kind])
    case = _linear(T, d_in, d_out, k=rng.choice((1, 2, 2, 2, 4)), x="clusters" if T > 256 else "rms",
                   temperature=rng.choice((1.0, 1.0, 15.0)), kind=kind)
    if kind == "linear":  # adapter counts and ranks of the variants table
        case["N"], case["r"] = rng.choice(((28, 8), (28, 8), (28, 8), (8, 8), (64, 8), (28, 16), (28, 32)))
    if kind == "train":
        case["k"] = rng.choice((2, 2, 4))  # top-1 passes no gradient to the gate
    return case


# ---- inputs ------------------------------------------------------------------------------------------------------

def _dtype(case):
    return torch.float32 if case.get("dtype") == "f32" else torch.bfloat16


def _tokens(g, T, d, how):
    x = torch.randn(T, d, device="cuda", generator=g)
    if how == "rms":
        x = x / x.pow(2).mean(dim=1, keepdim=True).sqrt()
    elif how == "clusters":  # four tasks in contiguous runs
        mean = torch.randn(4, d, device="cuda", generator=g)
        x = 0.5 * x + mean[torch.arange(T, device="cuda") * 4 // max(T, 1)]
    return x


def _activations(g, T, d, how, gates, k, dtype):
    """x[T, d] for layers with these gates; tokens within TIE_GAP of a tie among their picks are drawn again, because
    there the picks are the rounding's choice and not the input's."""
    x = _tokens(g, T, d, how).to(dtype)
    for _ in range(4):
        close = torch.zeros(T, dtype=torch.bool, device="cuda")
        for Wg in gates:
            top = (x.double() @ Wg.double().T).topk(min(k + 1, Wg.shape[0]), dim=1).values
            close |= (top[:, :-1] - top[:, 1:]).min(dim=1).values < TIE_GAP
        x = torch.where(close[:, None], _tokens(g, T, d, how).to(dtype), x)
    return x


def _weights(g, d_in, d_out, N, r, dtype):
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    return {"W0": (0.02 * rand(d_out, d_in)).to(dtype),
            "A": ((torch.rand(N, r, d_in, device="cuda", generator=g) * 2 - 1) / math.sqrt(d_in)).to(dtype),
            "B": (B_STD * rand(N, d_out, r)).to(dtype),
            "Wg": (rand(N, d_in) / math.sqrt(d_in)).to(dtype)}


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dtype, T, k, N, r = _dtype(case), case["T"], case["k"], case["N"], case["r"]
    s = {"case": case}
    if case["kind"] == "layer":
        w = {n: _weights(g, i, o, N, r, dtype) for n, (i, o) in dl.LINEARS.items()}
        s["linears"] = dl.LibraryLinears(w, k)
        s["x"] = [_activations(g, T, w[names[0]]["A"].shape[2], "rms", [w[n]["Wg"] for n in names], k, dtype)
                  for names in dl.GROUPS]
        return s
    d_in, d_out = case["d_in"], case["d_out"]
    w = s["w"] = _weights(g, d_in, d_out, N, r, dtype)
    s["x"] = _activations(g, T, d_in, case["x"], [w["Wg"]], k, dtype)
    s["workspace"] = mb.alloc_workspace(mb.make_shape(T, d_in, d_out, N, r, k, dtype, case["temperature"]))
    if case["kind"] == "train":
        s["dy"] = torch.randn(T, d_out, device="cuda", generator=g).to(dtype)
        s["Bt"] = mb.meteora_transpose_adapters_b(w["B"])  # the adapters are fixed while the gate trains
    if case["kind"] == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["y"] = torch.empty(T, d_out, dtype=dtype).pin_memory()
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------

def run(s):
    case = s["case"]
    k, x = case["k"], s["x"]
    if case["kind"] == "layer":
        lin, out = s["linears"], []
        for names, xi in zip(dl.GROUPS, x):
            out += lin.many(names, xi) if len(names) > 1 else [lin.one(names[0], xi)]
        return out + [lin.routing[n] for names in dl.GROUPS for n in names]
    w, tau = s["w"], case["temperature"]
    if case["kind"] == "linear":
        return mb.meteora_linear_forward(x, w["W0"], w["A"], w["B"], w["Wg"], k, tau, workspace=s["workspace"],
                                         return_routing=True)
    if case["kind"] == "host":
        return mb.meteora_linear_forward_host(x, w["W0"], w["A"], w["B"], w["Wg"], k, s["y"], s["workspace"], tau)
    if case["kind"] == "delta":
        idx, weight, _ = mb.meteora_gate_topk(x, w["Wg"], k, tau)
        counts, offsets, perm = mb.meteora_route(idx, case["N"])
        delta = mb.meteora_lora_delta(x, w["A"], w["B"], idx, weight, offsets, perm, workspace=s["workspace"])
        return idx, weight, counts, offsets, perm, delta
    y, idx, weight = mb.meteora_linear_forward(x, w["W0"], w["A"], w["B"], w["Wg"], k, tau, workspace=s["workspace"],
                                               return_routing=True)
    dWg, dlogit = mb.meteora_gate_backward(x, w["A"], w["B"], s["dy"], idx, weight, tau, Bt=s["Bt"])
    return y, idx, weight, dWg, dlogit


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def _linear_work(T, d_in, d_out, N, r, k, es, base=True, read_x=True):
    """Only the adapters that can have been picked are read; an expand and a shrink per pick."""
    touched = min(N, T * k)
    return {"bytes": es * ((d_in * d_out if base else 0) + N * d_in + touched * r * (d_in + d_out)
                           + (T * d_in if read_x else 0)) + (es if base else 4) * T * d_out + 8 * T * k,
            "flops": (2 * T * d_in * d_out if base else 0) + 2 * T * N * d_in + 2 * T * k * r * (d_in + d_out)}


def work(case):
    T, N, r, k = case["T"], case["N"], case["r"], case["k"]
    if case["kind"] == "layer":
        parts = [_linear_work(T, *dl.LINEARS[n], N, r, k, 2, read_x=n == names[0]) for names in dl.GROUPS for n in names]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    d_in, d_out, es = case["d_in"], case["d_out"], 4 if case["dtype"] == "f32" else 2
    got = _linear_work(T, d_in, d_out, N, r, k, es, base=case["kind"] != "delta")
    if case["kind"] == "delta":
        got["bytes"] += 4 * (T * k + 2 * N + 1)
    if case["kind"] == "train":  # dy and B^T in, dWg and dlogit out; <dy, B u> and dlogit^T x per pick
        got["bytes"] += es * (T * d_out + min(N, T * k) * r * d_out) + 4 * (N * d_in + T * k)
        got["flops"] += 2 * T * k * (r * d_out + r + d_in)
    return got


def tolerance(case):
    if case["kind"] == "delta":  # fp32 sums over up to 14336 products of bf16 values
        return {"rel": 3e-5, "max": 1e-3}
    if case.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 4e-4}
    # y is rounded once to bf16 (8 bits): one step of its last place at worst where two fp32 sums straddle a rounding
    # boundary, 1.1e-3 on average.  The picks are away from ties, so they are the same.
    return {"rel": 5e-3, "max": 2e-2}
