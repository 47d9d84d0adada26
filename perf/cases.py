"""Performance cases of the MoE layer: the calls an inference engine makes, over the range of sizes it makes them in.

A case is one pass of the layer (route -> dispatch layout -> grouped FFN -> combine) through the public entry points:
`MoeContext.layer` / `layer_fp8` on device tensors, `moe_layer_host` on pinned host buffers, or a prefill pass and a
few decode steps on two contexts and two streams.  The layer shapes are the repository's own: the tiny layer, the
DeepSeek-V3- and Qwen3-30B-A3B-shaped layers of `workloads`, and the paper's model shape (hidden 2560, 512 experts,
top-8) with the intermediate size the benchmark uses.  Data is synthetic, drawn from the seed on the GPU.
"""
import dataclasses
import functools
import math

import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

LAYERS = {
    "tiny": wl.C1,
    "v3": wl.C2,                                                    # selection bias, shared expert
    "v3-zipf": wl.C5,                                               # skewed expert popularity, shared expert
    "qwen3": wl.C3,
    "paper": wl.LayerShape("paper", T=1, H=2560, E=512, k=8, I=1024),
}
PD_D_TOKENS, PD_D_STEPS = 64, 4          # decode steps that run beside one prefill batch
PD_P_SMS, PD_D_SMS = 48, 100             # SM budgets of the two phases


def listed():
    return [
        # the smallest call: a short prompt through a small layer; latency and launches
        {"name": "prefill-tiny-64", "path": "device", "phase": "P", "layer": "tiny", "dtype": "bf16", "T": 64},
        # one sequence decoding: nine experts' weights are streamed for one row each
        {"name": "decode-v3-zipf-1", "path": "device", "phase": "D", "layer": "v3-zipf", "dtype": "bf16", "T": 1},
        # an ordinary decode batch on a large layer: most of the layer's weights are streamed
        {"name": "decode-v3-64", "path": "device", "phase": "D", "layer": "v3", "dtype": "bf16", "T": 64},
        # the largest decode batch, FP8 weights
        {"name": "decode-v3-fp8-128", "path": "device", "phase": "D", "layer": "v3", "dtype": "fp8", "T": 128},
        # an odd decode batch on a small layer: short K, sub-millisecond step
        {"name": "decode-qwen3-37", "path": "device", "phase": "D", "layer": "qwen3", "dtype": "bf16", "T": 37},
        # one ragged prompt chunk that comes from and goes back to pinned host buffers
        {"name": "host-qwen3-1531", "path": "host", "phase": "P", "layer": "qwen3", "dtype": "bf16", "T": 1531},
        # a full prefill batch on a small layer: tensor-bound, the benchmark's headline workload
        {"name": "prefill-qwen3-8192", "path": "device", "phase": "P", "layer": "qwen3", "dtype": "bf16", "T": 8192},
        # a ragged prefill batch with FP8 weights
        {"name": "prefill-qwen3-fp8-6007", "path": "device", "phase": "P", "layer": "qwen3", "dtype": "fp8", "T": 6007},
        # prefill over many small experts: 64 rows each
        {"name": "prefill-paper-4096", "path": "device", "phase": "P", "layer": "paper", "dtype": "bf16", "T": 4096},
        # prefill on the large layer: between weight streaming and tensor-bound
        {"name": "prefill-v3-4096", "path": "device", "phase": "P", "layer": "v3", "dtype": "bf16", "T": 4096},
        # a prefill batch with decode steps beside it on another stream, each phase on its share of the SMs
        {"name": "pd-v3-4096", "path": "pd", "phase": "PD", "layer": "v3", "dtype": "bf16", "T": 4096},
        # the largest batch: the prefill token budget with skewed expert popularity
        {"name": "prefill-v3-zipf-32768", "path": "device", "phase": "P", "layer": "v3-zipf", "dtype": "bf16", "T": 32768},
    ]


def draw(rng):
    """One more case of the same ranges: any layer, precision, phase and path, token counts log-uniform and mostly odd."""
    def tokens(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["tiny", "decode", "decode", "prefill", "prefill", "prefill", "host", "pd"])
    layer = rng.choice(["v3", "v3-zipf", "qwen3", "paper"])
    dtype = rng.choice(["bf16", "bf16", "fp8"])
    if kind == "tiny":
        return {"path": "device", "phase": rng.choice(["P", "D"]), "layer": "tiny", "dtype": "bf16", "T": tokens(1, 512)}
    if kind == "decode":
        return {"path": "device", "phase": "D", "layer": layer, "dtype": dtype, "T": tokens(1, 128)}
    if kind == "prefill":
        return {"path": "device", "phase": "P", "layer": layer, "dtype": dtype, "T": tokens(200, 32000)}
    if kind == "host":
        return {"path": "host", "phase": "P", "layer": rng.choice(["qwen3", "paper"]), "dtype": "bf16",
                "T": tokens(64, 8192)}
    return {"path": "pd", "phase": "PD", "layer": rng.choice(["v3", "v3-zipf"]), "dtype": "bf16", "T": tokens(512, 4096)}


def _context(shape, T, phase, fp8, stream=None, sm_budget=0):
    return B.MoeContext(B.make_config(shape.H, shape.E, shape.k, shape.I, shape.shared_I, T, phase, sm_budget=sm_budget,
                                      weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16),
                        stream=stream)


def _batch(shape, T, seed):
    """One batch's activations and the arrays its step writes."""
    a = wl.make_activations(shape, seed, "cuda", T=T)
    return {"a": a, "bufs": B.alloc_step_buffers(T, shape.k, shape.E, "cuda"),
            "out": torch.empty(T, shape.H, dtype=torch.bfloat16, device="cuda")}


def prepare(case, seed):
    shape, T, fp8 = LAYERS[case["layer"]], case["T"], case["dtype"] == "fp8"
    s = {"case": case, "w": (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 1000 + 2 * seed, "cuda")}
    if case["path"] == "pd":
        # the decode stream has priority, as in an engine that multiplexes the phases
        s["ctx"] = _context(shape, T, B.MOE_PHASE_PREFILL, fp8, torch.cuda.Stream(), PD_P_SMS)
        s["ctx_d"] = _context(shape, PD_D_TOKENS, B.MOE_PHASE_DECODE, fp8, torch.cuda.Stream(priority=-1), PD_D_SMS)
        s["batches_d"] = [_batch(shape, PD_D_TOKENS, 500_000 + 16 * seed + i) for i in range(PD_D_STEPS)]
    else:
        s["ctx"] = _context(shape, T, B.MOE_PHASE_DECODE if case["phase"] == "D" else B.MOE_PHASE_PREFILL, fp8)
    s["batch"] = _batch(shape, T, 2001 + 2 * seed)
    if case["path"] == "host":
        a = s["batch"]["a"]
        s["host"] = {"x": a["x"].cpu().pin_memory(), "logits": a["logits"].cpu().pin_memory(),
                     "out": torch.empty(T, shape.H, dtype=torch.bfloat16).pin_memory()}
    torch.cuda.current_stream().synchronize()  # the inputs are there for every stream
    return s


def _step(ctx, w, b):
    a = b["a"]
    if "wq_gate_up" in w:
        out, bufs = ctx.layer_fp8(a["x"], a["logits"], a["bias"], w, out=b["out"], bufs=b["bufs"])
    else:
        out, bufs = ctx.layer(a["x"], a["logits"], a["bias"], w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"],
                              out=b["out"], bufs=b["bufs"])
    return {"out": out, **bufs}


def run(state):
    w, path = state["w"], state["case"]["path"]
    if path == "host":
        h = state["host"]
        state["ctx"].moe_layer_host(h["logits"], state["batch"]["a"]["bias"], h["x"], w["w_gate_up"], w["w_down"],
                                    w["ws_gate_up"], w["ws_down"], h["out"])
        return h["out"]
    if path == "pd":
        p = _step(state["ctx"], w, state["batch"])
        return [p] + [_step(state["ctx_d"], w, b) for b in state["batches_d"]]
    return _step(state["ctx"], w, state["batch"])


@functools.lru_cache(maxsize=None)
def _experts_touched(layer, T):
    """Experts that get at least one of T tokens, with this layer's routing distribution."""
    shape = LAYERS[layer]
    a = wl.make_activations(dataclasses.replace(shape, H=1), 3, "cpu", T=T)
    key = a["logits"] if a["bias"] is None else a["logits"] + a["bias"][None, :]
    return int(torch.unique(key.topk(shape.k, dim=1).indices).numel())


def work(case):
    shape, T, wb = LAYERS[case["layer"]], case["T"], 1 if case["dtype"] == "fp8" else 2

    def one(T):
        """(bytes of activations, logits, routing arrays and output; flops) of one batch."""
        n = T * shape.k
        return (4 * T * shape.H + 4 * T * shape.E + 16 * n + 8 * shape.E,
                6 * n * shape.H * shape.I + 6 * T * shape.H * shape.shared_I)

    batches = [T] + ([PD_D_TOKENS] * PD_D_STEPS if case["path"] == "pd" else [])
    nbytes = flops = 0
    for t in batches:
        b, f = one(t)
        # a batch's experts are read once; the decode steps come one after the other and read theirs each
        b += wb * 3 * shape.H * (_experts_touched(case["layer"], t) * shape.I + shape.shared_I)
        nbytes, flops = nbytes + b, flops + f
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # The rows are stored in bf16 between the stages: a layer computed with exact sums and the same storage is
    # 2.9e-3 (2-norm) away from the exact result, and 2.3e-3 with FP8 weights; four times that.  Routing, counts and
    # permutation are integers and may not differ.
    return {"rel": 1.0e-2, "max": 0.15}
