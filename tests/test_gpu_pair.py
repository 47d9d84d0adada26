"""The two-CTA GEMM kernel, which AUTO takes where it was measured ahead: its results are those of the other two kernels, bit
for bit (the order of the sums is the same)."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import build as build_mod
from paper_2609_00993_b200 import workloads as wl
from helpers import check_layer, np_f32, np_i32, sample_tokens
from test_rules_cpu import rules  # noqa: F401  (fixture)

DEV = "cuda"
# H, I, E, k, T, shared_I, zipf, fp8: of each the passes named take the kernel
LAYERS = {
    "both passes, half a feature tile, ragged K": (1152, 704, 48, 4, 2101, 0, 0.0, False, (1, 1)),
    "shared expert of another length": (1344, 704, 48, 4, 2101, 320, 0.0, False, (1, 1)),
    "experts without rows and of several chunks": (768, 1536, 16, 2, 4211, 0, 1.2, False, (1, 0)),
    "many experts": (704, 128, 700, 8, 8600, 0, 0.0, False, (1, 0)),
    "FP8, half a k-block": (1344, 704, 48, 4, 2101, 320, 0.0, True, (1, 1)),
    "FP8, skewed": (2048, 1536, 16, 2, 4211, 0, 1.2, True, (1, 1)),
}


def _layer(name):
    H, I, E, k, T, shared, zipf, fp8, _ = LAYERS[name]
    shape = wl.LayerShape("t", T=T, H=H, E=E, k=k, I=I, shared_I=shared, zipf_s=zipf)
    return shape, fp8, (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 3, DEV), wl.make_activations(shape, 4, DEV)


def _ctx(shape, fp8, **kw):
    return B.MoeContext(B.make_config(shape.H, shape.E, shape.k, shape.I, shape.shared_I, shape.T,
                                      weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16, **kw))


def _run(ctx, fp8, w, a):
    out, _ = ctx.layer_fp8(a["x"], a["logits"], a["bias"], w) if fp8 else \
        ctx.layer(a["x"], a["logits"], a["bias"], w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])
    return out


def _taken(ctx):
    """Whether the last gated and the last down pass ran on the pair kernel."""
    g = ctx.moe_ctx_debug_gemm()
    return int(g["gated"] == B.MOE_KERNEL_PAIR), int(g["down"] == B.MOE_KERNEL_PAIR)


def _choice(H, I, E, k, T, fp8):
    R = f"{T * k}LL, {E}, 148"
    return f"moe::pair_is_faster({int(fp8)}, 1, {H}, {I}, {R})", f"moe::pair_is_faster({int(fp8)}, 0, {I}, {H}, {R})"


@pytest.mark.parametrize("H,I,E,k,T,fp8,gated,down", [
    # passes of which one side was measured at least 2 % ahead (csrc/rules.h has the times)
    (2048, 768, 128, 8, 30000, 0, 1, 1), (2048, 768, 128, 8, 1100, 0, 0, 0), (2048, 768, 128, 8, 8192, 0, 0, 1),
    (7168, 2048, 256, 8, 16000, 0, 0, 1), (4096, 1536, 128, 8, 16000, 0, 0, 1), (2560, 1024, 512, 8, 4096, 0, 0, 0),
    (2048, 768, 128, 8, 2500, 1, 1, 1), (2560, 1024, 512, 8, 12000, 1, 1, 1), (7168, 2048, 256, 8, 30000, 1, 0, 1),
    (7168, 512, 8, 2, 4500, 0, 0, 0), (512, 2048, 8, 2, 4500, 0, 0, 0),
    (4096, 1536, 128, 8, 6720, 0, 0, 1), (4096, 1536, 128, 8, 7680, 0, 0, 1), (2560, 1536, 128, 8, 7200, 0, 0, 1),
    (2048, 1408, 64, 6, 4800, 0, 0, 1), (2048, 1408, 64, 6, 3200, 0, 0, 0), (2560, 1536, 128, 8, 4800, 0, 0, 0),
    (1024, 512, 64, 4, 2500, 1, 0, 1), (1024, 512, 64, 4, 4160, 1, 0, 0), (1024, 512, 64, 4, 11200, 1, 0, 1), (1536, 512, 128, 8, 2560, 1, 1, 1),
    (2048, 768, 128, 8, 6720, 1, 1, 1), (2048, 768, 128, 8, 4160, 0, 0, 1),
] + [(*v[:5], int(v[7]), *v[8]) for v in LAYERS.values()])
def test_the_rule(rules, H, I, E, k, T, fp8, gated, down):  # noqa: F811
    assert rules(*_choice(H, I, E, k, T, fp8)) == [gated, down]


def test_no_barrier_between_warps_that_give_up_by_themselves():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(build_mod.CSRC, "gemm_pair.cu")).read())
    begin = text.index("if (warp == kProducerWarp) {")
    loops = text[begin:text.index("tc_fence_before();\n  __syncthreads();", begin)]
    assert "__syncthreads" not in loops and "cluster_sync" not in loops and "barrier.sync" not in loops


@pytest.mark.gpu
@pytest.mark.parametrize("name", LAYERS)
def test_auto_equals_both_variants(name):
    shape, fp8, w, a = _layer(name)
    outs = []
    for variant in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M, B.MOE_GEMM_LARGE_M, B.MOE_GEMM_AUTO):
        ctx = _ctx(shape, fp8, gemm_variant=variant)
        torch.cuda.synchronize()
        for _ in range(2):  # (the second step finds the tile counters as the first one left them)
            outs.append(_run(ctx, fp8, w, a))
        torch.cuda.synchronize()
        assert ctx.moe_ctx_status() == B.MOE_OK
        assert _taken(ctx) == (LAYERS[name][8] if variant == B.MOE_GEMM_AUTO else (0, 0))
        ctx.close()
    assert torch.isfinite(outs[0].float()).all()
    assert all(torch.equal(outs[0], o) for o in outs[1:])


@pytest.mark.gpu
def test_other_sizes_segments_budgets_and_graphs():
    """One context through sizes that take other kernels (they share the tensor maps), segments of experts, and a graph; and
    a context on part of the SMs."""
    name = "shared expert of another length"
    shape, fp8, w, a = _layer(name)
    ctx = _ctx(shape, fp8)
    torch.cuda.synchronize()
    ref = _run(ctx, fp8, w, a)
    assert _taken(ctx) == (1, 1)
    few = {k: (v[:300].contiguous() if k in ("x", "logits") else v) for k, v in a.items()}
    small = _run(ctx, fp8, w, few)
    assert _taken(ctx) == (0, 0)
    assert torch.equal(_run(ctx, fp8, w, a), ref)
    torch.cuda.synchronize()
    assert torch.equal(small, ref[:300])  # a token's result does not depend on the batch
    ctx.moe_ctx_set_segments(7)
    assert torch.equal(_run(ctx, fp8, w, a), ref) and _taken(ctx) == (1, 1)
    ctx.moe_ctx_set_segments(0)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.close()
    stream = torch.cuda.Stream()
    ctx = B.MoeContext(B.make_config(shape.H, shape.E, shape.k, shape.I, shape.shared_I, shape.T), stream=stream)
    bufs, out = B.alloc_step_buffers(shape.T, shape.k, shape.E, DEV), torch.empty_like(ref)
    step = lambda: ctx.layer(a["x"], a["logits"], a["bias"], w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"], out=out, bufs=bufs)
    torch.cuda.synchronize()
    step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    out.zero_()
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and ctx.moe_ctx_status() == B.MOE_OK and _taken(ctx) == (1, 1)
    ctx.close()
    ctx = _ctx(shape, fp8, sm_budget=37)
    torch.cuda.synchronize()
    assert torch.equal(_run(ctx, fp8, w, a), ref) and _taken(ctx) == (0, 0)
    ctx.close()


@pytest.mark.gpu
def test_pieces_of_the_down_pass():
    """moe_layer_host runs the down pass in ranges of features."""
    shape, fp8, w, a = _layer("both passes, half a feature tile, ragged K")
    ctx = _ctx(shape, fp8)
    torch.cuda.synchronize()
    ref = _run(ctx, fp8, w, a).cpu()
    x, logits, out = a["x"].cpu().pin_memory(), a["logits"].cpu().pin_memory(), torch.empty_like(ref).pin_memory()
    for _ in range(2):
        out.zero_()
        ctx.moe_layer_host(logits, None, x, w["w_gate_up"], w["w_down"], None, None, out)
        assert torch.equal(out, ref) and _taken(ctx) == (1, 1)
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["both passes, half a feature tile, ragged K", "FP8, half a k-block"])
def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable(name):
    shape, fp8, w, a = _layer(name)
    ctx = _ctx(shape, fp8)
    torch.cuda.synchronize()
    good = _run(ctx, fp8, w, a)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.moe_ctx_set_wait_limit(20_000)
    ctx.moe_ctx_debug_inject_stall(True)
    _run(ctx, fp8, w, a)
    torch.cuda.synchronize()
    assert _taken(ctx) == (1, 1)
    assert ctx.moe_ctx_status() == B.MOE_ERR_TIMEOUT
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.moe_ctx_debug_inject_stall(False)
    ctx.moe_ctx_set_wait_limit(0)
    again = _run(ctx, fp8, w, a)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK and torch.equal(again, good)
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("H,I,E,k,T,fp8,down", [
    (2560, 1536, 24, 8, 1050, False, B.MOE_GEMM_SMALL_M), (2560, 1536, 24, 8, 1051, False, B.MOE_KERNEL_PAIR),  # 350 rows
    (1024, 512, 147, 4, 7733, True, B.MOE_GEMM_LARGE_M), (1024, 512, 148, 4, 7733, True, B.MOE_KERNEL_PAIR),    # four waves
])
def test_down_passes_on_either_side_of_a_line(H, I, E, k, T, fp8, down):
    shape = wl.LayerShape("t", T=T, H=H, E=E, k=k, I=I)
    w, a = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 3, DEV), wl.make_activations(shape, 4, DEV)
    outs = []
    for variant in (B.MOE_GEMM_AUTO, B.MOE_GEMM_LARGE_M):
        ctx = _ctx(shape, fp8, gemm_variant=variant)
        torch.cuda.synchronize()
        outs.append(_run(ctx, fp8, w, a))
        torch.cuda.synchronize()
        assert ctx.moe_ctx_status() == B.MOE_OK
        assert ctx.moe_ctx_debug_gemm()["down"] == (down if variant == B.MOE_GEMM_AUTO else B.MOE_GEMM_LARGE_M)
        ctx.close()
    assert torch.isfinite(outs[0].float()).all() and torch.equal(*outs)


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["shared expert of another length", "FP8, half a k-block"])
def test_values_against_the_oracle(name):
    """Sampled tokens, among them the first and last rows of the most and the least loaded expert."""
    shape, fp8, w, a = _layer(name)
    ctx = _ctx(shape, fp8)
    torch.cuda.synchronize()
    out, bufs = ctx.layer_fp8(a["x"], a["logits"], a["bias"], w) if fp8 else \
        ctx.layer(a["x"], a["logits"], a["bias"], w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK and _taken(ctx) == (1, 1)
    tokens = sample_tokens(shape.T, np_i32(bufs["counts"]), np_i32(bufs["offsets"]), np_i32(bufs["perm"]).reshape(-1), shape.k, 12)
    x, logits = wl.bits(a["x"])[tokens], np_f32(a["logits"])[tokens]
    if fp8:
        ref = oracle.layer_fp8(x, logits, None, shape.k, *[w[n].cpu().numpy() for n in
                               ("wq_gate_up", "sw_gate_up", "wq_down", "sw_down", "wsq_gate_up", "sws_gate_up", "wsq_down", "sws_down")])
    else:
        ref = oracle.layer(x, logits, None, shape.k, *[wl.bits(w[n]) for n in ("w_gate_up", "w_down", "ws_gate_up", "ws_down")])
    assert np.array_equal(np_i32(bufs["topk_idx"])[tokens], ref["topk_idx"])
    check_layer(out[tokens], ref["out"], label=name)
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["shared expert of another length", "FP8, half a k-block"])
def test_nothing_is_written_outside_the_workspace_and_the_output(name):
    shape, fp8, w, a = _layer(name)
    cfg = B.make_config(shape.H, shape.E, shape.k, shape.I, shape.shared_I, shape.T,
                        weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16)
    guard, pattern, n_ws, n_out = 4096, 0xA5, B.moe_ctx_workspace_bytes(cfg), 2 * shape.T * shape.H
    raws = [torch.full((n + 2 * guard,), pattern, dtype=torch.uint8, device=DEV) for n in (n_ws, n_out)]
    out = raws[1][guard:guard + n_out].view(torch.bfloat16).view(shape.T, shape.H)
    ctx = B.MoeContext(cfg, workspace=raws[0][guard:guard + n_ws])
    bufs = B.alloc_step_buffers(shape.T, shape.k, shape.E, DEV)
    torch.cuda.synchronize()
    for segments in (0, 7):
        ctx.moe_ctx_set_segments(segments)
        if fp8:
            ctx.layer_fp8(a["x"], a["logits"], None, w, out=out, bufs=bufs)
        else:
            ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"], out=out, bufs=bufs)
        assert _taken(ctx) == (1, 1)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK and torch.isfinite(out.float()).all()
    for raw in raws:
        assert bool((raw[:guard] == pattern).all()) and bool((raw[-guard:] == pattern).all())
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["shared expert of another length", "FP8, half a k-block"])
def test_beside_decode_steps_of_another_context(name):
    """Prefill batches on all SMs beside decode steps on a stream of higher priority, whose CTAs take single SMs of the
    pairs: both phases give what they give alone."""
    shape, fp8, w, a = _layer(name)
    fmt = B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16
    few = {k: (v[:48].contiguous() if k in ("x", "logits") else v) for k, v in a.items()}
    cfg = lambda T, phase: B.make_config(shape.H, shape.E, shape.k, shape.I, shape.shared_I, T, phase, weight_format=fmt)
    p = B.MoeContext(cfg(shape.T, B.MOE_PHASE_PREFILL), stream=torch.cuda.Stream())
    d = B.MoeContext(cfg(48, B.MOE_PHASE_DECODE), stream=torch.cuda.Stream(priority=-1))
    torch.cuda.synchronize()
    alone = _run(p, fp8, w, a), _run(d, fp8, w, few)
    torch.cuda.synchronize()
    outs = []
    for _ in range(6):
        outs.append((_run(p, fp8, w, a), *[_run(d, fp8, w, few) for _ in range(3)]))
        assert _taken(p) == (1, 1)
    torch.cuda.synchronize()
    assert p.moe_ctx_status() == B.MOE_OK and d.moe_ctx_status() == B.MOE_OK
    assert all(torch.equal(o[0], alone[0]) and all(torch.equal(x, alone[1]) for x in o[1:]) for o in outs)
    p.close()
    d.close()
