"""Both passes and the combine of a few tokens in one launch, against the launches of the small-M kernel, bit for bit: groups of
one to sixty-four rows, one expert and 512, rows that end within a feature tile, more tiles than CTAs and fewer, both buffer
sets, steps on either side of the rule in turn (the launches tell which); infinities and NaN; a step whose waits run out."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _step(ctx, a, logits, bias, w, T):
    return ctx.layer(a["x"][:T], logits[:T], bias, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])


def _context(shape, phase, variant, budget):
    cfg = B.make_config(shape.H, shape.E, shape.k, shape.I, shape.shared_I, shape.T, phase, gemm_variant=variant, sm_budget=budget)
    return B.MoeContext(cfg, workspace=torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV))


# at_once: the largest T that the rule makes in one launch (148 SMs)
@pytest.mark.parametrize("E,k,H,I,shared,budget,at_once", [
    (1, 1, 64, 256, 0, 0, 64), (8, 2, 256, 512, 0, 0, 64), (5, 5, 192, 320, 256, 12, 17), (33, 4, 1344, 704, 320, 0, 3),
    (128, 8, 2048, 768, 0, 0, 3), (512, 8, 2560, 640, 512, 0, 17), (64, 16, 704, 2112, 0, 148, 1),
    (4, 2, 2048, 1024, 0, 0, 64), (2, 2, 1024, 1536, 512, 0, 64), (3, 3, 640, 2048, 192, 0, 64),  # groups of up to 64 rows, K up to 2048
    (64, 8, 2048, 1024, 0, 0, 17), (6, 3, 3072, 512, 0, 0, 33),                                   # ... of up to 17 and 33, more tiles than CTAs
    (8, 8, 128, 64, 0, 0, 64), (16, 16, 320, 64, 64, 0, 64), (16, 4, 1344, 128, 64, 0, 3),        # passes of one k-block and two
])
@pytest.mark.parametrize("phase", [B.MOE_PHASE_PREFILL, B.MOE_PHASE_DECODE])
def test_one_launch_is_the_small_m_kernels(E, k, H, I, shared, budget, at_once, phase):
    shape = wl.LayerShape("s", T=64, H=H, E=E, k=k, I=I, shared_I=shared)
    w, a = wl.make_weights(shape, 31, DEV), wl.make_activations(shape, 32, DEV)
    bias = torch.linspace(3.0, 0.0, E, device=DEV) if E > 8 else None  # experts of many rows and of none
    one, many = (_context(shape, phase, v, budget) for v in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M))
    torch.cuda.synchronize()
    for T in (1, 16, 3, 17, 64, 33, 63, 2):
        n0 = one.moe_ctx_launch_count()
        got, want = (_step(c, a, a["logits"], bias, w, T) for c in (one, many))
        assert one.moe_ctx_launch_count() - n0 == (2 if T <= at_once else 4), T
        torch.cuda.synchronize()
        assert one.moe_ctx_status() == B.MOE_OK and many.moe_ctx_status() == B.MOE_OK
        assert torch.equal(got[0], want[0]), T
        for name in want[1]:
            assert torch.equal(got[1][name], want[1][name]), (T, name)
    one.close(), many.close()


def test_infinities_and_nan_stay_in_their_rows():
    """A token of NaN, one of infinities and an expert with an infinite weight: the rows beside them in the same tiles do not see them."""
    E, k, H, I, T = 4, 2, 512, 256, 60
    shape = wl.LayerShape("s", T=T, H=H, E=E, k=k, I=I, shared_I=256)
    w, a = wl.make_weights(shape, 81, DEV), wl.make_activations(shape, 82, DEV)
    a["x"][7], a["x"][22, ::3] = float("nan"), float("inf")
    w["w_down"][3, 5, 17] = float("inf")
    one, many = (_context(shape, B.MOE_PHASE_DECODE, v, 0) for v in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M))
    torch.cuda.synchronize()
    got, want = (_step(c, a, a["logits"], None, w, T) for c in (one, many))
    torch.cuda.synchronize()
    assert one.moe_ctx_launch_count() == 2 and many.moe_ctx_launch_count() == 4
    assert torch.equal(torch.isnan(got[0]), torch.isnan(want[0])) and torch.equal(got[0].nan_to_num(0.0), want[0].nan_to_num(0.0))
    clean = torch.ones(T, H, dtype=torch.bool, device=DEV)
    clean[7] = clean[22] = False
    clean[(got[1]["topk_idx"] == 3).any(1), 5] = False
    assert torch.isfinite(got[0][clean]).all() and not torch.isfinite(got[0][~clean]).all()
    one.close(), many.close()


def test_a_wait_that_runs_out_is_reported_and_the_next_step_is_right():
    shape = wl.LayerShape("s", T=20, H=256, E=16, k=4, I=512, shared_I=256)
    w, a = wl.make_weights(shape, 41, DEV), wl.make_activations(shape, 42, DEV)
    ctx = _context(shape, B.MOE_PHASE_DECODE, B.MOE_GEMM_AUTO, 0)
    torch.cuda.synchronize()
    want = _step(ctx, a, a["logits"], None, w, 20)[0].clone()
    ctx.moe_ctx_set_wait_limit(20000)
    ctx.moe_ctx_debug_inject_stall(True)
    _step(ctx, a, a["logits"], None, w, 20)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_ERR_TIMEOUT
    ctx.moe_ctx_debug_inject_stall(False)
    got = _step(ctx, a, a["logits"], None, w, 20)[0]
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK and torch.equal(got, want)
    ctx.close()


def test_a_captured_step_starts_its_counters_anew():
    shape = wl.LayerShape("s", T=40, H=512, E=12, k=3, I=320, shared_I=256)
    w = wl.make_weights(shape, 71, DEV)
    args = (None, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])
    ctx = _context(shape, B.MOE_PHASE_PREFILL, B.MOE_GEMM_AUTO, 0)
    a = wl.make_activations(shape, 72, DEV)
    bufs, out = B.alloc_step_buffers(40, 3, 12, DEV), torch.empty(40, 512, dtype=torch.bfloat16, device=DEV)
    ctx.layer(a["x"], a["logits"], *args, out=out, bufs=bufs)
    torch.cuda.synchronize()
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    cap = B.MoeContext(B.make_config(512, 12, 3, 320, 256, 40), stream=s)
    with torch.cuda.stream(s):
        cap.layer(a["x"], a["logits"], *args, out=out, bufs=bufs)
    s.synchronize()
    with torch.cuda.graph(graph, stream=s):
        cap.layer(a["x"], a["logits"], *args, out=out, bufs=bufs)
    for seed in (73, 74, 75):
        b = wl.make_activations(shape, seed, DEV)
        want = ctx.layer(b["x"], b["logits"], *args)[0]
        a["x"].copy_(b["x"])
        a["logits"].copy_(b["logits"])
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    assert cap.moe_ctx_status() == B.MOE_OK
    ctx.close(), cap.close()
