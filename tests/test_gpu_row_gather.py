"""Whole prefill steps whose gated pass gathers its rows, against the kernel that reads moved rows, bit for bit: experts of no row, of one,
of a tile, of several and of all tokens; tiles that end within 8, 16 and 256 rows; the shared expert's rows; part of the SMs;
the rows and bounds at which the rule begins and ends; host buffers."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("H,E,k,I,shared,T,budget,gathers", [
    (1856, 64, 4, 704, 320, 2049, 0, True), (1856, 64, 4, 704, 320, 2048, 0, False),     # 8192 rows and more
    (1856, 64, 4, 704, 320, 2304, 0, True), (1856, 64, 4, 704, 320, 2305, 0, False),     # 144 rows per expert
    (1856, 64, 8, 512, 0, 2047, 0, True), (1856, 64, 8, 512, 0, 2048, 0, False),         # 256 rows per expert and fewer
    (2560, 512, 8, 320, 0, 1111, 0, True), (3072, 40, 9, 704, 576, 997, 0, True), (3072, 40, 9, 448, 576, 997, 37, False),
])
@pytest.mark.parametrize("skewed", [False, True])
def test_gathered_rows_are_the_moved_ones(H, E, k, I, shared, T, budget, gathers, skewed):
    shape = wl.LayerShape("g", T=T, H=H, E=E, k=k, I=I, shared_I=shared)
    w, a = wl.make_weights(shape, 51, DEV), wl.make_activations(shape, 52, DEV)
    # skewed: two experts get every token, the last third of the experts next to none
    bias = torch.cat([torch.full((2,), 9.0), torch.zeros(E - 2 - E // 3), torch.full((E // 3,), -4.0)]).to(DEV) if skewed else None
    res = []
    for variant in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M):
        cfg = B.make_config(H, E, k, I, shared, T, B.MOE_PHASE_PREFILL, gemm_variant=variant, sm_budget=budget)
        ctx = B.MoeContext(cfg, workspace=torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV))
        torch.cuda.synchronize()
        for _ in range(2):
            n0 = ctx.moe_ctx_launch_count()
            out, bufs = ctx.layer(a["x"], a["logits"], bias, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])
            n = ctx.moe_ctx_launch_count() - n0
        torch.cuda.synchronize()
        assert ctx.moe_ctx_status() == B.MOE_OK
        if variant == B.MOE_GEMM_AUTO:
            assert ctx.moe_ctx_debug_gemm()["gated"] == B.MOE_GEMM_SMALL_M
        res.append((out, bufs, ctx.moe_ctx_debug_ptrs()["act"][:T * k].clone(), n))
        ctx.close()
    got, want = res
    assert want[3] - got[3] == (1 if gathers else 0)
    assert torch.equal(got[2], want[2]) and torch.equal(got[0], want[0])
    assert all(torch.equal(got[1][n], want[1][n]) for n in want[1])


def test_gathered_from_host_buffers():
    shape = wl.LayerShape("g", T=1531, H=2048, E=128, k=8, I=256)
    w, a = wl.make_weights(shape, 53, DEV), wl.make_activations(shape, 54, DEV)
    ctx = B.MoeContext(B.make_config(2048, 128, 8, 256, 0, 1531, B.MOE_PHASE_PREFILL))
    want = ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])[0]
    x, logits = a["x"].cpu().pin_memory(), a["logits"].cpu().pin_memory()
    out = torch.empty(1531, 2048, dtype=torch.bfloat16).pin_memory()
    for _ in range(2):  # the call that creates the copy stream, and one that has it
        out.zero_()
        ctx.moe_layer_host(logits, None, x, w["w_gate_up"], w["w_down"], None, None, out)
        assert torch.equal(out, want.cpu())
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.close()


@pytest.mark.parametrize("H,E,k,I", [(2048, 128, 8, 768), (1024, 512, 8, 128)])
@pytest.mark.parametrize("then", ["", "segments", "preemption"])
@pytest.mark.parametrize("path", ["device", "host"])
def test_a_gathered_batch_leaves_nothing_to_the_next_one(H, E, k, I, then, path):
    """One context, batches that gather and batches that do not in turn, each against a context of its own."""
    sizes = (2001, 37, 2001, 64, 1, 300, 1531, 7)
    w = wl.make_weights(wl.LayerShape("g", T=1, H=H, E=E, k=k, I=I), 55, DEV)

    def context(switched):
        cfg = B.make_config(H, E, k, I, 0, max(sizes), B.MOE_PHASE_PREFILL)
        ctx = B.MoeContext(cfg, workspace=torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV))
        if switched:
            switch(ctx)
        return ctx

    def switch(ctx):
        if then == "segments":
            ctx.moe_ctx_set_segments(E // 2, lambda i, n: None)
        elif then == "preemption":
            ctx.moe_ctx_set_preemption(True)

    def step(ctx, a, T):
        if path == "device":
            out, bufs = ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])
            torch.cuda.synchronize()
            return {"out": out, **bufs}
        out = torch.zeros(T, H, dtype=torch.bfloat16).pin_memory()
        ctx.moe_layer_host(a["logits"].cpu().pin_memory(), None, a["x"].cpu().pin_memory(), w["w_gate_up"], w["w_down"], None, None, out)
        return {"out": out}

    kept = context(False)
    for i, T in enumerate(sizes):
        a = wl.make_activations(wl.LayerShape("g", T=T, H=H, E=E, k=k, I=I), 56 + i, DEV)
        fresh = context(i > 0)
        torch.cuda.synchronize()
        want, got = step(fresh, a, T), step(kept, a, T)
        assert fresh.moe_ctx_status() == B.MOE_OK and kept.moe_ctx_status() == B.MOE_OK
        assert torch.isfinite(want["out"].float()).all()
        for name in want:
            assert torch.equal(got[name], want[name]), (T, name)
        fresh.close()
        if i == 0:
            switch(kept)
    kept.close()


def test_a_step_whose_passes_are_refused_has_moved_its_rows():
    """The staged calls go on from there, as behind a step that does not gather."""
    T, H, E, k, I = 1100, 2048, 128, 8, 256
    shape = wl.LayerShape("g", T=T, H=H, E=E, k=k, I=I)
    w, a = wl.make_weights(shape, 57, DEV), wl.make_activations(shape, 58, DEV)
    cfg = B.make_config(H, E, k, I, 0, T, B.MOE_PHASE_PREFILL)
    ctx = B.MoeContext(cfg, workspace=torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV))
    bufs, out = B.alloc_step_buffers(T, k, E, DEV), torch.empty(T, H, dtype=torch.bfloat16, device=DEV)
    torch.cuda.synchronize()
    with pytest.raises(B.MoeError, match="weights are NULL"):
        ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], None, out=out, bufs=bufs)
    ctx.moe_grouped_ffn(w["w_gate_up"], w["w_down"], None, T=T)
    ctx.moe_combine(bufs["topk_w"], bufs["inv_perm"], out)
    want = ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])[0]
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    assert torch.isfinite(want.float()).all() and torch.equal(out, want)
    ctx.close()
