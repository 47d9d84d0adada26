"""A few tokens routed, laid out and moved in one launch (FP8 rows are quantised and moved in a second) against the calls
of the stages, bit for bit, and the oracle's layout: token counts at which the CTAs and clusters change, the last one and
the first behind it; expert counts that vectorise, that do not and that are too many; more pieces of a row than one and a
last piece that is not full; ties."""
import numpy as np
import pytest
import torch

import oracle
from helpers import np_i32
from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T,E,k,H", [
    (1, 1, 1, 64), (1, 256, 8, 7168), (4, 5, 5, 2112), (5, 33, 7, 64), (8, 512, 8, 2048), (9, 100, 4, 4160), (16, 128, 8, 4096),
    (17, 256, 2, 64), (31, 8, 2, 320), (32, 32, 32, 128), (33, 130, 3, 2112), (40, 512, 10, 64), (63, 16, 16, 2048), (64, 64, 16, 64),
    (64, 63, 17, 64), (65, 64, 2, 64), (16, 513, 2, 64),  # the three stages: too many slots, tokens, experts
])
@pytest.mark.parametrize("mode", ["bf16", "gather", "fp8"])
def test_one_launch_is_the_three_stages(T, E, k, H, mode):
    fp8, gather = mode == "fp8", mode == "gather"
    shape = wl.LayerShape("s", T=T, H=H, E=E, k=k, I=64, shared_I=64)
    w, a = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 61, DEV), wl.make_activations(shape, 62, DEV)
    g = torch.Generator(device=DEV).manual_seed(T * 1000 + E)
    bias = torch.randn(E, generator=g, device=DEV).round() if T % 2 else None
    logits = torch.where(torch.rand(T, E, generator=g, device=DEV) < 0.5, a["logits"], a["logits"].round())
    logits[T // 2] = 0.0 if T > 1 else logits[0]  # more keys tied than a warp's list holds
    ffn = [w[n] for n in ("wq_gate_up", "sw_gate_up", "wq_down", "sw_down", "wsq_gate_up", "sws_gate_up", "wsq_down", "sws_down")] if fp8 else \
        [w["w_gate_up"], w["w_down"], a["x"], w["ws_gate_up"], w["ws_down"]]
    res, launches = [], []
    for at_once in (True, False):
        cfg = B.make_config(H, E, k, 64, 64, 70, row_gather=int(gather),
                            # (AUTO could make the passes and the combine in one launch, too; the count is of the dispatch)
                            gemm_variant=B.MOE_GEMM_LARGE_M if gather else B.MOE_GEMM_SMALL_M,
                            weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16)
        ws = torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV)
        ctx = B.MoeContext(cfg, workspace=ws)
        bufs, out = B.alloc_step_buffers(T, k, E, DEV), torch.empty(T, H, dtype=torch.bfloat16, device=DEV)
        torch.cuda.synchronize()
        if at_once and fp8:
            ctx.layer_fp8(a["x"], logits, bias, w, out=out, bufs=bufs)
        elif at_once:
            ctx.layer(a["x"], logits, bias, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"], out=out, bufs=bufs)
        else:
            ctx.moe_route(logits, bias, bufs["topk_idx"], bufs["topk_w"])
            ctx.moe_dispatch_layout(bufs["topk_idx"], a["x"], bufs["counts"], bufs["offsets"], bufs["perm"], bufs["inv_perm"])
            ctx.moe_grouped_ffn_fp8(*ffn, T=T) if fp8 else ctx.moe_grouped_ffn(*ffn)
            ctx.moe_combine(bufs["topk_w"], bufs["inv_perm"], out)
        torch.cuda.synchronize()
        assert ctx.moe_ctx_status() == B.MOE_OK
        rows = {}
        if fp8:
            rows["xq"] = ctx.fp8_debug_view("xq", (T * k, H), torch.uint8).clone()
        elif not gather:
            rows["x_perm"] = ctx.moe_ctx_debug_ptrs()["x_perm"][:T * k].clone()
        launches.append(ctx.moe_ctx_launch_count())
        res.append({**bufs, "out": out, **rows})
        ctx.close()
    fits = T <= 64 and T * k <= 1024 and E <= 512
    assert launches[1] - launches[0] == (0 if not fits else 2 if mode == "bf16" else 1)
    for name, t in res[0].items():
        assert torch.equal(t, res[1][name]), name
    for got, want in zip((res[0][n] for n in ("counts", "offsets", "perm", "inv_perm")),
                         oracle.layout(np_i32(res[0]["topk_idx"]).reshape(-1), E)):
        assert np.array_equal(np_i32(got), want)
