"""The FP8 kernels' waits that run out, as for bf16: the status word reports it, and the same context computes a correct step
afterwards; CTAs of one tile and of many.  The CPU half: nothing that waits without a limit stands inside the roles' loops."""
import os
import re

import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import build as build_mod
from paper_2609_00993_b200 import workloads as wl

DEV = "cuda"


@pytest.mark.parametrize("name", ["gemm_tc.cu", "gemm_stream.cu"])
def test_no_named_barrier_between_warps_that_give_up_by_themselves(name):
    """A warp leaves its tile loop when its bounded wait runs out, so a barrier among some of the warps (which has no limit)
    may miss one for good; the roles meet at __syncthreads behind their loops only, where every warp arrives."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(build_mod.CSRC, name)).read())
    assert not re.search(r"\bbar(rier)?(\.cta)?\.(sync|red)\b|__barrier_sync|named_barrier", text)
    loops = text[text.index("if (warp == kProducerWarp) {"):text.index("tc_fence_before();\n  __syncthreads();", text.index("if (warp == kProducerWarp) {"))]
    assert "__syncthreads" not in loops


@pytest.mark.gpu
@pytest.mark.parametrize("sm_budget", [0, 2])
@pytest.mark.parametrize("variant", [B.MOE_GEMM_LARGE_M, B.MOE_GEMM_SMALL_M])
def test_an_fp8_wait_that_runs_out_is_reported_and_the_context_stays_usable(variant, sm_budget):
    shape = wl.LayerShape("t", T=64, H=256, E=8, k=2, I=128, shared_I=64)
    w, a = wl.make_weights_fp8(shape, 1, DEV), wl.make_activations(shape, 2, DEV)
    ctx = B.MoeContext(B.make_config(256, 8, 2, 128, 64, 64, B.MOE_PHASE_PREFILL, gemm_variant=variant, sm_budget=sm_budget,
                                     weight_format=B.MOE_WEIGHTS_FP8_E4M3), device=DEV)
    torch.cuda.synchronize()
    good = ctx.layer_fp8(a["x"], a["logits"], None, w)[0].clone()
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.moe_ctx_set_wait_limit(20_000)
    ctx.moe_ctx_debug_inject_stall(True)
    ctx.layer_fp8(a["x"], a["logits"], None, w)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_ERR_TIMEOUT
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.moe_ctx_debug_inject_stall(False)
    ctx.moe_ctx_set_wait_limit(0)
    again = ctx.layer_fp8(a["x"], a["logits"], None, w)[0]
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK and torch.equal(again, good)
    ctx.close()
