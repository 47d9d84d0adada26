"""Stage times are those of the kernels that a step launches without them: the same launches, and a bracket around each that
the stages name, where a few tokens are dispatched in one launch and where they are not."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T,fp8,stages", [
    (64, False, {"route", "ffn_combine"}),  # both passes and the combine in one launch
    (65, False, {"route", "layout", "permute", "gemm1_swiglu", "gemm2", "combine"}),
    (64, True, {"route", "quantize_x", "gemm1_swiglu", "quantize_act", "gemm2", "combine"}),
    (65, True, {"route", "layout", "quantize_x", "gemm1_swiglu", "quantize_act", "gemm2", "combine"}),
])
def test_stage_times_are_those_of_the_step(T, fp8, stages):
    _check(wl.LayerShape("t", T=T, H=256, E=8, k=2, I=128), fp8, stages)


@pytest.mark.parametrize("T,H,E,k,I,stages", [
    (3, 2048, 128, 8, 768, {"route", "ffn_combine"}),
    (64, 2048, 128, 8, 256, {"route", "gemm1_swiglu", "gemm2", "combine"}),  # too many slots for one launch
    (2047, 1856, 64, 8, 512, {"route", "layout", "gemm1_swiglu", "gemm2", "combine"}),             # the gated pass gathers
    (2048, 1856, 64, 8, 512, {"route", "layout", "permute", "gemm1_swiglu", "gemm2", "combine"}),
])
def test_stages_that_are_one_launch_or_none(T, H, E, k, I, stages):
    _check(wl.LayerShape("t", T=T, H=H, E=E, k=k, I=I), False, stages)


def _check(shape, fp8, stages):
    T = shape.T
    w, a = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 1, DEV), wl.make_activations(shape, 2, DEV)
    ctx = B.MoeContext(B.make_config(shape.H, shape.E, shape.k, shape.I, 0, T, weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16))
    torch.cuda.synchronize()
    outs, launches = [], []
    for profiling in (False, True):
        ctx.moe_ctx_set_profiling(profiling)
        n0 = ctx.moe_ctx_launch_count()
        out = ctx.layer_fp8(a["x"], a["logits"], None, w)[0] if fp8 else \
            ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])[0]
        torch.cuda.synchronize()
        outs.append(out)
        launches.append(ctx.moe_ctx_launch_count() - n0)
    prof = ctx.moe_ctx_read_profile()
    ctx.close()
    assert launches[0] == launches[1] == len(stages) and torch.equal(outs[0], outs[1])
    assert {name: calls for name, (_, calls) in prof.items() if calls} == {name: 1 for name in stages}
    assert all(prof[name][0] > 0 for name in stages)
