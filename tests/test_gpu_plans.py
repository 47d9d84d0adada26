"""The tensor maps a context keeps between steps: another T, other weights, another x and the other buffer set must each
be seen, and the rows a kept map reaches past the current batch must not matter, whatever they hold."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("phase", [B.MOE_PHASE_PREFILL, B.MOE_PHASE_DECODE])
@pytest.mark.parametrize("variant", [B.MOE_GEMM_SMALL_M, B.MOE_GEMM_LARGE_M])
def test_kept_maps_follow_every_operand(variant, phase, fp8):
    cap = 530  # three chunks of the dense group at the largest T, one box size of 16 rows at the smallest
    shape = wl.LayerShape("t", T=cap, H=128, E=6, k=2, I=128, shared_I=64)
    make = wl.make_weights_fp8 if fp8 else wl.make_weights
    weights = [make(shape, s, DEV) for s in (71, 72)]

    def step(ctx, a, w):
        if fp8:
            return ctx.layer_fp8(a["x"], a["logits"], None, w)[0]
        return ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])[0]

    def context():
        cfg = B.make_config(128, 6, 2, 128, 64, cap, phase, gemm_variant=variant,
                            weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16)
        ws = torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV)  # NaN in every format
        return B.MoeContext(cfg, workspace=ws)

    kept = context()
    for i, T in enumerate((cap, 3, 257, 16, 513, 1, 256, cap)):
        a = wl.make_activations(shape.with_tokens(T), 80 + i, DEV)
        fresh = context()
        torch.cuda.synchronize()
        w = weights[(i >> 1) & 1]
        want, got = step(fresh, a, w), step(kept, a, w)
        torch.cuda.synchronize()
        assert fresh.moe_ctx_status() == B.MOE_OK and kept.moe_ctx_status() == B.MOE_OK
        assert torch.isfinite(want.float()).all()
        assert torch.equal(want, got), f"T={T}"
        fresh.close()
    kept.close()
