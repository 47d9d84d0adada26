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


# AUTO takes the pair kernel for both passes of T = 2049 and more, and the small-M kernel below
PAIR_LAYER = dict(H=1344, E=48, k=4, I=704, shared_I=320)


def _pair_step(ctx, fp8, a, w, taken):
    if fp8:
        out, _ = ctx.layer_fp8(a["x"], a["logits"], None, w)
    else:
        out, _ = ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])
    g = ctx.moe_ctx_debug_gemm()
    assert (g["gated"], g["down"]) == (taken, taken)
    return out


def _pair_context(cap, fp8):
    p = PAIR_LAYER
    cfg = B.make_config(p["H"], p["E"], p["k"], p["I"], p["shared_I"], cap,
                        weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16)
    ws = torch.full((B.moe_ctx_workspace_bytes(cfg),), 0xFF, dtype=torch.uint8, device=DEV)  # NaN in every format
    return B.MoeContext(cfg, workspace=ws)


@pytest.mark.parametrize("fp8", [False, True])
def test_a_change_of_kernel_keeps_the_maps(fp8):
    """Batches that take the pair and the small-M kernel in turn: each kernel's maps are encoded once."""
    shape = wl.LayerShape("t", T=2101, **PAIR_LAYER)
    w = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 71, DEV)
    batches = [(wl.make_activations(shape.with_tokens(T), 80, DEV), taken)
               for T, taken in ((2101, B.MOE_KERNEL_PAIR), (300, B.MOE_GEMM_SMALL_M))]
    ctx = _pair_context(2101, fp8)
    torch.cuda.synchronize()
    first = [_pair_step(ctx, fp8, a, w, taken) for a, taken in batches]
    encoded = ctx.moe_ctx_debug_gemm()["maps_encoded"]
    for _ in range(3):
        assert all(torch.equal(_pair_step(ctx, fp8, a, w, taken), out) for (a, taken), out in zip(batches, first))
    assert ctx.moe_ctx_debug_gemm()["maps_encoded"] == encoded
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.close()


@pytest.mark.parametrize("fp8", [False, True])
def test_the_pair_kernels_maps_follow_every_operand(fp8):
    cap = 2700
    shape = wl.LayerShape("t", T=cap, **PAIR_LAYER)
    weights = [(wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, s, DEV) for s in (71, 72)]
    kept = _pair_context(cap, fp8)
    # nine to eleven chunks of the dense group, of 240 or 256 rows, the last one of 144 to 256
    for i, T in enumerate((cap, 2305, 3, 2321, 2304, 2556, 2064, cap)):
        a = wl.make_activations(shape.with_tokens(T), 80 + i, DEV)
        fresh = _pair_context(cap, fp8)
        torch.cuda.synchronize()
        w = weights[(i >> 1) & 1]
        taken = B.MOE_KERNEL_PAIR if T > 2048 else B.MOE_GEMM_SMALL_M
        want, got = _pair_step(fresh, fp8, a, w, taken), _pair_step(kept, fp8, a, w, taken)
        torch.cuda.synchronize()
        assert fresh.moe_ctx_status() == B.MOE_OK and kept.moe_ctx_status() == B.MOE_OK
        assert torch.isfinite(want.float()).all()
        assert torch.equal(want, got), f"T={T}"
        fresh.close()
    kept.close()
