"""AUTO on either side of the lines that depend on the number of tiles and on short K: whichever kernel it takes, the result
is that of both, bit for bit (the order of the sums is the same).  Which one it takes is asked on a context with part of the
SMs, which never takes the pair kernel."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl
from test_rules_cpu import rules  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("H,I,E,T,fp8", [
    (1152, 128, 221, 8300, False), (1152, 128, 222, 8300, False),    # one and a half waves of tiles, gated pass
    (1088, 128, 222, 14208, False), (1088, 128, 222, 14209, False),  # shorter K: 64 rows per expert
    (640, 128, 591, 38479, False), (640, 128, 592, 38481, False),    # ... or four waves
    (1024, 640, 222, 14208, False), (1024, 640, 222, 14209, False),  # down pass
    (1792, 128, 222, 14208, True), (1792, 128, 222, 14209, True),    # FP8, gated pass
    (2432, 256, 111, 22200, True), (2432, 256, 111, 22201, True),    # ... of few features: 200
])
def test_auto_equals_both_variants(H, I, E, T, fp8):
    shape = wl.LayerShape("t", T=T, H=H, E=E, k=1, I=I)
    w = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 3, DEV)
    a = wl.make_activations(shape, 4, DEV)
    outs = []
    for variant in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M, B.MOE_GEMM_LARGE_M):
        ctx = B.MoeContext(B.make_config(H, E, 1, I, 0, T, gemm_variant=variant,
                                         weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16))
        torch.cuda.synchronize()
        out, _ = ctx.layer_fp8(a["x"], a["logits"], None, w) if fp8 else \
            ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])
        torch.cuda.synchronize()
        assert ctx.moe_ctx_status() == B.MOE_OK
        outs.append(out)
        ctx.close()
    assert torch.isfinite(outs[0].float()).all()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


@pytest.mark.parametrize("H,I,k,fp8,below,above,down", [
    # (experts, tokens) on either side of a line of the context on 147 SMs, which never takes pairs; the pass that changes
    (2560, 1024, 8, False, (24, 1050), (24, 1051), True),      # down pass: 350 rows per expert
    (1024, 640, 1, False, (222, 14208), (222, 14209), True),   # ... of shorter K: 64
    (1152, 128, 1, False, (220, 8300), (221, 8300), False),    # gated pass: one and a half waves of tiles
    (1088, 128, 1, False, (222, 14208), (222, 14209), False),  # ... of shorter K: 64 rows per expert
    (640, 128, 1, False, (587, 38479), (588, 38479), False),   # ... or four waves
    (1792, 128, 1, True, (222, 14208), (222, 14209), False),   # FP8, gated pass: 64
    (2560, 1024, 8, True, (28, 1050), (28, 1051), False),      # ... of longer K: 300
    (2432, 256, 1, True, (111, 22200), (111, 22201), False),   # ... and few features: 200
    (2560, 1024, 8, True, (46, 1035), (46, 1036), True),       # FP8, down pass: 180
    (4096, 2048, 8, True, (21, 1050), (21, 1051), True),       # ... of longer K: 400
])
def test_a_context_on_part_of_the_sms_changes_over(rules, H, I, k, fp8, below, above, down):  # noqa: F811
    name = {B.MOE_GEMM_SMALL_M: 1, B.MOE_GEMM_LARGE_M: 0}
    taken = []
    for E, T in (below, above):
        shape = wl.LayerShape("t", T=T, H=H, E=E, k=k, I=I)
        w = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 3, DEV)
        a = wl.make_activations(shape, 4, DEV)
        outs = []
        for variant in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M):
            ctx = B.MoeContext(B.make_config(H, E, k, I, 0, T, gemm_variant=variant, sm_budget=147,
                                             weight_format=B.MOE_WEIGHTS_FP8_E4M3 if fp8 else B.MOE_WEIGHTS_BF16))
            torch.cuda.synchronize()
            out, _ = ctx.layer_fp8(a["x"], a["logits"], None, w) if fp8 else \
                ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])
            torch.cuda.synchronize()
            assert ctx.moe_ctx_status() == B.MOE_OK
            outs.append(out)
            if variant == B.MOE_GEMM_AUTO:
                g = ctx.moe_ctx_debug_gemm()
                taken.append([name[g["gated"]], name[g["down"]]])
            ctx.close()
        assert torch.isfinite(outs[0].float()).all() and torch.equal(outs[0], outs[1])
        rows = f"{T * k}LL, {E}, 147"
        assert taken[-1] == rules(f"moe::small_m_is_faster({int(fp8)}, 1, {H}, {I}, {rows})",
                                  f"moe::small_m_is_faster({int(fp8)}, 0, {I}, {H}, {rows})")
    assert taken[0][down] != taken[1][down] and taken[0][not down] == taken[1][not down]
