"""AUTO on either side of the lines that depend on the number of tiles and on short K: whichever kernel it takes, the result
is that of both, bit for bit (the order of the sums is the same).  Which one it takes is tested in test_rules_cpu.py."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

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
