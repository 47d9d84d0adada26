"""AUTO on either side of lines of the kernel choice: whichever kernel it takes, the result is that of the small-M and the large-M
kernel, bit for bit (the order of the sums is the same).  These contexts have all SMs, so beyond some of the lines it is the pair
kernel that takes over, and with the shortest K the lines named below are those of an older choice; test_gpu_variant_lines.py has
both sides of today's lines and asks which kernel ran."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("H,I,E,k,T,fp8", [
    (128, 64, 70, 2, 4200, False), (128, 64, 70, 2, 4201, False),     # short K: 120 rows per expert, and behind
    (128, 64, 42, 2, 4200, False), (128, 64, 42, 2, 4201, False),     # short K, down pass: 200
    (2560, 1024, 24, 8, 1050, False), (2560, 1024, 24, 8, 1051, False),  # middle K, down pass: 350
    (256, 2048, 4, 1, 8193, False),                                   # long down K, first size behind the launch overlap
    (2560, 1024, 28, 8, 1050, True), (2560, 1024, 28, 8, 1051, True),    # FP8, middle K, gated pass: 300
    (2560, 1024, 46, 8, 1035, True), (2560, 1024, 46, 8, 1036, True),    # FP8, middle K, down pass: 180
    (4096, 2048, 21, 8, 1050, True), (4096, 2048, 21, 8, 1051, True),    # FP8, long K, down pass: 400
])
def test_auto_equals_both_variants(H, I, E, k, T, fp8):
    shape = wl.LayerShape("t", T=T, H=H, E=E, k=k, I=I)
    w = (wl.make_weights_fp8 if fp8 else wl.make_weights)(shape, 3, DEV)
    a = wl.make_activations(shape, 4, DEV)
    outs = []
    for variant in (B.MOE_GEMM_AUTO, B.MOE_GEMM_SMALL_M, B.MOE_GEMM_LARGE_M):
        ctx = B.MoeContext(B.make_config(H, E, k, I, 0, T, gemm_variant=variant,
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
