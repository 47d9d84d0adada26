"""Quantisation of rows, bit for bit against the oracle, at the lengths where its kernels change: one warp per row with one
to four 16-element pieces a lane, one CTA per row behind 2048 elements, rows that do not fill their last piece; values
spread over many binades, zero rows, the row's largest value in its last element."""
import numpy as np
import pytest
import torch

import oracle
from helpers import np_f32, np_i32
from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("H,I", [(64, 512), (576, 1024), (1088, 1536), (1600, 2048), (2048, 2112), (2112, 4096), (4160, 6144),
                                 (6208, 8192), (8192, 64)])
@pytest.mark.parametrize("T,k,shared_I", [(1, 1, 0), (9, 3, 64), (67, 2, 0)])
def test_rows_of_every_length(H, I, T, k, shared_I):
    shape = wl.LayerShape("q", T=T, H=H, E=4, k=k, I=I, shared_I=shared_I)
    w8, a = wl.make_weights_fp8(shape, 21, DEV), wl.make_activations(shape, 22, DEV)
    g = torch.Generator(device=DEV).manual_seed(23)
    x = (a["x"].float() * torch.exp2(torch.randint(-20, 20, (T, H), generator=g, device=DEV).float())).to(torch.bfloat16)
    x[T // 2, -1] = 3.0e5 * 2.0 ** 20
    if T > 2:
        x[0] = 0
    ctx = B.MoeContext(B.make_config(H, 4, k, I, shared_I, T, weight_format=B.MOE_WEIGHTS_FP8_E4M3))
    torch.cuda.synchronize()
    _, bufs = ctx.layer_fp8(x, a["logits"], None, w8)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    N = T * k
    act = wl.bits(ctx.moe_ctx_debug_ptrs()["act"][:N])
    for name, scale, rows, n in (("xq", "sx", oracle.permute(wl.bits(x), np_i32(bufs["perm"]).reshape(-1), k), H),
                                 ("aq", "sa", act, I)):
        q_ref, s_ref = oracle.quantize_rows(rows)
        assert np.array_equal(ctx.fp8_debug_view(name, (N, n), torch.uint8).cpu().numpy(), q_ref), name
        assert np.array_equal(np_f32(ctx.fp8_debug_view(scale, (N,), torch.float32)), s_ref), scale
    ctx.close()
