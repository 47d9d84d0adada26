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


@pytest.mark.parametrize("T,I", [(1, 64), (5, 512), (66, 576), (7, 2112)])
def test_shared_rows_of_the_same_length_ride_along(T, I):
    """With shared_inter == inter the shared expert's activation is quantised in the routed rows' launch: the layer against
    the oracle's (worst case of the recipe: the bf16 layer's 5e-3), and bit for bit against a shared expert that cannot ride
    because it is padded with zero rows and columns (which add nothing to any sum)."""
    H, E, k = 256, 5, 2
    shape = wl.LayerShape("q", T=T, H=H, E=E, k=k, I=I, shared_I=I)
    w8, a = wl.make_weights_fp8(shape, 31, DEV, std=1.0), wl.make_activations(shape, 32, DEV)
    for name, fan in (("sw_gate_up", H), ("sws_gate_up", H), ("sw_down", I), ("sws_down", I)):
        w8[name] = (w8[name] / fan ** 0.5).contiguous()
    padded = dict(w8)
    g, u = w8["wsq_gate_up"][:I], w8["wsq_gate_up"][I:]
    z = torch.zeros(64, H, dtype=torch.uint8, device=DEV)
    padded["wsq_gate_up"] = torch.cat([g, z, u, z]).contiguous()
    one = torch.ones(64, device=DEV)
    padded["sws_gate_up"] = torch.cat([w8["sws_gate_up"][:I], one, w8["sws_gate_up"][I:], one]).contiguous()
    padded["wsq_down"] = torch.cat([w8["wsq_down"], torch.zeros(H, 64, dtype=torch.uint8, device=DEV)], dim=1).contiguous()
    outs = []
    for w, shared_I in ((w8, I), (padded, I + 64)):
        ctx = B.MoeContext(B.make_config(H, E, k, I, shared_I, T, weight_format=B.MOE_WEIGHTS_FP8_E4M3))
        torch.cuda.synchronize()
        out, _ = ctx.layer_fp8(a["x"], a["logits"], None, w)
        torch.cuda.synchronize()
        assert ctx.moe_ctx_status() == B.MOE_OK
        outs.append(out)
        ctx.close()
    assert torch.equal(outs[0], outs[1])
    h = {n: v.cpu().numpy() for n, v in w8.items()}
    ref = oracle.layer_fp8(wl.bits(a["x"]), np_f32(a["logits"]), None, k, h["wq_gate_up"], h["sw_gate_up"], h["wq_down"],
                           h["sw_down"], h["wsq_gate_up"], h["sws_gate_up"], h["wsq_down"], h["sws_down"])
    assert np.linalg.norm(np_f32(outs[0]) - ref["out"]) <= 5e-3 * np.linalg.norm(ref["out"])
