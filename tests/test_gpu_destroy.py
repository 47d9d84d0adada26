"""What moe_ctx_destroy asks about: the context's own launches, wherever its step stopped, and nothing that the caller put on
the stream behind them."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"
SHAPE = wl.LayerShape("t", T=96, H=128, E=6, k=2, I=64)


def _stop_at(ctx, where, w, a, bufs, out):
    lay = (bufs["counts"], bufs["offsets"], bufs["perm"], bufs["inv_perm"])
    if where == "failed layer":
        with pytest.raises(B.MoeError):
            ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], None, out=out, bufs=bufs)
        return
    if where == "layer":
        ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"], out=out, bufs=bufs)
        return
    ctx.moe_route(a["logits"], None, bufs["topk_idx"], bufs["topk_w"])
    if where == "route":
        return
    if where in ("notify", "move"):
        ctx.moe_dispatch_notify(bufs["topk_idx"], *lay)
        if where == "move":
            ctx.moe_dispatch_move(a["x"])
        return
    ctx.moe_dispatch_layout(bufs["topk_idx"], None if where == "layout" else a["x"], *lay)
    if where in ("ffn", "abandoned"):
        ctx.moe_grouped_ffn(w["w_gate_up"], w["w_down"], a["x"])
    if where == "abandoned":
        ctx.moe_ctx_abandon_step()


@pytest.mark.parametrize("where", ["route", "layout", "notify", "move", "rows", "ffn", "abandoned", "failed layer", "layer"])
@pytest.mark.parametrize("T", [3, 96])
def test_destroy_asks_about_the_contexts_own_launches(where, T):
    w, a = wl.make_weights(SHAPE, 1, DEV), wl.make_activations(SHAPE, 2, DEV, T=T)
    bufs, out = B.alloc_step_buffers(T, 2, 6, DEV), torch.empty(T, 128, dtype=torch.bfloat16, device=DEV)
    s = torch.cuda.Stream()
    for busy in (False, True):  # the stream busy behind the context's launches, then before them
        ctx = B.MoeContext(B.make_config(128, 6, 2, 64, 0, 96), stream=s)
        _stop_at(ctx, "layer", w, a, bufs, out)  # kernels loaded and configured
        torch.cuda.synchronize()
        if busy:
            with torch.cuda.stream(s):
                torch.cuda._sleep(60_000_000)  # about 30 ms
            _stop_at(ctx, where, w, a, bufs, out)
            with pytest.raises(B.MoeError) as err:
                ctx.destroy()
            assert err.value.status == B.MOE_ERR_STATE
            s.synchronize()
        else:
            _stop_at(ctx, where, w, a, bufs, out)
            s.synchronize()
            with torch.cuda.stream(s):
                torch.cuda._sleep(60_000_000)
        ctx.destroy()
        assert s.query() == busy
        s.synchronize()


@pytest.mark.parametrize("T", [0, 5])
def test_a_context_may_go_as_soon_as_the_host_path_returns(T):
    w, a = wl.make_weights(SHAPE, 1, DEV), wl.make_activations(SHAPE, 2, DEV, T=T)
    hl, hx, out = a["logits"].cpu().pin_memory(), a["x"].cpu().pin_memory(), torch.empty(T, 128, dtype=torch.bfloat16).pin_memory()
    for _ in range(5):
        ctx = B.MoeContext(B.make_config(128, 6, 2, 64, 0, 96))
        torch.cuda.synchronize()
        ctx.moe_layer_host(hl, None, hx, w["w_gate_up"], w["w_down"], None, None, out)
        ctx.destroy()
