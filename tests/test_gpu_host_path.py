"""moe_layer_host against the device path, bit for bit, where its pieces and chunks have edges: one piece and several, a
last piece narrower than the others, one chunk and two (the second ragged), a decode context, pageable buffers."""
import pytest
import torch

from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"
P, D = B.MOE_PHASE_PREFILL, B.MOE_PHASE_DECODE


@pytest.mark.parametrize("phase,T,H,shared_I,pinned", [
    (P, 5, 256, 0, True),        # one piece
    (P, 700, 1216, 64, True),    # two pieces (768 + 448 columns), shared expert
    (P, 1700, 2112, 64, True),   # four pieces of 768 columns at most: three are enough, the last narrower
    (P, 4099, 1088, 0, True),    # two chunks of tokens, the second ragged
    (D, 1100, 1088, 64, True),   # a decode context: pieces, never chunks
    (P, 700, 1216, 64, False),   # pageable buffers: neither
])
def test_host_path_equals_device_path(phase, T, H, shared_I, pinned):
    shape = wl.LayerShape("t", T=T, H=H, E=12, k=2, I=128, shared_I=shared_I, select_bias=True)
    w, a = wl.make_weights(shape, 91, DEV), wl.make_activations(shape, 92, DEV)
    wargs = (w["w_gate_up"], w["w_down"], w["ws_gate_up"], w["ws_down"])
    ctx = B.MoeContext(B.make_config(H, 12, 2, 128, shared_I, T, phase))
    torch.cuda.synchronize()
    want, _ = ctx.layer(a["x"], a["logits"], a["bias"], *wargs)
    torch.cuda.synchronize()
    pin = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    hl, hx = pin(a["logits"].cpu()), pin(a["x"].cpu())
    for _ in range(2):  # twice: the second call finds the staging buffers used
        out = pin(torch.full((T, H), 7.0, dtype=torch.bfloat16))
        ctx.moe_layer_host(hl, a["bias"], hx, *wargs, out)
        assert torch.equal(out, want.cpu())
    assert ctx.moe_ctx_status() == B.MOE_OK
    ctx.close()
