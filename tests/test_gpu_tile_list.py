"""The small-M kernel's tile list (experts by size class) where it can go wrong: expert counts around the group size of
32 and at the limit, experts of every size class from empty to several chunks, ties within a class."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_layer_strict, np_f32, np_i32
from paper_2609_00993_b200 import binding as B
from paper_2609_00993_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T,E,k,zipf", [
    (17, 1, 1, 0.0),       # the first size at which the list is ordered
    (65, 31, 3, 0.0),
    (700, 32, 4, 1.6),     # one expert of several 256-row chunks, the rest down to a few rows
    (300, 33, 2, 1.2),     # one expert past a group of 32
    (260, 511, 2, 0.0),    # most experts empty or of one row
    (2000, 1024, 4, 1.2),  # the largest E
])
def test_ordered_tile_list(T, E, k, zipf):
    shape = wl.LayerShape("t", T=T, H=64, E=E, k=k, I=64, zipf_s=zipf)
    w, a = wl.make_weights(shape, 61, DEV), wl.make_activations(shape, 62, DEV)
    for n in ("w_gate_up", "w_down"):
        w[n] = (w[n].float() * (1.0 / (0.02 * 8.0))).to(torch.bfloat16)  # unit-variance pre-activations
    ctx = B.MoeContext(B.make_config(64, E, k, 64, 0, T, B.MOE_PHASE_DECODE))
    torch.cuda.synchronize()
    out, bufs = ctx.layer(a["x"], a["logits"], None, w["w_gate_up"], w["w_down"])
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_OK
    ref = oracle.layer(wl.bits(a["x"]), np_f32(a["logits"]), None, k, wl.bits(w["w_gate_up"]), wl.bits(w["w_down"]))
    assert np.array_equal(np_i32(bufs["counts"]), ref["counts"])
    check_layer_strict(out, ref, f"T={T} E={E} k={k}")
    ctx.close()
