"""The dispatch layout at the edges of its chunks: one step per warp and several, one CTA and many, the last size whose
CTAs count every chunk themselves and the first that counts in a launch of its own, expert counts that vectorise and not."""
import numpy as np
import pytest
import torch

import oracle
from helpers import np_i32
from paper_2609_00993_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T,E,k", [
    (31, 5, 1), (1023, 7, 1), (512, 256, 2), (1025, 33, 1),     # one CTA up to 1024 slots, two behind
    (2047, 64, 8), (16384, 3, 1), (16385, 3, 1),                # 16384: the other chunks recounted; behind: a count launch
    (8200, 130, 8), (65537, 9, 1), (40000, 1024, 2),            # E % 4 != 0; several steps per warp; the largest E
    (300000, 6, 1),                                             # more chunks than the target, 4096 slots each
])
@pytest.mark.parametrize("static", [False, True])
def test_layout_at_chunk_edges(T, E, k, static):
    g = torch.Generator(device=DEV).manual_seed(T * 7 + E)
    idx = (torch.rand(T, k, generator=g, device=DEV) ** 2 * E).int().clamp_(0, E - 1)  # skewed, repeats within a token
    bufs = B.alloc_step_buffers(T, k, E, DEV)
    if static:
        if -(-T * k // 256) * E > 65536:
            pytest.skip("beyond the limit of the static entry point")
        torch.cuda.synchronize()
        assert B.moe_dispatch_layout_static(idx, E, bufs["counts"], bufs["offsets"], bufs["perm"], bufs["inv_perm"]) == B.MOE_OK
    else:
        ctx = B.MoeContext(B.make_config(64, E, k, 64, 0, T))
        torch.cuda.synchronize()
        for _ in range(2):
            ctx.moe_dispatch_layout(idx, None, bufs["counts"], bufs["offsets"], bufs["perm"], bufs["inv_perm"], T=T)
        assert ctx.moe_ctx_status() == B.MOE_OK
        ctx.close()
    torch.cuda.synchronize()
    counts, offsets, perm, inv = oracle.layout(np_i32(idx).reshape(-1), E)
    assert np.array_equal(np_i32(bufs["counts"]), counts) and np.array_equal(np_i32(bufs["offsets"]), offsets)
    assert np.array_equal(np_i32(bufs["perm"]), perm) and np.array_equal(np_i32(bufs["inv_perm"]), inv)
