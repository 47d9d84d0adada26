"""The dispatch layout where its chunks grow with the batch: the last size with chunks of 4096 slots, the first behind it,
and one of many steps per warp; chunks that end within a warp's run."""
import numpy as np
import pytest
import torch

import oracle
from helpers import np_i32
from paper_2609_00993_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T,E,k", [(148 * 4096 // 8, 256, 8), (148 * 4096 // 8 + 1, 256, 8), (606209, 33, 1), (400003, 1024, 8)])
def test_layout_with_large_chunks(T, E, k):
    g = torch.Generator(device=DEV).manual_seed(T + E)
    idx = (torch.rand(T, k, generator=g, device=DEV) ** 2 * E).int().clamp_(0, E - 1)
    idx[T - 1, 0] = E  # dropped: the last token's first slot
    bufs = B.alloc_step_buffers(T, k, E, DEV)
    ctx = B.MoeContext(B.make_config(64, E, k, 64, 0, T))
    torch.cuda.synchronize()
    ctx.moe_dispatch_layout(idx, None, bufs["counts"], bufs["offsets"], bufs["perm"], bufs["inv_perm"], T=T)
    torch.cuda.synchronize()
    assert ctx.moe_ctx_status() == B.MOE_ERR_BAD_INDEX
    ctx.close()
    flat = np_i32(idx).reshape(-1)
    drop = (T - 1) * k
    kept = np.delete(np.arange(T * k), drop)
    counts, offsets, perm, inv = oracle.layout(flat[kept], E)
    assert np.array_equal(np_i32(bufs["counts"]), counts) and np.array_equal(np_i32(bufs["offsets"]), offsets)
    assert np.array_equal(np_i32(bufs["perm"]).reshape(-1)[:-1], kept[perm])
    got = np_i32(bufs["inv_perm"]).reshape(-1)
    assert got[drop] == -1 and np.array_equal(got[kept], inv)
