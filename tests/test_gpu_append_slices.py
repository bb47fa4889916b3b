"""The KV append's split of a request's block over CTAs: blocks of one partial slice, of
exactly one, and of many, and a bad page id found by every slice's CTA."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import softmax_desc
from paper_2606_01774_gb300 import flare, workloads
from test_gpu_append import _bits, _with_room

pytestmark = pytest.mark.gpu
BASE = workloads.WORKLOADS["serving_batch64"]


# 16-byte chunks of a request: 8, 512 (one slice of 256 threads x 2), 520, 4096, 12288
@pytest.mark.parametrize("dtype, heads, dim, block", [("bf16", 1, 64, 1), ("bf16", 2, 256, 8),
                                                      ("bf16", 5, 64, 13), ("bf16", 2, 256, 64),
                                                      ("f32", 3, 256, 64)])
def test_slices_write_every_row_once(dtype, heads, dim, block):
    spec = BASE.replace(num_requests=5, prefix_lo=1, prefix_hi=300, page_size=16, act_dtype=dtype,
                        num_q_heads=heads, num_kv_heads=heads, head_dim=dim, block_len=block,
                        seed=58)
    w = _with_room(spec)
    sb = w.softmax[0]
    n = torch.tensor([block, 0, 1, (block + 1) // 2, block], dtype=torch.int32).cuda()
    last = (int(w.prefix_len[4]) + block - 1) // spec.page_size
    ref = oracle.append_kv(sb.k_blk.cpu(), sb.v_blk.cpu(), w.k_pool.cpu(), w.v_pool.cpu(),
                           w.page_table.cpu(), w.prefix_len.cpu(),
                           torch.cat([n[:4].cpu(), torch.zeros(1, dtype=torch.int32)]))
    w.page_table[4, last] = w.k_pool.shape[0]  # one past the pool: request 4 writes nothing
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    flare.check(flare.flare_append_kv(softmax_desc(spec, w), sb.k_blk, sb.v_blk, w.k_pool, w.v_pool,
                                      w.page_table, w.prefix_len, n, st))
    assert flare.flare_read_status(st)[1] == flare.FLARE_DEV_BAD_PAGE
    for got, want in zip((w.k_pool, w.v_pool), ref):
        assert np.array_equal(_bits(got).cpu().numpy().view(np.uint8),
                              np.ascontiguousarray(want).view(np.uint8))
