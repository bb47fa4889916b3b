"""The attention kernels' own ordering of the requests and page check: batches on
each side of the on-chip limit (512), with bad prefix lengths and page ids among
them, whole and split prefixes."""
import pytest
import torch

from gpu_helpers import assert_out_close, gen, oracle_softmax, softmax_desc
from paper_2606_01774_gb300 import flare, workloads

pytestmark = pytest.mark.gpu
LARGE = workloads.WORKLOADS["serving_batch64"]
SMALL = workloads.WORKLOADS["small_model_batch256"]


@pytest.mark.parametrize("base,requests,block,hi", [
    (SMALL, 512, 1, 150), (SMALL, 513, 1, 150), (LARGE, 511, 20, 150),  # unsplit
    (LARGE, 5, 32, 4000), (SMALL, 7, 16, 3000)])  # split
def test_bad_requests_are_left_out_and_the_rest_served(base, requests, block, hi):
    spec = base.replace(num_requests=requests, block_len=block, prefix_lo=1, prefix_hi=hi, seed=92)
    w = gen(spec)
    lens = w.prefix_len.clone()
    long = int(lens.argmax())
    bad_len = {0: -1, requests - 1: w.page_table.shape[1] * spec.page_size + 1}
    bad_len.pop(long, None)
    for r, n in bad_len.items():
        w.prefix_len[r] = n
    # a page id out of range at the very end of the longest prefix, negative in another
    w.page_table[long, (int(lens[long]) - 1) // spec.page_size] = w.k_pool.shape[0]
    other = next(r for r in range(1, requests) if r != long and r not in bad_len)
    w.page_table[other, 0] = -7
    bad = set(bad_len) | {long, other}
    sb, desc = w.softmax[0], softmax_desc(spec, w)
    n = flare.flare_softmax_workspace_size(desc)
    ws = torch.empty(max(n, 1), dtype=torch.uint8, device="cuda")
    out = torch.full_like(sb.q, 5.0)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    flare.check(flare.flare_block_softmax_attn(desc, sb.q, sb.k_blk, sb.v_blk, w.k_pool, w.v_pool,
                                               w.page_table, w.prefix_len, out, None, ws, n, st))
    _, bits = flare.flare_read_status(st)
    assert bits == flare.FLARE_DEV_BAD_PAGE | flare.FLARE_DEV_BAD_PREFIX_LEN
    for r in bad:
        assert (out[r] == 5.0).all()
    good = [r for r in range(requests) if r not in bad][:: max(1, requests // 12)]
    ref, _ = oracle_softmax(w, 0, good)
    assert_out_close(out[good], ref, "bf16", "good requests")
    rest = [r for r in range(requests) if r not in bad]
    assert torch.isfinite(out[rest].float()).all() and not (out[rest] == 5.0).all(-1).any()
