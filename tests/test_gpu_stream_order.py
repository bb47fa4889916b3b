"""The library's kernels are launched as programmatic dependents: set up while the kernel
ahead drains, they read and write memory only once it is done.  Chains in which each
call reads what the one before wrote, with large kernels of PyTorch's ahead and
behind, give bit for bit what the same calls give with the device idle between
them, on one stream, on two ordered by an event, and in a graph."""
import pytest
import torch

from gpu_helpers import gen, install_states, linear_desc, status_word
from paper_2606_01774_gb300 import flare, workloads

pytestmark = pytest.mark.gpu
LARGE = workloads.WORKLOADS["serving_batch64"]


@pytest.mark.parametrize("requests, block", [(1, 8), (1, 32), (24, 32), (24, 64)])
def test_chained_calls_see_each_other(requests, block):
    spec = LARGE.replace(num_requests=requests, block_len=block, prefix_lo=64, prefix_hi=128,
                         seed=270 + block)
    w = gen(spec)
    install_states(w, [0])
    b, pool0 = w.commit, w.state_pool.nan_to_num()
    desc, n = linear_desc(spec, pool0.shape[0]), torch.full((requests,), block, dtype=torch.int32).cuda()
    big = torch.randn(64 << 20, device="cuda")
    # everything that the chain touches has its address before a graph is captured
    pool, v, out, st = pool0.clone(), b.v.clone(), torch.empty_like(b.v), status_word("cuda")
    res = torch.empty_like(b.v, dtype=torch.float32)

    def chain(fence, other=None):
        pool.copy_(pool0)
        v.copy_(b.v)
        for _ in range(4):
            big.mul_(1.0)
            fence()
            v.mul_(0.5).add_(0.25)
            fence()
            flare.check(flare.flare_commit_state(desc, b.q, b.k, v, b.log_decay, b.beta, pool,
                                                 w.state_slot, n, out, st))
            fence()
            flare.check(flare.flare_block_linear_attn(desc, b.q, b.k, out, b.log_decay, b.beta, pool,
                                                      w.state_slot, v, st))
            fence()
            if other is not None:
                other.wait_stream(torch.cuda.current_stream())
                with torch.cuda.stream(other):
                    big.mul_(1.0)
                    v.mul_(2.0)
                torch.cuda.current_stream().wait_stream(other)
            else:
                v.mul_(2.0)
            fence()
        res.copy_(v)
        return pool.clone(), res.clone()

    want = chain(torch.cuda.synchronize)
    for other in (None, torch.cuda.Stream()):
        got = chain(lambda: None, other)
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(got, want))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(lambda: None)
    for _ in range(3):
        pool.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(pool, want[0]) and torch.equal(res, want[1])
    assert int(st) == 0
