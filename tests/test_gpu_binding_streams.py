"""The stream a binding call runs on when none is given: torch's current stream of
the calling thread, looked up at every call."""
import threading

import pytest
import torch

from gpu_helpers import gen, linear_desc, status_word
from paper_2606_01774_gb300 import flare, workloads

pytestmark = pytest.mark.gpu


def test_default_stream_is_torchs_current_one_in_every_thread():
    w = gen(workloads.WORKLOADS["tiny_fp32"].replace(num_requests=4))
    w.state_pool.zero_()
    assert flare._stream(None) == torch.cuda.current_stream().cuda_stream
    seen = {}

    def work(name, stream):
        with torch.cuda.stream(stream):
            seen[name] = flare._stream(None)
            blk, out, st = w.denoise[0], torch.empty_like(w.denoise[0].v), status_word("cuda")
            # the call has to wait behind this stream's own work: its values are copied here
            v = torch.zeros_like(blk.v)
            torch.cuda._sleep(20_000_000)
            v.copy_(blk.v)
            flare.check(flare.flare_block_linear_attn(
                linear_desc(w.spec, w.state_pool.shape[0]), blk.q, blk.k, v, blk.log_decay,
                blk.beta, w.state_pool, w.state_slot, out, st))
            stream.synchronize()
            seen[name + "_out"] = out

    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(f"s{i}", s)) for i, s in enumerate(streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, s in enumerate(streams):
        assert seen[f"s{i}"] == s.cuda_stream
    assert torch.equal(seen["s0_out"], seen["s1_out"]) and seen["s0_out"].abs().sum() > 0
    assert flare._stream(streams[0]).value == streams[0].cuda_stream
