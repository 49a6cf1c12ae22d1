"""Dense + mass on the one-stream kernel costs about the same at blocks of 128 and
below: the column sums of smaller blocks need registers, and an instance that
spills them shows here (head dim 128, 83 heads of 512 tokens: blocks of 64 18.6 us
against 15.4 with 80 bytes of stack, 15.5 without)."""
import statistics

import pytest
import torch

from paper_2609_27373_gb300 import wise

pytestmark = pytest.mark.gpu


def _time(d, blk):
    s = wise.Shape(1, 512, 83, 83, d, blk)
    q, k, v = (torch.randn((1, 83, 512, d), device="cuda").to(torch.bfloat16) for _ in range(3))
    o, mass = torch.empty_like(q), torch.empty((1, 83, 512 // blk, 512 // blk), device="cuda")
    wise.wise_full_attn_accumulate(s, q, k, v, o, mass, 0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(20):
            wise.wise_full_attn_accumulate(s, q, k, v, o, mass, 0)
    ms = []
    for _ in range(9):
        a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        z.record()
        z.synchronize()
        ms.append(a.elapsed_time(z))
    return statistics.median(ms)


@pytest.mark.parametrize("d", [64, 96, 128])
def test_small_blocks_cost_no_more(d):
    t = {blk: _time(d, blk) for blk in (128, 64, 32)}
    assert wise.wise_get_status() == wise.WISE_OK
    assert max(t[64], t[32]) <= 1.1 * t[128], t
