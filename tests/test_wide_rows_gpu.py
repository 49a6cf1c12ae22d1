"""Support lists in rows much wider than their counts, as working sets come
(rows of n_blocks): the same attention as from tight rows, bit for bit, whatever
stands behind the counts, at no multiple of the time."""
import statistics

import numpy as np
import pytest
import torch

from paper_2609_27373_gb300 import synth, wise
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _widen(idx, counts, cap, junk):
    """The lists in rows of width cap; behind the counts -1, or valid-looking blocks."""
    b, h, nb, _ = idx.shape
    wide = np.full((b, h, nb, cap), -1, dtype=np.int32)
    if junk:
        wide[:] = np.random.default_rng(1).integers(0, nb, wide.shape, dtype=np.int32)
    for x in range(idx.shape[-1]):
        live = counts > x
        wide[..., x][live] = idx[..., x][live]
    return wide


# batch, heads, kv heads, seqlen, head dim, block: at least 4 x 152 query tiles;
# rows of 32 (one pass) to several passes, lists around the passes' edges.
@pytest.mark.parametrize("b,h,hkv,L,d,blk", [(1, 40, 40, 2048, 64, 32), (1, 32, 16, 2560, 96, 64), (1, 24, 24, 4096, 128, 32),
                                             (2, 20, 20, 2048, 128, 128)])
@pytest.mark.parametrize("n", [1, 31, 33, 64])
def test_wide_rows_equal_tight_ones(b, h, hkv, L, d, blk, n):
    s = wise.Shape(b, L, h, hkv, d, blk)
    nb = s.n_blocks
    n = min(n, nb)
    q, k, v = (to_dev(x) for x in synth.random_qkv(b, h, hkv, L, d, seed=n))
    idx, counts = synth.random_support(b, hkv, nb, n, seed=n, n_sink=0, density=0.9)
    counts[0, 0, nb // 2] = 0
    dc = torch.from_numpy(counts).cuda()
    outs = []
    for lists in (idx, _widen(idx, counts, nb + 3, False), _widen(idx, counts, max(n, 32), True), _widen(idx, counts, nb + 97, True)):
        o = torch.empty_like(q)
        wise.wise_sparse_attn(s, q, k, v, torch.from_numpy(lists).cuda(), dc, o)
        assert wise.wise_get_status() == wise.WISE_OK
        outs.append(o)
    assert all(torch.equal(o, outs[0]) for o in outs[1:])


def test_wide_rows_cost_no_more_than_tight_ones():
    # 32K, block 32, lists of three entries in rows of 1024 against rows of 4: 1024 / 160 us
    # when every row was walked to its end.  The bound of twice the time leaves
    # room for the wide rows' scattered reads.
    L, h, d = 32768, 8, 128
    s = wise.Shape(1, L, h, h, d, 32)
    nb = s.n_blocks
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v = (torch.randn((1, h, L, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    o = torch.empty_like(q)
    rows = torch.arange(nb, dtype=torch.int32, device="cuda")
    tight = torch.stack([rows * 0, rows // 2, rows, rows * 0 - 1], -1)
    counts = torch.full((1, h, nb), 3, dtype=torch.int32, device="cuda")
    tight[:2, 1:] = -1  # blocks 0 and 1 have no third distinct block
    tight[1, 1] = 1
    counts[..., 0], counts[..., 1] = 1, 2
    tight = tight.expand(1, h, nb, 4).contiguous()
    wide = torch.full((1, h, nb, nb), -1, dtype=torch.int32, device="cuda")
    wide[..., :4] = tight
    times = {}
    for name, idx in (("tight", tight), ("wide", wide)):
        ms = []
        for i in range(9):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                wise.wise_sparse_attn(s, q, k, v, idx, counts, o)
            z.record()
            z.synchronize()
            ms.append(a.elapsed_time(z))
        times[name] = statistics.median(ms)
    assert wise.wise_get_status() == wise.WISE_OK
    assert times["wide"] <= 2.0 * times["tight"], times
