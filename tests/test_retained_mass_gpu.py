"""The retained mass of few and many rows (eight lanes a row, one lane a row),
well-formed and malformed lists: the sums in list order, bit for bit; and the
cost of many rows of short lists."""
import statistics

import pytest
import torch

from paper_2609_27373_gb300 import wise

pytestmark = pytest.mark.gpu


def _want(mass, idx, counts, group):
    """fp32 sums in list order over the entries in [0, q] above every accepted one before them."""
    B, H, nb, _ = mass.shape
    idx, counts = idx.repeat_interleave(group, 1), counts.repeat_interleave(group, 1)
    q = torch.arange(nb, device=idx.device)
    acc = torch.zeros((B, H, nb), device=idx.device)
    prev = torch.full((B, H, nb), -1, device=idx.device)
    bad = (counts < 0) | (counts > idx.shape[-1])
    n = counts.clamp(0, idx.shape[-1])
    for i in range(idx.shape[-1]):
        v = idx[..., i]
        live = i < n
        ok = live & (v >= 0) & (v <= q) & (v > prev)
        got = mass.gather(-1, v.clamp(0, nb - 1).long()[..., None])[..., 0]
        acc = torch.where(ok, acc + got, acc)
        prev = torch.where(ok, v, prev)
        bad |= live & ~ok
    return acc, bool(bad.any())


# 32768 rows and the next above, row widths 16 and 17, groups of heads, one block.
@pytest.mark.parametrize("B,H,Hkv,nb,cap", [(8, 64, 64, 64, 12), (1, 993, 331, 33, 16), (1, 993, 331, 33, 17), (64, 16, 4, 40, 8),
                                            (3, 12345, 12345, 1, 1), (2, 36, 12, 500, 16)])
@pytest.mark.parametrize("malformed", [False, True])
def test_sums(B, H, Hkv, nb, cap, malformed):
    g = torch.Generator(device="cuda").manual_seed(nb)
    mass = torch.rand((B, H, nb, nb), generator=g, device="cuda")
    key = torch.rand((B, Hkv, nb, nb), generator=g, device="cuda")
    q = torch.arange(nb, device="cuda")
    key = key.masked_fill(q[None, :] > q[:, None], 2.0)
    n = torch.minimum(torch.randint(0, cap + 1, (B, Hkv, nb), generator=g, device="cuda"), q + 1).clamp(max=min(cap, nb))
    low = key.sort(-1).indices[..., :min(cap, nb)]
    order = torch.where(torch.arange(low.shape[-1], device="cuda") < n[..., None], low, nb + 1).sort(-1).values
    idx = torch.full((B, Hkv, nb, cap), -1, dtype=torch.int32, device="cuda")
    idx[..., :low.shape[-1]] = torch.where(order <= nb, order, -1).int()
    counts = n.int()
    if malformed:
        hit = torch.rand(idx.shape, generator=g, device="cuda") < 0.05
        idx[hit] = torch.randint(-2, nb + 3, idx.shape, generator=g, device="cuda", dtype=torch.int32)[hit]
        counts[0, 0, 0], counts[-1, -1, -1] = -1, cap + 1
    out = torch.full((B, H, nb), -7.0, device="cuda")
    wise.wise_support_mass(wise.Shape(B, nb * 32, H, Hkv, 64, 32), mass, idx, counts, out)
    want, bad = _want(mass, idx, counts, H // Hkv)
    assert bad == malformed
    assert wise.wise_get_status() == (wise.WISE_ERR_BAD_SUPPORT if bad else wise.WISE_OK)
    assert torch.equal(out, want)


def test_many_rows_of_short_lists():
    # 131072 rows against 1024, lists of two entries: 8.6 / 2.1 us with eight lanes for
    # each, 3.3 / 1.9 here.
    t = {}
    for B, H in ((1, 16), (64, 32)):
        s = wise.Shape(B, 64 * 32, H, H, 64, 32)
        rows = torch.arange(64, dtype=torch.int32, device="cuda")
        idx = torch.full((B, H, 64, 12), -1, dtype=torch.int32, device="cuda")
        idx[..., 0], idx[..., 1] = 0, rows
        counts = torch.full((B, H, 64), 2, dtype=torch.int32, device="cuda")
        counts[..., 0] = 1
        mass, out = torch.rand((B, H, 64, 64), device="cuda"), torch.empty((B, H, 64), device="cuda")
        wise.wise_support_mass(s, mass, idx, counts, out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(50):
                wise.wise_support_mass(s, mass, idx, counts, out)
        ms = []
        for _ in range(9):
            x, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            x.record()
            graph.replay()
            z.record()
            z.synchronize()
            ms.append(x.elapsed_time(z))
        t[B] = statistics.median(ms)
    assert wise.wise_get_status() == wise.WISE_OK
    assert t[64] <= 2.8 * t[1], t
