"""The support overlap over the shapes that take its kernels in turn (merge, 8
and 32 lanes a row, clusters of 1 to 8 CTAs), with lists that end at and around
its chunks and with malformed ones: equal to the oracle's; and the cost of many
small batch elements."""
import statistics

import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2609_27373_gb300 import synth, wise

pytestmark = pytest.mark.gpu


def _lists(B, Hkv, nb, cap, seed):
    """Ascending lists of 0 .. cap blocks out of [0, q] in rows of width cap."""
    rng = np.random.default_rng(seed)
    q = np.tile(np.arange(nb), B * Hkv)
    key = rng.random((len(q), nb)) + (np.arange(nb)[None, :] > q[:, None]) * 2.0
    n = np.minimum(rng.integers(0, cap + 1, len(q)), q + 1)
    take = np.argsort(np.argsort(key, 1), 1) < n[:, None]
    idx = np.full((len(q), cap), -1, dtype=np.int32)
    for r in range(len(q)):
        idx[r, :n[r]] = np.flatnonzero(take[r])
    return idx.reshape(B, Hkv, nb, cap), n.astype(np.int32).reshape(B, Hkv, nb)


def _run(s, B, lists):
    out = torch.full((B, 2), -1, dtype=torch.int64, device="cuda")
    t = [torch.from_numpy(x).cuda() for x in lists]
    wise.wise_support_overlap(s, t[0], t[1], t[2], t[3], out)
    return out.cpu().numpy()


# batch, kv heads, blocks, row widths: one row, rows that are no multiple of a warp's,
# 255 to 257 and 1024 / 1025 blocks, row widths that sum to 24 and 25, 31 and 257 rows
# an element, 1023 / 1024 rows, 19 / 20 elements.
@pytest.mark.parametrize("B,Hkv,nb,ca,cb", [
    (1, 1, 1, 1, 1), (1, 3, 37, 9, 8), (1, 33, 31, 31, 8), (1, 32, 32, 32, 9), (5, 7, 255, 40, 17), (2, 9, 256, 8, 33),
    (2, 9, 257, 33, 65), (1, 2, 1024, 64, 31), (1, 2, 1025, 64, 31), (128, 2, 16, 16, 8), (128, 2, 16, 17, 8),
    (160, 1, 31, 12, 12), (16, 1, 256, 12, 12), (17, 1, 257, 12, 12), (19, 4, 64, 64, 7), (20, 4, 64, 64, 7),
    (300, 1, 5, 5, 3), (2000, 1, 3, 3, 2)])
@pytest.mark.parametrize("malformed", [False, True])
def test_overlap(B, Hkv, nb, ca, cb, malformed):
    ia, na = _lists(B, Hkv, nb, ca, 1)
    ib, nb_ = _lists(B, Hkv, nb, cb, 2)
    if malformed:
        rng = np.random.default_rng(3)
        for idx, n in ((ia, na), (ib, nb_)):
            hit = rng.random(idx.shape) < 0.1
            idx[hit] = rng.integers(-2, nb + 3, int(hit.sum()))
            n[rng.random(n.shape) < 0.05] = idx.shape[-1] + 2
        na[0, 0, 0] = -1
    got = _run(wise.Shape(B, nb * 32, Hkv, Hkv, 64, 32), B, (ia, na, ib, nb_))
    assert wise.wise_get_status() == (wise.WISE_ERR_BAD_SUPPORT if malformed else wise.WISE_OK)
    assert np.array_equal(got, orc.support_overlap(ia, na, ib, nb_))


def test_many_small_elements():
    # 256 elements of 128 rows against one: 70 / 3.5 us with eight full CTAs for each,
    # 6.2 / 2.3 here.
    t = {}
    for B in (1, 256):
        s = wise.Shape(B, 16 * 32, 8, 8, 64, 32)
        a = [torch.from_numpy(x).cuda() for x in synth.random_support(1, 8, 16, 16, seed=1, density=0.9)]
        b = [torch.from_numpy(x).cuda() for x in synth.random_support(1, 8, 16, 8, seed=2, density=0.9)]
        (ia, na), (ib, nb) = ([x.expand(B, *x.shape[1:]).contiguous() for x in y] for y in (a, b))
        out = torch.empty((B, 2), dtype=torch.int64, device="cuda")
        wise.wise_support_overlap(s, ia, na, ib, nb, out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                wise.wise_support_overlap(s, ia, na, ib, nb, out)
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
    assert t[256] <= 6.0 * t[1], t
