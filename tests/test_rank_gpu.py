"""Selection and working sets at the sizes where the ranking changes its method
(32 blocks and fewer, few picks, many picks), the fixed-point conversion at its
edges, and the support overlap on long lists and on more than 1024 blocks: all
integers, equal to the oracle's."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2609_27373_gb300 import synth, wise

pytestmark = pytest.mark.gpu


def _masses(steps, B, H, nb, seed, kind):
    rng = np.random.default_rng(seed)
    m = rng.random((steps, B, H, nb, nb), dtype=np.float32)
    if kind == "peaked":
        m = (m ** 12).astype(np.float32)
    elif kind == "ties":
        m = (np.floor(m * 4) / 4).astype(np.float32)
    elif kind == "edges":
        # Zeros, negatives, NaN, infinity, denormals, masses around 2^-32 and
        # around the clip at 4096, neighbours that differ below 2^-32.
        pool = np.array([0.0, -0.0, -1.0, np.nan, np.inf, 1e-45, 1e-38, 2.0 ** -33, 2.0 ** -32,
                         np.nextafter(np.float32(2.0 ** -32), np.float32(0)), 1.5 * 2.0 ** -31, 4095.9998, 4096.0, 5000.0,
                         1.0, np.nextafter(np.float32(1), np.float32(2)), 3.0 * 2.0 ** -30, 0.25 + 2.0 ** -26],
                        dtype=np.float32)
        m = pool[rng.integers(0, len(pool), m.shape)]
    return np.ascontiguousarray(m)


@pytest.mark.parametrize("kind", ["flat", "peaked", "ties", "edges"])
@pytest.mark.parametrize("nb,H,Hkv", [(31, 3, 3), (32, 4, 2), (33, 2, 2), (64, 6, 2), (129, 2, 1), (300, 2, 2), (1000, 1, 1)])
def test_selection_matches_oracle(nb, H, Hkv, kind):
    B, block = 1, 32
    m = _masses(1, B, H, nb, nb, kind)[0]
    dev = torch.from_numpy(m).cuda()
    s = wise.Shape(B, nb * block, H, Hkv, 64, block)
    for mode, topk, eta, cap, sink, local in ((0, 3, 0.0, 5, 1, 1), (0, 200, 0.0, 60, 0, 2), (1, 0, 0.95, 12, 1, 1),
                                              (1, 0, 0.7, 400, 0, 1), (1, 0, 1.0, 1100, 2, 3)):
        idx = torch.full((B, Hkv, nb, cap), -9, dtype=torch.int32, device="cuda")
        counts = torch.full((B, Hkv, nb), -9, dtype=torch.int32, device="cuda")
        wise.wise_select_support(s, wise.Select(sink, local, mode, topk, eta, cap), dev, idx, counts)
        wi, wc = orc.select_support(m, Hkv, block, mode, sink, local, topk, eta, cap)
        assert np.array_equal(counts.cpu().numpy(), wc), (mode, topk, eta, cap)
        assert np.array_equal(idx.cpu().numpy(), wi), (mode, topk, eta, cap)


@pytest.mark.parametrize("kind", ["flat", "ties", "edges"])
@pytest.mark.parametrize("nb,H,Hkv", [(32, 2, 1), (70, 2, 2), (130, 1, 1)])
def test_working_sets_match_oracle(nb, H, Hkv, kind):
    B, block = 1, 32
    m = _masses(3, B, H, nb, nb + 1, kind)
    dev = torch.from_numpy(m).cuda()
    s = wise.Shape(B, nb * block, H, Hkv, 64, block)
    ri, rc = synth.random_support(B, Hkv, nb, nb, seed=nb, density=0.4)
    for mode, steps, kw in ((wise.WS_UNION, 3, {}), (wise.WS_STATIC, 1, dict(n_sink=1, n_local=2)),
                            (wise.WS_MASS_MATCHED, 1, dict(ref=True)), (wise.WS_SIZE_MATCHED, 1, dict(ref=True))):
        ref = kw.pop("ref", False)
        idx = torch.full((B, Hkv, nb, nb), -9, dtype=torch.int32, device="cuda")
        counts = torch.full((B, Hkv, nb), -9, dtype=torch.int32, device="cuda")
        wise.wise_select_working_set(s, mode, dev[:steps].contiguous(), idx, counts, eta=0.9,
                                     ref_idx=torch.from_numpy(ri).cuda() if ref else None,
                                     ref_counts=torch.from_numpy(rc).cuda() if ref else None, **kw)
        wi, wc = orc.working_set(mode, m[:steps], Hkv, eta=0.9, ref_idx=ri if ref else None,
                                 ref_counts=rc if ref else None, **kw)
        assert np.array_equal(counts.cpu().numpy(), wc), mode
        assert np.array_equal(idx.cpu().numpy(), wi), mode
    assert wise.wise_get_status() == wise.WISE_OK


@pytest.mark.parametrize("B,Hkv,nb,cap_a,cap_b", [(1, 1, 1, 1, 1), (3, 2, 40, 40, 7), (2, 3, 100, 33, 100),
                                                  (1, 2, 1024, 70, 9), (1, 1, 1100, 40, 64)])
def test_overlap_matches_oracle(B, Hkv, nb, cap_a, cap_b):
    s = wise.Shape(B, nb * 32, Hkv, Hkv, 64, 32)
    ia, ca = synth.random_support(B, Hkv, nb, cap_a, seed=1, density=0.5)
    ib, cb = synth.random_support(B, Hkv, nb, cap_b, seed=2, density=0.5, n_sink=0)
    # A repeated and an out-of-range entry in the last row, where they fit.
    bad = cap_a >= 3
    if bad:
        ia[-1, -1, -1, :3], ca[-1, -1, -1] = [0, 0, nb + 1], 3
    out = torch.full((B, 2), -1, dtype=torch.int64, device="cuda")
    t = [torch.from_numpy(x).cuda() for x in (ia, ca, ib, cb)]
    wise.wise_support_overlap(s, t[0], t[1], t[2], t[3], out)
    assert wise.wise_get_status() == (wise.WISE_ERR_BAD_SUPPORT if bad else wise.WISE_OK)
    assert np.array_equal(out.cpu().numpy(), orc.support_overlap(ia, ca, ib, cb))


@pytest.mark.parametrize("nb,cap", [(1, 1), (9, 8), (60, 17), (200, 200)])
def test_retained_mass_in_list_order(nb, cap):
    B, H, Hkv = 2, 4, 2
    s = wise.Shape(B, nb * 32, H, Hkv, 64, 32)
    m = _masses(1, B, H, nb, 5, "flat")[0]
    idx, counts = synth.random_support(B, Hkv, nb, cap, seed=nb, density=0.6)
    counts[0, 0, 0] = 0
    out = torch.full((B, H, nb), -7.0, device="cuda")
    wise.wise_support_mass(s, torch.from_numpy(m).cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(counts).cuda(), out)
    assert wise.wise_get_status() == wise.WISE_OK
    want = np.zeros((B, H, nb), dtype=np.float32)
    for b in range(B):
        for h in range(H):
            for q in range(nb):
                acc = np.float32(0)
                for v in idx[b, h // 2, q, :counts[b, h // 2, q]]:
                    acc = np.float32(acc + m[b, h, q, v])
                want[b, h, q] = acc
    assert np.array_equal(out.cpu().numpy(), want)
