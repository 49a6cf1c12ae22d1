"""The two-stream attention kernel (attn_duo.cuh), which launches with several
query tiles per SM take: dense, dense + mass and sparse against the oracle at
the sizes where its pairing, tile and schedule code can go wrong.  Every shape
here has at least 4 x 152 query tiles, so that it runs on any GB300, or is a
short sequence with 1.5 to 2 query tiles per SM.

Tolerances are those of the parity tests (gpu_helpers)."""
import numpy as np
import pytest
import torch

from gpu_helpers import (MASS_MAX_ABS, assert_close_o, bf16_dev_to_f64, empty_like_q, sample_units, to_dev, units_of)
from oracle import oracle as orc
from paper_2609_27373_gb300 import synth, wise

pytestmark = pytest.mark.gpu

# batch, heads, kv heads, seqlen, head dim, block: unpaired heads with an odd
# and an even number of query tiles, odd and even groups (head pairs), ragged
# last tiles at block 32 and 64, one-tile units, more units than a CTA stages,
# unpaired heads of 96 (boxes of their own) over several tiles.
SHAPES = [
    (4, 52, 52, 384, 128, 128), (2, 40, 40, 1024, 128, 128), (4, 33, 11, 640, 128, 128), (4, 64, 16, 384, 128, 128),
    (4, 55, 55, 384, 96, 128), (3, 54, 9, 544, 96, 32), (4, 40, 40, 576, 64, 64), (4, 64, 32, 416, 64, 32),
    (8, 80, 80, 128, 64, 128), (10, 64, 8, 96, 64, 32), (2, 37, 37, 1120, 96, 32),
    (1, 125, 125, 256, 128, 128), (2, 36, 36, 416, 64, 32), (4, 16, 16, 512, 96, 64), (3, 40, 8, 160, 128, 32),
]


def _data(i, shape):
    b, h, hkv, L, d, blk = shape
    return synth.random_qkv(b, h, hkv, L, d, seed=100 + i)


@pytest.mark.parametrize("i", range(len(SHAPES)))
def test_dense_and_mass(i):
    b, h, hkv, L, d, blk = SHAPES[i]
    s = wise.Shape(b, L, h, hkv, d, blk)
    nb = s.n_blocks
    Q, K, V = _data(i, SHAPES[i])
    q, k, v = map(to_dev, (Q, K, V))
    o1, o2 = empty_like_q(Q), empty_like_q(Q)
    mass = torch.full((b, h, nb, nb), 7.0, dtype=torch.float32, device="cuda")
    wise.wise_full_attn_accumulate(s, q, k, v, o1)
    wise.wise_full_attn_accumulate(s, q, k, v, o2, mass, 0)
    first = mass.clone()
    wise.wise_full_attn_accumulate(s, q, k, v, o2, mass, 1)
    assert wise.wise_get_status() == wise.WISE_OK
    if blk == 128:  # smaller blocks sum each key block's row part by itself
        assert torch.equal(o1, o2)
    assert torch.equal(mass, first + first)
    m = first.cpu().numpy().astype(np.float64)
    assert np.abs(m.sum(-1) - 1.0).max() <= 1e-5
    pick = sample_units(b, h, nb, 12, seed=i)
    for bb, hh, qq in pick:
        g = hh // (h // hkv)
        want_o, want_m = orc.full_attention(Q[bb:bb + 1, hh:hh + 1], K[bb:bb + 1, g:g + 1], V[bb:bb + 1, g:g + 1], blk,
                                            with_mass=True)
        rows = slice(qq * blk, (qq + 1) * blk)
        for o in (o1, o2):
            assert_close_o(bf16_dev_to_f64(o[bb, hh, rows]), np.asarray(want_o).reshape(L, d)[rows])
        assert np.abs(m[bb, hh, qq] - np.asarray(want_m).reshape(nb, nb)[qq]).max() <= MASS_MAX_ABS


@pytest.mark.parametrize("i", range(len(SHAPES)))
def test_sparse(i):
    b, h, hkv, L, d, blk = SHAPES[i]
    s = wise.Shape(b, L, h, hkv, d, blk)
    nb = s.n_blocks
    cap = max(2, min(nb, 5) if i % 2 else nb + 40)  # also lists longer than a warp
    Q, K, V = _data(i, SHAPES[i])
    idx, counts = synth.random_support(b, hkv, nb, cap, seed=i, density=0.5)
    counts[0, 0, nb // 2] = 0  # a query block that attends nothing
    q, k, v = map(to_dev, (Q, K, V))
    o = empty_like_q(Q)
    wise.wise_sparse_attn(s, q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(counts).cuda(), o)
    assert wise.wise_get_status() == wise.WISE_OK
    pick = sample_units(b, h, nb, 40, seed=i) + [(0, 0, nb // 2)]
    want = orc.sparse_attention(Q, K, V, idx, counts, blk, units=pick)
    got = bf16_dev_to_f64(o)
    assert_close_o(units_of(got, pick, blk), np.asarray(want))
    # Every admissible block: the dense result, bit for bit.
    fi, fc = synth.all_blocks_support(b, hkv, nb)
    od = empty_like_q(Q)
    wise.wise_sparse_attn(s, q, k, v, torch.from_numpy(fi).cuda(), torch.from_numpy(fc).cuda(), o)
    wise.wise_full_attn_accumulate(s, q, k, v, od)
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(o, od)


@pytest.mark.parametrize("i", [0, 3, 5, 6])
def test_malformed_lists_are_skipped_and_reported(i):
    b, h, hkv, L, d, blk = SHAPES[i]
    s = wise.Shape(b, L, h, hkv, d, blk)
    nb = s.n_blocks
    Q, K, V = _data(i, SHAPES[i])
    idx, counts = synth.random_support(b, hkv, nb, nb + 3, seed=50 + i, density=0.4)
    bad, bad_counts = idx.copy(), counts.copy()
    for q in range(nb):  # entries out of range, out of order and repeated, and a count over the cap
        n = int(counts[-1, -1, q])
        bad[-1, -1, q, :n + 3] = np.concatenate([[nb + 5, -3], idx[-1, -1, q, :n], idx[-1, -1, q, :1]])
        bad_counts[-1, -1, q] = nb + 9 if q == nb - 1 else n + 3
    q, k, v = map(to_dev, (Q, K, V))
    o, want = empty_like_q(Q), empty_like_q(Q)
    wise.wise_sparse_attn(s, q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(counts).cuda(), want)
    assert wise.wise_get_status() == wise.WISE_OK
    wise.wise_sparse_attn(s, q, k, v, torch.from_numpy(bad).cuda(), torch.from_numpy(bad_counts).cuda(), o)
    assert wise.wise_get_status() == wise.WISE_ERR_BAD_SUPPORT
    assert torch.equal(o, want)


@pytest.mark.parametrize("i", [1, 4, 6])
def test_output_aligned_to_16_bytes(i):
    b, h, hkv, L, d, blk = SHAPES[i]
    s = wise.Shape(b, L, h, hkv, d, blk)
    Q, K, V = _data(i, SHAPES[i])
    q, k, v = map(to_dev, (Q, K, V))
    want = empty_like_q(Q)
    wise.wise_full_attn_accumulate(s, q, k, v, want)
    raw = torch.zeros(want.numel() + 32, dtype=torch.bfloat16, device="cuda")
    off = next(o for o in range(8, 24, 8) if (raw.data_ptr() + 2 * o) % 32 == 16)
    o = raw[off:off + want.numel()].view(want.shape)
    wise.wise_full_attn_accumulate(s, q, k, v, o)
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(o, want)
    assert not raw[:off].any() and not raw[off + want.numel():].any()
