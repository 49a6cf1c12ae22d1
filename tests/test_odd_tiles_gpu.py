"""Dense launches whose heads have an odd number of query tiles, one of which has
no partner in the two-stream kernel: against the oracle on both sides of the
rule that says which one, and no slower than one tile more per head."""
import statistics

import numpy as np
import pytest
import torch

from gpu_helpers import (MASS_MAX_ABS, assert_close_o, bf16_dev_to_f64, empty_like_q, sample_units, to_dev)
from oracle import oracle as orc
from paper_2609_27373_gb300 import synth, wise

pytestmark = pytest.mark.gpu


# 456 to 608 query tiles (the first one alone), more (the last), three tiles, a
# ragged last tile, an odd group.
@pytest.mark.parametrize("b,h,hkv,L,d,blk", [
    (1, 92, 92, 640, 128, 128), (2, 46, 46, 608, 64, 32), (1, 120, 40, 640, 96, 64), (3, 27, 9, 864, 128, 32),
    (1, 123, 123, 640, 64, 64), (1, 156, 156, 352, 96, 32), (1, 60, 60, 1088, 96, 64)])
def test_dense_and_mass(b, h, hkv, L, d, blk):
    s = wise.Shape(b, L, h, hkv, d, blk)
    nb = s.n_blocks
    Q, K, V = synth.random_qkv(b, h, hkv, L, d, seed=L)
    q, k, v = map(to_dev, (Q, K, V))
    o1, o2 = empty_like_q(Q), empty_like_q(Q)
    mass = torch.full((b, h, nb, nb), 7.0, dtype=torch.float32, device="cuda")
    wise.wise_full_attn_accumulate(s, q, k, v, o1)
    wise.wise_full_attn_accumulate(s, q, k, v, o2, mass, 0)
    assert wise.wise_get_status() == wise.WISE_OK
    m = mass.cpu().numpy().astype(np.float64)
    assert np.abs(m.sum(-1) - 1.0).max() <= 1e-5
    full, fc = (torch.from_numpy(x).cuda() for x in synth.all_blocks_support(b, hkv, nb))
    o = empty_like_q(Q)
    wise.wise_sparse_attn(s, q, k, v, full, fc, o)
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(o, o1)
    for bb, hh, qq in sample_units(b, h, nb, 12, seed=1) + [(b - 1, 0, 0), (0, 0, 128 // blk)]:
        g = hh // (h // hkv)
        want_o, want_m = orc.full_attention(Q[bb:bb + 1, hh:hh + 1], K[bb:bb + 1, g:g + 1], V[bb:bb + 1, g:g + 1], blk,
                                            with_mass=True)
        rows = slice(qq * blk, (qq + 1) * blk)
        for got in (o1, o2):
            assert_close_o(bf16_dev_to_f64(got[bb, hh, rows]), np.asarray(want_o).reshape(L, d)[rows])
        assert np.abs(m[bb, hh, qq] - np.asarray(want_m).reshape(nb, nb)[qq]).max() <= MASS_MAX_ABS


# One query tile per head: dense runs on the one-stream kernel, dense + mass and
# sparse on the two-stream one, with the same output.
@pytest.mark.parametrize("b,h,hkv,L,d,blk", [(1, 460, 460, 128, 64, 128), (2, 300, 100, 96, 128, 32), (3, 160, 160, 64, 96, 64)])
def test_one_tile(b, h, hkv, L, d, blk):
    s = wise.Shape(b, L, h, hkv, d, blk)
    Q, K, V = synth.random_qkv(b, h, hkv, L, d, seed=L)
    q, k, v = map(to_dev, (Q, K, V))
    full, fc = (torch.from_numpy(x).cuda() for x in synth.all_blocks_support(b, hkv, s.n_blocks))
    o, od, om = (empty_like_q(Q) for _ in range(3))
    mass = torch.empty((b, h, s.n_blocks, s.n_blocks), device="cuda")
    wise.wise_full_attn_accumulate(s, q, k, v, od)
    wise.wise_full_attn_accumulate(s, q, k, v, om, mass, 0)
    wise.wise_sparse_attn(s, q, k, v, full, fc, o)
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(o, od)
    want, _ = orc.full_attention(Q[:1], K[:1], V[:1], blk, with_mass=False)
    for got in (od, om):
        assert_close_o(bf16_dev_to_f64(got[:1]), np.asarray(want).reshape(1, h, L, d))


def _graph_time(s, q, k, v, o, *mass):
    wise.wise_full_attn_accumulate(s, q, k, v, o, *mass)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(20):
            wise.wise_full_attn_accumulate(s, q, k, v, o, *mass)
    ms = []
    for _ in range(9):
        a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        z.record()
        z.synchronize()
        ms.append(a.elapsed_time(z))
    return statistics.median(ms)


def test_a_tile_less_per_head_costs_less():
    # 92 heads of 5 tiles against 6, head dim 128: 15 key tiles a head against 21, two
    # thirds of them on the critical path.  20.8 / 20.9 us with the last of five
    # tiles alone, 17.0 / 20.9 with the first.
    t = {}
    for L in (640, 768):
        s = wise.Shape(1, L, 92, 92, 128, 128)
        q, k, v = (torch.randn((1, 92, L, 128), device="cuda").to(torch.bfloat16) for _ in range(3))
        t[L] = _graph_time(s, q, k, v, torch.empty_like(q))
    assert wise.wise_get_status() == wise.WISE_OK
    assert t[640] <= 0.93 * t[768], t


def test_one_tile_without_mass_costs_less_than_with():
    # 912 heads x 128 tokens, head dim 96: 19.4 / 19.1 us with dense on the two-stream
    # kernel, 17.5 / 19.1 on the other.
    s = wise.Shape(1, 128, 912, 912, 96, 128)
    q, k, v = (torch.randn((1, 912, 128, 96), device="cuda").to(torch.bfloat16) for _ in range(3))
    o, mass = torch.empty_like(q), torch.empty((1, 912, 1, 1), device="cuda")
    plain, with_mass = _graph_time(s, q, k, v, o), _graph_time(s, q, k, v, o, mass, 0)
    assert wise.wise_get_status() == wise.WISE_OK
    assert plain <= 0.96 * with_mass, (plain, with_mass)
