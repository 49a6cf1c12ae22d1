"""The one-stream attention kernel (attn_kernel.cuh) where it is dispatched:
launches below 3 query tiles per SM, several tiles to a CTA, and sequences of
more than 256 query tiles; and the time-out path of both kernels in the forms
that have code of their own.

A CTA of this kernel takes its units one after the other: the two softmax
warpgroups share the staging boxes that O is written through, and the block
masses' column sums are double-buffered across units.  A missing order between
one unit's reads and the next one's writes shows up here as wrong or
unrepeatable rows; units of one or two key tiles make the warpgroups change
places at every tile.

Tolerances are those of the parity tests (gpu_helpers)."""
import numpy as np
import pytest
import torch

from gpu_helpers import (MASS_MAX_ABS, MASS_ROWSUM, O_MAX_ABS, assert_close_o, bf16_dev_to_f64, empty_like_q, sample_units,
                         to_dev, units_of)
from oracle import oracle as orc
from paper_2609_27373_gb300 import synth, wise

pytestmark = pytest.mark.gpu

# batch, heads, kv heads, seqlen, head dim, block: 160 to 448 query tiles, neither 2 nor 4
# of them to a head; ragged last tiles, head groups, 128 key blocks and more (the
# column sums in shared and in global memory).
SHAPES = [
    (1, 24, 24, 2048, 128, 128), (1, 12, 4, 1952, 64, 32), (2, 10, 10, 1216, 96, 64), (1, 20, 10, 1536, 128, 64),
    (3, 14, 14, 1152, 64, 128), (1, 16, 8, 3072, 96, 32), (1, 4, 4, 5120, 128, 32), (1, 28, 28, 2048, 64, 64),
]


def _dev(*arrays):
    return [torch.from_numpy(x).cuda() for x in arrays]


@pytest.mark.parametrize("i", range(len(SHAPES)))
def test_dense_and_mass(i):
    b, h, hkv, L, d, blk = SHAPES[i]
    s = wise.Shape(b, L, h, hkv, d, blk)
    nb = s.n_blocks
    Q, K, V = synth.random_qkv(b, h, hkv, L, d, seed=200 + i)
    q, k, v = map(to_dev, (Q, K, V))
    o1, o2 = empty_like_q(Q), empty_like_q(Q)
    mass = torch.full((b, h, nb, nb), 7.0, dtype=torch.float32, device="cuda")
    wise.wise_full_attn_accumulate(s, q, k, v, o1)
    wise.wise_full_attn_accumulate(s, q, k, v, o2, mass, 0)
    first = mass.clone()
    wise.wise_full_attn_accumulate(s, q, k, v, o2, mass, 1)
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(mass, first + first)
    m = first.cpu().numpy().astype(np.float64)
    assert np.abs(m.sum(-1) - 1.0).max() <= MASS_ROWSUM
    for bb, hh, qq in sample_units(b, h, nb, 10, seed=i):
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
    Q, K, V = synth.random_qkv(b, h, hkv, L, d, seed=300 + i)
    q, k, v = map(to_dev, (Q, K, V))
    pick = sample_units(b, h, nb, 60, seed=i) + [(0, 0, nb // 2)]
    # Lists that are staged (blocks of 32 and 64, at most 128 entries a tile) and that are merged.
    for cap in (6, nb + 5):
        idx, counts = synth.random_support(b, hkv, nb, cap, seed=i + cap, density=0.4)
        counts[0, 0, nb // 2] = 0  # a query block that attends nothing
        outs = []
        for _ in range(3):
            o = empty_like_q(Q)
            wise.wise_sparse_attn(s, q, k, v, *_dev(idx, counts), o)
            outs.append(o)
        assert wise.wise_get_status() == wise.WISE_OK
        assert all(torch.equal(o, outs[0]) for o in outs[1:])
        want = orc.sparse_attention(Q, K, V, idx, counts, blk, units=pick)
        assert_close_o(units_of(bf16_dev_to_f64(outs[0]), pick, blk), np.asarray(want))
    # Every admissible block: the dense result, bit for bit.
    od = empty_like_q(Q)
    wise.wise_sparse_attn(s, q, k, v, *_dev(*synth.all_blocks_support(b, hkv, nb)), o)
    wise.wise_full_attn_accumulate(s, q, k, v, od)
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(o, od)


@pytest.mark.parametrize("h,hkv,L,d,blk", [(24, 24, 2048, 128, 128), (24, 24, 2048, 128, 32), (26, 26, 2048, 96, 128),
                                           (24, 8, 2048, 64, 64)])
@pytest.mark.parametrize("sink", [False, True])
def test_units_of_one_and_two_tiles(h, hkv, L, d, blk, sink):
    """Each query block attends itself, every third one the first block too.  V is
    drawn with std 0.5: such rows are close to one V row, whose half bf16 ulp
    would exceed the bound at |V| > 4."""
    s = wise.Shape(1, L, h, hkv, d, blk)
    nb = s.n_blocks
    Q, K, V = synth.random_qkv(1, h, hkv, L, d, seed=19, std=1.3, v_std=0.5)
    q, k, v = map(to_dev, (Q, K, V))
    idx = np.full((1, hkv, nb, 2), -1, dtype=np.int32)
    counts = np.ones((1, hkv, nb), dtype=np.int32)
    idx[..., 0] = np.arange(nb)
    if sink:
        two = np.arange(1, nb, 3)
        idx[:, :, two, 0], idx[:, :, two, 1], counts[:, :, two] = 0, two, 2
    di, dc = _dev(idx, counts)
    outs = []
    for _ in range(4):
        o = empty_like_q(Q)
        wise.wise_sparse_attn(s, q, k, v, di, dc, o)
        outs.append(o)
    assert wise.wise_get_status() == wise.WISE_OK
    assert all(torch.equal(o, outs[0]) for o in outs[1:])
    assert_close_o(bf16_dev_to_f64(outs[0]), np.asarray(orc.sparse_attention(Q, K, V, idx, counts, blk)))


# On either side of 256 query tiles: two heads of 256 and 257 tiles.  The reference
# is plain PyTorch in fp64 on sampled query blocks.
@pytest.mark.parametrize("L", [32768, 32896])
@pytest.mark.parametrize("blk", [128, 32])
def test_long_sequences(L, blk):
    h, d = 2, 64
    s = wise.Shape(1, L, h, h, d, blk)
    nb = s.n_blocks
    g = torch.Generator(device="cuda").manual_seed(L + blk)
    q, k, v = (torch.randn((1, h, L, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    o, om, os_ = (torch.empty_like(q) for _ in range(3))
    mass = torch.full((1, h, nb, nb), 7.0, device="cuda")
    cap = 9
    key = torch.rand((1, h, nb, nb), generator=g, device="cuda")
    qb = torch.arange(nb, device="cuda")
    key = key.masked_fill(qb[None, :] > qb[:, None], 2.0).masked_fill(qb[None, :] == qb[:, None], -1.0)
    low = key.argsort(-1)[..., :cap]
    counts = (qb + 1).clamp(max=cap).expand(1, h, nb).int().contiguous()
    idx = torch.where(torch.arange(cap, device="cuda") < counts[..., None], low, nb).sort(-1).values
    idx = torch.where(idx < nb, idx, -1).int().contiguous()
    wise.wise_full_attn_accumulate(s, q, k, v, o)
    wise.wise_full_attn_accumulate(s, q, k, v, om, mass, 0)
    wise.wise_sparse_attn(s, q, k, v, idx, counts, os_)
    assert wise.wise_get_status() == wise.WISE_OK
    assert (mass.double().sum(-1) - 1.0).abs().max() <= MASS_ROWSUM
    for head, block in ((0, 0), (1, nb // 2), (0, nb - 2), (1, nb - 1), (0, nb - 1), (1, 37 % nb)):
        rows = torch.arange(block * blk, (block + 1) * blk, device="cuda")
        n = (block + 1) * blk
        logits = q[0, head, rows].double() @ k[0, head, :n].double().T / d ** 0.5
        logits = logits.masked_fill(torch.arange(n, device="cuda")[None, :] > rows[:, None], -torch.inf)
        a = torch.softmax(logits, -1)
        for got in (o, om):
            assert (got[0, head, rows].double() - a @ v[0, head, :n].double()).abs().max() <= O_MAX_ABS
        r = a.reshape(blk, block + 1, blk).sum((0, 2)) / blk
        assert (mass[0, head, block, :block + 1].double() - r).abs().max() <= MASS_MAX_ABS
        assert not mass[0, head, block, block + 1:].any()
        keep = torch.zeros(nb, dtype=torch.bool, device="cuda")
        keep[idx[0, head, block, :int(counts[0, head, block])].long()] = True
        a = torch.softmax(logits.masked_fill(~keep[:block + 1].repeat_interleave(blk)[None, :], -torch.inf), -1)
        want = a @ v[0, head, :n].double()
        # A row with few keys may be close to one V row: half a bf16 ulp of it on top.
        assert (os_[0, head, rows].double() - want).abs().max() <= O_MAX_ABS + 2.0 ** -9 * float(want.abs().max())


# One-stream kernel; two streams: head pairs, unpaired heads of 96 (two V tiles a
# stream), of 64 (rings of two K tiles), tile pairs with the first tile alone.
@pytest.mark.parametrize("h,hkv,L,d,blk", [(24, 24, 2048, 128, 128), (24, 24, 2048, 96, 32), (64, 16, 2048, 128, 128),
                                           (40, 40, 2048, 96, 128), (40, 40, 2048, 64, 32), (92, 92, 640, 128, 64)])
@pytest.mark.parametrize("mode", ["dense", "dense_mass", "sparse"])
def test_a_wait_that_runs_out(h, hkv, L, d, blk, mode):
    """As in test_timeout_gpu: with a limit of 1 ns the kernel gives up, reports it
    and unwinds; afterwards the same call gives the same output as before."""
    s = wise.Shape(1, L, h, hkv, d, blk)
    nb = s.n_blocks
    q, k, v = (to_dev(x) for x in synth.random_qkv(1, h, hkv, L, d, seed=5))
    o, mass = torch.empty_like(q), torch.zeros((1, h, nb, nb), device="cuda")
    idx, counts = _dev(*synth.random_support(1, hkv, nb, 8, seed=6, density=0.5))

    def call():
        if mode == "sparse":
            wise.wise_sparse_attn(s, q, k, v, idx, counts, o)
        else:
            wise.wise_full_attn_accumulate(s, q, k, v, o, mass if mode == "dense_mass" else None, 0)

    call()
    assert wise.wise_get_status() == wise.WISE_OK
    want, want_mass = o.clone(), mass.clone()
    status = wise.WISE_OK
    wise.wise_set_wait_limit_ns(1)
    try:
        for _ in range(10):  # a wait that ends within its first probe never looks at the clock
            call()
            status = wise.wise_get_status()
            if status != wise.WISE_OK:
                break
    finally:
        wise.wise_set_wait_limit_ns(0)
    assert status == wise.WISE_ERR_TIMEOUT
    o.zero_()
    call()
    assert wise.wise_get_status() == wise.WISE_OK
    assert torch.equal(o, want) and torch.equal(mass, want_mass)
