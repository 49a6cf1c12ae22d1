"""The limit of the attention kernels' internal waits (wise_set_wait_limit_ns)
at both ends of its range, on launches of either kernel: a healthy launch never
runs out of time, whatever the limit is above the time of one of its steps."""
import contextlib

import pytest
import torch

from paper_2609_27373_gb300 import synth, wise
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def wait_limit(ns):
    wise.wise_set_wait_limit_ns(ns)
    try:
        yield
    finally:
        wise.wise_set_wait_limit_ns(0)


# 1024 query tiles (two-stream kernel: heads unpaired or tiles paired), head
# pairs, unpaired heads of 96; 96 query tiles (one-stream kernel).
@pytest.mark.parametrize("H,Hkv,L,D", [(32, 32, 4096, 128), (64, 8, 1024, 64), (64, 64, 1024, 96), (12, 12, 1024, 128)])
@pytest.mark.parametrize("ns", [2 ** 64 - 1, 2 ** 63, 2 ** 62, 10 ** 12])
def test_a_long_limit_is_no_limit(H, Hkv, L, D, ns):
    shape = wise.Shape(1, L, H, Hkv, D, 128)
    nb = shape.n_blocks
    Q, K, V = (to_dev(x) for x in synth.random_qkv(1, H, Hkv, L, D, seed=3))
    idx, counts = (torch.from_numpy(x).cuda() for x in synth.random_support(1, Hkv, nb, 6, seed=4, density=0.5))
    mass = torch.empty((1, H, nb, nb), dtype=torch.float32, device="cuda")
    outs = []
    for limit in (0, ns):
        O = [torch.zeros_like(Q) for _ in range(3)]
        with wait_limit(limit):
            wise.wise_full_attn_accumulate(shape, Q, K, V, O[0])
            wise.wise_full_attn_accumulate(shape, Q, K, V, O[1], mass, 0)
            wise.wise_sparse_attn(shape, Q, K, V, idx, counts, O[2])
            assert wise.wise_get_status() == wise.WISE_OK
        outs.append(O)
    assert all(torch.equal(a, b) for a, b in zip(*outs))


# Launches of a few hundred us whose steps take a few us each, under limits
# between the two.  One-tile units leave one stream of a CTA without work for
# the whole launch; units without a tile have no product to issue.
@pytest.mark.parametrize("mode", ["dense", "dense_mass"])
def test_a_stream_without_work_is_not_a_stalled_one(mode):
    H, L, D = 24576, 128, 64
    shape = wise.Shape(1, L, H, H, D, 128)
    g = torch.Generator(device="cuda").manual_seed(1)
    Q, K, V = (torch.randn((1, H, L, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    mass = torch.zeros((1, H, 1, 1), device="cuda") if mode == "dense_mass" else None
    O = torch.empty_like(Q)
    wise.wise_full_attn_accumulate(shape, Q, K, V, O, mass, 0)  # loads the kernel, allocates the scratch
    assert wise.wise_get_status() == wise.WISE_OK
    with wait_limit(100_000):
        wise.wise_full_attn_accumulate(shape, Q, K, V, O, mass, 0)
        assert wise.wise_get_status() == wise.WISE_OK
    want = torch.nn.functional.scaled_dot_product_attention(Q[:, :64].float(), K[:, :64].float(), V[:, :64].float(),
                                                            is_causal=True)
    assert (O[:, :64].float() - want).abs().max() <= 1e-2 * max(1.0, float(want.abs().max()))


@pytest.mark.parametrize("H,Hkv", [(256, 256), (256, 128)])
def test_units_without_a_tile_are_progress(H, Hkv):
    L, D, cap = 32768, 64, 4
    shape = wise.Shape(1, L, H, Hkv, D, 128)
    Q = torch.zeros((1, H, L, D), dtype=torch.bfloat16, device="cuda")
    K, V = Q[:, :Hkv].contiguous(), Q[:, :Hkv].contiguous()
    idx = torch.full((1, Hkv, L // 128, cap), -1, dtype=torch.int32, device="cuda")
    counts = torch.zeros((1, Hkv, L // 128), dtype=torch.int32, device="cuda")
    O = torch.ones_like(Q)
    wise.wise_sparse_attn(shape, Q, K, V, idx, counts, O)
    assert wise.wise_get_status() == wise.WISE_OK
    O.fill_(1.0)
    with wait_limit(100_000):
        wise.wise_sparse_attn(shape, Q, K, V, idx, counts, O)
        assert wise.wise_get_status() == wise.WISE_OK
    assert not O.any()
