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
