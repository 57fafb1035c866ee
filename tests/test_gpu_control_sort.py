"""The control's bucket sort at the edges of its variants: one block up to
4096 samples, the four launches beyond, one and two scan tiles (4096 buckets
each: 65,536 samples up), and the wider buckets past 2^23 samples.  A
permutation is exact: every output equals the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1802_01685_gb300 import bf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


@pytest.mark.parametrize("n", [1023, 1025, 4095, 4096, 4097, 8193, 65535, 65537, 131073, 2 ** 23, 2 ** 23 + 1])
def test_control_at_the_edges_of_its_variants(ctx, n):
    x = np.arange(n, dtype=np.float32)              # exact in FP32 up to 2^24: every sample is its own index
    xd = torch.from_numpy(x).cuda()
    yd = torch.full_like(xd, -1.0)
    for seed in (9, 2 ** 63 + 11):
        bf.bf_control_randomize(ctx, xd, seed, yd)
        np.testing.assert_array_equal(yd.cpu().numpy(), oracle.permute(x, seed))
