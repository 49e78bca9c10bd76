"""Activations of any K: rows that start at any byte and end in the middle of a 32-column unit, and the end of X, in the
default, packed and wide staging forms. X ends exactly at its last byte in a buffer whose rest is poisoned."""
import numpy as np
import pytest

import oracle
from paper_2608_09291_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K", [1, 2, 15, 31, 33, 63, 100, 129, 1000, 1001, 1023, 2047, 4104])
@pytest.mark.parametrize("fmt", [(16, 128, 2, 1), (16, 384, 2, 1), (16, 1024, 2, 1), (16, 512, 2, 2)])
def test_any_k(K, fmt):
    from paper_2608_09291_b200 import binding as b
    M = 200
    W = workloads.make_weight(M, K, 0.4, seed=K)
    X = workloads.make_x(K, 40, seed=K)
    sw = b.SparseWeight(W, fmt=fmt, max_N=40)
    try:
        for N in (1, 5, 8, 11, 24, 40):
            packed = b.pack_int4(X[:N])
            buf = torch.full((packed.size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
            buf[: packed.size] = torch.from_numpy(packed.reshape(-1)).cuda()
            y = sw.spmm(buf[: packed.size].view(N, -1), N).cpu().numpy()
            sw.check()
            assert (y == oracle.spmm_dense(W, X[:N])).all(), (N, K, fmt)
    finally:
        sw.close()


def test_plan_counts_the_largest_share():
    """5008 x 3008 has CTAs of nine tiles: all its warps at once, not eight in half an SM; 4096 x 4096 has eight."""
    from paper_2608_09291_b200 import binding as b
    for M, K, wide in ((5008, 3008, True), (4096, 4096, False)):
        W = workloads.make_weight(M, K, 0.5, seed=1)
        h = b.us_encode(W, fmt=(16, 1024, 2, 2), max_N=8)
        assert (b.us_launch_info(h, 8)["block"] > 384) == wide
        b.us_destroy(h)
