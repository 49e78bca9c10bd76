"""Activations of any K: rows that start at any byte and end in the middle of a 32-column unit, and the end of X, in the
default, packed and wide staging forms. X ends exactly at its last byte in a buffer whose rest is poisoned."""
import os
import subprocess
import sys
from pathlib import Path

import numpy as np
import pytest

import oracle
from paper_2608_09291_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = Path(__file__).resolve().parent.parent


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


def run_largest_share():
    from paper_2608_09291_b200 import binding as b
    for M, K, wide in ((512, 8192, True), (1500, 6000, True), (4096, 4096, False), (2304, 4096, False)):
        W = workloads.make_weight(M, K, 0.5, seed=1)
        X = workloads.make_x(K, 8, seed=1)
        sw = b.SparseWeight(W, max_N=8)
        info = b.us_launch_info(sw.handle, 8)
        assert b.us_launch_kernel(sw.handle, 8) == "us_spmm_kernel"
        assert (info["smem_bytes"] > 114 * 1024) == wide, (M, K, info)
        y = sw.spmm(torch.from_numpy(b.pack_int4(X)).cuda(), 8).cpu().numpy()
        sw.check()
        assert (y == oracle.spmm_dense(W, X)).all(), (M, K)
        sw.close()


def test_plan_counts_the_largest_share():
    """512 x 8192 (one strip of 32 tiles to a CTA) and 1500 x 6000 (12 tiles): all warps of the SM; 4096 x 4096 (eight
    tiles) and 2304 x 4096 (one strip to a CTA, none gets two): half an SM. The plans are us_spmm_kernel's: a child process
    keeps the decode-ahead kernel off these shapes."""
    r = subprocess.run([sys.executable, "-c", "import sys; sys.path[:0] = ['.', 'tests']; import test_gpu_ragged; test_gpu_ragged.run_largest_share()"],
                       cwd=ROOT, env=dict(os.environ, US_AHEAD="0"), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-1500:] + r.stderr[-1500:]
