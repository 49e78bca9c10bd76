"""The tensor-memory kernel at the edges of its ranges, against the CPU oracle: token groups (one more than a multiple
of 8 or 16), partial 128-row and 256-row blocks, odd and single mask words per tile, ragged K, CTAs that enter a tile in
its middle, and the rule that chooses it. A child process forces it wherever it can run."""
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

# (M, K, sparsity, N, format, flags)
EDGES = [
    (16, 128, 0.5, 9, (16, 128, 2, 1), 0), (1, 1, 0.0, 23, (16, 128, 2, 1), 0), (128, 256, 0.5, 16, (16, 256, 2, 1), 0),
    (130, 300, 0.5, 17, (16, 256, 2, 1), 0), (257, 1000, 0.5, 64, (16, 384, 2, 1), 0), (1030, 4100, 0.3, 24, (16, 1024, 2, 1), 2),
    (4096, 4096, 0.3, 32, (16, 1024, 2, 1), 0),      # as many ring slots as warps and a few: slots change owner
    (2000, 9000, 0.3, 48, (16, 512, 2, 1), 4), (500, 3001, 0.6, 33, (16, 256, 2, 2), 2), (1030, 4096, 0.5, 40, (16, 1024, 2, 2), 0),
    (333, 700, 0.5, 56, (16, 512, 2, 2), 8), (2048, 8200, 0.7, 16, (16, 1024, 2, 2), 8),
]


def run_edges():
    from paper_2608_09291_b200 import binding as b
    for M, K, s, N, fmt, flags in EDGES:
        W = (workloads.make_weight_w2 if flags & 8 else workloads.make_weight)(M, K, s, seed=M + K + N)
        X = workloads.make_x(K, N, seed=N)
        s_w, s_x = workloads.make_scales(M, N, seed=M)
        sw = b.SparseWeight(W, s_w, fmt=fmt, max_N=N, flags=flags)
        assert b.us_launch_info(sw.handle, N)["block"] in (800, 896)
        Xd, xs = torch.from_numpy(b.pack_int4(X)).cuda(), torch.from_numpy(s_x.copy()).cuda()
        ref = oracle.spmm_dense(W, X)
        for _ in range(2):     # the second call checks the self-cleaning workspace
            y32 = sw.spmm(Xd, N).cpu().numpy()
            sw.check()
            assert (y32 == ref).all(), (M, K, N, fmt, flags, int((y32 != ref).sum()))
        y16 = sw.spmm(Xd, N, xs).cpu().numpy()
        assert oracle.fp16_within_tolerance(y16, ref, s_w, s_x).all(), (M, K, N, fmt, flags)
        if fmt[3] == 1:        # chained call: the absmax of the outputs
            am = b.new_amax()
            y = sw.spmm_requant(torch.from_numpy(workloads.make_x_f16(K, N, seed=3)).cuda(), N,
                                b.absmax_f16(torch.from_numpy(workloads.make_x_f16(K, N, seed=3)).cuda()), y_amax=am)
            got = np.abs(y.cpu().numpy()).max(axis=1)
            assert (b.amax_values(am, N) == got.view(np.uint16)).all(), (M, K, N)
        sw.close()


@pytest.mark.parametrize("octets", ["2", "3"])
def test_edges_forced(octets):
    r = subprocess.run([sys.executable, "-c", "import sys; sys.path[:0] = ['.', 'tests']; import test_gpu_tc; test_gpu_tc.run_edges()"],
                       cwd=ROOT, env=dict(os.environ, US_TC="2", US_TC_OCT=octets), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-1500:] + r.stderr[-1500:]


def test_rule_and_withheld_copy():
    """28672 x 4096 at N = 40 takes this kernel, N = 8 does not; a copy that never comes is reported, not waited for."""
    from paper_2608_09291_b200 import binding as b
    W = workloads.make_weight(28672, 4096, 0.5, seed=7)
    X = workloads.make_x(4096, 40, seed=7)
    sw = b.SparseWeight(W, None, max_N=40)
    try:
        assert b.us_launch_info(sw.handle, 40)["block"] == 800 and b.us_launch_info(sw.handle, 8)["block"] <= 640
        Xd = torch.from_numpy(b.pack_int4(X)).cuda()
        ref = oracle.spmm_dense(W, X)
        for position in (0, 1000):
            b.us_debug_withhold_copy(sw.handle, position, wait_us=2000)
            sw.spmm(Xd, 40)
            assert b.us_last_error(sw.handle) == 7
            b.us_debug_withhold_copy(sw.handle, -1)
            y = sw.spmm(Xd, 40).cpu().numpy()
            sw.check()
            assert (y == ref).all()
    finally:
        sw.close()


@pytest.mark.parametrize("s,fmt", [(0.5, (16, 512, 2, 2)), (0.3, (16, 512, 2, 1))])
def test_idle_warps_keep_off_tiles_in_use(s, fmt):
    """The last row block has 14 strips for 16 warps, and the tile ring a number of slots (between 16 and 32) that 16 does
    not divide: the two idle warps refill slots that other warps decode from, at two stages per tile."""
    from paper_2608_09291_b200 import binding as b
    M, K, N = 8160, 9216, 64
    W = workloads.make_weight(M, K, s, seed=11)
    X = workloads.make_x(K, N, seed=11)
    sw = b.SparseWeight(W, fmt=fmt, max_N=N)
    try:
        assert b.us_launch_info(sw.handle, N)["block"] == 800
        Xd = torch.from_numpy(b.pack_int4(X)).cuda()
        ref = torch.from_numpy(oracle.spmm_dense(W, X)).cuda()
        for _ in range(20):
            y = sw.spmm(Xd, N)
            sw.check()
            assert torch.equal(y, ref), int((y != ref).sum())
    finally:
        sw.close()


def test_sums_stay_exact_at_the_largest_k():
    """37888 x 131072 gives every CTA one row block of 512 stages, whose sums of extreme values would leave 32 bits by one:
    the other kernel takes it. (Nearly all rows are empty, so that the matrix costs no host memory.)"""
    from paper_2608_09291_b200 import binding as b
    M, K = 37888, 131072
    W = np.zeros((M, K), np.int8)
    rows = [0, 8, 20000, 37887]     # both halves of a strip
    W[rows] = -8
    X = workloads.make_x(K, 64, seed=3)
    X[0], X[1] = -8, 7
    sw = b.SparseWeight(W, max_N=64)
    try:
        Xd = torch.from_numpy(b.pack_int4(X)).cuda()
        want = torch.from_numpy((-8 * X.astype(np.int64).sum(axis=1)).astype(np.int32)).cuda()
        for N in (16, 64):
            y = sw.spmm(Xd[:N], N)
            sw.check()
            assert all(torch.equal(y[:, r], want[:N]) for r in rows), (N, y[:2, rows].tolist(), want[:2].tolist())
            y[:, rows] = 0
            assert int(y.count_nonzero()) == 0, N
            assert b.us_launch_info(sw.handle, N)["block"] <= 512
    finally:
        sw.close()
