"""The decode-ahead kernel at its edges: one tile and many rounds per warp, tiles parked and not, activations over the tile
slots and beside them, K cut in ranges (sums through the workspace), ragged rows, every format, chained calls among plain ones."""
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


# (half an SM's shared memory, and the threads: 384 and 512 at N <= 8 and N <= 16, 320 with two column areas and at N <= 32)
@pytest.mark.parametrize("M,K,fmt,w2,N,block", [
    (16, 256, (16, 128, 2, 1), False, 8, 384),         # one CTA, two tiles
    (2300, 1100, (16, 128, 2, 1), False, 7, 384),      # nine segments, ragged rows
    (4096, 4096, None, False, 1, 384),
    (11008, 2048, None, False, 3, 384),
    (4096, 3000, (16, 384, 2, 1), False, 9, 512),      # three mask words, columns past K
    (9000, 5120, None, False, 16, 512),                # later tiles decoded when their turn comes
    (2048, 16384, None, False, 16, 512),               # K in ranges
    (1600, 16001, (16, 1024, 2, 1), False, 11, 512),   # the same with ragged rows
    (3000, 4096, None, False, 32, 320),                # activations over the slots
    (3000, 4095, (16, 1024, 2, 2), False, 25, 320),
    (5003, 3001, (16, 1024, 2, 2), False, 8, 320),
    (4096, 4096, (16, 512, 2, 2), True, 8, 320),
    (1500, 2100, (16, 2048, 2, 2), True, 16, 320),     # parked tiles of 128 columns
])
def test_decode_ahead(M, K, fmt, w2, N, block):
    from paper_2608_09291_b200 import binding as b
    W = (workloads.make_weight_w2 if w2 else workloads.make_weight)(M, K, 0.5, seed=M + K)
    X = workloads.make_x(K, N, seed=K)
    s_w, s_x = workloads.make_scales(M, N, seed=K)
    sw = b.SparseWeight(W, s_w, fmt=fmt, max_N=N, flags=b.US_ENCODE_W2 if w2 else 0)
    try:
        info = b.us_launch_info(sw.handle, N)
        assert b.us_launch_kernel(sw.handle, N) == "us_spmm_ahead_kernel"
        assert info["block"] == block and info["smem_bytes"] <= 114 * 1024, info
        ref = oracle.spmm_dense(W, X)
        Xd, sd = torch.from_numpy(b.pack_int4(X)).cuda(), torch.from_numpy(s_x).cuda()
        outs = [sw.spmm(Xd, N) if i % 2 else sw.spmm(Xd, N, sd) for i in range(6)]   # back to back: each beside the one before
        torch.cuda.synchronize()
        sw.check()
        for i, y in enumerate(outs):
            if i % 2:
                assert (y.cpu().numpy() == ref).all(), i
            else:   # (one rounding to fp16)
                assert oracle.fp16_within_tolerance(y.cpu().numpy(), ref, s_w, s_x).all(), i
    finally:
        sw.close()


@pytest.mark.parametrize("M,K,N", [(1024, 1024, 8), (2304, 2304, 16), (2048, 2048, 32)])
def test_dependent_chain_of_decode_ahead_calls(M, K, N):
    """Every call reads what the one before wrote, and the weights of several handles are decoded meanwhile."""
    from paper_2608_09291_b200 import binding as b
    s_w = workloads.make_chain_weight_scales(M, K, 3)
    Ws = [workloads.make_weight(M, K, 0.5, seed=i) for i in range(3)]
    sws = [b.SparseWeight(W, s_w, max_N=N) for W in Ws]
    try:
        x0 = workloads.make_x_f16(K, N, seed=1)
        a, src, ys, amaxes = b.absmax_f16(torch.from_numpy(x0).cuda()), torch.from_numpy(x0).cuda(), [], []
        for sw in sws:
            left = b.new_amax()
            y = sw.spmm_requant(src, N, a, y_amax=left, amax_range=(0, M))
            ys.append(y); amaxes.append(left)
            src, a = y, left
        torch.cuda.synchronize()
        prev = x0
        for W, sw, y, left in zip(Ws, sws, ys, amaxes):
            sw.check()
            q, s = oracle.requant_int4(prev)
            prev = y.cpu().numpy()
            assert oracle.fp16_within_tolerance(prev, oracle.spmm_dense(W, q), s_w, s).all()
            assert (b.amax_values(left, N) == oracle.absmax_f16(prev).view(np.uint16)).all()
    finally:
        for sw in sws:
            sw.close()


WITHHELD = [
    (1024, 4096, None, 8),                    # one K range, activations beside the slots, every tile parked
    (2048, 16384, None, 16),                  # K in ranges: partial sums and arrivals are left in the workspace
    (3000, 4096, None, 32),                   # activations over the slots: they are fetched as the wait runs out
    (1600, 16001, (16, 1024, 2, 1), 11),      # K in ranges, ragged rows
    (9000, 5120, None, 16),                   # later tiles, for which helpers wait on slots
    (5003, 3001, (16, 1024, 2, 2), 8),        # two column areas, ragged rows
]


def run_withheld(M, K, fmt, N, kernel):
    from paper_2608_09291_b200 import binding as b
    W, V = workloads.make_weight(M, K, 0.5, seed=M + K), workloads.make_weight(4096, 2048, 0.5, seed=5)
    X, Z = workloads.make_x(K, N, seed=K), workloads.make_x(2048, 8, seed=6)
    sw, other = b.SparseWeight(W, None, fmt=fmt, max_N=N), b.SparseWeight(V, None, max_N=8)
    try:
        assert b.us_launch_kernel(sw.handle, N) == kernel
        ref, ref_other = oracle.spmm_dense(W, X), oracle.spmm_dense(V, Z)
        Xd, Zd = torch.from_numpy(b.pack_int4(X)).cuda(), torch.from_numpy(b.pack_int4(Z)).cuda()
        n_tiles = sw.stats["n_tiles"]
        for position in (0, n_tiles // 2 + 3, n_tiles - 1):
            b.us_debug_withhold_copy(sw.handle, position, wait_us=2000)
            sw.spmm(Xd, N)
            ys = [other.spmm(Zd, 8) for _ in range(4)]
            torch.cuda.synchronize()
            assert b.us_last_error(sw.handle) == 7, position      # US_ERR_DEVICE_TIMEOUT
            assert b.us_last_error(sw.handle) == 0
            other.check()
            for y in ys:
                assert (y.cpu().numpy() == ref_other).all(), position
            b.us_debug_withhold_copy(sw.handle, -1)
            for _ in range(2):
                y = sw.spmm(Xd, N)
            torch.cuda.synchronize()
            sw.check()
            assert (y.cpu().numpy() == ref).all(), position
    finally:
        sw.close()
        other.close()


@pytest.mark.parametrize("M,K,fmt,N", WITHHELD)
def test_withheld_tile_ends_the_call_and_leaves_its_neighbours_alone(M, K, fmt, N):
    """A tile that is never copied: the call ends with its error, nothing of it (activations still on their way) reaches the
    CTAs of the calls behind it on the stream, and the handle's next call is correct."""
    run_withheld(M, K, fmt, N, "us_spmm_ahead_kernel")


def test_withheld_tile_of_the_other_kernel():
    """The same shapes on us_spmm_kernel: sums in shared memory, K in ranges, half an SM and all of it. (A child process: which
    kernels may run is read once.)"""
    code = ("import sys; sys.path[:0] = ['.', 'tests']; import test_gpu_ahead as t\n"
            "for case in t.WITHHELD + [(24000, 1024, None, 8)]: t.run_withheld(*case, 'us_spmm_kernel')")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, US_AHEAD="0", US_TC="0"), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-1500:] + r.stderr[-1500:]


def test_time_of_earlier_work_is_not_counted_against_a_wait():
    """Two calls that take two seconds each by giving up (test hook), a third behind them, resident from the start: its helpers
    wait for slots that come free behind its own MMAs, four seconds later, with a limit of two for what is its own."""
    from paper_2608_09291_b200 import binding as b
    M, K, N = 148 * 96, 5120, 16           # six strips, 30 tiles to each of 148 CTAs, of which 16 are parked; seven slots
    W, X = workloads.make_weight(M, K, 0.5, seed=3), workloads.make_x(K, N, seed=3)
    sws = [b.SparseWeight(W, None, max_N=N) for _ in range(3)]
    try:
        info = b.us_launch_info(sws[0].handle, N)
        if info["grid"] != 148:
            pytest.skip("laid out for 148 SMs")
        Xd = torch.from_numpy(b.pack_int4(X)).cuda()
        ys = [torch.empty((N, M), dtype=torch.int32, device="cuda") for _ in sws]
        torch.cuda.synchronize()
        b.us_debug_withhold_copy(sws[0].handle, 0, wait_us=2_000_000)      # a tile that is decoded ahead
        b.us_debug_withhold_copy(sws[1].handle, 29, wait_us=2_000_000)     # one whose turn comes when the first call has ended
        for sw, y in zip(sws, ys):
            sw.spmm(Xd, N, out=y)
        torch.cuda.synchronize()
        assert [b.us_last_error(sw.handle) for sw in sws] == [7, 7, 0]     # US_ERR_DEVICE_TIMEOUT where a tile was withheld
        assert (ys[2].cpu().numpy() == oracle.spmm_dense(W, X)).all()
    finally:
        for sw in sws:
            sw.close()


@pytest.mark.parametrize("M,K,s", [(20480, 5120, 0.5), (27648, 5120, 0.5),     # 45 and 59 tiles to a CTA, six and five slots
                                   (8192, 8192, 0.5), (8200, 8191, 0.5)])      # K in ranges where the other kernel has one; ragged rows
def test_call_that_follows_its_neighbour_to_half_an_sm(M, K, s):
    """Behind a call of half an SM on the same stream the call takes half an SM itself, twice running; on another stream, behind
    another kernel of the library or a clear it does not. The sums are the same in both forms."""
    from paper_2608_09291_b200 import binding as b
    N = 16
    W, (s_w, s_x) = workloads.make_weight(M, K, s, seed=M), workloads.make_scales(M, N, seed=K)
    X = workloads.make_x(K, N, seed=K)
    sw = b.SparseWeight(W, s_w, max_N=N)
    small = b.SparseWeight(workloads.make_weight(2048, 2048, 0.5, seed=1), workloads.make_chain_weight_scales(2048, 2048, 1), max_N=N)
    other = torch.cuda.Stream()
    try:
        Xd, xs = torch.from_numpy(b.pack_int4(X)).cuda(), torch.from_numpy(s_x.copy()).cuda()
        Zd = torch.from_numpy(b.pack_int4(workloads.make_x(2048, N, seed=2))).cuda()
        z16 = torch.from_numpy(workloads.make_x_f16(2048, N, seed=3)).cuda()
        amax = b.absmax_f16(z16)
        out = torch.empty((N, 2048), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()

        def kernel(stream=None):
            return b.us_launch_kernel(sw.handle, N, stream)

        ref = torch.from_numpy(oracle.spmm_dense(W, X)).cuda()
        assert kernel() == "us_spmm_kernel"
        first = sw.spmm(Xd, N, xs)
        for _ in range(3):
            assert torch.equal(sw.spmm(Xd, N), ref)
            small.spmm(Zd, N, out=out)
            assert kernel() == "us_spmm_ahead_kernel" and kernel(other.cuda_stream) == "us_spmm_kernel"
            assert torch.equal(sw.spmm(Xd, N), ref)
            assert kernel() == "us_spmm_ahead_kernel"
            assert torch.equal(sw.spmm(Xd, N, xs), first)
            assert kernel() == "us_spmm_kernel"
            assert torch.equal(sw.spmm(Xd, N), ref)
            for between in (lambda: small.spmm_requant(z16, N, amax), lambda: b.quantize_f16(z16, amax), lambda: b.absmax_f16(z16)):
                small.spmm(Zd, N, out=out)
                between()
                assert kernel() == "us_spmm_kernel"
            small.spmm(Zd, N, out=out)
            y = torch.empty_like(ref)
            b.us_spmm_static_scratch(sw.handle, Xd.data_ptr(), N, None, y.data_ptr())
            assert kernel() == "us_spmm_kernel" and torch.equal(y, ref)
        sw.check()
        small.check()
        assert oracle.fp16_within_tolerance(first.cpu().numpy(), ref.cpu().numpy(), s_w, s_x).all()
    finally:
        sw.close()
        small.close()
