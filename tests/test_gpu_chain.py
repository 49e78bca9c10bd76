"""Chained calls (fp16 in, per-token INT4 inside, fp16 out) against the CPU oracle. The quantised
codes, steps and absmax words are integers decided in fp32 on both sides: they must agree bit for
bit. The fp16 outputs are checked stage by stage from the device's own previous output, within
max(2e-3 relative, 1 fp16 ulp) of the exactly rounded reference."""
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


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2608_09291_b200 import binding
    torch.cuda.set_device(0)
    return binding


def _unpack(Xq: np.ndarray, K: int) -> np.ndarray:
    nib = np.empty((Xq.shape[0], 2 * Xq.shape[1]), dtype=np.int16)
    nib[:, 0::2] = Xq & 0xF
    nib[:, 1::2] = Xq >> 4
    nib = nib[:, :K]
    return np.where(nib >= 8, nib - 16, nib).astype(np.int8)


def _amax_words(a16: np.ndarray) -> np.ndarray:
    return a16.view(np.uint16)


@pytest.mark.parametrize("N,K,pad,off", [(8, 4096, 0, 0), (16, 5120, 10240, 5120), (5, 1000, 24, 0),
                                         (3, 1001, 6, 1), (1, 7, 0, 0), (64, 256, 0, 0)])
def test_absmax_and_quantize_bit_exact(b, N, K, pad, off):
    """Aligned and unaligned rows, ragged K, a column window of a wider buffer."""
    full = workloads.make_x_f16(K + pad, N, seed=900 + K)
    full[0, off] = 0.0
    if N > 2:
        full[2, off:off + K] = 0.0                       # an all-zero token
        full[1, off:off + K] *= np.float16(2.0 ** -14)   # a token deep in the small range
    Xd = torch.from_numpy(full).cuda()
    view = Xd[:, off:off + K]
    x = full[:, off:off + K]
    amax = b.absmax_f16(view)
    Xq, sc = b.quantize_f16(view, amax)
    torch.cuda.synchronize()
    a_ref = oracle.absmax_f16(x)
    assert np.array_equal(b.amax_values(amax, N), _amax_words(a_ref))
    q_ref, s_ref = oracle.requant_int4(x)
    assert np.array_equal(sc.cpu().numpy().view(np.uint16), s_ref.view(np.uint16))
    assert np.array_equal(_unpack(Xq.cpu().numpy(), K), q_ref)


def _check_requant_call(b, sw, W, s_w, x16, N, m0, m1, reps=2):
    """One chained call on activations x16 (numpy (N, K) fp16): output within the bar, absmax words
    exact for the values the device stored."""
    Xd = torch.from_numpy(np.ascontiguousarray(x16)).cuda()
    amax = b.absmax_f16(Xd)
    y_amax = torch.full((b.US_AMAX_BYTES // 4,), -1, dtype=torch.int32, device="cuda")   # junk: never cleared
    q, s = oracle.requant_int4(x16)
    ref = oracle.spmm_dense(W, q)
    for rep in range(reps):
        Y = sw.spmm_requant(Xd, N, amax, y_amax=y_amax, amax_range=(m0, m1))
        torch.cuda.synchronize()
        sw.check()
        got = Y.cpu().numpy()
        ok = oracle.fp16_within_tolerance(got, ref, s_w, s, rel=2e-3)
        assert ok.all(), f"rep {rep}: {int((~ok).sum())} fp16 outputs outside tolerance"
        assert np.array_equal(b.amax_values(y_amax, N), _amax_words(oracle.absmax_f16(got, m0, m1))), f"rep {rep}"
    return got


@pytest.mark.parametrize("M,K,N,s,rng_m", [
    (1024, 1024, 8, 0.5, (0, 1024)),
    (4096, 4096, 1, 0.5, (100, 3000)),
    (4096, 4096, 16, 0.3, (0, 4096)),
    (2000, 1000, 5, 0.5, (7, 1993)),        # ragged rows and columns
    (1030, 2056, 12, 0.6, (0, 0)),          # empty range: the words stay zero
    (5120, 13824, 16, 0.5, (0, 5120)),      # the 13B down projection
    (11008, 4096, 32, 0.5, (11008 - 16, 11008)),
    (4096, 11008, 32, 0.5, (0, 4096)),      # global split-K path
    (4096, 4096, 64, 0.5, (1, 4095)),
])
def test_spmm_requant(b, M, K, N, s, rng_m):
    seed = 700 + M % 97 + K % 89 + N
    W = workloads.make_weight(M, K, s, seed=seed)
    s_w, _ = workloads.make_scales(M, N, seed=seed)
    x16 = workloads.make_x_f16(K, N, seed=seed)
    sw = b.SparseWeight(W, s_w, max_N=N)
    try:
        _check_requant_call(b, sw, W, s_w, x16, N, *rng_m)
        # the plain entry point fed with the separately quantised codes gives the same fp16 values
        Xd = torch.from_numpy(x16).cuda()
        amax = b.absmax_f16(Xd)
        Xq, sc = b.quantize_f16(Xd, amax)
        y_plain = sw.spmm(Xq, N, sc)
        y_chain = sw.spmm_requant(Xd, N, amax)
        torch.cuda.synchronize()
        sw.check()
        assert torch.equal(y_plain, y_chain)
    finally:
        sw.close()


def test_requant_argument_errors(b):
    W = workloads.make_weight(256, 256, 0.5, seed=5)
    s_w, _ = workloads.make_scales(256, 8, seed=5)
    sw = b.SparseWeight(W, s_w, max_N=8)
    bare = b.SparseWeight(W, None, max_N=8)
    try:
        X = torch.zeros((8, 256), dtype=torch.float16, device="cuda")
        a = b.new_amax()
        a2 = b.new_amax()
        Y = torch.zeros((8, 256), dtype=torch.float16, device="cuda")
        call = b._lib.us_spmm_requant
        assert call(sw.handle, X.data_ptr(), 255, a.data_ptr(), 8, Y.data_ptr(), None, 0, 0, None) == 1   # ldx < K
        assert call(sw.handle, X.data_ptr(), 256, a.data_ptr(), 9, Y.data_ptr(), None, 0, 0, None) == 1   # N > max_N
        assert call(sw.handle, X.data_ptr(), 256, a.data_ptr(), 8, Y.data_ptr(), a2.data_ptr(), 0, 257, None) == 1
        assert call(sw.handle, X.data_ptr(), 256, a.data_ptr(), 8, Y.data_ptr(), a2.data_ptr(), 9, 3, None) == 1
        assert call(sw.handle, X.data_ptr(), 256, a.data_ptr(), 8, Y.data_ptr(), a.data_ptr(), 0, 8, None) == 1   # same buffer
        assert call(sw.handle, None, 256, a.data_ptr(), 8, Y.data_ptr(), None, 0, 0, None) == 1
        assert call(bare.handle, X.data_ptr(), 256, a.data_ptr(), 8, Y.data_ptr(), None, 0, 0, None) == 1  # no weight scales
        assert b._lib.us_absmax_f16(X.data_ptr(), 100, 8, 256, a.data_ptr(), None) == 1
        assert b._lib.us_quantize_f16(X.data_ptr(), 256, 0, 256, a.data_ptr(), Y.data_ptr(), None, None) == 1
        torch.cuda.synchronize()
        sw.check()
    finally:
        sw.close()
        bare.close()


@pytest.mark.parametrize("j,s", [(0, 0.3), (1, 0.5), (2, 0.7)])
def test_layer_13b_chain(b, j, s):
    """The projections of one 13B-shaped decoder layer as a chain of four launches on one stream,
    no synchronisation in between: [Q;K;V] stacked (15360 x 5120) -> O (5120 x 5120, reads the Q
    columns) -> [gate;up] stacked (27648 x 5120) -> down (5120 x 13824, reads the gate columns).
    The attention and the gating between them are not this library's work: the chain carries the
    data flow and the re-quantisation. Each stage is checked against the oracle from the device's
    own previous output."""
    N, H, F = 16, 5120, 13824
    shapes = [("qkv", 3 * H, H, (0, H)), ("o", H, H, (0, H)), ("gate_up", 2 * F, H, (0, F)), ("down", H, F, (0, 0))]
    mats = []
    try:
        for i, (name, M, K, rng_m) in enumerate(shapes):
            seed = 800 + 10 * j + i
            W = workloads.make_weight(M, K, s, seed=seed)
            s_w = workloads.make_chain_weight_scales(M, K, seed=seed)
            mats.append(dict(W=W, s_w=s_w, sw=b.SparseWeight(W, s_w, max_N=N), M=M, K=K, rng=rng_m,
                             Y=torch.zeros((N, M), dtype=torch.float16, device="cuda"),
                             amax=b.new_amax()))
        x0 = workloads.make_x_f16(H, N, seed=800 + 10 * j)
        X0 = torch.from_numpy(x0).cuda()
        a0 = b.new_amax()
        for rnd in range(2):
            b.absmax_f16(X0, out=a0)
            src, src_amax = X0, a0
            for m in mats:
                m["sw"].spmm_requant(src, N, src_amax, out=m["Y"], y_amax=m["amax"], amax_range=m["rng"])
                src, src_amax = m["Y"][:, m["rng"][0]:m["rng"][1]], m["amax"]
            torch.cuda.synchronize()
            prev = x0
            for m in mats:
                m["sw"].check()
                got = m["Y"].cpu().numpy()
                q, st = oracle.requant_int4(prev)
                ref = oracle.spmm_dense(m["W"], q)
                assert np.isfinite(got).all() and np.abs(got).max() > 0
                ok = oracle.fp16_within_tolerance(got, ref, m["s_w"], st, rel=2e-3)
                assert ok.all(), f"pass {rnd}: {int((~ok).sum())} outputs outside tolerance"
                m0, m1 = m["rng"]
                assert np.array_equal(b.amax_values(m["amax"], N), _amax_words(oracle.absmax_f16(got, m0, m1)))
                prev = got[:, m0:m1]
    finally:
        for m in mats:
            m["sw"].close()


def run_half_sm_plan(M, K, fmt, warps):
    from paper_2608_09291_b200 import binding as b
    W = workloads.make_weight(M, K, 0.5, seed=M + K)
    s_w = workloads.make_chain_weight_scales(M, K, 5)
    sw = b.SparseWeight(W, s_w, fmt=fmt, max_N=8)
    try:
        info = b.us_launch_info(sw.handle, 8)
        assert b.us_launch_kernel(sw.handle, 8) == "us_spmm_kernel"
        assert info["smem_bytes"] <= 114 * 1024 and info["block"] == 32 * warps, info
        X = workloads.make_x(K, 8, seed=1)
        ref = oracle.spmm_dense(W, X)
        for N in (1, 8):
            y = sw.spmm(torch.from_numpy(b.pack_int4(X[:N])).cuda(), N).cpu().numpy()
            sw.check()
            assert (y == ref[:N]).all(), N
        if fmt is None or fmt[3] == 1:
            _check_requant_call(b, sw, W, s_w, workloads.make_x_f16(K, 8, seed=2), 8, 0, M)
    finally:
        sw.close()


@pytest.mark.parametrize("M,K,fmt,warps", [(2048, 2048, None, 10),                    # local mode
                                           (10000, 1000, (16, 512, 2, 1), 10),        # local mode, one range of two segments, 10 tiles per CTA
                                           (24000, 1024, None, 11),                   # direct mode, 11 tiles per CTA
                                           (4001, 2500, (16, 512, 2, 2), 10)])        # two column areas, K no multiple of 32
def test_half_sm_plan_counts_the_registers_of_every_kernel(M, K, fmt, warps):
    """Plain, single-token and chained calls are different kernels under one plan: its warps are what two CTAs of each of
    them share an SM with (10 in local mode, whose kernels take 81 to 96 registers since a mask word's activations are one load;
    12 fit 80. 11500 x 1000, 12 tiles per CTA, has the whole SM so). The plan is us_spmm_kernel's: a child process keeps
    the decode-ahead kernel off these shapes."""
    code = f"import sys; sys.path[:0] = ['.', 'tests']; import test_gpu_chain; test_gpu_chain.run_half_sm_plan({M}, {K}, {fmt}, {warps})"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, US_AHEAD="0"), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-1500:] + r.stderr[-1500:]


@pytest.mark.parametrize("M,K,fmt,N", [(1024, 1024, None, 8), (2048, 4096, None, 16), (2048, 2048, None, 32),   # resident beside two launches
                                       (24000, 1024, None, 8),                                                  # half an SM, the other kernel
                                       (1600, 4001, None, 5), (4001, 2500, (16, 512, 2, 2), 3),                 # ragged rows
                                       (2048, 4096, None, 64), (1100, 4099, None, 40)])                         # the tensor-memory kernel
def test_activations_are_written_while_the_call_is_resident(b, M, K, fmt, N):
    """Chained calls on one handle, back to back: the quantiser writes the same buffer of codes and steps again for every one
    of them, while the product that reads it is already resident and the one before has just read the old ones."""
    W = workloads.make_weight(M, K, 0.5, seed=M + K)
    s_w = workloads.make_chain_weight_scales(M, K, 5)
    sw = b.SparseWeight(W, s_w, fmt=fmt, max_N=N)
    try:
        xs = [workloads.make_x_f16(K, N, seed=10 + i) * np.float16(2.0 ** (i % 5 - 2)) for i in range(6)]
        Xd = [torch.from_numpy(x).cuda() for x in xs]
        amax = [b.absmax_f16(x) for x in Xd]
        ref = []
        for x, a in zip(Xd, amax):
            torch.cuda.synchronize()
            ref.append(sw.spmm_requant(x, N, a))
        torch.cuda.synchronize()
        ys = [sw.spmm_requant(x, N, a) for _ in range(4) for x, a in zip(Xd, amax)]
        torch.cuda.synchronize()
        sw.check()
        for i, y in enumerate(ys):
            assert torch.equal(y, ref[i % 6]), i
        q, st = oracle.requant_int4(xs[0])
        assert oracle.fp16_within_tolerance(ref[0].cpu().numpy(), oracle.spmm_dense(W, q), s_w, st, rel=2e-3).all()
    finally:
        sw.close()
