"""The encoder on the GPU against the encoder on the host (which the CPU tests pin to the oracle): same statistics, same
row order, same matrix back, for ragged shapes, every kernel format and flag, chunk edges of the upload; errors; threads."""
import threading

import numpy as np
import pytest

import oracle
from paper_2608_09291_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def b():
    from paper_2608_09291_b200 import binding
    torch.cuda.set_device(0)
    return binding


@pytest.mark.parametrize("M,K,s,fmt,flags", [
    (1, 1, 0.0, (16, 128, 2, 1), 0), (17, 129, 0.5, (16, 128, 2, 1), 2), (333, 1001, 0.3, (16, 256, 2, 1), 6),
    (1024, 1024, 0.5, None, 0), (700, 3000, 0.95, (16, 384, 2, 1), 4), (48, 512, 1.0, (16, 512, 2, 1), 0),
    (5, 200001, 0.5, (16, 1024, 2, 1), 2),                  # rows longer than an upload chunk
    (3000, 1100, 0.5, (16, 1024, 2, 1), 2),
    (500, 777, 0.5, (16, 256, 2, 2), 2), (100, 5000, 0.7, (16, 2048, 2, 2), 0), (500, 777, 0.5, (16, 512, 2, 2), 10),
])
def test_same_as_host_encoder(b, M, K, s, fmt, flags):
    W = (workloads.make_weight_w2 if flags & 8 else workloads.make_weight)(M, K, s, seed=M + K)
    dev = b.us_encode(W, fmt=fmt, max_N=8, flags=flags)
    st = b.us_get_stats(dev)
    host = b.us_encode(W, fmt=st["fmt"], max_N=8, flags=flags | b.US_ENCODE_HOST_ONLY)
    try:
        assert st == b.us_get_stats(host)
        assert (b.us_get_row_order(dev) == b.us_get_row_order(host)).all()
        assert (b.us_decode(dev) == W).all()
        assert b.us_spmm_bytes(dev, 8, False) == b.us_spmm_bytes(host, 8, False)
    finally:
        b.us_destroy(dev)
        b.us_destroy(host)


@pytest.mark.parametrize("bad,at,flags", [(9, (3, 5), 0), (-9, (999, 1000), 0), (8, (0, 0), 2), (-3, (7, 1000), 8), (2, (500, 64), 8)])
def test_value_range(b, bad, at, flags):
    W = np.zeros((1000, 1001), np.int8)
    W[at] = bad
    with pytest.raises(b.UsError) as e:
        b.us_encode(W, fmt=(16, 256, 2, 2) if flags & 8 else None, flags=flags)
    assert e.value.status == 2


def test_concurrent_loads_and_products(b):
    """Handles made, used and destroyed by several threads at once, each on its own stream."""
    W = [workloads.make_weight(600 + 40 * i, 2000, 0.5, seed=i) for i in range(4)]
    X = workloads.make_x(2000, 8, seed=1)
    ref = [oracle.spmm_dense(w, X) for w in W]
    wrong = []

    def work(i):
        torch.cuda.set_device(0)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            Xd = torch.from_numpy(b.pack_int4(X)).cuda()
            for _ in range(6):
                sw = b.SparseWeight(W[i], max_N=8)
                y = sw.spmm(Xd, 8)
                sw.close()                       # the product may still be running
                stream.synchronize()
                if not (y.cpu().numpy() == ref[i]).all():
                    wrong.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_concurrent_decodes_of_one_handle(b):
    """Reading a handle is no call on it that must not overlap: several threads decode the same one."""
    W = workloads.make_weight(3000, 2000, 0.5, seed=9)
    h = b.us_encode(W, max_N=8)
    wrong = []

    def work():
        if not (b.us_decode(h) == W).all():
            wrong.append(1)

    try:
        threads = [threading.Thread(target=work) for _ in range(8)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not wrong
    finally:
        b.us_destroy(h)


def test_first_call_of_a_thread(b):
    """A thread whose first use of CUDA is a launch: it has no context yet."""
    W = workloads.make_weight(512, 1024, 0.5, seed=4)
    X = workloads.make_x(1024, 24, seed=4)
    h = b.us_encode(W, max_N=24)
    try:
        Xd = torch.from_numpy(b.pack_int4(X)).cuda()
        Y = torch.zeros((24, 512), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        failed = []

        def work():
            try:
                b.us_spmm(h, Xd.data_ptr(), 24, None, Y.data_ptr(), None)
            except Exception as e:
                failed.append(e)

        t = threading.Thread(target=work)
        t.start()
        t.join()
        assert not failed, failed
        assert b.us_last_error(h) == 0
        assert (Y.cpu().numpy() == oracle.spmm_dense(W, X)).all()
    finally:
        b.us_destroy(h)
