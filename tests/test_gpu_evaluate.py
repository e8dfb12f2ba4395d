"""Error sampler and logical test at the edges of their tiles: row lengths around words, 16-byte chunks and
segments, batches around a tile, rates 0 and 1, buffers at any byte offset (all exact)."""
import ctypes

import numpy as np
import pytest

from paper_2508_07879_gb300 import gf2
from paper_2508_07879_gb300 import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    from paper_2508_07879_gb300 import qldpc
    return qldpc


def ring(m, n):
    """m checks on n variables, check i on variables i, i+1 and i+5 (mod n)."""
    cols = [sorted({i % n, (i + 1) % n, (i + 5) % n}) for i in range(m)]
    rp = np.cumsum([0] + [len(c) for c in cols]).astype(np.int32)
    return w.CSR(rp, np.concatenate(cols).astype(np.int32), m, n)


@pytest.mark.parametrize("offset", [0, 1, 6])
@pytest.mark.parametrize("m,n,batch", [(2, 3, 1), (5, 17, 31), (33, 32, 32), (31, 95, 33), (40, 1023, 65),
                                       (1025, 1028, 40), (1030, 2049, 7), (4, 144, 4900),
                                       (5, 17, 2431), (33, 32, 2432), (31, 95, 2433), (40, 1023, 2465), (1300, 2049, 2440)])
def test_sampler_rows(q, m, n, batch, offset):
    h = ring(m, n)
    g = q.Graph.from_csr(h)
    pad = 64
    err = torch.full((batch * n + 2 * pad,), 7, dtype=torch.uint8, device="cuda")
    syn = torch.full((batch * m + 2 * pad,), 7, dtype=torch.uint8, device="cuda")
    for lo, hi in ((0.02, 0.3), (0.05, 0.05), (0.0, 0.0), (1.0, 1.0), (0.0, 1.0)):
        err.fill_(7)
        syn.fill_(7)
        q.check(q.qldpc_sample_errors(g.handle, ctypes.c_uint64(77), 12345, batch, lo, hi,
                                      ctypes.c_void_p(err.data_ptr() + pad + offset),
                                      ctypes.c_void_p(syn.data_ptr() + pad + offset), q._stream_handle(None)))
        ref, _ = w.iid_x_errors_prange(n, lo, hi, batch, seed=77, first_shot=12345)
        for got, want in ((err, ref), (syn, w.syndromes(h, ref))):
            got = got.cpu().numpy()
            at = pad + offset
            np.testing.assert_array_equal(got[at:at + want.size].reshape(want.shape), want)
            assert (got[:at] == 7).all() and (got[at + want.size:] == 7).all()


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("offset", [0, 3])
@pytest.mark.parametrize("k,n,batch", [(1, 1, 1), (1, 31, 63), (33, 32, 64), (5, 33, 65), (16, 400, 700), (140, 512, 130),
                                       (32, 513, 33), (140, 1054, 333), (3, 2048, 31), (2, 2049, 17), (47, 8192, 40),
                                       (46, 8193, 9), (512, 64, 70), (513, 64, 70), (3000, 90, 129)])
def test_logical_tiles(q, k, n, batch, offset, dense):
    rng = np.random.default_rng(k * 10007 + n)
    L = (rng.random((k, n)) < min(0.5, 3.0 / n)).astype(np.uint8)
    e = (rng.random((batch, n)) < 0.3).astype(np.uint8)
    # residuals that often commute: a bit here and there (none in every third shot), or many bits, in
    # every second shot only on qubits that no operator touches
    r = (rng.random((batch, n)) < min(0.5, 0.3 / n)).astype(np.uint8)
    r[::3] = 0
    if dense:
        L[:, n // 2:] = 0                                   # half of the qubits touch no operator
        r = (rng.random((batch, n)) < 0.5).astype(np.uint8)
        r[::2, :n // 2] = 0
    d = e ^ r
    ok = (rng.random(batch) < 0.8).astype(np.uint8)
    junk = lambda a: a | (rng.integers(0, 128, a.shape, dtype=np.uint8) << 1)   # only bit 0 of an error counts

    def at(a):   # the array at a byte offset of a device buffer
        t = torch.zeros(a.size + 32, dtype=torch.uint8, device="cuda")
        t[offset:offset + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
        return t, ctypes.c_void_p(t.data_ptr() + offset)

    bufs = [at(L * 5), at(junk(e)), at(junk(d)), at(ok * 3)]            # any byte but 0 counts in L and ok
    fail = torch.full((batch + 2,), 9, dtype=torch.uint8, device="cuda")
    q.check(q.qldpc_logical_failures(bufs[0][1], k, n, bufs[1][1], bufs[2][1], bufs[3][1], batch,
                                     ctypes.c_void_p(fail.data_ptr() + 1), q._stream_handle(None)))
    want = (ok == 0) | gf2.logical_failures(r, L)
    got = fail.cpu().numpy()
    np.testing.assert_array_equal(got[1:-1], want.astype(np.uint8))
    assert got[0] == 9 and got[-1] == 9
