"""decode_host / decode_pair_host with every kind of buffer a caller may pass, and from a thread that has made no CUDA call:
the same results as from device tensors."""
import threading

import numpy as np
import pytest

from paper_2508_07879_gb300 import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def pinned(a, lead=0):
    """A page-locked copy of a, `lead` bytes into its allocation."""
    t = torch.empty(a.nbytes + lead + 3, dtype=torch.uint8, pin_memory=True).numpy()
    v = t[lead:lead + a.nbytes].view(a.dtype).reshape(a.shape)
    v[...] = a
    return v


def read_only(a):
    b = a.copy()
    b.flags.writeable = False
    return b


INPUTS = {"pageable": lambda a: a.copy(), "read_only": read_only, "pinned": pinned, "pinned_slice": lambda a: pinned(a, 4),
          "strided": lambda a: np.repeat(a, 2, axis=-1)[..., ::2]}


@pytest.mark.parametrize("thread", [False, True])
@pytest.mark.parametrize("outputs", ["none", "pageable", "pinned", "mixed"])
@pytest.mark.parametrize("inputs", list(INPUTS))
@pytest.mark.parametrize("batch", [0, 1, 300])
def test_buffers(batch, inputs, outputs, thread):
    from paper_2508_07879_gb300 import qldpc as q
    code = w.bb_code(12, 6)
    ex, ez = w.depolarizing_errors(code.n, 0.05, max(batch, 1), seed=3)
    hs = (code.hz_csr, code.hx_csr)
    s = [w.syndromes(h, e)[:batch] for h, e in zip(hs, (ex, ez))]
    gs = [q.Graph.from_csr(h) for h in hs]
    prior = np.full(code.n, w.prior_llr(0.03), dtype=np.float32)
    ref = [q.decode(g, torch.from_numpy(x).cuda(), torch.from_numpy(prior).cuda(), 20)[:3] for g, x in zip(gs, s)]
    ref = [[t.cpu().numpy() for t in r] for r in ref]

    def out():
        kinds = {"pageable": [0, 0, 0], "pinned": [1, 1, 1], "mixed": [1, 0, 1]}[outputs]
        blank = (np.zeros((batch, code.n), np.uint8), np.zeros(batch, np.int32), np.zeros(batch, np.uint8))
        return tuple(pinned(a) if k else a for a, k in zip(blank, kinds))

    make, got = INPUTS[inputs], {}

    def work():
        try:
            got["one"] = q.decode_host(gs[0], make(s[0]), make(prior), 20, out=None if outputs == "none" else out())
            got["two"] = q.decode_pair_host(*gs, make(s[0]), make(s[1]), make(prior), make(prior), 20,
                                            out=None if outputs == "none" else (out(), out()))
        except Exception as e:      # (raised in the test's own thread below)
            got["error"] = e

    if thread:
        t = threading.Thread(target=work)
        t.start()
        t.join()
    else:
        work()
    if "error" in got:
        raise got["error"]
    for res, want in ((got["one"], ref[0]), (got["two"][0], ref[0]), (got["two"][1], ref[1])):
        for a, b in zip(res, want):
            np.testing.assert_array_equal(a, b)
