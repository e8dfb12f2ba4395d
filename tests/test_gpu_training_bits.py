"""A shot's weight gradient to the last bit.  The sum over shots has no fixed order, but a shot's own gradient is one
chain of operations: the same bits alone and in every batch, the bits of the release before two shots per block
(tests/golden/nms_grad_crc.txt), and an error against 64 bits that the exponential of a code explains.  Last bits matter here:
a minimum that changes place after the next step moves the whole gradient."""
import os
import zlib

import numpy as np
import pytest

import oracle
from helpers import GOLDEN
from paper_2508_07879_gb300 import workloads as w

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CODES = {"rows6": lambda: w.bb_code(12, 6).hz_csr, "rows7": lambda: w.hgp_code(400).hz_csr,
         "rows8": lambda: w.lp_code(1054).hz_csr}
SHOTS, T = 5, 8


def inputs(h, llr=w.prior_llr(0.04), iters=T, shots=SHOTS, seed=71):
    """Errors, syndromes, priors and weights (exact steps of 2^-10) of a few shots."""
    e = w.iid_x_errors(h.n, 0.05, shots, seed=seed)
    weights = np.random.default_rng(seed).integers(512, 1024, (iters, h.nnz)).astype(np.float32) / 1024
    return e, w.syndromes(h, e), np.full(h.n, llr, np.float32), weights


def gradients(h, e, s, prior, weights, loss, batch, shots):
    """Gradient of each of `shots` in a batch of `batch` whose other shots have no weight in the sum."""
    from paper_2508_07879_gb300 import qldpc as q
    g, iters = q.Graph.from_csr(h), weights.shape[0]
    rows = np.arange(batch) % len(s)
    ed, sd, pd, wd = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (e[rows], s[rows], prior, weights))
    ws = torch.empty(q.nms_workspace_bytes(g, batch, iters), dtype=torch.uint8, device="cuda")
    q.nms_forward(g, sd, ed, pd, wd, ws, loss=loss)
    out = []
    for b in shots:
        one = torch.zeros(batch, device="cuda")
        one[b] = 1.0
        out.append(q.nms_backward(g, sd, ed, pd, iters, one, ws, loss=loss).cpu().numpy())
    return out


def crc(a):
    return zlib.crc32(np.ascontiguousarray(a).tobytes())


@pytest.mark.parametrize("loss", ["error", "syndrome"])
@pytest.mark.parametrize("code", list(CODES))
def test_bits(code, loss):
    h = CODES[code]()
    e, s, prior, weights = inputs(h)
    alone = [gradients(h, e[b:b + 1], s[b:b + 1], prior, weights, loss, 1, [0])[0] for b in range(SHOTS)]
    with open(os.path.join(GOLDEN, "nms_grad_crc.txt")) as f:
        want = {tuple(x[:2]): [int(c, 16) for c in x[2:]] for x in map(str.split, f) if x and x[0] != "#"}
    assert [crc(a) for a in alone] == want[code, loss]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for batch in (3 * sms, 3 * sms + 1, 3 * sms + 2):    # one shot per block up to 3 per SM, then two
        shots = list(range(SHOTS)) + [batch - 2, batch - 1]
        for b, got in zip(shots, gradients(h, e, s, prior, weights, loss, batch, shots)):
            np.testing.assert_array_equal(got.view(np.uint32), alone[b % SHOTS].view(np.uint32), err_msg=f"{batch} {b}")


@pytest.mark.parametrize("code", list(CODES))
def test_small_llr_gradient_error(code):
    """Q near 0, where tanh(Q / 2) comes from x = exp(-|Q|) just below 1: x is good to some 2.5e-8 (root mean square of an
    error of at most one unit, 6e-8), which is 2.5e-8 / |Q| of 1 - x, so of each of the other d - 1 factors of a check of
    degree d; |Q| is about 1.5 priors after an iteration.  The factors' errors are independent."""
    h, llr, shots = CODES[code](), 0.01, 24
    e, s, prior, weights = inputs(h, llr, 2, shots, 5)
    off = []
    for b in range(shots):
        got = gradients(h, e[b:b + 1], s[b:b + 1], prior, weights, "syndrome", 1, [0])[0]
        ref = oracle.nms_train(h.row_ptr, h.col_idx, h.m, h.n, s[b:b + 1], e[b:b + 1], prior, weights, grad_loss=np.ones(1),
                               precision="f32", loss="syndrome")["grad"]
        off.append(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    degree = h.nnz // h.m
    assert np.mean(off) <= 2.5e-8 / (1.5 * llr) * np.sqrt(degree - 1), off
