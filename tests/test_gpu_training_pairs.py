"""Training kernels with two shots per block, and one, at odd and even batches on both sides of the rule that chooses
(3 shots per SM), for every form of row: forward LLRs bit-exact, losses and gradients within the bounds of the
one-shot tests, which hold for any batch."""
import numpy as np
import pytest

import oracle
from paper_2508_07879_gb300 import workloads as w
from test_gpu_learned import grad_tolerance, irregular_code, train_case

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def short_rows(seed=5):
    """Rows of degree 2..8 (the row-degree bucket 8), columns of degree up to 12."""
    rng = np.random.default_rng(seed)
    h, deg = np.zeros((48, 90), np.uint8), np.zeros(90, int)
    for i in range(48):
        cols = rng.choice(np.nonzero(deg < 12)[0], rng.integers(2, 9), replace=False)
        h[i, cols] = 1
        deg[cols] += 1
    return w.csr_from_dense(h)


CODES = {"rows6": lambda: w.bb_code(12, 6).hz_csr, "rows7": lambda: w.hgp_code(400).hz_csr,
         "rows8": lambda: w.lp_code(1054, L=7).hz_csr, "short": short_rows, "long": irregular_code}


@pytest.mark.parametrize("loss", ["error", "syndrome"])
@pytest.mark.parametrize("batch", [1, 455, 456, 457, 458, 911])
@pytest.mark.parametrize("code", list(CODES))
def test_batches(code, batch, loss):
    from paper_2508_07879_gb300 import qldpc as q
    h, T = CODES[code](), 4
    g, ws, (e, s, prior, weights, gl), (sd, ed, pd, wd, gd) = train_case(q, h, batch, T, 61 + batch)
    got, post = q.nms_forward(g, sd, ed, pd, wd, ws, want_post=True, loss=loss)
    grad = q.nms_backward(g, sd, ed, pd, T, gd, ws, loss=loss).cpu().numpy()
    ref = oracle.nms_train(h.row_ptr, h.col_idx, h.m, h.n, s, e, prior, weights, grad_loss=gl.astype(np.float64),
                           precision="f32", loss=loss, post=True, threads=16)
    np.testing.assert_array_equal(post.cpu().numpy().view(np.uint32), ref["post"][:, T - 1].view(np.uint32))
    np.testing.assert_allclose(got.cpu().numpy(), ref["loss"], rtol=2e-5 if loss == "error" else 1e-4, atol=1e-6)
    assert (np.abs(grad - ref["grad"]) <= grad_tolerance(ref["grad"])).all()
