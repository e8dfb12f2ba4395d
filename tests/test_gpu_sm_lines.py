"""Rules that count SMs, on both sides of their lines whatever the number of SMs: training with one and two shots per block
(3 shots per SM), the sampler by shot and by tile (a tile of 32 shots for every second SM); and the sampler's last shots."""
import numpy as np
import pytest

import oracle
from paper_2508_07879_gb300 import workloads as w
from test_gpu_evaluate import ring
from test_gpu_learned import grad_tolerance, train_case
from test_gpu_training_pairs import CODES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("loss", ["error", "syndrome"])
@pytest.mark.parametrize("past", [-1, 0, 1, 2])
@pytest.mark.parametrize("code", ["rows7", "short", "long"])
def test_training_line(code, past, loss):
    from paper_2508_07879_gb300 import qldpc as q
    h, T, batch = CODES[code](), 3, 3 * sms() + past
    g, ws, (e, s, prior, weights, gl), (sd, ed, pd, wd, gd) = train_case(q, h, batch, T, 83 + past)
    _, post = q.nms_forward(g, sd, ed, pd, wd, ws, want_post=True, loss=loss)
    grad = q.nms_backward(g, sd, ed, pd, T, gd, ws, loss=loss).cpu().numpy()
    ref = oracle.nms_train(h.row_ptr, h.col_idx, h.m, h.n, s, e, prior, weights, grad_loss=gl.astype(np.float64),
                           precision="f32", loss=loss, post=True, threads=16)
    np.testing.assert_array_equal(post.cpu().numpy().view(np.uint32), ref["post"][:, T - 1].view(np.uint32))
    assert (np.abs(grad - ref["grad"]) <= grad_tolerance(ref["grad"])).all()


@pytest.mark.parametrize("last", [False, True])
@pytest.mark.parametrize("past", [-1, 0, 1, 33])
@pytest.mark.parametrize("m,n", [(5, 17), (40, 1023)])
def test_sampler_line(m, n, past, last):
    from paper_2508_07879_gb300 import qldpc as q
    h, batch = ring(m, n), 32 * (sms() // 2) + past
    first = 2 ** 63 - 1 - batch if last else 4
    err, syn = q.sample_errors(q.Graph.from_csr(h), 91, first, batch, 0.02, 0.3)
    want, _ = w.iid_x_errors_prange(n, 0.02, 0.3, batch, seed=91, first_shot=first)
    np.testing.assert_array_equal(err.cpu().numpy(), want)
    np.testing.assert_array_equal(syn.cpu().numpy(), w.syndromes(h, want))
