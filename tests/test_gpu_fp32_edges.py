"""FP32 check step where its minima meet: ties, zeros, subnormal and huge magnitudes, in every kernel and row form
(bit-exact against the oracle; nothing overflows in the iterations run)."""
import numpy as np
import pytest

import oracle
from paper_2508_07879_gb300 import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def uneven(m, n, lo, hi, seed):
    rng = np.random.default_rng(seed)
    h, deg = np.zeros((m, n), np.uint8), np.zeros(n, int)
    for i in range(m):
        cols = rng.choice(np.nonzero(deg < 12)[0], rng.integers(lo, hi + 1), replace=False)
        h[i, cols] = 1
        deg[cols] += 1
    return w.csr_from_dense(h)


GRAPHS = {"rows6": lambda: w.bb_code(12, 6).hz_csr, "rows7": lambda: w.hgp_code(400).hz_csr,
          "rows8": lambda: w.lp_code(1054).hz_csr, "rows9": lambda: w.data_syndrome_csr(w.lp_code(1054).hz_csr),
          "uneven8": lambda: uneven(40, 100, 2, 8, 1), "uneven16": lambda: uneven(40, 130, 2, 15, 2),
          "uneven32": lambda: uneven(20, 90, 2, 32, 3)}
PRIORS = {"ties": lambda r, n: r.choice([-1.0, 1.0, 2.0], n), "zeros": lambda r, n: r.choice([0.0, -0.0, 1.5], n),
          "subnormal": lambda r, n: r.normal(0, 1e-40, n), "huge": lambda r, n: r.normal(0, 1e30, n)}


@pytest.mark.parametrize("prior", list(PRIORS))
@pytest.mark.parametrize("graph", list(GRAPHS))
def test_minima(graph, prior):
    from paper_2508_07879_gb300 import qldpc as q
    h = GRAPHS[graph]()
    rng = np.random.default_rng(len(graph) * 31 + len(prior))
    gamma = PRIORS[prior](rng, h.n).astype(np.float32)
    s = rng.integers(0, 2, (35, h.m)).astype(np.uint8)
    g = q.Graph.from_csr(h)
    st, pr = torch.from_numpy(s).cuda(), torch.from_numpy(gamma).cuda()
    for schedule in ("flooding", "layered"):
        ref = oracle.msa(h.row_ptr, h.col_idx, h.m, h.n, s, gamma, 4, 0.75, "f32", early_stop=False, schedule=schedule)
        for kernel in ("auto", "batch", "latency", "packed") if schedule == "flooding" else ("auto",):
            try:
                g.set_launch(kernel)
            except q.QldpcError:      # (the single-shot kernel does not hold every graph)
                assert kernel == "latency"
                continue
            err, iters, ok, post = q.decode(g, st, pr, 4, 0.75, early_stop=False, want_post=True,
                                            layered=schedule == "layered")
            np.testing.assert_array_equal(post.cpu().numpy(), ref["post"])     # (zeros compare equal whatever their sign)
            np.testing.assert_array_equal(err.cpu().numpy(), ref["err"])
            np.testing.assert_array_equal(ok.cpu().numpy(), ref["ok"])
        g.set_launch("auto")


@pytest.mark.parametrize("kernel", ["batch", "latency"])
@pytest.mark.parametrize("graph", list(GRAPHS))
def test_learned_rows(graph, kernel):
    """Learned weights reach their edges for every row form (groups of four edges, the last one not always full)."""
    from paper_2508_07879_gb300 import qldpc as q
    h = GRAPHS[graph]()
    rng = np.random.default_rng(len(graph))
    s = rng.integers(0, 2, (35, h.m)).astype(np.uint8)
    gamma = rng.uniform(0.5, 3.0, h.n).astype(np.float32)
    weights = rng.uniform(0.3, 1.0, (3, h.nnz)).astype(np.float32)
    ref = oracle.nms_decode(h.row_ptr, h.col_idx, h.m, h.n, s, gamma, weights, 3, 0.75, threads=4)
    g = q.Graph.from_csr(h)
    g.set_weights(weights)
    try:
        g.set_launch(kernel)
    except q.QldpcError:      # (the single-shot kernel does not hold every graph)
        assert kernel == "latency"
        return
    got = q.decode(g, torch.from_numpy(s).cuda(), torch.from_numpy(gamma).cuda(), 3, 0.75, learned=True,
                   want_post=True)
    for name, t in zip(("err", "iters", "ok", "post"), got):
        np.testing.assert_array_equal(t.cpu().numpy(), ref[name], err_msg=name)
