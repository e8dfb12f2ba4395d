"""The automatic launch choice on both sides of each of its lines (shots per SM): the same results bit for bit as the
one-shot-per-block kernel at a fixed shape, for single decodes, pairs and learned weights."""
import numpy as np
import pytest

from paper_2508_07879_gb300 import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODES = {"hgp400": lambda: w.hgp_code(400), "lp1054": lambda: w.lp_code(1054), "bb144": lambda: w.bb_code(12, 6),
         "lp2040": lambda: w.lp_code(7, L=60)}


def same(a, b):
    return all(x is y is None or torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", ["fp32", "int16", "int8"])
@pytest.mark.parametrize("code", list(CODES))
def test_lines(code, precision):
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    c = CODES[code]()
    hz, hx = c.hz_csr, c.hx_csr
    gz, gx = q.Graph.from_csr(hz), q.Graph.from_csr(hx)
    rng = np.random.default_rng(5)
    gz.set_weights(rng.uniform(0.5, 1.0, (4, hz.nnz)).astype(np.float32))
    most = 64 * sms + 1
    s = torch.from_numpy(w.syndromes(hz, w.iid_x_errors(hz.n, 0.04, most, seed=9))).cuda()
    sx = torch.from_numpy(w.syndromes(hx, w.iid_x_errors(hx.n, 0.04, most // 2 + 1, seed=10))).cuda()
    prior = torch.full((hz.n,), w.prior_llr(0.04), device="cuda")
    how = dict(max_iter=12, alpha=0.75, precision=precision, want_post=True)
    gz.set_launch("batch", 128)
    ref = q.decode(gz, s, prior, **how)
    gx.set_launch("batch", 128)
    ref_x = q.decode(gx, sx, prior, **how)
    ref_w = q.decode(gz, s, prior, learned=True, **how) if precision == "fp32" else None
    gz.set_launch("auto")
    gx.set_launch("auto")
    for per_sm in (1, 4, 12, 24, 40, 48, 64):
        for batch in (per_sm * sms, per_sm * sms + 1):
            assert same(q.decode(gz, s[:batch], prior, **how), [t[:batch] for t in ref]), batch
            if ref_w:
                assert same(q.decode(gz, s[:batch], prior, learned=True, **how), [t[:batch] for t in ref_w]), batch
        for batch in (per_sm * sms // 2, per_sm * sms // 2 + 1):
            a, b = q.decode_pair(gz, gx, s[:batch], sx[:batch], prior, prior, **how)
            assert same(a, [t[:batch] for t in ref]) and same(b, [t[:batch] for t in ref_x]), batch


@pytest.mark.parametrize("precision", ["fp32", "int16", "int8"])
@pytest.mark.parametrize("code", ["lp1054", "hgp400", "bb144"])
def test_layered_line(code, precision):
    """40 shots per SM (80 in blocks of two warps): the register-resident kernel up to there, the shared-memory kernel
    past it."""
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    h = CODES[code]().hz_csr
    h = w.csr_rows(h, w.layer_order(h)) if code != "lp1054" else h
    g = q.Graph.from_csr(h)
    assert g.layers() <= 8
    n = (40 if code == "lp1054" else 80) * sms
    s = torch.from_numpy(w.syndromes(h, w.iid_x_errors(h.n, 0.04, n + 1, seed=11))).cuda()
    prior = torch.full((h.n,), w.prior_llr(0.04), device="cuda")
    for early in (True, False):
        how = dict(max_iter=9, alpha=0.75, precision=precision, early_stop=early, want_post=True, layered=True)
        past = q.decode(g, s, prior, **how)
        assert same(q.decode(g, s[:n], prior, **how), [t[:n] for t in past])
        assert same(q.decode(g, s[:sms + 1], prior, **how), [t[:sms + 1] for t in past])


@pytest.mark.parametrize("precision", ["fp32", "int16", "int8"])
@pytest.mark.parametrize("lo,hi", [(2, 8), (9, 9), (2, 15), (17, 32)])
def test_layered_rows(lo, hi, precision):
    """Rows of one, two and four 16-byte groups of the layered edge lists, against the oracle."""
    import oracle
    from paper_2508_07879_gb300 import qldpc as q
    rng = np.random.default_rng(hi)
    d, deg = np.zeros((37, 150), np.uint8), np.zeros(150, int)
    for i in range(37):
        cols = rng.choice(np.nonzero(deg < 12)[0], rng.integers(lo, hi + 1), replace=False)
        d[i, cols] = 1
        deg[cols] += 1
    h = w.csr_from_dense(d)
    s = rng.integers(0, 2, (400, h.m)).astype(np.uint8)
    s[::4] = w.syndromes(h, w.iid_x_errors(h.n, 0.02, 100, seed=12))
    prior = rng.normal(2, 1.5, h.n).astype(np.float32)
    ref = oracle.msa(h.row_ptr, h.col_idx, h.m, h.n, s, prior, 6, 0.75, {"fp32": "f32", "int16": "i16", "int8": "i8"}[precision],
                     threads=8, schedule="layered")
    err, iters, ok, post = q.decode(q.Graph.from_csr(h), torch.from_numpy(s).cuda(), torch.from_numpy(prior).cuda(), 6,
                                    0.75, precision, want_post=True, layered=True)
    np.testing.assert_array_equal(err.cpu().numpy(), ref["err"])
    np.testing.assert_array_equal(iters.cpu().numpy(), ref["iters"])
    np.testing.assert_array_equal(ok.cpu().numpy(), ref["ok"])
    np.testing.assert_array_equal(post.cpu().numpy() * {"fp32": 1, "int16": 256, "int8": 4}[precision], ref["post"])


@pytest.mark.parametrize("precision,per_sm", [("fp32", 320), ("int16", 80), ("int8", 40)])
@pytest.mark.parametrize("code", ["hgp400", "lp1054"])
def test_pair_line(code, precision, per_sm):
    """One shot per block up to the line, two past it (an odd batch: the last block has one)."""
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    h = CODES[code]().hz_csr
    g = q.Graph.from_csr(h)
    most = per_sm * sms + 1
    s = torch.from_numpy(w.syndromes(h, w.iid_x_errors(h.n, 0.04, most, seed=11))).cuda()
    prior = torch.full((h.n,), w.prior_llr(0.04), device="cuda")
    how = dict(max_iter=8, alpha=0.75, precision=precision, want_post=True)
    g.set_launch("batch", 128)
    ref = q.decode(g, s, prior, **how)
    g.set_launch("auto")
    for batch in (most - 1, most - most % 2 - 1, most):
        assert same(q.decode(g, s[:batch], prior, **how), [t[:batch] for t in ref]), batch
