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
