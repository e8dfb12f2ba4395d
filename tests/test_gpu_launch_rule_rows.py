"""The automatic launch choice for rows of other degrees than 6 to 9: on both sides of each line the same results bit for
bit as one shot per block at a fixed shape, and never far from the fastest kernel."""
import numpy as np
import pytest

from paper_2508_07879_gb300 import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def regular(dc, dv, m, seed=1):
    """A random matrix of m rows of degree dc, columns of degree dv."""
    rng, n = np.random.default_rng(seed), m * dc // dv
    rows = rng.permutation(np.repeat(np.arange(n), dv)).reshape(m, dc)
    for _ in range(10000):                                  # swap repeats out of their rows
        bad = [i for i in range(m) if len(set(rows[i])) < dc]
        if not bad:
            break
        i = bad[0]
        j = np.nonzero(np.bincount(rows[i])[rows[i]] > 1)[0][0]
        a, b = rng.integers(m), rng.integers(dc)
        rows[i, j], rows[a, b] = rows[a, b], rows[i, j]
    assert all(len(set(r)) == dc for r in rows)
    return w.CSR(np.arange(0, m * dc + 1, dc).astype(np.int32), np.sort(rows, 1).reshape(-1).astype(np.int32), m, n)


CODES = {"rows4": (4, 2, 100), "rows12": (12, 4, 240), "rows24": (24, 4, 120)}


def case(q, code, rate, batch, seed):
    h = regular(*CODES[code])
    p = rate * min(1.0, 8.0 / CODES[code][0])
    g = q.Graph.from_csr(h)
    g.set_weights(np.random.default_rng(2).uniform(0.6, 0.8, (20, h.nnz)).astype(np.float32))
    s = torch.from_numpy(w.syndromes(h, w.iid_x_errors(h.n, p, batch, seed=seed))).cuda()
    return g, s, torch.full((h.n,), w.prior_llr(p), device="cuda")


MODES = ["fp32", "int16", "int8", "learned"]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("code", list(CODES))
def test_lines(code, mode):
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = 80 * sms + 1
    g, s, prior = case(q, code, 0.05, most, 7)
    how = dict(max_iter=9, alpha=0.75, precision="fp32" if mode == "learned" else mode, learned=mode == "learned", want_post=True)
    g.set_launch("batch", 128)
    ref = q.decode(g, s, prior, **how)
    g.set_launch("auto")
    for per_sm in (1, 2, 4, 24, 40, 64, 80):
        for batch in (per_sm * sms, per_sm * sms + 1):
            got = q.decode(g, s[:batch], prior, **how)
            assert all(torch.equal(a, b[:batch]) for a, b in zip(got, ref)), batch


@pytest.mark.parametrize("mode,lines", [("int16", (80, 240)), ("int8", (40, 90))])
def test_few_checks_lines(mode, lines):
    """192 checks of degree 7: one shot per block up to the second line, where larger codes stop at the first: the same results."""
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    h = w.hgp_code(400).hz_csr
    g = q.Graph.from_csr(h)
    s = torch.from_numpy(w.syndromes(h, w.iid_x_errors(h.n, 0.01, lines[1] * sms + 1, seed=15))).cuda()
    prior = torch.full((h.n,), w.prior_llr(0.01), device="cuda")
    how = dict(max_iter=20, alpha=0.75, precision=mode, want_post=True)
    g.set_launch("batch", 128)
    ref = q.decode(g, s, prior, **how)
    g.set_launch("auto")
    for batch in (lines[0] * sms, lines[0] * sms + 1, lines[1] * sms, lines[1] * sms + 1):
        got = q.decode(g, s[:batch], prior, **how)
        assert all(torch.equal(a, b[:batch]) for a, b in zip(got, ref)), batch


def microseconds(f):
    f()
    f()
    took = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        took.append(a.elapsed_time(b) * 1e3)
    return min(took)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("code", ["rows12", "rows24"])
@pytest.mark.parametrize("per_sm", [7, 16])
def test_no_far_slower_kernel(code, mode, per_sm):
    """1000 and 2400 noisy shots: within half as much again of the faster throughput kernel (a wrong choice here cost two to
    five times; block sizes alone differ by a fifth)."""
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g, s, prior = case(q, code, 0.05, per_sm * sms, 3)
    how = dict(max_iter=40, alpha=0.75, precision="fp32" if mode == "learned" else mode, learned=mode == "learned")
    took = {}
    for kernel in ("auto", "batch") + (() if mode == "learned" else ("packed",)):
        g.set_launch(kernel)
        took[kernel] = microseconds(lambda: q.decode(g, s, prior, **how))
    assert took["auto"] <= 1.5 * min(took.values()), took


@pytest.mark.parametrize("mode", ["fp32", "int16", "int8"])
@pytest.mark.parametrize("code", ["lp1054", "hgp400"])
def test_layered_lines(code, mode):
    """Register-resident up to the line, shared-memory past it: the same results."""
    from paper_2508_07879_gb300 import qldpc as q
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    h = (w.lp_code(1054) if code == "lp1054" else w.hgp_code(400)).hz_csr
    h = w.csr_rows(h, w.layer_order(h)) if code == "hgp400" else h
    g = q.Graph.from_csr(h)
    lines = (16, 24, 40) if code == "lp1054" else (80, 100)
    s = torch.from_numpy(w.syndromes(h, w.iid_x_errors(h.n, 0.05, (lines[-1] + 1) * sms, seed=13))).cuda()
    prior = torch.full((h.n,), w.prior_llr(0.05), device="cuda")
    how = dict(max_iter=30, alpha=0.75, precision=mode, layered=True, want_post=True)
    for per_sm in lines:
        n, more = per_sm * sms, per_sm * sms + sms
        past = q.decode(g, s[:more], prior, **how)
        assert all(torch.equal(a, b[:n]) for a, b in zip(q.decode(g, s[:n], prior, **how), past))
