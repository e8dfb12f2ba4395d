"""Workloads whose time matters to a user of the decoder, each through the public entry points.

A case is a dict of plain values.  ``kind`` names the call:

  decode    ``qldpc.decode`` on device tensors: flooding, layered or learned schedule
  pair      ``qldpc.decode_pair``: the X and Z halves of a CSS syndrome round in one launch
  host      ``qldpc.decode_host``: the whole call from page-locked host buffers
  pair_host ``qldpc.decode_pair_host``: the same for both halves
  soft      ``qldpc.decode_soft`` on the data-syndrome graph [H | I]
  train     ``NeuralMinSum.train_step``: forward, backward and Adam of the learned decoder
  evaluate  ``qldpc.sample_errors`` and ``qldpc.logical_failures``: the two ends of the loop that
            measures a logical error rate, around a decode

The codes are the four of ``workloads.CONFIG_CODES``.  Noise rates, iteration limits and batch sizes
span the decoder's configurations: single shots (a control loop's syndrome round), tens to thousands
of shots (simulation in steps, several patches at once), 65536 (Monte Carlo).

The persistent server is left out: its worker kernel stays resident after a call, so a device-wide
wait after a pass would time the workers' idle timeout.  It runs the single-shot decoders that the
``host`` cases time.
"""
import functools
import math

import numpy as np
import torch

from paper_2508_07879_gb300 import learned, qldpc, workloads

ALPHA = 0.75
READ_ERROR = 0.01        # rate at which a syndrome bit is misread (kind "soft")
LARGEST_OPS = 4.4e10     # operations of the largest listed case: no drawn case has more
LEARNED_ITERS = 20
_OPS = 10                # per edge and iteration: |q|, sign, parity, two minima (3), select, scale, two sums


# ------------------------------------------------------------------------------------------------
# Codes
# ------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _code(name):
    return workloads.CONFIG_CODES[name]()


@functools.lru_cache(maxsize=None)
def _matrix(name, side="z", form="plain"):
    """H_Z (decodes X errors) or H_X of a code; form "layers": its rows in an order with few layers
    (what a user of the layered schedule passes; LP-1054's natural order already has few), "soft":
    the data-syndrome graph [H | I]."""
    h = _code(name).hz_csr if side == "z" else _code(name).hx_csr
    if form == "layers" and name != "lp1054":
        h = workloads.csr_rows(h, workloads.layer_order(h))
    return workloads.data_syndrome_csr(h) if form == "soft" else h


@functools.lru_cache(maxsize=None)
def _logicals(name):
    return learned.z_logicals(_code(name))


def _columns(h, device):
    """Columns of every row, [m, degree] (every row of these codes has the same degree)."""
    return torch.as_tensor(np.asarray(h.col_idx).reshape(h.m, -1), device=device).long()


def _form(case):
    return "layers" if case.get("schedule") == "layered" else "plain"


def _seeded(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _flips(batch, n, rate, gen):
    """Independent flips at ``rate`` (a number, or one rate per shot), uint8 [batch, n]."""
    return (torch.rand(batch, n, device="cuda", generator=gen) < rate).to(torch.uint8)


def _syndromes(h, errors):
    cols = _columns(h, errors.device)
    out = torch.empty(errors.shape[0], h.m, dtype=torch.uint8, device=errors.device)
    for b in range(0, errors.shape[0], 16384):
        out[b:b + 16384] = errors[b:b + 16384][:, cols].sum(dim=2, dtype=torch.uint8) & 1
    return out


def _llr(p, n):
    return torch.full((n,), workloads.prior_llr(p), dtype=torch.float32, device="cuda")


def _inputs(case, seed):
    """Syndromes and priors of a case from the seed alone (device tensors)."""
    gen, name, p, batch = _seeded(seed), case["code"], case["p"], case["batch"]
    if case["kind"] in ("pair", "pair_host"):   # depolarizing noise: X, Y and Z at p/3 each
        hz, hx = _matrix(name), _matrix(name, "x")
        u = torch.rand(batch, hz.n, device="cuda", generator=gen)
        ex = (u < 2 * p / 3).to(torch.uint8)
        ez = ((u >= p / 3) & (u < p)).to(torch.uint8)
        prior = _llr(2 * p / 3, hz.n)
        return {"s": (_syndromes(hz, ex), _syndromes(hx, ez)), "prior": prior}
    h = _matrix(name, "z", _form(case))
    if case["kind"] == "train":                 # one rate per shot over the range of the training
        rate = 0.02 + 0.04 * torch.rand(batch, 1, device="cuda", generator=gen)
        e = _flips(batch, h.n, rate, gen)
        w = 0.7 + 0.05 * torch.randn(case["iters"], h.nnz, device="cuda", generator=gen)
        m = 1e-6 * torch.randn(case["iters"], h.nnz, device="cuda", generator=gen)
        return {"s": _syndromes(h, e), "e": e, "w": w, "m": m, "prior": _llr(0.04, h.n)}
    e = _flips(batch, h.n, p, gen)
    s = _syndromes(h, e)
    got = {"s": s, "e": e, "prior": _llr(p, h.n)}
    if case["kind"] == "soft":
        got["s"] = s ^ _flips(batch, h.m, READ_ERROR, gen)
        got["read_llr"] = _llr(READ_ERROR, h.m)
    if case.get("schedule") == "learned":       # as trained: a damped first iteration, 0.7 after it
        w = 0.7 + 0.04 * torch.randn(LEARNED_ITERS, h.nnz, device="cuda", generator=gen)
        w[0] -= 0.28
        got["w"] = w
    return got


# ------------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # one syndrome round of a control loop, transfers included: the latency the paper quotes
        {"name": "host_single_lp1054", "kind": "host", "code": "lp1054", "batch": 1, "precision": "fp32",
         "p": 0.03, "max_iter": 50, "early_stop": True},
        # the paper's timed mode: both halves of one round, a fixed number of iterations
        {"name": "pair_host_single_bb144", "kind": "pair_host", "code": "bb144", "batch": 1,
         "precision": "fp32", "p": 0.05, "max_iter": 10, "early_stop": False},
        # a handful of patches decoded together on device buffers
        {"name": "decode_lp1054_64", "kind": "decode", "schedule": "flooding", "code": "lp1054", "batch": 64,
         "precision": "fp32", "p": 0.03, "max_iter": 50, "early_stop": True, "post": False},
        # the hypergraph-product configuration, with the a-posteriori LLRs a second stage reads
        {"name": "decode_hgp400_1000", "kind": "decode", "schedule": "flooding", "code": "hgp400",
         "batch": 1000, "precision": "fp32", "p": 0.05, "max_iter": 32, "early_stop": True, "post": True},
        # a simulation step in the fixed point of the paper's integer proposal
        {"name": "decode_lp1054_4096_int16", "kind": "decode", "schedule": "flooding", "code": "lp1054",
         "batch": 4096, "precision": "int16", "p": 0.03, "max_iter": 50, "early_stop": True, "post": False},
        # Monte Carlo at the noisiest rate of the benchmark: the largest batch
        {"name": "decode_lp1054_65536", "kind": "decode", "schedule": "flooding", "code": "lp1054",
         "batch": 65536, "precision": "fp32", "p": 0.05, "max_iter": 50, "early_stop": True, "post": False},
        # both halves of many bivariate-bicycle rounds, an odd number of them, 8-bit messages
        {"name": "pair_bb288_10001_int8", "kind": "pair", "code": "bb288", "batch": 10001, "precision": "int8",
         "p": 0.05, "max_iter": 64, "early_stop": True},
        # the row-serial schedule, which needs half the iterations
        {"name": "layered_lp1054_16384", "kind": "decode", "schedule": "layered", "code": "lp1054",
         "batch": 16384, "precision": "fp32", "p": 0.03, "max_iter": 50, "early_stop": True, "post": False},
        # misread syndrome bits: the longer rows of [H | I] and many more iterations
        {"name": "soft_lp1054_8191", "kind": "soft", "code": "lp1054", "batch": 8191, "precision": "fp32",
         "p": 0.01, "max_iter": 50, "early_stop": True, "post": True},
        # trained weights first, plain min-sum for what they leave
        {"name": "learned_lp1054_16384", "kind": "decode", "schedule": "learned", "code": "lp1054",
         "batch": 16384, "precision": "fp32", "p": 0.03, "max_iter": 50, "early_stop": True, "post": False},
        # one training step of the configured run
        {"name": "train_lp1054_4096", "kind": "train", "code": "lp1054", "batch": 4096, "iters": 20,
         "loss": "syndrome", "p": 0.04},
        # fresh shots for a logical error rate, and the logical test of decoded ones
        {"name": "evaluate_lp1054_65536", "kind": "evaluate", "code": "lp1054", "batch": 65536, "p": 0.03},
    ]


_PRECISIONS = ("fp32", "fp32", "int16", "int8")


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("decode", "decode", "decode", "pair", "host", "pair_host", "soft", "train", "evaluate"))
    code = rng.choice(("lp1054", "lp1054", "hgp400", "bb144", "bb288"))
    case = {"kind": kind, "code": code, "batch": 1, "p": round(rng.uniform(0.01, 0.05), 4)}
    if kind == "train":
        case.update(p=0.04, iters=rng.randint(4, 20), loss=rng.choice(("syndrome", "error")))
        case["batch"] = size(64, 4096)
        return case
    if kind == "evaluate":
        case["batch"] = size(1000, 65536)
        return case
    case["precision"] = rng.choice(_PRECISIONS)
    case["early_stop"] = rng.random() < 0.8
    case["max_iter"] = rng.randint(20, 64) if case["early_stop"] else rng.randint(5, 20)
    if kind == "decode":
        case["schedule"] = rng.choice(("flooding", "flooding", "flooding", "layered", "learned"))
        if case["schedule"] == "learned":
            case.update(precision="fp32", early_stop=True)
    if kind in ("decode", "soft"):
        case["post"] = rng.random() < 0.3
    lo, hi = {"host": (1, 32), "pair_host": (1, 32), "pair": (1, 20000), "soft": (1, 16384)}.get(kind, (1, 65536))
    hi = min(hi, int(LARGEST_OPS / (work(case)["flops"] + 1)))
    case["batch"] = size(lo, hi)
    return case


def _iterations(case):
    """Iterations a shot runs on average (measured over the declared rates, rounded)."""
    if not case.get("early_stop", True):
        return case["max_iter"]
    p, code = case["p"], case["code"]
    if case["kind"] == "soft":
        k = 20 + 700 * (p - 0.01)
    elif code == "lp1054":
        k = 1 + 9500 * max(p, 0.01) ** 2.15
    elif code == "hgp400":
        k = 1 + 700 * (p - 0.008)
    else:
        k = 0.5 + 3800 * p ** 2
    return max(1.0, min(float(case["max_iter"]), k * (0.55 if case.get("schedule") == "layered" else 1.0)))


def work(case):
    kind, batch = case["kind"], case["batch"]
    h = _matrix(case["code"], "z", "soft" if kind == "soft" else "plain")
    if kind == "train":
        T = case["iters"]
        moved = batch * (h.m + (h.n if case["loss"] == "error" else 0) + 4) + 4 * T * h.nnz * 8 + 4 * h.n
        return {"bytes": moved, "flops": 30.0 * h.nnz * T * batch}
    if kind == "evaluate":
        k = _logicals(case["code"]).shape[0]
        moved = batch * (h.n + h.m) + batch * (2 * h.n + 2) + k * h.n
        return {"bytes": moved, "flops": float(batch) * (20 * h.n + h.nnz + 2 * k * math.ceil(h.n / 32))}
    sides = 2 if kind in ("pair", "pair_host") else 1
    moved = batch * (h.m + h.n + 5 + (4 * h.n if case.get("post") else 0)) + 4 * h.n
    return {"bytes": sides * moved, "flops": float(sides) * batch * _OPS * h.nnz * _iterations(case)}


# ------------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------------
def _pinned(t):
    return t.cpu().pin_memory().numpy()


def _pinned_out(batch, n):
    return tuple(torch.empty(shape, dtype=dt, pin_memory=True).numpy()
                 for shape, dt in (((batch, n), torch.uint8), ((batch,), torch.int32), ((batch,), torch.uint8)))


def prepare(case, seed):
    kind, name = case["kind"], case["code"]
    st = {"case": case, "seed": seed}
    if kind == "evaluate":
        h = _matrix(name)
        st["graph"] = qldpc.Graph.from_csr(h)
        st["logicals"] = torch.as_tensor(_logicals(name), device="cuda")
        got = _inputs(case, seed)
        st["errors"] = got["e"]
        st["decisions"], _, st["ok"], _ = qldpc.decode(st["graph"], got["s"], got["prior"], 30, ALPHA)
        return st
    got = _inputs(case, seed)
    st.update(got)
    if kind in ("pair", "pair_host"):
        st["graphs"] = qldpc.Graph.from_csr(_matrix(name)), qldpc.Graph.from_csr(_matrix(name, "x"))
        if kind == "pair_host":
            n = _matrix(name).n
            st["s"] = tuple(_pinned(s) for s in got["s"])
            st["prior"] = _pinned(got["prior"])
            st["out"] = _pinned_out(case["batch"], n), _pinned_out(case["batch"], n)
        return st
    if kind == "train":
        h = _matrix(name)
        model = learned.NeuralMinSum(h, got["prior"].cpu().numpy(), T=case["iters"], max_batch=case["batch"],
                                     loss=case["loss"])
        with torch.no_grad():                   # in the middle of a run: weights and moments as they come
            model.weights.copy_(got["w"])
            model.exp_avg.copy_(got["m"])
            model.exp_avg_sq.fill_(1e-11)
        model.step = 50
        st["model"] = model
        return st
    h = _matrix(name, "z", "soft" if kind == "soft" else _form(case))
    st["graph"] = qldpc.Graph.from_csr(h)
    if "w" in got:
        st["graph"].set_weights(got["w"])
    if kind == "host":
        st["graph"].reserve(case["batch"])
        st["s"], st["prior"] = _pinned(got["s"]), _pinned(got["prior"])
        st["out"] = _pinned_out(case["batch"], h.n)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "evaluate":
        fresh = qldpc.sample_errors(state["graph"], state["seed"], 0, case["batch"], case["p"])
        failed = qldpc.logical_failures(state["logicals"], state["errors"], state["decisions"], state["ok"])
        return {"errors": fresh[0], "syndromes": fresh[1], "failed": failed}
    if kind == "train":
        model = state["model"]
        loss = model.train_step(state["s"], state["e"])
        return {"loss": loss, "grad": model.weights.grad, "weights": model.weights, "exp_avg": model.exp_avg,
                "exp_avg_sq": model.exp_avg_sq}
    how = dict(alpha=ALPHA, precision=case["precision"], early_stop=case["early_stop"])
    if kind == "host":
        return qldpc.decode_host(state["graph"], state["s"], state["prior"], case["max_iter"], out=state["out"], **how)
    if kind == "pair_host":
        return qldpc.decode_pair_host(*state["graphs"], *state["s"], state["prior"], state["prior"],
                                      case["max_iter"], out=state["out"], **how)
    if kind == "pair":
        return qldpc.decode_pair(*state["graphs"], *state["s"], state["prior"], state["prior"], case["max_iter"], **how)
    if kind == "soft":
        return qldpc.decode_soft(state["graph"], state["s"], state["prior"], state["read_llr"], case["max_iter"],
                                 want_post=case["post"], **how)
    return qldpc.decode(state["graph"], state["s"], state["prior"], case["max_iter"], want_post=case["post"],
                        learned=case["schedule"] == "learned", layered=case["schedule"] == "layered", **how)


# ------------------------------------------------------------------------------------------------
# The same in 64 bits, plain torch
# ------------------------------------------------------------------------------------------------
class _Flooding:
    """Algorithm 1 in float64 on all edges of a batch: r and q are [batch, m, degree]."""

    def __init__(self, h, syndromes):
        self.cols = _columns(h, "cuda")
        self.m, self.d = self.cols.shape
        flat = self.cols.reshape(-1)
        order = torch.argsort(flat, stable=True)
        count = torch.bincount(flat, minlength=h.n)
        place = torch.arange(flat.numel(), device="cuda") - (torch.cumsum(count, 0) - count)[flat[order]]
        self.edges = torch.full((h.n, int(count.max())), flat.numel(), device="cuda")
        self.edges[flat[order], place] = order          # edges of each variable, padded with one past the last
        self.flip = 1.0 - 2.0 * syndromes.double().unsqueeze(2)
        self.s = syndromes.bool()

    def check(self, q, scale):
        mag = q.abs()
        i1 = mag.detach().argmin(2, keepdim=True)
        i2 = mag.detach().scatter(2, i1, math.inf).argmin(2, keepdim=True)
        m1, m2 = mag.gather(2, i1), mag.gather(2, i2)
        here = torch.arange(self.d, device="cuda") == i1
        sign = torch.where(q < 0, -1.0, 1.0).double()
        return scale * torch.where(here, m2, m1) * (sign * (sign.prod(2, keepdim=True) * self.flip))

    def total(self, prior, r):
        flat = torch.cat([r.reshape(r.shape[0], -1), r.new_zeros(r.shape[0], 1)], 1)
        return prior + flat[:, self.edges].sum(2)

    def met(self, Q):
        odd = (Q < 0)[:, self.cols].sum(2) % 2 == 1
        return (odd == self.s).all(1)

    def decode(self, prior, max_iter, early, alpha, learned_w=None):
        """A-posteriori LLRs of the iteration each shot stops at."""
        batch = self.s.shape[0]
        start = prior.expand(batch, -1)
        phases = [(alpha, max_iter)]
        if learned_w is not None:
            phases.insert(0, (None, learned_w.shape[0]))
        post = start.clone()
        done = self.met(start) if early else torch.zeros(batch, dtype=torch.bool, device="cuda")
        for scale, limit in phases:
            q = start[:, self.cols]
            if limit:
                post[~done] = start[~done]
            for k in range(limit):
                r = self.check(q, learned_w[k].view(self.m, self.d) if scale is None else scale)
                Q = self.total(prior, r)
                post[~done] = Q[~done]
                if early:
                    done |= self.met(Q)
                    if bool(done.all()):
                        break
                q = Q[:, self.cols] - r
        return post


def _exact_train(case, seed):
    got = _inputs(case, seed)
    h = _matrix(case["code"])
    T, batch = case["iters"], case["batch"]
    w = got["w"].double().requires_grad_(True)
    prior = got["prior"].double()
    mean = 0.0
    for b in range(0, batch, 512):                      # the mean loss is a sum over shots
        s, e = got["s"][b:b + 512], got["e"][b:b + 512]
        f = _Flooding(h, s)
        q = prior.expand(s.shape[0], -1)[:, f.cols]
        loss = 0.0
        for k in range(T):
            r = f.check(q, w[k].view(f.m, f.d))
            Q = f.total(prior, r)
            if case["loss"] == "error":
                loss = loss + torch.where(e.bool(), torch.nn.functional.softplus(Q),
                                          torch.nn.functional.softplus(-Q)).sum() / h.n
            else:
                match = (1.0 + f.flip.squeeze(2) * torch.tanh(Q / 2)[:, f.cols].prod(2)) / 2
                loss = loss - torch.log(match.clamp_min(1e-7)).sum() / h.m
            q = Q[:, f.cols] - r
        part = loss / (T * batch)
        part.backward()
        mean = mean + part.detach()
    g, step, b1, b2, lr, eps = w.grad, 51, 0.9, 0.999, 1e-3, 1e-8
    m = got["m"].double() + (1 - b1) * (g - got["m"].double())
    v = b2 * torch.full_like(g, 1e-11) + (1 - b2) * g * g
    new = w.detach() - lr / (1 - b1 ** step) * m / (v.sqrt() / math.sqrt(1 - b2 ** step) + eps)
    return {"loss": mean, "grad": g, "weights": new, "exp_avg": m, "exp_avg_sq": v}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if not case.get("post") or case["precision"] != "fp32" or case.get("schedule") == "layered":
        return None       # decisions, counts and bytes, or values of another number format or schedule
    got = _inputs(case, seed)
    h = _matrix(case["code"], "z", "soft" if case["kind"] == "soft" else "plain")
    prior = got["prior"].double()
    if case["kind"] == "soft":
        prior = torch.cat([prior, got["read_llr"].double()])
    w = got["w"].double() if "w" in got else None
    parts = [_Flooding(h, got["s"][b:b + 4096]).decode(prior, case["max_iter"], case["early_stop"], ALPHA, w)
             for b in range(0, case["batch"], 4096)]
    post = torch.cat(parts)
    return (None, None, None, None, post) if case["kind"] == "soft" else (None, None, None, post)
