"""Workloads of the TIM / TIM+ engine whose speed is tracked.

Each case is one thing a program does with the library through its public calls
(paper_1404_0900_gb300.tim): answering an influence-maximisation query on a small or a
large graph, sampling RR sets, selecting seeds over a store, scoring a seed set by
forward cascades, answering many queries at once, training the start-round network.
Graphs are seeded synthetic ones of the families and sizes that the repository's
configurations, tests and benchmark use (R-MAT scales 12 to 20, directed Chung-Lu graphs up
to a tenth of the Twitter-size configuration), drawn on the GPU.

A case is a dict of plain values:
  op       query | load_query | sample | select | select_noalloc | spread | batch | train
  graph    rmat (scale, degree) or chung_lu (n, degree)
  weights  wc (IC, 1/indeg), triv (IC, {0.1, 0.01, 0.001}), inv (LT, 1/indeg), rand (LT,
           random normalised), trig (a general triggering model of small option sets)
and the sizes of its op (k, eps, theta, cascades, queries, mix, samples, steps).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1404_0900_gb300 import inputs, tim

ELL = 1.0
SELECT_SIDS = 3 << 56  # set ids of Algorithm 1's RR sets
SCORE_SIDS = 7 << 56   # set ids kept apart for scoring a chosen seed set
HIDDEN = 64


def listed():
    return [
        # an interactive query on a small graph that is already loaded: the smallest whole
        # call, where launches and read-backs count
        dict(name="query_small", op="query", graph="rmat", scale=14, degree=16, weights="wc",
             k=10, eps=0.5),
        # a new graph of a million nodes, loaded and answered, weighted cascade
        dict(name="step_ic_wc", op="load_query", graph="rmat", scale=20, degree=16,
             weights="wc", k=50, eps=0.1),
        # the same under the linear threshold model
        dict(name="step_lt", op="load_query", graph="rmat", scale=20, degree=16, weights="inv",
             k=50, eps=0.1),
        # the largest: a tenth of the Twitter-size graph, trivalency, whose RR sets range
        # from one node to a large part of the graph
        dict(name="step_ic_triv", op="load_query", graph="chung_lu", n=4_160_000, degree=35,
             weights="triv", k=50, eps=0.2),
        # the stepwise calls: sampling into the store and the coverage counts over it; an odd
        # node count, weights that differ within an in-list
        dict(name="sample_lt_rand", op="sample", graph="chung_lu", n=1_000_003, degree=16,
             weights="rand", theta=1_500_007),
        # the same for a general triggering model, a medium graph
        dict(name="sample_trig", op="sample", graph="rmat", scale=16, degree=16, weights="trig",
             theta=60_001),
        # seed selection over a large store of small and medium RR sets
        dict(name="select", op="select", graph="rmat", scale=20, degree=16, weights="wc", k=50,
             theta=2_000_003),
        # selection on buffers of the caller's, in a budget without allocations
        dict(name="select_noalloc", op="select_noalloc", n=150_001, sets=250_007, mean=6, k=50),
        # scoring 50 seeds by forward cascades, independent cascade
        dict(name="spread_ic", op="spread", graph="rmat", scale=18, degree=16, weights="wc",
             k=50, cascades=2_000),
        # and linear threshold
        dict(name="spread_lt", op="spread", graph="rmat", scale=18, degree=16, weights="inv",
             k=50, cascades=1_000),
        # a batch of independent queries on graphs of uneven sizes, half IC and half LT
        dict(name="batch", op="batch", queries=24, lo=12, hi=17, mix=1),
        # training the start-round network on the labelled set's size
        dict(name="train", op="train", samples=3_924, steps=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph(rng, lo, hi):
    """A graph of about lo to hi nodes (both powers of two: 2^lo .. 2^hi)."""
    if rng.random() < 0.5:
        return dict(graph="rmat", scale=rng.randint(lo, hi), degree=rng.choice([4, 8, 16]))
    return dict(graph="chung_lu", n=_log(rng, 2 ** lo, 2 ** hi) | 1, degree=rng.randint(4, 24))


def draw(rng):
    op = rng.choice(["query", "load_query", "load_query", "sample", "sample", "select",
                     "select_noalloc", "spread", "spread", "batch", "train"])
    if op == "query":
        return dict(op=op, **_graph(rng, 12, 16), weights=rng.choice(["wc", "inv", "rand"]),
                    k=rng.randint(1, 50), eps=round(rng.uniform(0.2, 0.5), 3))
    if op == "load_query":
        weights = rng.choice(["wc", "inv", "rand", "triv"])
        if weights == "triv":
            g = dict(graph="chung_lu", n=_log(rng, 100_000, 2_000_000) | 1, degree=35)
            return dict(op=op, **g, weights=weights, k=rng.randint(10, 50),
                        eps=round(rng.uniform(0.2, 0.5), 3))
        return dict(op=op, **_graph(rng, 16, 20), weights=weights, k=rng.randint(10, 50),
                    eps=round(rng.uniform(0.1, 0.4), 3))
    if op == "sample":
        weights = rng.choice(["wc", "inv", "rand", "trig"])
        hi = 16 if weights == "trig" else 19
        top = 60_000 if weights == "trig" else 1_500_000
        return dict(op=op, **_graph(rng, 13, hi), weights=weights,
                    theta=_log(rng, 1_000, top))
    if op == "select":
        return dict(op=op, **_graph(rng, 14, 20), weights=rng.choice(["wc", "inv", "rand"]),
                    k=rng.randint(1, 50), theta=_log(rng, 10_000, 2_000_000))
    if op == "select_noalloc":
        return dict(op=op, n=_log(rng, 1_000, 262_000), sets=_log(rng, 1_000, 300_000),
                    mean=rng.randint(2, 6), k=rng.randint(1, 50))
    if op == "spread":
        return dict(op=op, **_graph(rng, 13, 18), weights=rng.choice(["wc", "inv", "rand"]),
                    k=rng.randint(1, 50), cascades=_log(rng, 50, 1_000))
    if op == "batch":
        lo = rng.randint(12, 14)
        return dict(op=op, queries=rng.randint(2, 24), lo=lo, hi=lo + rng.randint(1, 3),
                    mix=rng.randint(2, 10 ** 6))
    return dict(op=op, samples=_log(rng, 100, 8_000), steps=rng.randint(20, 200))


# ----------------------------------------------------------------- inputs

def _draw_graph(case, seed):
    if case["graph"] == "rmat":
        return inputs.rmat_device(case["scale"], case["degree"], seed=seed)
    n = case["n"]
    return inputs.chung_lu_device(n, n * case["degree"], 2.1, seed=seed)


def _weights(g, kind, seed):
    """(model, per-edge weights) of one kind."""
    if kind == "wc":
        return tim.TIM_IC, inputs.weighted_cascade_device(g)
    if kind == "triv":
        return tim.TIM_IC, inputs.trivalency_device(g, seed=seed)
    if kind == "inv":
        return tim.TIM_LT, inputs.weighted_cascade_device(g)
    return tim.TIM_LT, inputs.lt_random_normalised_device(g, seed=seed)


def _triggering(g, seed):
    """Triggering options of every node on the host: its in-edges in runs of one to three,
    each run one option, with random probabilities that sum to 0.9 per node."""
    order = torch.argsort(g.dst.to(torch.int64), stable=True)
    node = g.dst[order].to(torch.int64).cpu().numpy()
    order = order.cpu().numpy().astype(np.int64)
    m = node.shape[0]
    r = np.random.Generator(np.random.Philox(seed))
    first = np.ones(m, dtype=bool)
    first[1:] = node[1:] != node[:-1]
    at = np.arange(m) - np.maximum.accumulate(np.where(first, np.arange(m), 0))
    start = at % int(r.integers(2, 4)) == 0  # the first in-edge of an option
    opt_edge_rowptr = np.append(np.flatnonzero(start), m).astype(np.int64)
    opt_node = node[start]
    opt_rowptr = np.zeros(g.n + 1, dtype=np.int64)
    np.cumsum(np.bincount(opt_node, minlength=g.n), out=opt_rowptr[1:])
    p = r.random(opt_node.shape[0]) + 0.05
    total = np.bincount(opt_node, weights=p, minlength=g.n)
    return opt_rowptr, (0.9 * p / total[opt_node]).astype(np.float32), opt_edge_rowptr, order


def _load(eng, s):
    tim.tim_load_graph_device(eng.ctx, s["n"], s["m"], s["rowptr"], s["dst"], s["weight"],
                              s["model"])


def _top_sources(g, k):
    """The k nodes of largest out-degree (ties: smallest id)."""
    deg = g.rowptr[1:] - g.rowptr[:-1]
    return torch.sort(deg, descending=True, stable=True).indices[:k].cpu().numpy().astype(np.int32)


def _store_csr(case, seed):
    """RR sets of skewed sizes over skewed nodes as a CSR, members distinct in a set."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, sets = case["n"], case["sets"]
    u = torch.rand(sets, generator=gen, device="cuda", dtype=torch.float64)
    size = (1.0 + (2 * case["mean"] - 2) * u * u * 1.5).to(torch.int64)
    sid = torch.repeat_interleave(torch.arange(sets, device="cuda"), size)
    v = torch.rand(sid.shape[0], generator=gen, device="cuda", dtype=torch.float64)
    node = (n * v * v * v).to(torch.int64).clamp_(max=n - 1)
    key = torch.unique(sid * n + node)  # distinct members, ascending by set
    off = torch.zeros(sets + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(key // n, minlength=sets), 0)
    return off, (key % n).to(torch.int32)


def _train_inputs(case, seed):
    """Features and targets as the start-round network sees them (12 standardised features;
    a smooth target with noise), initial parameters, scaling."""
    r = np.random.Generator(np.random.Philox(seed))
    n, d = case["samples"], 12
    x = (r.normal(size=(n, d)) * 2.0 + 3.0).astype(np.float32)
    z = (x.astype(np.float64) - 3.0) / 2.0
    y = 4.0 + np.tanh(z @ r.normal(size=d) * 0.4) * 2.0 + 0.3 * z[:, 0] * z[:, 1]
    y = (y + 0.1 * r.normal(size=n)).astype(np.float32)
    parts = []
    for fan_out, fan_in in ((HIDDEN, d), (HIDDEN, HIDDEN), (1, HIDDEN)):
        lim = 1.0 / math.sqrt(fan_in)
        parts += [r.uniform(-lim, lim, size=fan_out * fan_in), np.zeros(fan_out)]
    params = np.concatenate(parts).astype(np.float32)
    mu = np.full(d, 3.0, dtype=np.float32)
    isd = np.full(d, 0.5, dtype=np.float32)
    return dict(x=x, y=y, params=params, mu=mu, isd=isd, out_mu=4.0, out_sd=2.0, lr=3e-3)


def _batch_specs(case, seed):
    """Scales, k and eps of a batch's queries (from its mix), graph seeds; even queries IC,
    odd ones LT."""
    r = np.random.Generator(np.random.Philox(case["mix"]))
    return [dict(scale=int(r.integers(case["lo"], case["hi"] + 1)), k=int(r.integers(1, 51)),
                 eps=float(r.choice([0.1, 0.2, 0.3, 0.5])), weights="wc" if q % 2 == 0 else "inv",
                 seed=seed * 256 + q, tag=q + 1) for q in range(case["queries"])]


def prepare(case, seed):
    op = case["op"]
    s = dict(op=op, seed=seed)
    if op == "train":
        s.update(_train_inputs(case, seed), steps=case["steps"])
        s["eng"] = tim.Engine(0)
        s["mlp"] = tim.tim_mlp_create(s["eng"].ctx, 12)
        tim.tim_mlp_set_scaling(s["eng"].ctx, s["mlp"], s["mu"], s["isd"], s["out_mu"],
                                s["out_sd"])
        return s
    if op == "select_noalloc":
        s["off"], s["mem"] = _store_csr(case, seed)
        s.update(n=case["n"], sets=case["sets"], k=case["k"])
        s["seeds"] = torch.zeros(case["k"], dtype=torch.int32, device="cuda")
        s["covered"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        return s
    if op == "batch":
        s["queries"], s["engines"] = [], []
        for q in _batch_specs(case, seed):
            g = inputs.rmat_device(q["scale"], 16, seed=q["seed"])
            model, w = _weights(g, q["weights"], q["seed"])
            torch.cuda.synchronize()
            eng = tim.Engine(0)
            tim.tim_load_graph_device(eng.ctx, g.n, g.m, g.rowptr, g.dst, w, model)
            s["engines"].append(eng)
            s["queries"].append(dict(ctx=eng.ctx, k=q["k"], eps=q["eps"], ell=ELL, tag=q["tag"]))
        return s
    g = _draw_graph(case, seed)
    s.update(n=g.n, m=g.m, k=case.get("k", 0), eps=case.get("eps", 0.0))
    s["eng"] = eng = tim.Engine(0)
    if case["weights"] == "trig":
        opts = _triggering(g, seed)
        tim.tim_load_graph_triggering(eng.ctx, g.n, g.rowptr.cpu().numpy(), g.dst.cpu().numpy(),
                                      *opts)
    else:
        model, w = _weights(g, case["weights"], seed + 1)
        s.update(rowptr=g.rowptr, dst=g.dst, weight=w, model=model)
        torch.cuda.synchronize()  # the engine's stream is its own
        if op != "load_query":
            _load(eng, s)
            for name in ("rowptr", "dst", "weight"):
                del s[name]
    if op in ("sample", "select"):
        s["theta"] = case["theta"]
    if op == "select":
        tim.tim_sample_rr(eng.ctx, s["theta"], seed, SELECT_SIDS)
    if op == "spread":
        s["cascades"] = case["cascades"]
        s["seeds"] = _top_sources(g, case["k"])
    return s


# ----------------------------------------------------------------- one pass

def _answer(seeds, frac, st):
    """What a caller reads of a query's answer."""
    out = dict(seeds=seeds, fraction=float(frac))
    for name in ("lambda", "kpt_star", "kpt_plus", "eps_prime"):
        out[name] = float(st[name])
    for name in ("kpt_round", "theta_prime", "covered_prime", "theta", "covered",
                 "members_select", "width_select", "sets_total"):
        out[name] = int(st[name])
    return out


def run(s):
    op = s["op"]
    if op == "train":
        ctx = s["eng"].ctx
        tim.tim_mlp_set_params(ctx, s["mlp"], s["params"])
        history = tim.tim_mlp_train(ctx, s["mlp"], s["x"], s["y"], s["steps"], s["lr"])
        return dict(history=history, params=tim.tim_mlp_get_params(ctx, s["mlp"]))
    if op == "select_noalloc":
        tim.tim_node_select_noalloc(0, None, s["n"], s["sets"], s["off"], s["mem"], s["k"],
                                    s["seeds"], s["covered"])
        return dict(seeds=s["seeds"], covered=s["covered"])
    if op == "batch":
        out, st = tim.tim_run_batch(s["queries"], s["seed"])
        answers = [_answer(*q) for q in out]
        return {name: (np.concatenate([a[name] for a in answers]) if name == "seeds" else
                       np.array([a[name] for a in answers])) for name in answers[0]}
    ctx = s["eng"].ctx
    if op in ("query", "load_query"):
        if op == "load_query":
            _load(s["eng"], s)
        return _answer(*tim.tim_run(ctx, s["k"], s["eps"], ELL, s["seed"]))
    if op == "sample":
        total = tim.tim_sample_rr(ctx, s["theta"], s["seed"], SELECT_SIDS)
        return dict(members=total, counts=tim.tim_coverage_counts(ctx, s["n"]))
    if op == "select":
        seeds, frac, covered = tim.tim_node_select(ctx, s["k"])
        return dict(seeds=seeds, fraction=float(frac), covered=covered)
    mean, total, counts = tim.tim_spread_mc(ctx, s["seeds"], s["cascades"], s["seed"], SCORE_SIDS,
                                            want_counts=True)
    return dict(mean=float(mean), total=total, counts=counts)


# ----------------------------------------------------------------- work and exact values

def _nodes(case):
    return 2 ** case["scale"] if case["graph"] == "rmat" else case["n"]


def work(case):
    """Inputs read once and outputs written once (a graph is 8 B per node and 8 B per edge;
    a few duplicate draws are dropped from the edges counted here). Where the work depends
    on what is drawn (RR sets, cascades), a set or cascade counts with its record alone."""
    op = case["op"]
    if op == "train":
        p = HIDDEN * 12 + HIDDEN + HIDDEN * HIDDEN + HIDDEN + HIDDEN + 1
        n, steps = case["samples"], case["steps"]
        # forward, gradient of the weights, gradient of the activations
        flops = 2.0 * n * steps * (2 * HIDDEN * 12 + 3 * HIDDEN * HIDDEN + 3 * HIDDEN)
        return dict(bytes=4.0 * (13 * n + steps + 2 * p), flops=flops)
    if op == "select_noalloc":
        return dict(bytes=8.0 * (case["sets"] + 1) + 4.0 * case["sets"] * case["mean"] +
                    4.0 * case["k"] + 8, flops=0)
    if op == "batch":
        scale = 0.5 * (case["lo"] + case["hi"])
        return dict(bytes=case["queries"] * 2.0 ** scale * (8 + 8 * 16), flops=0)
    n = _nodes(case)
    graph = 8.0 * (n + 1) + 8.0 * n * case["degree"]
    if op == "spread":
        return dict(bytes=graph + 4.0 * (case["cascades"] + case["k"]), flops=0)
    if op == "sample":
        return dict(bytes=graph + 24.0 * case["theta"] + 4.0 * n, flops=0)
    if op == "select":
        return dict(bytes=24.0 * case["theta"] + 4.0 * n, flops=0)
    return dict(bytes=graph + 4.0 * case["k"], flops=0)


def _lambda(n, k, eps):
    """Eq. 4 of the paper, l = 1."""
    lnc = math.fsum(math.log((n - i) / (k - i)) for i in range(k))
    return (8.0 + 2.0 * eps) * n * (ELL * math.log(n) + lnc + math.log(2.0)) / eps ** 2


def _eps_prime(k, eps):
    return 5.0 * (ELL * eps * eps / (k + ELL)) ** (1.0 / 3.0)


def _bf16(t):
    return t.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _train_exact(case, seed):
    """Full-batch Adam in 64 bits, weight matrices used rounded to bfloat16."""
    i = _train_inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float64)).to(dev)  # noqa: E731
    x, y = (f(i["x"]) - f(i["mu"])) * f(i["isd"]), (f(i["y"]) - i["out_mu"]) / i["out_sd"]
    n, d, h = x.shape[0], 12, HIDDEN
    shapes = [(h, d), (h,), (h, h), (h,), (1, h), (1,)]
    sizes = [math.prod(v) for v in shapes]
    w = [t.reshape(v).clone() for t, v in zip(torch.split(f(i["params"]), sizes), shapes)]
    m1 = [torch.zeros_like(t) for t in w]
    m2 = [torch.zeros_like(t) for t in w]
    history = []
    phi = lambda t: 0.5 * (1.0 + torch.erf(t / math.sqrt(2.0)))  # noqa: E731
    dgelu = lambda t: phi(t) + t * torch.exp(-0.5 * t * t) / math.sqrt(2 * math.pi)  # noqa: E731
    for step in range(1, case["steps"] + 1):
        w1, w2, w3 = _bf16(w[0]), _bf16(w[2]), _bf16(w[4])
        a1 = x @ w1.T + w[1]
        h1 = a1 * phi(a1)
        a2 = h1 @ w2.T + w[3]
        h2 = a2 * phi(a2)
        diff = (h2 @ w3.T + w[5])[:, 0] - y
        history.append(0.5 * (diff * diff).mean())
        dz = diff[:, None] / n
        d2 = dz @ w3 * dgelu(a2)
        d1 = d2 @ w2 * dgelu(a1)
        grads = [d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dz.T @ h2, dz.sum(0)]
        for t, g, a, b in zip(w, grads, m1, m2):
            a.mul_(0.9).add_(0.1 * g)
            b.mul_(0.999).add_(0.001 * g * g)
            t -= i["lr"] * (a / (1 - 0.9 ** step)) / ((b / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return dict(history=torch.stack(history), params=torch.cat([t.reshape(-1) for t in w]))


def exact(case, seed):
    """What has a value apart from the sets that are drawn: Eq. 4 and the network."""
    op = case["op"]
    if op == "train":
        return _train_exact(case, seed)
    if op in ("query", "load_query"):
        n = _nodes(case)
        return {"lambda": _lambda(n, case["k"], case["eps"]),
                "eps_prime": _eps_prime(case["k"], case["eps"])}
    if op == "batch":
        q = _batch_specs(case, seed)
        return {"lambda": np.array([_lambda(2 ** v["scale"], v["k"], v["eps"]) for v in q]),
                "eps_prime": np.array([_eps_prime(v["k"], v["eps"]) for v in q])}
    return None
