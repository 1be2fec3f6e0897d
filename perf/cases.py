"""The work a user of this framework has it do, as measurable cases.

A program that learns a Bayesian-network structure builds the local-score tables of its
data sets, scores batches of node orders against a table (a search of its own, or the
re-scoring of stored orders), runs the Metropolis-Hastings sampler over orders, and may
train and use a network that proposes swaps.  Each case below is one such call, or one
such sequence of calls, through the package's public functions.

The networks are random DAGs (in-degree <= 3, CPT rows ~ Dirichlet(1)) with forward
samples, the shapes those of the repository's workloads: 6 to 60 nodes, 2 to 4 states,
100 to 5,000 rows, parent sets of up to 4 nodes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1210_5128_gb300 as bn

FULL, PRUNED, SLICED, SORTED = "full", "pruned", "sliced", "sorted"
_MODE = {FULL: bn.SCAN_FULL, PRUNED: bn.SCAN_PRUNED, SLICED: bn.SCAN_SLICED, SORTED: bn.SCAN_SORTED}
_BUILD_ROWS = 60 * 489406 * 1000        # row visits of the largest table build


# ---- the cases -----------------------------------------------------------------------
def listed():
    net = dict(arity=3, m=1000, k=4, bdeu=0.0, gamma=0.0, prior=False)
    return [
        # one order of the smallest network a learner is run on in earnest, host arrays in and
        # out: a search that scores one proposal at a time; latency alone
        dict(name="score_n13_one", kind="score", n=13, B=1, mode=FULL, where="host", **net),
        # one order over the largest table (29.4 M entries): one step of a search on 60 nodes
        dict(name="score_n60_one", kind="score", n=60, B=1, mode=FULL, where="cuda", **net),
        # a ragged batch over a 40-node table in the default scan: re-scoring a population
        dict(name="score_n40_777", kind="score", n=40, B=777, mode=FULL, where="cuda", **(net | dict(m=2000))),
        # a large population on the pruned table of 60 nodes, host arrays in and out
        dict(name="score_pruned_n60_4096", kind="score", n=60, B=4096, mode=PRUNED, where="host", **net),
        # the sum over graphs instead of the best graph, for a handful of orders
        dict(name="sum_n60_8", kind="sum", n=60, B=8, where="cuda", **net),
        # the preprocessing step: every local score of the largest network, read out whole
        dict(name="build_n60", kind="build", n=60, where="cuda", **net),
        # learning a network end to end from host data: a 37-node network of 2 to 4 states,
        # BDeu score and a pairwise prior, pruning, 64 chains, posterior edge frequencies
        dict(name="learn_n37", kind="learn", n=37, chains=64, steps=2000, **(net | dict(arity=0, bdeu=1.0, prior=True))),
        # the sampler on a table the program keeps: 256 chains over 60 nodes
        dict(name="mcmc_n60_256", kind="mcmc", n=60, chains=256, steps=1000, mode=PRUNED, **net),
        # the same sampler on a table as it is after the build (default scan), 512 chains
        dict(name="mcmc_full_n40_512", kind="mcmc", n=40, chains=512, steps=64, mode=FULL, **(net | dict(m=2000))),
        # a dozen data sets of uneven size learned together: 10 to 60 nodes, 2 to 4 states
        dict(name="learn_batch_12", kind="batch", count=12, n=60, chains=32, steps=1024, m=5000),
        # training the proposal network: 16 steps of forward, backward and Adam
        dict(name="train_n60_256", kind="train", n=60, B=256, hidden=512, d=32, steps=16),
        # the sampler with the learned proposal inside its MH ratio
        dict(name="learned_n60_256", kind="learned", n=60, chains=256, steps=256, hidden=512, d=32, **net),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _table(rng, lo=6, hi=60):
    n = rng.randint(lo, hi)
    k = min(n - 1, rng.choice([2, 3, 4, 4, 4]))
    m = _log(rng, 100, 5000)
    c = dict(n=n, k=k, arity=rng.choice([0, 2, 3, 3, 4]), bdeu=rng.choice([0.0, 0.0, 1.0, 10.0]),
             gamma=rng.choice([0.0, 0.0, -0.5]), prior=rng.random() < 0.3)
    rows = n * _num_sets(n - 1, k)
    if c["arity"] in (0, 4):
        rows *= 4                       # counts of up to 1,024 cells a set, against 243
    c["m"] = max(50, min(m, _BUILD_ROWS // rows))
    return c


def draw(rng):
    kind = rng.choice(["score", "score", "score", "sum", "build", "build", "learn", "mcmc", "mcmc", "batch", "train", "learned"])
    if kind == "score":
        c = _table(rng)
        c["mode"] = rng.choice([FULL, FULL, PRUNED, SLICED, SORTED])
        B = _log(rng, 1, 8192)
        if c["mode"] == FULL:           # 5 ms of the mask-test scan at most
            B = min(B, max(1, 1000 * 60 * 489406 // (c["n"] * _num_sets(c["n"] - 1, c["k"]))))
        return dict(kind=kind, B=B, where=rng.choice(["host", "cuda"]), **c)
    if kind == "sum":
        return dict(kind=kind, B=_log(rng, 1, 64), where=rng.choice(["host", "cuda"]), **_table(rng))
    if kind == "build":
        return dict(kind=kind, where=rng.choice(["host", "cuda"]), **_table(rng))
    if kind == "learn":
        return dict(kind=kind, chains=_log(rng, 1, 256), steps=_log(rng, 200, 2000), **_table(rng, 6, 50))
    if kind == "mcmc":
        c = _table(rng)
        c["mode"] = rng.choice([FULL, PRUNED, PRUNED, SORTED])
        steps = _log(rng, 200, 4000) if c["mode"] == PRUNED else _log(rng, 8, 64)
        chains = _log(rng, 1, 512)
        if c["mode"] == FULL:
            chains = min(chains, max(1, 512 * 40 * 92171 // (c["n"] * _num_sets(c["n"] - 1, c["k"]))))
        return dict(kind=kind, chains=chains, steps=steps, **c)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 10), n=rng.randint(20, 50), chains=_log(rng, 1, 32),
                    steps=_log(rng, 100, 1024), m=_log(rng, 200, 5000))
    if kind == "train":
        return dict(kind=kind, n=rng.randint(6, 60), B=_log(rng, 16, 512), hidden=rng.choice([128, 256, 512]),
                    d=rng.choice([8, 16, 32]), steps=rng.randint(1, 12))
    c = _table(rng, 10, 60)
    return dict(kind="learned", chains=_log(rng, 1, 256), steps=_log(rng, 16, 256), hidden=rng.choice([128, 256, 512]),
                d=rng.choice([8, 16, 32]), **c)


# ---- inputs --------------------------------------------------------------------------
def _num_sets(N, k):
    return sum(math.comb(N, j) for j in range(min(N, k) + 1))


def _network(n, arity, m, seed):
    """Forward samples (m, n) uint8 of a random DAG, and the arities (arity 0: 2 to 4 each)."""
    rng = np.random.default_rng(seed)
    ar = np.full(n, arity, np.uint8) if arity else rng.integers(2, 5, n).astype(np.uint8)
    topo = rng.permutation(n)
    x = np.zeros((m, n), np.uint8)
    adj = np.zeros((n, n), bool)
    for p, v in enumerate(topo):
        ps = rng.choice(topo[:p], size=int(rng.integers(0, min(3, p) + 1)), replace=False) if p else []
        cfg, q = np.zeros(m, np.int64), 1
        for u in ps:
            cfg += x[:, u].astype(np.int64) * q
            q *= int(ar[u])
            adj[v, u] = True
        cdf = np.cumsum(rng.dirichlet(np.ones(int(ar[v])), size=q), axis=1)
        x[:, v] = np.minimum((rng.random(m)[:, None] >= cdf[cfg]).sum(1), int(ar[v]) - 1)
    return x, ar, adj


def _prior(adj, seed):
    """Interface matrix: a tenth of the true edges at 1, a tenth of the others at 0, else 0.5."""
    u = np.random.default_rng(seed).random(adj.shape)
    R = np.where(u < 0.1, np.where(adj, 1.0, 0.0), 0.5)
    np.fill_diagonal(R, 0.5)
    return R


def _inputs(case, seed):
    x, ar, adj = _network(case["n"], case["arity"], case["m"], seed)
    R = _prior(adj, seed + 1) if case["prior"] else None
    opt = dict(score_kind=1 if case["bdeu"] else 0, ess=case["bdeu"] or 1.0, log10_gamma=case["gamma"])
    return x, ar, R, opt


def _orders(n, B, seed):
    return np.random.default_rng(seed).permuted(np.tile(np.arange(n, dtype=np.uint8), (B, 1)), axis=1)


def _weights(n, d, H, seed):
    rng = np.random.default_rng(seed)
    P = n * (n - 1) // 2

    def uni(shape, fan):
        return (rng.uniform(-1, 1, shape) / math.sqrt(fan)).astype(np.float32)
    return dict(E=uni((n, d), 1), W1=uni((H, n * d), n * d), b1=uni(H, n * d), W2=uni((H, H), H), b2=uni(H, H),
                W3=uni((P, H), H), b3=uni(P, H))


def _place(a, where):
    return torch.from_numpy(a).cuda() if where == "cuda" else a


def _batch_networks(case, seed):
    rng = np.random.default_rng([case["count"], case["n"], case["m"]])      # the sizes are the case's own
    nets = []
    for t in range(case["count"]):
        n = case["n"] if t == 0 else int(rng.integers(10, case["n"] + 1))
        # the largest network is a ternary one with m = 1,000, as in the largest single build
        m = min(1000, case["m"]) if n > 45 else int(round(math.exp(rng.uniform(math.log(200), math.log(case["m"] + 1)))))
        x, ar, _ = _network(n, 3 if n > 45 else 0, m, seed + 10 * t + 1)
        nets.append((x, ar, 4 if t == 0 else int(rng.integers(3, 5)), None))
    return nets


def _train_batch(case, seed):
    n, B, T = case["n"], case["B"], case["steps"]
    rng = np.random.default_rng(seed + 5)
    pairs = rng.integers(0, n * (n - 1) // 2, (T, B)).astype(np.uint32)
    # acceptance probabilities of logged swaps: many are 0 (no-ops and bad moves), some are 1
    alpha = np.minimum(1.0, 10.0 ** rng.normal(-2.0, 4.0, (T, B))).astype(np.float32)
    return _orders(n, T * B, seed + 6).reshape(T, B, n), pairs, alpha


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "batch":
        s["nets"] = _batch_networks(case, seed)
        return s
    if kind == "train":
        s["net"] = bn.mlp_create(case["n"], _weights(case["n"], case["d"], case["hidden"], seed), hidden=case["hidden"],
                                 d=case["d"], batch_cap=case["B"], lr=3e-4)
        s["orders"], s["pairs"], s["alpha"] = _train_batch(case, seed)
        return s
    x, ar, R, opt = _inputs(case, seed)
    if kind in ("build", "learn"):
        where = case.get("where", "host")
        s.update(x=_place(x, where), ar=_place(ar, where), R=None if R is None else _place(R, where), opt=opt)
        return s
    t = bn.build_scores(x, ar, case["k"], R=R, **opt)
    mode = PRUNED if kind == "learned" else case.get("mode", FULL)
    if mode != FULL:
        bn.table_set_scan(t, _MODE[mode])
    s["table"] = t
    if kind in ("score", "sum"):
        s["orders"] = _place(_orders(case["n"], case["B"], seed + 2), case["where"])
    if kind == "learned":
        s["net"] = bn.mlp_create(case["n"], _weights(case["n"], case["d"], case["hidden"], seed + 3),
                                 hidden=case["hidden"], d=case["d"], batch_cap=case["chains"], lr=1e-3)
    return s


# ---- one pass ------------------------------------------------------------------------
def _result(r):
    return dict(best_order=r["best_order"], best_dag=r["best_dag"], best_score=r["best_score"], edge_freq=r["edge_freq"])


def run(state):
    case, kind, seed = state["case"], state["case"]["kind"], state["seed"]
    if kind == "score":
        return bn.score_orders(state["table"], state["orders"])
    if kind == "sum":
        return bn.score_orders_sum(state["table"], state["orders"])
    if kind == "build":
        t = bn.build_scores(state["x"], state["ar"], case["k"], R=state["R"], **state["opt"])
        return bn.table_scores(t, device="cuda")
    if kind == "learn":
        t = bn.build_scores(state["x"], state["ar"], case["k"], R=state["R"], **state["opt"])
        bn.table_set_scan(t, bn.SCAN_PRUNED)
        return _result(bn.mcmc_run(t, case["chains"], case["steps"], seed, burn_in=case["steps"] // 4))
    if kind == "batch":
        ts = bn.build_scores_batch(state["nets"])
        for t in ts:
            bn.table_set_scan(t, bn.SCAN_PRUNED)
        return [_result(r) for r in bn.mcmc_run_batch(ts, case["chains"], case["steps"], seed, burn_in=case["steps"] // 4)]
    if kind == "train":
        net, loss = state["net"], []
        for i in range(case["steps"]):
            loss.append(bn.mlp_loss_grad(net, state["orders"][i], state["pairs"][i], state["alpha"][i]))
            bn.mlp_adam_step(net)
        return dict(loss=np.array(loss), **{w: bn.mlp_read(net, w) for w in bn.MLP_TENSORS})
    if kind == "mcmc" and case["mode"] == PRUNED:
        return _result(bn.mcmc_run(state["table"], case["chains"], case["steps"], seed, burn_in=case["steps"] // 4))
    c = bn.chains_create(state["table"], case["chains"], seed, burn_in=case["steps"] // 4)
    outs = ["orders", "scores", "best_orders", "best_scores", "best_ranks", "edge_counts", "accepts"]
    if kind == "learned":
        bn.chains_set_proposal(c, state["net"], bn.PROPOSAL_LEARNED, eps_mix=0.1)
        outs.append("logits")
    bn.chains_step(c, case["steps"])
    return {w: bn.chains_read(c, w) for w in outs}


# ---- what a pass cannot do without ---------------------------------------------------
def work(case):
    kind, n = case["kind"], case["n"]
    if kind in ("train", "learned"):
        P, H, nd = n * (n - 1) // 2, case["hidden"], n * case["d"]
        params = n * case["d"] + H * nd + H * H + P * H + 2 * H + P
        if kind == "train":
            # three products per layer and step; weights and both moments read and written once
            return dict(bytes=24.0 * params + case["steps"] * case["B"] * (n + 8.0),
                        flops=case["steps"] * (6.0 * case["B"] * (H * nd + H * H) + 2.0 * case["B"] * H * P + 4.0 * case["B"] * H))
        C = case["chains"]
        return dict(bytes=2.0 * params + C * (n * (2 + 4 + 4.0 * n) + 4.0 * P + 24),
                    flops=case["steps"] * 2.0 * C * (4 * H * case["d"] + H * H + H * P))
    if kind == "batch":
        # the data in, the results out; every table's counts and one order score per step
        per = case["m"] * 30.0 + 9.0 * 35 * 35
        return dict(bytes=case["count"] * per, flops=case["count"] * (math.comb(35, 4) * 1000.0 + case["chains"] * case["steps"] * 35.0))
    S = _num_sets(n - 1, case["k"])
    # every joint count table of up to k + 1 nodes, one addition per row; one entry per set
    count = _num_sets(n, case["k"] + 1) * float(case["m"]) + n * S
    if kind == "build":
        return dict(bytes=case["m"] * n + 8.0 * n * S, flops=count)
    if kind == "learn":
        return dict(bytes=case["m"] * n + 9.0 * n * n, flops=count + case["chains"] * case["steps"] * float(n))
    if kind == "sum":
        # every entry once (8 bytes), the orders, the scores
        return dict(bytes=8.0 * n * S + case["B"] * (n + 8.0 * n + 8), flops=case["B"] * n * S / 5.0)
    io = case.get("B", 0) * (n + 4.0 * n + 8)
    if kind == "score":
        if case["mode"] != FULL and case["mode"] != SLICED:
            return dict(bytes=io + n * 64.0, flops=case["B"] * float(n))
        # every entry's place in its node's score order, 4 bytes
        return dict(bytes=io + 4.0 * n * S, flops=case["B"] * float(n))
    steps = case["steps"]
    evals = case["chains"] * steps * float(n)
    out = case["chains"] * n * (2 + 4 + 4.0 * n)
    if case["mode"] == FULL:
        return dict(bytes=steps * 4.0 * n * S + out, flops=evals)
    return dict(bytes=n * 64.0 + 9.0 * n * n, flops=evals)


# ---- the same in 64 bits, by plain torch ----------------------------------------------
def _colex(N, k):
    """Per size j <= k the j-subsets of range(N) as rows, in colex order (the table's rank order)."""
    rows = [np.zeros((1, 0), np.int64)]
    for j in range(1, min(N, k) + 1):
        prev = rows[-1]
        rows.append(np.concatenate([np.concatenate([prev[:math.comb(a, j - 1)], np.full((math.comb(a, j - 1), 1), a)], axis=1)
                                    for a in range(j - 1, N)]))
    return rows


def _exact_table(case, seed, dev):
    """(n, S) float64 scores and the (n, S) parent masks in node space."""
    x, ar, R, opt = _inputs(case, seed)
    n, k, m = case["n"], case["k"], case["m"]
    X = torch.from_numpy(x).to(dev).t().contiguous().to(torch.int32)
    A = torch.from_numpy(ar.astype(np.int64)).to(dev)
    classes = [torch.from_numpy(c).to(dev) for c in _colex(n - 1, k)]
    ppf = None if R is None else torch.from_numpy(100.0 * (R - 0.5) ** 3).to(dev)
    out, masks = [], []
    for i in range(n):
        r = int(ar[i])
        for j, sets in enumerate(classes):
            par = sets + (sets >= i).long()
            qs = torch.ones(len(par), dtype=torch.int64, device=dev)
            strides = []
            for t in range(j):
                strides.append(r * qs)
                qs = qs * A[par[:, t]]
            W = int(qs.max()) * r
            step = max(1, min((1 << 26) // max(m, 1), (1 << 26) // W))
            for a in range(0, len(par), step):
                p, q = par[a:a + step], qs[a:a + step]
                c = len(p)
                cell = X[i].expand(c, m) + (torch.arange(c, device=dev, dtype=torch.int32) * W)[:, None]
                for t in range(j):
                    cell = cell + X[p[:, t]] * strides[t][a:a + step, None].to(torch.int32)
                cnt = torch.bincount(cell.reshape(-1), minlength=c * W).view(c, W // r, r).double()
                if opt["score_kind"]:
                    a_cell, a_cfg = opt["ess"] / (q * r).double(), opt["ess"] / q.double()
                else:
                    a_cell, a_cfg = torch.ones(c, dtype=torch.float64, device=dev), torch.full((c,), float(r), dtype=torch.float64, device=dev)
                tot = cnt.sum(2)
                g = lambda v, al: torch.where(v > 0, torch.lgamma(v + al) - torch.lgamma(al), torch.zeros((), dtype=torch.float64, device=dev))  # noqa: E731
                ls = g(cnt, a_cell[:, None, None]).sum((1, 2)) - g(tot, a_cfg[:, None]).sum(1)
                ls = ls / math.log(10.0) + j * opt["log10_gamma"]
                if ppf is not None:
                    for t in range(j):
                        ls = ls + ppf[i, p[:, t]]
                out.append(ls)
                masks.append((torch.ones_like(p) << p).sum(1) if j else torch.zeros(c, dtype=torch.int64, device=dev))
    S = _num_sets(n - 1, k)
    return torch.cat(out).view(n, S), torch.cat(masks).view(n, S)


def _exact_score(case, seed, dev):
    T, M = _exact_table(case, seed, dev)
    n, B = case["n"], case["B"]
    o = torch.from_numpy(_orders(n, B, seed + 2).astype(np.int64)).to(dev)
    bits = torch.ones_like(o) << o
    pred = torch.empty_like(o).scatter_(1, o, torch.cumsum(bits, 1) - bits)   # [b, v] = v's predecessors
    node = torch.empty((B, n), dtype=torch.float64, device=dev)
    step = max(1, (1 << 28) // T.shape[1])
    for i in range(n):
        for b in range(0, B, step):
            ok = (M[i][None, :] & ~pred[b:b + step, i, None]) == 0
            v = torch.where(ok, T[i][None, :], torch.full((), -math.inf, dtype=torch.float64, device=dev))
            if case["kind"] == "score":
                node[b:b + step, i] = v.amax(1)
            else:
                node[b:b + step, i] = torch.logsumexp(v * math.log(10.0), 1) / math.log(10.0)
    return node


def _exact_train(case, seed, dev):
    n, H, d, B = case["n"], case["hidden"], case["d"], case["B"]
    w = {k: torch.from_numpy(v).to(dev).double().requires_grad_() for k, v in _weights(n, d, H, seed).items()}
    mom = {k: (torch.zeros_like(v), torch.zeros_like(v)) for k, v in w.items()}
    orders, pairs, alpha = _train_batch(case, seed)
    losses = []
    for t in range(case["steps"]):
        o = torch.from_numpy(orders[t].astype(np.int64)).to(dev)
        p = torch.from_numpy(pairs[t].astype(np.int64)).to(dev)
        al = torch.from_numpy(alpha[t]).to(dev).double()
        h = torch.relu(w["E"][o].reshape(B, n * d) @ w["W1"].t() + w["b1"])
        h = torch.relu(h @ w["W2"].t() + w["b2"])
        l = (h * w["W3"][p]).sum(1) + w["b3"][p]
        loss = torch.nn.functional.binary_cross_entropy_with_logits(l, al)
        grads = torch.autograd.grad(loss, list(w.values()))
        losses.append(float(loss.detach()))
        with torch.no_grad():
            for (k, v), g in zip(w.items(), grads):
                a, b = mom[k]
                a.mul_(0.9).add_(0.1 * g)
                b.mul_(0.999).add_(0.001 * g * g)
                v.sub_(3e-4 * (a / (1 - 0.9 ** (t + 1))) / ((b / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8))
    return dict(loss=np.array(losses), **{k: v.detach() for k, v in w.items()})


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("learn", "mcmc", "batch", "learned"):
        return None                     # thousands of dependent steps of a sampler
    if kind == "train":
        return _exact_train(case, seed, dev)
    if dev == "cpu" and case["n"] > 20:
        return None
    if kind == "build":
        return _exact_table(case, seed, dev)[0]
    node = _exact_score(case, seed, dev)
    return (None, node.sum(1)) if kind == "score" else (node.sum(1), node)
