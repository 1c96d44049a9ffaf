"""The work a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values.  ``prepare`` builds what a program holds before the call (a graph
handle, seed sets, a surrogate network), ``run`` makes the call through the package's entry points,
``work`` says what the call cannot do without and ``exact`` recomputes the floating outputs in 64 bits.

Simulation outputs are integers (spreads, counts, edge checks, chosen seeds), so ``exact`` has no value
for them.  The network's floating outputs are recomputed in fp64 from the definition in include/cnd.h
with its bf16 inputs (features, weight matrices) and no rounding of what is computed from them.
"""
import math

import numpy as np
import torch

import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

H, D0 = 64, 16


def listed():
    return [
        # one small what-if question from host arrays, as an interactive user asks it: G(1000, 10000), p = 0.1
        {"name": "ic_er_1k", "kind": "sim", "model": "ic", "graph": "er", "n": 1000, "m": 10000, "p": "0.1",
         "pick": "uniform", "seeds": 10, "trials": 1000, "mode": "host", "first_trial": 0},
        # the run-time table's small-world network: p ~ U[0, 1], 100 seeds, 1,000 runs, host arrays
        {"name": "ic_ws_10k", "kind": "sim", "model": "ic", "graph": "ws", "n": 10000, "k": 10, "p": "ur1",
         "pick": "uniform", "seeds": 100, "trials": 1000, "mode": "host", "first_trial": 0},
        # a mid-size social graph, weighted cascade, many trials, device arrays, one graph launch per call
        {"name": "ic_ba_100k", "kind": "sim", "model": "ic", "graph": "ba", "n": 100000, "k": 5, "p": "wc",
         "pick": "top", "seeds": 50, "trials": 10000, "mode": "graph", "first_trial": 0},
        # the same network under LT (weighted cascade: every node's in-weights equal)
        {"name": "lt_ba_100k", "kind": "sim", "model": "lt", "graph": "ba", "n": 100000, "k": 5, "p": "wc",
         "pick": "top", "seeds": 50, "trials": 10000, "mode": "device", "first_trial": 0},
        # LT with measured (unequal) influence weights, a ragged number of trials
        {"name": "lt_uneven_rmat_17", "kind": "sim", "model": "lt", "graph": "rmat", "scale": 17, "factor": 15,
         "p": "uneven", "pick": "top", "seeds": 50, "trials": 999, "mode": "device", "first_trial": 0},
        # a large web-like graph, IC with uniform p = 0.01, one shard's trial range
        {"name": "ic_rmat_21", "kind": "sim", "model": "ic", "graph": "rmat", "scale": 21, "factor": 16, "p": "0.01",
         "pick": "top", "seeds": 100, "trials": 1024, "mode": "device", "first_trial": 1024},
        # the same graph shape under LT: the largest call here
        {"name": "lt_rmat_21", "kind": "sim", "model": "lt", "graph": "rmat", "scale": 21, "factor": 16, "p": "wc",
         "pick": "top", "seeds": 100, "trials": 1000, "mode": "device", "first_trial": 0},
        # scoring many candidate seed sets of uneven size and trial count in one call
        {"name": "batch_rmat_20", "kind": "batch", "model": "ic", "graph": "rmat", "scale": 20, "factor": 16,
         "p": "ur0.1", "items": 16, "size": 100, "trials": 1024, "counts": False},
        # choosing seeds: CELF, k = 10, 1,000 common trials on the random 7-regular graph
        {"name": "celf_rr_5k", "kind": "celf", "model": "ic", "graph": "rr", "n": 5000, "k": 7, "p": "wc",
         "picks": 10, "trials": 1000},
        # surrogate inference: every node's predicted activation for one seed set on a large graph
        {"name": "sur_forward_rmat_20", "kind": "forward", "graph": "rmat", "scale": 20, "factor": 16, "p": "wc",
         "seeds": 100},
        # one training example's loss and gradient at the size the surrogate is trained on
        {"name": "sur_grad_rmat_17", "kind": "grad", "graph": "rmat", "scale": 17, "factor": 16, "p": "wc",
         "seeds": 50},
        # screening: every node's first-order gain, as each round of the screened greedy asks for it
        {"name": "sur_scores_rmat_17", "kind": "scores", "graph": "rmat", "scale": 17, "factor": 16, "p": "wc",
         "seeds": 25},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_graph(rng, names, scales=(10, 21)):
    kind = rng.choice(names)
    if kind == "er":
        n = _log(rng, 300, 20000)
        return {"graph": "er", "n": n, "m": n * rng.randint(4, 10)}
    if kind == "ws":
        return {"graph": "ws", "n": _log(rng, 500, 40000), "k": 2 * rng.randint(2, 5)}
    if kind == "ba":
        return {"graph": "ba", "n": _log(rng, 2000, 100000), "k": rng.randint(2, 5)}
    if kind == "rr":
        return {"graph": "rr", "n": 2 * _log(rng, 100, 2500), "k": rng.randint(3, 7)}
    return {"graph": "rmat", "scale": rng.randint(*scales), "factor": rng.randint(8, 16)}


def draw(rng):
    kind = rng.choice(["sim", "sim", "sim", "sim", "batch", "celf", "forward", "grad", "scores", "onehop"])
    if kind == "sim":
        c = _draw_graph(rng, ["er", "ws", "ba", "rmat", "rmat"])
        model = rng.choice(["ic", "lt"])
        p = rng.choice(["wc", "ur1", "tv", "0.1", "0.01"] if model == "ic" else ["wc", "wc", "uneven"])
        if p == "uneven" and c["graph"] == "rmat":
            c["scale"] = min(c["scale"], 18)
        big = c["graph"] == "rmat" and c["scale"] > 17
        return {**c, "kind": "sim", "model": model, "p": p, "pick": rng.choice(["uniform", "top"]),
                "seeds": _log(rng, 1, 100), "trials": _log(rng, 64, 1000 if big or p == "uneven" else 10000),
                "mode": rng.choice(["host", "device", "graph"]), "first_trial": 64 * rng.randint(0, 1000)}
    if kind == "batch":
        c = _draw_graph(rng, ["ba", "rmat"], (12, 20))
        return {**c, "kind": "batch", "model": rng.choice(["ic", "ic", "lt"]) if c["graph"] == "ba" else "ic",
                "p": rng.choice(["wc", "tv"]) if c["graph"] == "ba" else "ur0.1", "items": rng.randint(2, 16),
                "size": _log(rng, 4, 100), "trials": _log(rng, 256, 1024), "counts": rng.random() < 0.5}
    if kind == "celf":
        c = _draw_graph(rng, ["rr"])
        return {**c, "kind": "celf", "model": rng.choice(["ic", "lt"]), "p": "wc", "picks": rng.randint(1, 10),
                "trials": _log(rng, 100, 1000)}
    c = _draw_graph(rng, ["ba", "rmat"], (12, 20 if kind == "forward" else 18))
    return {**c, "kind": kind, "p": "wc", "seeds": _log(rng, 1, 100)}


# ------------------------------------------------------------------------------------ inputs
def _graph(case, seed):
    kind = case["graph"]
    if kind == "er":
        return I.erdos_renyi_m(case["n"], case["m"], graph_seed=seed)
    if kind == "ws":
        return I.watts_strogatz(case["n"], case["k"], 0.007, graph_seed=seed)
    if kind == "ba":
        return I.barabasi_albert(case["n"], case["k"], graph_seed=seed)
    if kind == "rr":
        return I.random_regular(case["n"], case["k"], graph_seed=seed)
    return I.rmat(case["scale"], case["factor"] << case["scale"], graph_seed=seed)


def _ic_prob(case, g, seed):
    p = case["p"]
    if p == "wc":
        return I.ic_weighted_cascade(g)
    if p == "tv":
        return I.ic_trivalency(g, graph_seed=seed)
    if p.startswith("ur"):
        return I.ic_uniform_random(g, float(p[2:]), graph_seed=seed)
    return I.ic_uniform(g, float(p))


def _lt_weight(case, g, seed):
    return I.lt_random(g, 1.0, graph_seed=seed) if case["p"] == "uneven" else I.lt_weighted_cascade(g)


def _params(seed):
    # the initial network with the head's bias a trained one has: most nodes are predicted inactive
    w = I.surrogate_init(seed)
    w[-1] = -3.0
    return w


def _sur_inputs(case, seed):
    g = _graph(case, seed)
    prob = _ic_prob(case, g, seed)
    seeds = I.uniform_seeds(g.n, min(case["seeds"], g.n), seed)
    rng = np.random.Generator(np.random.Philox(seed + 77))
    y = (rng.random(g.n, dtype=np.float32) ** 4).astype(np.float32)  # activation frequencies: most near 0
    y[seeds] = 1.0
    return g, prob, seeds, y, _params(seed)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "key": seed % (1 << 31)}
    if kind in ("forward", "grad", "scores", "onehop"):
        g, prob, seeds, y, params = _sur_inputs(case, seed)
        s["G"] = P.cnd_graph_create(g.n, g.row_ptr, g.col, prob)
        s["sur"] = P.cnd_sur_create(s["G"], params)
        s["seeds"], s["y"] = seeds, y
        return s
    g = _graph(case, seed)
    prob = _ic_prob(case, g, seed) if case["model"] == "ic" else None
    weight = _lt_weight(case, g, seed) if case["model"] == "lt" else None
    s["G"] = P.cnd_graph_create(g.n, g.row_ptr, g.col, prob, weight)
    if kind == "sim":
        k = min(case["seeds"], g.n)
        seeds = I.top_degree_seeds(g, k) if case["pick"] == "top" else I.uniform_seeds(g.n, k, seed)
        s["seeds"] = seeds if case["mode"] == "host" else torch.from_numpy(seeds).cuda()
    elif kind == "batch":
        t = case["trials"]
        off, seeds, trials, keys = I.batch_items(g.n, case["items"], 1, case["size"], (t // 4, t, 4 * t),
                                                 graph_seed=seed)
        # the same total work whatever the seed: trial counts in turn instead of drawn
        trials = np.array([(t // 4, t, 4 * t)[i % 3] for i in range(case["items"])], dtype=np.int32)
        s.update(off=off, seeds=torch.from_numpy(seeds).cuda(), trials=trials, keys=keys + np.uint64(s["key"]))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "forward":
        yhat, spread = P.cnd_sur_forward(s["sur"], s["seeds"])
        return {"yhat": yhat, "spread": spread}
    if kind == "grad":
        loss, grad = P.cnd_sur_loss_grad(s["sur"], s["seeds"], s["y"])
        return {"loss": loss, "grad": grad}
    if kind == "scores":
        return {"scores": P.cnd_sur_scores(s["sur"], s["seeds"])}
    if kind == "onehop":
        return {"scores": P.cnd_sur_onehop(s["sur"], s["seeds"])}
    ic = case["model"] == "ic"
    if kind == "celf":
        f = P.cnd_ic_im_celf if ic else P.cnd_lt_im_celf
        r = f(s["G"], case["picks"], case["trials"], s["key"])
        return {"seeds": r.seeds, "f": r.f, "evaluations": r.evaluations, "edge_checks": r.edge_checks}
    if kind == "batch":
        f = P.cnd_ic_simulate_batch if ic else P.cnd_lt_simulate_batch
        r = f(s["G"], s["off"], s["seeds"], s["trials"], s["keys"], node_count=case["counts"], edge_checks=True)
        return {"spread": r.spread, "node_count": r.node_count, "edge_checks": r.edge_checks}
    if case["mode"] == "host":
        f = P.cnd_ic_simulate_ex if ic else P.cnd_lt_simulate_ex
        r = f(s["G"], s["seeds"], case["trials"], s["key"], first_trial=case["first_trial"])
        return {"spread": r.spread, "node_count": r.node_count}
    f = P.cnd_ic_simulate_ex if ic else P.cnd_lt_simulate_ex
    r = f(s["G"], s["seeds"], case["trials"], s["key"], first_trial=case["first_trial"], edge_checks=True,
          level_counts_len=64, graph=1 if case["mode"] == "graph" else 0)
    return {"spread": r.spread, "node_count": r.node_count, "edge_checks": r.edge_checks, "levels": r.level_counts}


# ------------------------------------------------------------------------------------ work
def _size(case):
    if case["graph"] == "er":
        return case["n"], case["m"]
    if case["graph"] == "rmat":
        return 1 << case["scale"], case["factor"] << case["scale"]  # a few per cent of the samples repeat
    if case["graph"] == "ba":
        return case["n"], 2 * case["k"] * (case["n"] - case["k"])
    return case["n"], case["n"] * case["k"]


def work(case):
    n, m = _size(case)
    graph = 4 * (n + 1) + 8 * m  # offsets; target and probability (or weight) of every edge
    kind = case["kind"]
    if kind == "sim":
        return {"bytes": graph + 4 * (case["seeds"] + case["trials"] + n), "flops": 0}
    if kind == "batch":
        t = case["trials"]
        trials = sum((t // 4, t, 4 * t)[i % 3] for i in range(case["items"]))
        return {"bytes": graph + 4 * trials + (4 * n * case["items"] if case["counts"] else 0), "flops": 0}
    if kind == "celf":
        return {"bytes": graph + 12 * case["picks"], "flops": 0}
    # the network: three dense maps of a node, two 64-wide sums over its in-edges (the first layer's
    # inputs are fixed but for the seeds); backward: dW and dX of each map, two sums over its out-edges
    dense = 2 * H * (2 * D0 + 2 * H + 2 * H) * n
    edges = 2 * 2 * H * m
    params = 4 * 18689
    if kind == "forward":
        return {"bytes": graph + params + 4 * n, "flops": dense + edges}
    if kind == "grad":
        return {"bytes": graph + 2 * params + 4 * n, "flops": 3 * dense + 2 * edges}
    if kind == "scores":
        return {"bytes": graph + params + 4 * n, "flops": 2 * dense + 2 * edges}
    return {"bytes": graph + params + 4 * n, "flops": dense + edges + 2 * m}


# ------------------------------------------------------------------------------------ 64 bits
def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


class _Net:
    """The network of include/cnd.h in fp64 on the GPU."""

    def __init__(self, g, prob, seeds, params):
        dev = "cuda"
        self.n = g.n
        self.src = torch.from_numpy(g.src().astype(np.int64)).to(dev)
        self.dst = torch.from_numpy(g.col.astype(np.int64)).to(dev)
        p = torch.from_numpy(prob).to(dev).double()
        self.q = torch.where(p == 1, p, torch.floor(p * 2.0**32).float().double() * 2.0**-32)
        self.s = torch.zeros(g.n, dtype=torch.float64, device=dev)
        self.s[torch.from_numpy(seeds.astype(np.int64)).to(dev)] = 1.0
        one = torch.ones(g.m, dtype=torch.float64, device=dev)
        degree = [torch.zeros(g.n, dtype=torch.float64, device=dev).index_add_(0, i, one) for i in (self.dst, self.src)]
        zero = torch.zeros(g.n, 13, dtype=torch.float64, device=dev)
        self.x = torch.cat([self.s[:, None], _bf16(torch.log1p(degree[0]))[:, None],
                            _bf16(torch.log1p(degree[1]))[:, None], zero], 1)
        self.flat = torch.from_numpy(params.astype(np.float64)).to(dev)

    def split(self, flat):
        out, at = [], 0
        for name, r, c in I.SURROGATE_SHAPES:
            w = flat[at:at + r * c]
            at += r * c
            out.append(w.reshape(r, c) if name[0] == "W" else w)
        return out

    def weights(self):
        # the matrices as the bf16 values the network multiplies with
        return torch.cat([(_bf16(w) if w.dim() == 2 else w).reshape(-1) for w in self.split(self.flat)])

    def sum_in(self, h):
        out = torch.zeros_like(h)
        step = 1 << 22
        for k in range(0, self.q.numel(), step):
            e = slice(k, k + step)
            out = out.index_add(0, self.dst[e], self.q[e, None] * h[self.src[e]])
        return out

    def forward(self, flat, x):
        w = self.split(flat)
        h = x
        for i in range(3):
            h = torch.relu(h @ w[3 * i].T + self.sum_in(h) @ w[3 * i + 1].T + w[3 * i + 2])
        return h @ w[9] + w[10]


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("forward", "grad", "scores", "onehop"):
        return None
    g, prob, seeds, y, params = _sur_inputs(case, seed)
    net = _Net(g, prob, seeds, params)
    flat, x = net.weights(), net.x
    if kind in ("forward", "onehop"):
        with torch.no_grad():
            yhat = net.s + (1 - net.s) * torch.sigmoid(net.forward(flat, x))
            if kind == "forward":
                return {"yhat": yhat.cpu().numpy(), "spread": float(yhat.sum())}
            hop = torch.zeros_like(yhat).index_add(0, net.src, net.q * (1 - yhat[net.dst]))
            return {"scores": ((1 - yhat) * (1 + hop)).cpu().numpy()}
    if kind == "grad":
        flat.requires_grad_(True)
        yhat = net.s + (1 - net.s) * torch.sigmoid(net.forward(flat, x))
        loss = (yhat - torch.from_numpy(y).cuda().double()).square().mean()
        loss.backward()
        return {"loss": float(loss), "grad": flat.grad.cpu().numpy()}
    x.requires_grad_(True)
    o = net.forward(flat, x)
    (net.s + (1 - net.s) * torch.sigmoid(o)).sum().backward()
    with torch.no_grad():
        direct = (1 - net.s) * (1 - torch.sigmoid(o))
        return {"scores": (direct + x.grad[:, 0]).cpu().numpy()}
