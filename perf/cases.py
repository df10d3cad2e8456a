"""The planner's work, as a user's program has it done, case by case.

A case is a dict of plain values.  `kind` says what is called:

  plan    pp_plan_run on an instance that is kept (an epoch's planning)
  epoch   the same from new host arrays: pp_instance_create, plan, destroy
  replan  pp_replan: the epoch update against an incumbent placement
  update  one coordinate update of a batch of workers against the others'
          targets: pp_marginals, pp_tree_dp, pp_traceback (an external
          scheduler, or a program that refines a placement by itself)
  dp      pp_tree_dp + pp_traceback on the caller's own profits
  score   pp_objective and pp_marginals of a batch of placements

`tree` is the family of the prefix tree (the three of the synthetic
workloads), n chunks, W workers, k slots per worker, chunk weights 1..wmax,
`source` whether transfer costs depend on the source worker.  Sizes are those
of the repository's workloads (2,000 to 200,000 chunks, 4 to 32 workers,
budgets 77 to 8,192, 1 to 16 starts, up to 6 sweeps), odd ones among them.
Everything is whole numbers, so every output is compared bit for bit.
"""
import math

import numpy as np
import torch

from paper_2608_01655_gb300 import binding as pp
from paper_2608_01655_gb300 import workloads as wl


def _case(name, kind, tree, n, W, k, wmax=1, source=False, starts=1, rounds=0, batch=1):
    return dict(name=name, kind=kind, tree=tree, n=n, W=W, k=k, wmax=wmax, source=source, starts=starts,
                rounds=rounds, batch=batch)


def listed():
    return [
        # one start, few workers: the smallest plan, all latency
        _case("plan-tiny", "plan", "grown", 2000, 4, 256, starts=1, rounds=3),
        # retrieval-augmented serving, requester-side costs with the safeguards
        _case("plan-rag", "plan", "rag", 10_000, 8, 1024, starts=4, rounds=5),
        # the same family with source-dependent costs and chunks of two sizes
        _case("plan-source", "plan", "rag", 20_000, 16, 2048, wmax=2, source=True, starts=8, rounds=5),
        # the paper-scale plan: multi-turn conversations under shared prefixes
        _case("plan-paper", "plan", "mixed", 50_000, 16, 4096, source=True, starts=16, rounds=6),
        # a large cluster's tree, weighted chunks, a bounded number of starts
        _case("plan-large", "plan", "mixed", 200_000, 16, 8192, wmax=4, source=True, starts=2, rounds=1),
        # chunks of up to nine slots, odd sizes
        _case("plan-heavy", "plan", "grown", 3001, 3, 1500, wmax=9, starts=2, rounds=2),
        # an epoch begins: demand and costs arrive on the host
        _case("epoch-rag", "epoch", "rag", 9973, 8, 1000, source=True, starts=4, rounds=3),
        # an epoch ends: keep the incumbent or move
        _case("replan-rag", "replan", "rag", 10_000, 8, 1024, starts=4, rounds=5),
        # one worker refined alone, ragged sizes
        _case("update-one", "update", "mixed", 20_011, 12, 2001, source=True, batch=1),
        # every worker's best response at the paper's scale, one batch
        _case("update-batch", "update", "mixed", 50_000, 16, 4096, source=True, batch=16),
        # the smallest call: one small tree
        _case("dp-small", "dp", "grown", 501, 1, 77, batch=1),
        # scoring of candidate placements
        _case("score", "score", "rag", 20_000, 16, 2048, source=True, batch=8),
    ]


def draw(rng):
    def size(lo, hi):                     # over the logarithm, odd values among them
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plan", "plan", "plan", "epoch", "replan", "update", "update", "dp", "dp", "score"])
    tree = rng.choice(["grown", "rag", "mixed"])
    source = rng.random() < 0.5 and kind != "dp"
    wmax = rng.choice([1, 1, 1, 2, 4])
    if kind in ("plan", "epoch", "replan"):
        n = size(2000, 50_000)
        W = rng.choice([3, 4, 8, 11, 16])
        starts, rounds, batch = rng.randint(1, 16 if n <= 20_000 else 8), rng.randint(0, 6 if n <= 20_000 else 3), 1
    else:
        n = size(500, 50_000)
        W = 1 if kind == "dp" else rng.choice([2, 7, 12, 16])
        starts, rounds, batch = 1, 0, rng.randint(1, 16)
    if n <= 5000 and rng.random() < 0.25:
        wmax = rng.randint(5, 9)
    k = min(size(77, 8192), max(8, n // 3))
    if wmax > 4:
        k = min(k, 2000)
    c = _case("", kind, tree, n, W, k, wmax, source, starts, rounds, batch)
    del c["name"]
    return c


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _tree(rng, case):
    n = case["n"]
    if case["tree"] == "grown":
        return wl._grow_random(rng, n, min(8, n), 24, lambda r: int(r.geometric(0.5)))
    if case["tree"] == "rag":
        return wl._rag_tree(rng, n, n_docs=max(50, min(2000, n // 5)))
    return wl._mixed_tree(rng, n)


def _host(case, seed):
    """The arrays of an instance: tree, weights, demand, costs, budgets."""
    rng = np.random.default_rng(seed)
    n, W = case["n"], case["W"]
    parent = _tree(rng, case)
    weight = rng.integers(1, case["wmax"] + 1, size=n).astype(np.int32)
    classes = [m % 3 for m in range(W)]
    depth = np.zeros(n, np.int64)
    tokens = np.zeros(n, np.int64)                       # prefix length before each chunk
    par, wt = parent.tolist(), weight.tolist()
    d, t = depth.tolist(), tokens.tolist()
    for v in range(n):                                   # parents precede children
        p = par[v]
        d[v] = 1 if p < 0 else d[p] + 1
        t[v] = 0 if p < 0 else t[p] + wt[p] * wl.CHUNK_TOKENS
    depth, tokens = np.asarray(d, np.int64), np.asarray(t, np.int64)
    counts = wl._leaf_demand(rng, parent, W, 0.9 if case["tree"] == "rag" else 1.0, case["tree"] == "mixed")
    demand = wl._propagate_up(parent, counts, depth)
    recompute = wl._recompute(weight, tokens, classes)
    if case["source"]:
        transfer = wl._transfer_source(rng, weight, W, 0.5)
    else:
        transfer = wl._transfer_requester(rng, weight, W, 0.3)
    budget = np.full(W, case["k"], np.int32)
    return dict(parent=parent, weight=weight, demand=demand, recompute=recompute,
                transfer=np.ascontiguousarray(transfer), mode=int(case["source"]), budget=budget)


def _instance(h):
    return pp.Instance(h["parent"], h["weight"], h["demand"], h["recompute"], h["transfer"], h["mode"], h["budget"])


def _placement(rng, h, W, frac):
    """Parent-closed, within-budget targets, the popular chunks first: what a
    refinement in progress holds."""
    n = len(h["parent"])
    par = h["parent"].tolist()
    out = np.zeros((W, n), np.uint8)
    for m in range(W):
        pop = np.log1p(h["demand"][m]) * rng.uniform(0.5, 1.5, n)
        want = (pop >= np.quantile(pop, 1.0 - frac)).tolist()
        keep = [False] * n
        for v in range(n):
            keep[v] = want[v] and (par[v] < 0 or keep[par[v]])
        got = np.asarray(keep)
        used = np.cumsum(np.where(got, h["weight"], 0))
        out[m] = got & (used <= h["budget"][m])
    return out


def _masks(placement):
    m = np.zeros(placement.shape[-1], np.uint32)
    for x in range(placement.shape[0]):
        m |= placement[x].astype(np.uint32) << np.uint32(x)
    return m


def _inputs(case, seed):
    """All host inputs of a case."""
    h = _host(case, seed)
    rng = np.random.default_rng(seed + 1_000_003)
    n, W, B, kind = case["n"], case["W"], case["batch"], case["kind"]
    if kind == "replan":
        h["incumbent"] = _placement(rng, h, W, 0.1)
    if kind in ("update", "score"):
        h["workers"] = ((np.arange(B) + int(rng.integers(W))) % W).astype(np.int32)
        h["placements"] = np.stack([_placement(rng, h, W, f) for f in rng.uniform(0.02, 0.12, 1 if kind == "update" else B)])
    if kind == "update":
        h["placements"] = np.repeat(h["placements"], B, axis=0)
    if kind == "dp":
        # a caller's own scores: saved time per chunk, a fifth of the chunks
        # already covered elsewhere and worth nothing here
        h["profits"] = np.stack([h["demand"][0] * h["recompute"][0] * (rng.random(n) < 0.8) for _ in range(B)])
    if kind in ("update", "dp"):
        k = case["k"]
        lo = k - k // 8 if B > 1 else k
        h["k_item"] = rng.integers(lo, k + 1, size=B).astype(np.int32)
    return h


def prepare(case, seed):
    h = _inputs(case, seed)
    s = dict(case=case)
    kind, B, n = case["kind"], case["batch"], case["n"]
    if kind == "epoch":
        s["host"] = h
        return s
    s["inst"] = _instance(h)
    if kind == "replan":
        s["incumbent"] = h["incumbent"]
    if kind in ("update", "score"):
        s["workers"] = torch.from_numpy(h["workers"]).cuda()
        s["masks"] = torch.from_numpy(np.stack([_masks(p) for p in h["placements"]]).view(np.int32)).cuda()
        s["profit"] = torch.zeros((B, n), dtype=torch.int64, device="cuda")
    if kind == "score":
        s["placements"] = torch.from_numpy(h["placements"]).cuda()
        s["objective"] = torch.zeros(B, dtype=torch.int64, device="cuda")
    if kind == "dp":
        s["profit"] = torch.from_numpy(h["profits"]).cuda()
    if kind in ("update", "dp"):
        s["k"] = torch.from_numpy(h["k_item"]).cuda()
        s["best"] = torch.zeros(B, dtype=torch.int64, device="cuda")
        s["bits"] = torch.zeros(pp.pp_dp_bits_size(s["inst"], B, case["k"]) // 4, dtype=torch.int32, device="cuda")
        s["chosen"] = torch.zeros((B, n), dtype=torch.uint8, device="cuda")
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def _plan_outputs(r):
    return [r.placement, r.objective, r.best_start, r.per_start_objective, r.per_start_sweeps,
            r.per_start_accepted, r.orders]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "epoch":
        inst = _instance(state["host"])
        out = _plan_outputs(pp.pp_plan_run(inst, case["starts"], None, case["rounds"]))
        inst.close()
        return out
    inst = state["inst"]
    if kind == "plan":
        return _plan_outputs(pp.pp_plan_run(inst, case["starts"], None, case["rounds"]))
    if kind == "replan":
        r = pp.pp_replan(inst, state["incumbent"], case["starts"], case["rounds"], wl.REQUESTS_PER_EPOCH,
                         10 * wl.REQUESTS_PER_EPOCH)
        return [r.placement, r.incumbent_objective, r.new_objective, r.materialization_cost,
                r.break_even_requests, r.adopted]
    if kind == "score":
        pp.pp_objective(inst, state["placements"], state["objective"])
        pp.pp_marginals(inst, state["workers"], state["masks"], state["profit"])
        return [state["objective"], state["profit"]]
    out = []
    if kind == "update":
        pp.pp_marginals(inst, state["workers"], state["masks"], state["profit"])
        out = [state["profit"]]
    pp.pp_tree_dp(inst, state["profit"], state["k"], case["k"], state["best"], state["bits"])
    pp.pp_traceback(inst, state["bits"], state["k"], case["k"], state["chosen"])
    return out + [state["best"], state["chosen"]]


def work(case):
    """Each input read once, each output written once; the additions and
    comparisons of the marginals (W per chunk and update) and at least one per
    chunk of an exact update."""
    n, W, B, kind = case["n"], case["W"], case["batch"], case["kind"]
    table = 8 * n * (W * W if case["source"] else 2 * W + 1)
    if kind in ("plan", "epoch", "replan"):
        updates = case["starts"] * W * (1 + min(case["rounds"], 1)) + (0 if case["source"] else 3 * W)
        host = table + 16 * W * n if kind == "epoch" else 0
        inc = W * n if kind == "replan" else 0
        return dict(bytes=host + table + 8 * n + inc + W * n, flops=updates * n * (2 * W + 1))
    per_item = 8 * n                                        # profits
    if kind == "dp":
        return dict(bytes=B * (per_item + n) + 8 * n, flops=2 * B * n)
    if kind == "update":
        return dict(bytes=table + B * (4 * n + per_item + n) + 8 * n, flops=B * n * (2 * W + 2))
    return dict(bytes=table + B * (W * n + 4 * n + per_item), flops=B * n * 4 * W)


def tolerance(case):
    return "exact"                                          # integers throughout


# ----------------------------------------------------------------------------
# the same in plain numpy (Algorithm 1 and Eq. 2-10 from their definitions)
# ----------------------------------------------------------------------------
def _preorder(parent):
    n = len(parent)
    kids = [[] for _ in range(n)]
    roots = []
    for v, p in enumerate(parent.tolist()):
        (roots if p < 0 else kids[p]).append(v)
    order, end, stack = [], [0] * n, list(reversed(roots))
    while stack:
        v = stack.pop()
        if v < 0:
            end[~v] = len(order)
            continue
        order.append(v)
        stack.append(~v)
        stack.extend(reversed(kids[v]))
    order = np.asarray(order, np.int64)
    return order, np.asarray(end, np.int64)[order]


def _rooted_dp(order, nxt, weight, profit, k):
    """Eq. 9 with backtracking: take only when strictly better."""
    n = len(order)
    w, p, nx = weight[order].tolist(), profit[order].tolist(), nxt.tolist()
    D = [None] * (n + 1)
    D[n] = np.zeros(k + 1, np.int64)
    take = np.zeros((n, k + 1), bool)
    for i in range(n - 1, -1, -1):
        row = D[nx[i]].copy()
        c = w[i]
        if c <= k:
            t = D[i + 1][:k + 1 - c] + p[i]
            take[i, c:] = t > row[c:]
            np.maximum(row[c:], t, out=row[c:])
        D[i] = row
    chosen = np.zeros(n, np.uint8)
    i, j = 0, k
    while i < n and j > 0:
        if take[i, j]:
            chosen[order[i]] = 1
            j -= w[i]
            i += 1
        else:
            i = nx[i]
    return int(D[0][k]), chosen


class _Reference:
    def __init__(self, h):
        self.h, self.W, self.n = h, len(h["budget"]), len(h["parent"])
        self.order, self.nxt = _preorder(h["parent"])
        lam, w, f = h["demand"], h["recompute"], h["transfer"]
        if h["mode"] == 0:
            self.a = lam * np.minimum(w, f)
            self.own = lam * np.maximum(w - f, 0)
            self.delta = self.own.sum(0)
        else:
            q = np.maximum(w[None] - f, 0)                  # [source][requester][chunk]
            for m in range(self.W):
                q[m, m] = w[m]
            self.g = lam[None] * q

    def marginal(self, h, pl):
        others = pl.astype(bool).copy()
        others[h] = False
        if self.h["mode"] == 0:
            return self.a[h] + np.where(others.any(0), 0, self.delta)
        v = np.where(others[:, None, :], self.g, 0).max(0)
        return np.maximum(self.g[h] - v, 0).sum(0)

    def objective(self, pl):
        on = pl.astype(bool)
        if self.h["mode"] == 0:
            return int((self.a * on).sum() + (self.delta * on.any(0)).sum())
        return int(np.where(on[:, None, :], self.g, 0).max(0).sum())

    def dp(self, profit, k):
        return _rooted_dp(self.order, self.nxt, self.h["weight"], profit, int(k))

    def orders(self, S):
        W = self.W
        out = np.tile(np.arange(W, dtype=np.int32), (S, 1))
        if S == 1:
            return out
        none = np.zeros((W, self.n), np.uint8)
        score = [self.dp(self.marginal(m, none), self.h["budget"][m])[0] for m in range(W)]
        out[0] = sorted(range(W), key=lambda m: (-score[m], m))
        out[1] = out[0][::-1]
        mask = (1 << 64) - 1
        for s in range(2, S):
            x = s
            for i in range(W - 1, 0, -1):                   # Fisher-Yates driven by SplitMix64
                x = (x + 0x9E3779B97F4A7C15) & mask
                z = x
                z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
                z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
                j = (z ^ (z >> 31)) % (i + 1)
                out[s, [i, j]] = out[s, [j, i]]
        return out

    def start(self, order, R):
        pl = np.zeros((self.W, self.n), np.uint8)
        sweeps = accepted = 0
        for r in range(R + 1):
            got = 0
            for m in order.tolist():
                p = self.marginal(m, pl)
                best, ch = self.dp(p, self.h["budget"][m])
                if r == 0 or best > int(p[pl[m].astype(bool)].sum()):
                    pl[m] = ch
                    got += r > 0
            sweeps += r > 0
            accepted += got
            if r > 0 and got == 0:
                break
        return pl, self.objective(pl), sweeps, accepted

    def safeguards(self):
        out, lam = [], self.h["demand"]
        for profit in (self.a + self.own, lam):
            out.append(np.stack([self.dp(profit[m], self.h["budget"][m])[1] for m in range(self.W)]))
        pl = np.zeros((self.W, self.n), np.uint8)
        for m in range(self.W):
            p = self.a[m] + np.where(pl[:m].any(0), 0, self.own[m])
            pl[m] = self.dp(p, self.h["budget"][m])[1]
        return out + [pl]

    def plan(self, S, R):
        orders = self.orders(S)
        starts = [self.start(o, R) for o in orders]
        cand = [(s[1], s[0]) for s in starts]
        if self.h["mode"] == 0:
            cand += [(self.objective(pl), pl) for pl in self.safeguards()]
        best = max(range(len(cand)), key=lambda c: (cand[c][0], -c))
        return [cand[best][1], cand[best][0], best, np.asarray([s[1] for s in starts], np.int64),
                np.asarray([s[2] for s in starts], np.int32), np.asarray([s[3] for s in starts], np.int32), orders]


def _seconds(case):
    """What the numpy reference takes, roughly."""
    n, k = case["n"], case["k"]
    dps = case["batch"]
    if case["kind"] == "score":
        return 1.0
    if case["kind"] in ("plan", "epoch", "replan"):
        dps = case["W"] * (1 + case["starts"] * (1 + case["rounds"]) + (0 if case["source"] else 3))
    return dps * n * (15e-6 + 5e-9 * k)


def exact(case, seed):
    if _seconds(case) > 15 or case["n"] * case["k"] > 40_000_000:
        return None
    h = _inputs(case, seed)
    ref = _Reference(h)
    kind = case["kind"]
    if kind in ("plan", "epoch"):
        return ref.plan(case["starts"], case["rounds"])
    if kind == "replan":
        pl, new = ref.plan(case["starts"], case["rounds"])[:2]
        old = h["incumbent"]
        was = ref.objective(old)
        cost = 0
        for m in range(ref.W):
            fetch = np.full(ref.n, np.iinfo(np.int64).max)
            for x in range(ref.W):
                f = h["transfer"][x, m] if h["mode"] else h["transfer"][m]
                if x != m:
                    fetch = np.where(old[x].astype(bool), np.minimum(fetch, f), fetch)
            added = pl[m].astype(bool) & ~old[m].astype(bool)
            cost += int(np.minimum(h["recompute"][m], fetch)[added].sum())
        gain, E = new - was, wl.REQUESTS_PER_EPOCH
        adopted = gain > 0 and gain * 10 * E > cost * E
        return [pl if adopted else old, was, new, cost, -(-cost * E // gain) if gain > 0 else -1, adopted]
    if kind == "score":
        return [np.asarray([ref.objective(p) for p in h["placements"]], np.int64),
                np.stack([ref.marginal(int(w), p) for w, p in zip(h["workers"], h["placements"])])]
    if kind == "update":
        profits = np.stack([ref.marginal(int(w), p) for w, p in zip(h["workers"], h["placements"])])
    else:
        profits = h["profits"]
    got = [ref.dp(profits[b], h["k_item"][b]) for b in range(case["batch"])]
    out = [profits] if kind == "update" else []
    return out + [np.asarray([g[0] for g in got], np.int64), np.stack([g[1] for g in got])]
