"""Performance cases of the MaxSAT engine: the calls its users make, over the
sizes its configurations, tests and benchmark use.

A case is one call pattern ("kind") on one instance family:

  step     Solver.step(K), optionally followed by the tensor-core evaluation
           of the rounded x, then the updated x read back: the optimizer loop
           of a long run, which looks at its state every K steps
  solve    Solver.solve (Algorithm 1 by chunks, with its best-cost trace) and
           the best assignments
  oneshot  host arrays in, answer out: create a Solver, step it, read the
           costs and the best assignments, close it
  grad     msat_loss forward and backward through autograd, for callers that
           run their own optimizer on x
  eval     Solver.evaluate of a batch of given assignments, clause-list or
           tensor-core backend
  serve    a burst of requests through the continuous-batching Server

Families: uniform random k-SAT ("ksat"), weighted Zipf clauses of 2 to 20
literals ("zipf": skewed occurrence counts, weights 1..1000), the ordering
principle ("gt") and pigeonhole ("php") formulas.  Instances are drawn on the
GPU from the case's seed and handed over as the host arrays Solver takes.
"""
import math

import numpy as np
import torch

import paper_2402_03640_gb300 as msat

# clause / variable ratio at the satisfiability threshold of random k-SAT,
# where the serving stream and the benchmark's instances lie
RATIO = {3: 4.3, 4: 10.0, 5: 21.3}


def listed():
    return [
        # the oracle-sized instance: one small formula, many steps (latency of a step)
        dict(name="step_n50_b1", kind="step", family="ksat", n=50, m=215, k=3, B=1, steps=500, dense=False),
        # a small formula with several restarts, as most serving requests are
        dict(name="step_n301_b16", kind="step", family="ksat", n=301, m=1290, k=3, B=16, steps=200, dense=False),
        # batched restarts of a medium formula, each look at the state with the
        # tensor-core evaluation of the rounded batch
        dict(name="step_n5000_b256_dense", kind="step", family="ksat", n=5000, m=21500, k=3, B=256, steps=50,
             dense=True),
        # the largest configuration: a million variables, 16 restarts
        dict(name="step_n1e6_b16", kind="step", family="ksat", n=1000000, m=4300000, k=3, B=16, steps=100,
             dense=False),
        # weighted, skewed, clauses of different lengths, a single restart
        dict(name="step_zipf_b1", kind="step", family="zipf", n=200000, m=1000000, k=0, B=1, steps=200, dense=False),
        # a structured formula under the time-limited solver, 8 restarts
        dict(name="solve_gt30_b8", kind="solve", family="gt", n=930, m=27466, k=30, B=8, steps=512),
        # one answer from host arrays: creation, 20 steps, costs, best assignments
        dict(name="oneshot_n1e6_b16", kind="oneshot", family="ksat", n=1000000, m=4300000, k=3, B=16, steps=20),
        # the differentiable layer at its test size: small calls
        dict(name="grad_n1000_b8", kind="grad", family="ksat", n=1000, m=4300, k=3, B=8),
        # the differentiable layer on longer clauses and an odd size
        dict(name="grad_k5_n30011_b64", kind="grad", family="ksat", n=30011, m=639234, k=5, B=64),
        # scoring a given batch of assignments on the tensor cores
        dict(name="eval_dense_n5000_nb256", kind="eval", family="ksat", n=5000, m=21500, k=3, nb=256,
             backend="dense"),
        # the same from the clause list: a weighted instance far too large to
        # be dense, a batch that is no multiple of the warp
        dict(name="eval_sparse_zipf_nb100", kind="eval", family="zipf", n=200000, m=1000000, k=0, nb=100,
             backend="sparse"),
        # a burst of k in {3, 4, 5} requests, n in [100, 50000], 8 restarts each
        dict(name="serve_32_b8", kind="serve", family="ksat", requests=32, n_lo=100, n_hi=50000, B=8, steps=250),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "solve", "oneshot", "grad", "eval", "eval", "serve"])
    if kind == "serve":
        return dict(kind="serve", family="ksat", requests=rng.randint(8, 32), n_lo=100, n_hi=_logint(rng, 1000, 50000),
                    B=8, steps=_logint(rng, 50, 250))
    if kind == "solve":
        k = rng.randint(10, 30)
        if rng.random() < 0.5:
            return dict(kind="solve", family="gt", n=(k + 1) * k, m=_gt_clauses(k), k=k,
                        B=8, steps=64 * rng.randint(2, 8))
        return dict(kind="solve", family="php", n=k * (k + 1), m=k + 1 + k * (k * (k + 1) // 2), k=k,
                    B=8, steps=64 * rng.randint(2, 8))
    family = rng.choice(["ksat", "ksat", "zipf"])
    k = rng.choice([3, 3, 4, 5]) if family == "ksat" else 0
    if kind == "eval":
        backend = rng.choice(["dense", "sparse"])
        n = _logint(rng, 300, 6000 if backend == "dense" else 200000)
        nb = _logint(rng, 1, 300)
    else:
        n = _logint(rng, 50, 1000000)
        nb = 0
    m = int(n * (RATIO[k] if k else 5.0) * rng.uniform(0.93, 1.07))
    if m * max(k, 4) > 12900000:  # no more clause literals than the largest listed case
        n = int(n * 12900000 / (m * max(k, 4)))
        m = int(n * (RATIO[k] if k else 5.0))
    if kind == "eval":
        return dict(kind="eval", family=family, n=n, m=m, k=k, nb=nb, backend=backend)
    # restarts: as many as keep a step at or below the largest listed case's
    most = max(0, min(8, int(math.log2(max(1.0, 12900000 * 16 / (m * max(k, 4)))))))
    B = 1 << rng.randint(0, most)
    if kind == "grad":
        return dict(kind="grad", family=family, n=n, m=m, k=k, B=B)
    if kind == "oneshot":
        return dict(kind="oneshot", family=family, n=n, m=m, k=k, B=B, steps=_logint(rng, 5, 20))
    return dict(kind="step", family=family, n=n, m=m, k=k, B=B, steps=_logint(rng, 20, 100),
                dense=bool(n <= 6000 and rng.random() < 0.5))


# ------------------------------------------------------------ instances

def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + salt)


def _ksat_vars(n, m, k, gen):
    """m rows of k distinct variables, uniform: the p-th draw is uniform over
    the n - p values not taken by the row's earlier draws."""
    rows = torch.empty((m, k), dtype=torch.int64, device="cuda")
    taken = None
    for p in range(k):
        v = torch.randint(0, n - p, (m,), device="cuda", generator=gen)
        for q in range(p):  # earlier draws in ascending order
            v += (v >= taken[:, q]).to(torch.int64)
        rows[:, p] = v
        taken = torch.sort(rows[:, :p + 1], dim=1).values
    return rows


def _zipf(n, m, gen):
    """Clause lengths 2 + Geom(1/3) up to 20 and distinct Zipf(1.2) variables."""
    u = torch.rand(m, device="cuda", generator=gen, dtype=torch.float64)
    top = 1.0 - (2.0 / 3.0) ** 19
    lens = 2 + torch.clamp((torch.log1p(-u * top) / math.log(2.0 / 3.0)).floor().to(torch.int64), 0, 18)
    lens = torch.minimum(lens, torch.full_like(lens, max(2, n // 2)))
    cdf = torch.cumsum(torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** -1.2, 0)
    perm = torch.randperm(n, device="cuda", generator=gen)
    V = torch.full((m, 20), -1, dtype=torch.int64, device="cuda")
    for p in range(20):
        todo = torch.nonzero(lens > p).reshape(-1)
        for _ in range(4096):
            if todo.numel() == 0:
                break
            r = torch.rand(todo.numel(), device="cuda", generator=gen, dtype=torch.float64) * cdf[-1]
            v = perm[torch.clamp(torch.searchsorted(cdf, r, right=True), max=n - 1)]
            V[todo, p] = v
            clash = (V[todo, :p] == v[:, None]).any(dim=1) if p else torch.zeros(todo.numel(), dtype=torch.bool,
                                                                                 device="cuda")
            todo = todo[clash]
    return lens, V[V >= 0]


def _gt_clauses(size):
    N = size + 1
    return N * (N - 1) // 2 + N * (N - 1) * (N - 2) + N


def _gt(size):
    """The ordering principle on size + 1 elements: antisymmetry,
    transitivity, every element has a predecessor."""
    N = size + 1
    idx = np.cumsum(~np.eye(N, dtype=bool).reshape(-1)).reshape(N, N)  # x(a, b), a != b
    a, b = np.triu_indices(N, 1)
    two = np.stack([-idx[a, b], -idx[b, a]], 1)
    a, b, c = (v.reshape(-1) for v in np.meshgrid(np.arange(N), np.arange(N), np.arange(N), indexing="ij"))
    ok = (a != b) & (b != c) & (a != c)
    a, b, c = a[ok], b[ok], c[ok]
    three = np.stack([-idx[a, b], -idx[b, c], idx[a, c]], 1)
    last = np.stack([idx[np.arange(N) != e, e] for e in range(N)])
    return [two, three, last]


def _php(h):
    """h + 1 pigeons, h holes."""
    p = np.arange(1, (h + 1) * h + 1).reshape(h + 1, h)
    i, j = np.triu_indices(h + 1, 1)
    pairs = np.stack([-p[i], -p[j]], 2).transpose(1, 0, 2).reshape(-1, 2)
    return [p, pairs]


class _Cnf:
    def __init__(self, n, off, lits, weights=None):
        self.n, self.off, self.lits, self.weights = n, off, lits, weights


def _instance(case, seed):
    """The case's clause set as host arrays (structured families are fixed)."""
    n, m = case["n"], case["m"]
    if case["family"] in ("gt", "php"):
        parts = _gt(case["k"]) if case["family"] == "gt" else _php(case["k"])
        lens = np.concatenate([np.full(len(p), p.shape[1], np.int64) for p in parts])
        off = np.concatenate([np.zeros(1, np.int64), np.cumsum(lens)])
        return _Cnf(n, off, np.concatenate([p.reshape(-1) for p in parts]).astype(np.int32))
    gen = _gen(seed, 1)
    if case["family"] == "zipf":
        lens, V = _zipf(n, m, gen)
        w = torch.randint(1, 1001, (m,), device="cuda", generator=gen).cpu().numpy()
        off = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(lens, 0)]).cpu().numpy()
    else:
        V = _ksat_vars(n, m, case["k"], gen).reshape(-1)
        w = None
        off = np.arange(m + 1, dtype=np.int64) * case["k"]
    sign = torch.randint(0, 2, (V.numel(),), device="cuda", generator=gen) * 2 - 1
    return _Cnf(n, off, ((V + 1) * sign).to(torch.int32).cpu().numpy(), w)


def _request_sizes(case):
    """(k, n, m) of the burst: k in {3, 4, 5} in turn, n spread evenly over the
    logarithm of its range, m / n around the threshold."""
    out = []
    for r in range(case["requests"]):
        k = 3 + (2 * r) % 3
        n = int(math.exp(math.log(case["n_lo"]) + (r + 0.5) / case["requests"] * math.log(case["n_hi"] / case["n_lo"])))
        out.append((k, n, int(n * RATIO[k] * (0.93 + 0.14 * ((7 * r) % 11) / 10))))
    return out


def _requests(case, seed):
    """The burst's clause sets, in an order of the seed's."""
    out = [_instance(dict(family="ksat", n=n, m=m, k=k), seed * 1009 + r)
           for r, (k, n, m) in enumerate(_request_sizes(case))]
    return [out[i] for i in np.random.RandomState(seed % 2 ** 32).permutation(len(out))]


# ---------------------------------------------------------------- cases

def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return dict(case=case, seed=seed, cnfs=_requests(case, seed), server=msat.Server(restarts=case["B"]))
    cnf = _instance(case, seed)
    st = dict(case=case, seed=seed, cnf=cnf)
    if kind == "oneshot":
        return st
    st["solver"] = msat.Solver.from_cnf(cnf, restarts=case.get("B", 1), seed_x=seed + 1)
    if kind == "grad":
        st["x"] = _grad_x(case, seed).requires_grad_(True)
    if kind == "eval":
        st["assign"] = _assignments(case, seed)
    return st


def _grad_x(case, seed):
    return torch.rand((case["n"], case["B"]), device="cuda", generator=_gen(seed, 2)) * 2 - 1


def _assignments(case, seed):
    a = torch.randint(0, 2, (case["n"], case["nb"]), device="cuda", generator=_gen(seed, 3), dtype=torch.int8)
    return a * 2 - 1


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        s = state["solver"]
        loss, cost = s.step(case["steps"])
        out = dict(loss=loss, cost=cost, x=s.x())
        if case["dense"]:
            out["dense_cost"] = s.evaluate_x("dense")
        return out
    if kind == "solve":
        s = state["solver"]
        r = s.solve(case["steps"], chunk=64)
        assign, best = s.best()
        return dict(steps=r["steps"], trace=r["trace_best_cost"], assign=assign, best=best, x=s.x())
    if kind == "oneshot":
        with msat.Solver.from_cnf(state["cnf"], restarts=case["B"], seed_x=state["seed"] + 1) as s:
            loss, cost = s.step(case["steps"])
            assign, best = s.best()
        return dict(loss=loss, cost=cost, assign=assign, best=best)
    if kind == "grad":
        x = state["x"]
        x.grad = None
        loss = msat.msat_loss(x, state["solver"])
        loss.sum().backward()
        return dict(loss=loss.detach(), grad=x.grad)
    if kind == "eval":
        return dict(cost=state["solver"].evaluate(state["assign"], case["backend"]))
    srv = state["server"]
    tickets = [srv.submit(c, case["steps"], seed_x=state["seed"] + i) for i, c in enumerate(state["cnfs"])]
    res = [srv.wait(t) for t in tickets]
    return dict(best=np.stack([r["best_costs"] for r in res]), assign=np.concatenate([r["assignment"] for r in res]))


def _mean_literals(case):
    return case["k"] if case["family"] == "ksat" else 4.0 if case["family"] == "zipf" else 3.0


def _step_work(n, m, nnz, B, steps, weighted=False):
    """Bytes and flops of `steps` optimizer steps: the clause lists and their
    transpose, x, both moments and tanh(x) read and written.  A working set
    that fits the chip's caches has to cross HBM once a call, a larger one
    once a step.  Per literal and restart: an addition each in the clause and
    the variable pass and a product; per variable and restart about 40
    operations of Adam and tanh."""
    once = 8 * nnz + 4 * (n + 1) + (8 * m if weighted else 0) + 32 * n * B + m * B / 4
    fits = once + 4 * m * B < 100e6
    return once * (1 if fits else max(1, steps)), float(steps) * (3 * nnz * B + 40 * n * B)


def work(case):
    kind = case["kind"]
    if kind == "serve":
        b = f = 0.0
        for k, n, m in _request_sizes(case):
            x, y = _step_work(n, m, m * k, case["B"], case["steps"])
            b, f = b + x, f + y
        return dict(bytes=b, flops=f)
    n, m, nnz = case["n"], case["m"], case["m"] * _mean_literals(case)
    weighted = case["family"] == "zipf"
    if kind == "eval":
        if case["backend"] == "dense":  # the product of the clause matrix (4 bits an entry) and the batch
            return dict(bytes=m * n / 2 + n * case["nb"] + 8 * m + 8 * case["nb"], flops=2.0 * m * n * case["nb"])
        return dict(bytes=4 * nnz + n * case["nb"] + (8 * m if weighted else 0), flops=2.0 * nnz * case["nb"])
    if kind == "grad":
        b, f = _step_work(n, m, nnz, case["B"], 1, weighted)
        return dict(bytes=8 * nnz + 4 * (n + 1) + 8 * n * case["B"] + m * case["B"] / 4, flops=f)
    b, f = _step_work(n, m, nnz, case["B"], case["steps"], weighted)
    if kind == "oneshot":
        b += 12 * nnz + 8 * m + n * case["B"]
    if case.get("dense"):
        b += m * n / 2 + n * case["B"] / 2
        f += 2.0 * m * n * case["B"]
    return dict(bytes=b, flops=f)


# ------------------------------------------------------ 64-bit reference

def _start_x(n, B, seed):
    """The random start: x[i][b] = k 2^-23 - 1, k the top 24 bits of output
    b n + i of the SplitMix64 stream seeded with `seed`."""
    c = (np.arange(n, dtype=np.uint64)[:, None] + np.arange(B, dtype=np.uint64)[None, :] * np.uint64(n))
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (c + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z >> np.uint64(40)).astype(np.float64) * 2.0 ** -23 - 1.0).cuda()


class _Objective:
    """Masked mean squared clause value and its gradient in 64 bits."""

    def __init__(self, cnf):
        lits = torch.from_numpy(np.asarray(cnf.lits)).cuda().to(torch.int64)
        lens = torch.from_numpy(np.diff(cnf.off)).cuda()
        self.n, self.m = cnf.n, lens.numel()
        self.var, self.neg = lits.abs() - 1, (lits < 0)
        self.clause = torch.repeat_interleave(torch.arange(self.m, device="cuda"), lens)
        self.w = (torch.ones(self.m, device="cuda", dtype=torch.float64) if cnf.weights is None
                  else torch.from_numpy(np.asarray(cnf.weights)).cuda().to(torch.float64))

    def __call__(self, x):
        """(loss [B], gradient [n][B], cost [B]) at x [n][B], 8 restarts at a time."""
        loss, grad, cost = [], [], []
        for xb in x.split(8, dim=1):
            t = torch.tanh(xb)
            tv = t[self.var]
            tv[self.neg] *= -1.0
            f = torch.zeros((self.m, xb.shape[1]), device="cuda", dtype=torch.float64).index_add_(0, self.clause, tv)
            true = torch.zeros((self.m, xb.shape[1]), device="cuda", dtype=torch.float64)
            true.index_add_(0, self.clause, (tv > 0).to(torch.float64))
            wu = self.w[:, None] * (true == 0)
            c = wu.sum(0)
            safe = torch.clamp(c, min=1.0)
            loss.append((wu * f * f).sum(0) / safe)
            g = (2.0 * wu * f / safe)[self.clause]
            g[self.neg] *= -1.0
            s = torch.zeros_like(t).index_add_(0, self.var, g)
            grad.append(s * (1.0 - t * t))
            cost.append(c)
        return torch.cat(loss), torch.cat(grad, 1), torch.cat(cost)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None  # whole numbers only
    cnf = _instance(case, seed)
    if kind == "eval":
        obj = _Objective(cnf)
        cost = []
        for a in _assignments(case, seed).to(torch.float64).split(8, dim=1):
            tv = a[obj.var]
            tv[obj.neg] *= -1.0
            true = torch.zeros((obj.m, a.shape[1]), device="cuda", dtype=torch.float64)
            true.index_add_(0, obj.clause, (tv > 0).to(torch.float64))
            cost.append((obj.w[:, None] * (true == 0)).sum(0))
        return dict(cost=torch.cat(cost).round().to(torch.int64))
    obj = _Objective(cnf)
    if kind == "grad":
        loss, grad, _ = obj(_grad_x(case, seed).to(torch.float64))
        return dict(loss=loss, grad=grad)
    if case["m"] * _mean_literals(case) * case["B"] * case["steps"] > 3e10:
        return None
    x = _start_x(case["n"], case["B"], seed + 1)
    mom, vel = torch.zeros_like(x), torch.zeros_like(x)
    lr, b1, b2, eps = 1e-4, 0.9, 0.999, 1e-8
    for t in range(1, case["steps"] + 1):
        loss, g, cost = obj(x)
        mom = b1 * mom + (1.0 - b1) * g
        vel = b2 * vel + (1.0 - b2) * g * g
        step = lr / (1.0 - b1 ** t) * mom / (torch.sqrt(vel / (1.0 - b2 ** t)) + eps)
        x = torch.where((cost > 0)[None, :], x - step, x)
    if kind == "solve":  # no assignment satisfies these formulas, so every step is taken
        return dict(steps=None, trace=None, assign=None, best=None, x=x)
    out = dict(loss=loss, cost=None)
    if kind == "oneshot":
        return dict(out, assign=None, best=None)
    out["x"] = x
    if case["dense"]:
        out["dense_cost"] = None
    return out
