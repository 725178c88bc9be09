"""The work a user of this framework has it do, as measurable cases: whole
detection runs, single requests, batches, a served stream, and the scoring of
given labellings, through the package's public entry points.

Every graph is an LFR-style one (Sec. 5.2 of the paper): power-law degrees
with a given mean and maximum, communities of power-law sizes, a fraction
1 - mu of each node's stubs wired inside its community. ``tau`` 0 gives every
node the mean degree (the planted-partition shape). All inputs are drawn from
the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_01752_gb300 as mocd

NOALLOC_CELLS = mocd.NOALLOC_MAX_CELLS


def listed():
    return [
        # The smallest ordinary run: ten communities of a hundred nodes, the
        # paper's parameters. A generation is a few short launches.
        _detect("detect-1k", n=1000, deg=11.4, dmax=20, mu=0.2, tau=0.0, cmin=100, cmax=100, gens=100),
        # The paper's benchmark graph (n = 40,000, mean degree 20, maximum 50)
        # with its parameters: N_p 100, E_S 4, C_P 0.8, M_P 0.2, G 100.
        _detect("detect-40k", n=40_000, deg=20.0, dmax=50, mu=0.3, cmin=20, cmax=100, gens=100),
        # Mixing so strong that neighbours rarely agree, on a graph whose
        # label matrices no longer fit the L2 cache.
        _detect("detect-170k-mixed", n=170_001, deg=16.0, dmax=100, mu=0.6, cmin=20, cmax=1000, gens=60),
        # The largest graph of the framework's benchmark.
        _detect("detect-1m", n=1_000_000, deg=16.0, dmax=200, mu=0.3, cmin=20, cmax=2000, gens=60),
        # A social-network shape: a heavy tail with hubs of thousands of
        # neighbours, an odd population, three parents, the seeded start.
        _detect("detect-hubs", n=30_011, deg=14.0, dmax=5000, mu=0.3, cmin=20, cmax=1000, gens=60,
                np=50, es=3, init=1),
        # A dense network (every degree above a warp's width), a full-width
        # population and more parents.
        _detect("detect-dense", n=4001, deg=90.0, dmax=256, mu=0.4, cmin=100, cmax=600, gens=60, np=128, es=6),
        # One request from host arrays to the answer: upload and validation,
        # the run, the front, release.
        dict(_detect("request-5k", n=5003, deg=16.0, dmax=50, mu=0.4, cmin=20, cmax=100, gens=100), kind="request"),
        # Many uneven jobs of 10^3 to 5 x 10^4 nodes run together.
        dict(name="batch-16", kind="batch", jobs=16, n_min=1000, n_max=50_000, mu=0.35, gens=20, np=100, es=4),
        # A queue of requests of mixed sizes through the server.
        dict(name="serve-12", kind="serve", jobs=12, n_min=1000, n_max=100_000, mu=0.35, gens=30, np=100, es=4),
        # Scoring given labellings from the host.
        dict(name="evaluate-40k", kind="evaluate", n=40_000, deg=20.0, dmax=50, mu=0.3, tau=2.0, cmin=20, cmax=100,
             count=100),
        # Scoring a population that is already on the device, without any
        # device allocation.
        dict(name="evaluate-device-40k", kind="noalloc", n=40_000, deg=20.0, dmax=50, mu=0.3, tau=2.0, cmin=20,
             cmax=100, count=100),
        # Resuming a saved population, its front's community statistics and
        # the member two criteria prefer.
        dict(name="statistics-40k", kind="stats", n=40_000, deg=20.0, dmax=50, mu=0.3, tau=2.0, cmin=20, cmax=100,
             count=100),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["detect", "detect", "detect", "request", "batch", "serve", "evaluate", "noalloc", "stats"])
    mu = round(rng.uniform(0.1, 0.6), 3)
    if kind in ("batch", "serve"):
        return dict(kind=kind, jobs=rng.randint(2, 16), n_min=log(500, 2000), n_max=log(10_000, 50_000), mu=mu,
                    gens=rng.randint(10, 30), np=rng.choice([50, 64, 100]), es=rng.choice([2, 3, 4]))
    deg = round(rng.uniform(8.0, 30.0), 2)
    shape = dict(deg=deg, dmax=log(2.0 * deg, 300), mu=mu, tau=rng.choice([0.0, 2.0, 2.0, 2.5]), cmin=20,
                 cmax=log(60, 1000))
    if kind == "detect":
        n = log(1000, 400_000)
        if n < 50_000 and rng.random() < 0.3:  # a heavier tail
            shape["dmax"] = log(300, n // 6 + 300)
        return _detect(None, n=n, gens=rng.randint(20, 60), np=rng.choice([33, 64, 100, 100, 128]),
                       es=rng.choice([2, 3, 4, 4, 4, 5]), init=rng.randint(0, 1), **shape)
    if kind == "request":
        return dict(_detect(None, n=log(1000, 100_000), gens=rng.randint(20, 100), **shape), kind="request")
    n = log(1000, 200_000)
    count = rng.randint(20, 128)
    if kind == "noalloc":
        count = min(count, NOALLOC_CELLS // n)
    return dict(kind=kind, n=n, count=count, **shape)


def _detect(name, *, n, deg, dmax, mu, cmin, cmax, gens, tau=2.0, np=100, es=4, init=0):
    case = dict(kind="detect", n=n, deg=deg, dmax=dmax, mu=mu, tau=tau, cmin=cmin, cmax=cmax, gens=gens, np=np, es=es,
                init=init)
    return case if name is None else dict(case, name=name)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _power_mean(a, b, tau):
    if abs(tau - 2.0) < 1e-12:
        return math.log(b / a) / (1.0 / a - 1.0 / b)
    return (1 - tau) / (2 - tau) * (b ** (2 - tau) - a ** (2 - tau)) / (b ** (1 - tau) - a ** (1 - tau))


def _power_min(mean, b, tau):
    lo, hi = 0.05, float(b)
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if _power_mean(mid, b, tau) < mean else (lo, mid)
    return lo


def _pairs(stubs, tag, group, n_groups):
    """Stubs paired at random within their group (an odd one is left out)."""
    order = torch.argsort(group * (1 << 32) + tag)
    stubs, group = stubs[order], group[order]
    counts = torch.bincount(group, minlength=n_groups)
    pos = torch.arange(stubs.numel(), device=stubs.device) - (torch.cumsum(counts, 0) - counts)[group]
    first = torch.nonzero((pos % 2 == 0) & (pos + 1 < counts[group])).flatten()
    return stubs[first], stubs[first + 1]


def graph(n, deg, dmax, mu, tau, cmin, cmax, seed):
    """(row_ptr int64 [n + 1], col_idx int32 [2m], member [n]) on the GPU; node ids are in random order."""
    dev = "cuda"
    gen = torch.Generator(device=dev).manual_seed(seed)
    dmax = min(dmax, n - 1)

    def rand(size):
        return torch.rand(size, generator=gen, device=dev, dtype=torch.float64)

    def words(size):
        return torch.randint(0, 1 << 32, (size,), generator=gen, device=dev)

    if tau == 0.0:
        degree = torch.floor(deg + rand(n)).long()
    else:
        a = _power_min(deg, dmax, tau)
        e = 1.0 - tau
        degree = torch.round((a ** e + rand(n) * (dmax ** e - a ** e)) ** (1.0 / e)).long()
    degree = degree.clamp(1, dmax)
    r = rand(n // cmin + 2)  # community sizes: power law of exponent 1
    sizes = torch.round(cmin * (cmax / cmin) ** r).long()
    member = torch.bucketize(torch.arange(n, device=dev), torch.cumsum(sizes, 0), right=True)
    member = member[torch.argsort(words(n))]
    n_comm = int(member.max()) + 1
    sizes = torch.bincount(member, minlength=n_comm)
    inside = torch.minimum(torch.round((1.0 - mu) * degree).long(), sizes[member] - 1).clamp(min=0)
    nodes = torch.arange(n, device=dev)
    stubs = torch.repeat_interleave(nodes, inside)
    u0, v0 = _pairs(stubs, words(stubs.numel()), member[stubs], n_comm)
    stubs = torch.repeat_interleave(nodes, degree - inside)
    u1, v1 = _pairs(stubs, words(stubs.numel()), torch.zeros_like(stubs), 1)
    # A ring through a few nodes keeps the smallest graph from having no edge.
    ring = torch.arange(min(n, 3), device=dev)
    u, v = torch.cat([u0, u1, ring[:-1]]), torch.cat([v0, v1, ring[1:]])
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    u, v = key // n, key % n
    key = torch.sort(torch.cat([u * n + v, v * n + u])).values
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    row_ptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return row_ptr, (key % n).int(), member


def labellings(member, count, seed):
    """[count][n] int32 on the GPU: a population as a run holds it. Each
    labelling follows the communities (named by one of their nodes), some of
    them merged, with a fraction of the nodes on labels of their own."""
    dev = member.device
    n = member.numel()
    gen = torch.Generator(device=dev).manual_seed(seed + 77)
    n_comm = int(member.max()) + 1
    name = torch.zeros(n_comm, dtype=torch.int64, device=dev)
    name.scatter_reduce_(0, member, torch.arange(n, device=dev), "amax", include_self=False)
    out = torch.empty((count, n), dtype=torch.int32, device=dev)
    for k in range(count):
        merged = torch.div(torch.arange(n_comm, device=dev), 1 + k % 7, rounding_mode="floor") * (1 + k % 7)
        lab = name[merged][member]
        stray = torch.rand(n, generator=gen, device=dev) < 0.004 * (k % 25)
        other = torch.randint(0, n, (n,), generator=gen, device=dev)
        out[k] = torch.where(stray, other, lab).int()
    return out


def _shape(case):
    return {k: case[k] for k in ("n", "deg", "dmax", "mu", "tau", "cmin", "cmax")}


def _host(t):
    return t.cpu().numpy()


def _params(case, seed):
    return mocd.Params(pop_size=case["np"], n_parents=case["es"], seed=seed, init_mode=case.get("init", 0))


def _jobs(case):
    """The uneven jobs of a batch or a stream: sizes log-spaced, mean degrees 10 to 30."""
    jobs = case["jobs"]
    for k in range(jobs):
        t = k / max(1, jobs - 1)
        deg = 10.0 + 20.0 * ((7 * k) % jobs) / jobs
        yield dict(n=int(round(case["n_min"] * (case["n_max"] / case["n_min"]) ** t)), deg=deg,
                   dmax=int(round(2.5 * deg)), mu=case["mu"], tau=2.0, cmin=20, cmax=100)


class Context:
    """An uploaded graph, released with its last reference."""

    def __init__(self, row_ptr, col_idx):
        self.handle = mocd.graph_upload(row_ptr, col_idx)

    def __del__(self):
        mocd.destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        graphs = [graph(seed=seed * 1009 + k, **job)[:2] for k, job in enumerate(_jobs(case))]
        graphs = [(_host(rp), _host(ci)) for rp, ci in graphs]
        params = [_params(case, seed + k) for k in range(len(graphs))]
        state = dict(kind=kind, graphs=graphs, params=params, gens=case["gens"])
        if kind == "batch":
            state["contexts"] = [Context(rp, ci) for rp, ci in graphs]
        return state
    row_ptr, col_idx, member = graph(seed=seed, **_shape(case))
    if kind in ("detect", "request"):
        state = dict(kind=kind, graph=(_host(row_ptr), _host(col_idx)), params=_params(case, seed), gens=case["gens"])
        if kind == "detect":
            state["context"] = Context(*state["graph"])
        return state
    labels = labellings(member, case["count"], seed)
    if kind == "noalloc":
        count, n = labels.shape
        rows = torch.zeros((n, (count + 3) // 4 * 4), dtype=torch.int32, device="cuda")
        rows[:, :count] = labels.t()
        out = torch.zeros((2, count), dtype=torch.int64, device="cuda")
        return dict(kind=kind, n=n, count=count, row_ptr=row_ptr.int(), col_idx=col_idx, rows=rows, out=out)
    return dict(kind=kind, context=Context(_host(row_ptr), _host(col_idx)), labels=_host(labels),
                params=mocd.Params(pop_size=case["count"], seed=seed))


def _whole(a):
    # A front's arrays are views of buffers of N_p entries, zero past its
    # members: the buffer has the same shape however many members there are.
    return a if a.base is None else a.base


def _front(front):
    return dict(labels=_whole(front.labels), f1=_whole(front.f1), f2=_whole(front.f2), intra=_whole(front.intra),
                sumsq=_whole(front.sumsq), best=front.best)


def run(state):
    kind = state["kind"]
    if kind == "detect":
        ctx = state["context"].handle
        mocd.population_init(ctx, state["params"])
        mocd.generation(ctx, state["gens"])
        return _front(mocd.pareto_front(ctx))
    if kind == "request":
        ctx = mocd.graph_upload(*state["graph"])
        try:
            mocd.population_init(ctx, state["params"])
            mocd.generation(ctx, state["gens"])
            return _front(mocd.pareto_front(ctx))
        finally:
            mocd.destroy(ctx)
    if kind == "batch":
        handles = [c.handle for c in state["contexts"]]
        for ctx, params in zip(handles, state["params"]):
            mocd.population_init(ctx, params)
        batch = mocd.batch_create(handles)
        try:
            mocd.batch_configure(batch, 8, 1)
            mocd.batch_generation(batch, state["gens"])
            mocd.batch_synchronize(batch)
        finally:
            mocd.batch_destroy(batch)
        fronts = [mocd.pareto_front(ctx) for ctx in handles]
        return [[_whole(f.labels), _whole(f.intra), _whole(f.sumsq)] for f in fronts]
    if kind == "serve":
        server = mocd.Server(1 << 34, max_running=4, depth=2)
        try:
            ids = [server.submit(rp, ci, params, state["gens"])
                   for (rp, ci), params in zip(state["graphs"], state["params"])]
            while True:
                running, queued, _ = server.step()
                if not running and not queued:
                    break
            fronts = [server.result(j) for j in ids]
        finally:
            server.close()
        return [[_whole(f.labels), _whole(f.intra), _whole(f.sumsq)] for f in fronts]
    if kind == "evaluate":
        return list(mocd.evaluate(state["context"].handle, state["labels"]))
    if kind == "noalloc":
        out = state["out"]
        mocd.evaluate_noalloc(state["row_ptr"].data_ptr(), state["col_idx"].data_ptr(), state["n"],
                              state["rows"].data_ptr(), state["count"], out[0].data_ptr(), out[1].data_ptr(),
                              torch.cuda.current_stream())
        return [out[0], out[1]]
    ctx = state["context"].handle
    mocd.set_population(ctx, state["params"], state["labels"], 0)
    stats = mocd.front_stats(ctx)
    chosen = [mocd.select_solution(ctx, c) for c in (mocd.SELECT_MODULARITY, mocd.SELECT_MEAN_CONDUCTANCE)]
    return dict(communities=_whole(stats.communities), size_sumsq=_whole(stats.size_sumsq),
                mean=_whole(stats.mean_conductance), max=_whole(stats.max_conductance), chosen=chosen)


# ---------------------------------------------------------------------------
# What a pass cannot do without, and what its numbers are in 64 bits
# ---------------------------------------------------------------------------

def _run_work(n, deg, np, es, gens):
    """Per generation: the parents are read and the crossed children written,
    these are read again for the mutation (its neighbours' labels are other
    nodes' rows), the children written, and read for the evaluation; the
    adjacency is read for the mutation and, an edge once, for the evaluation.
    Operations are label comparisons: E_S per child and node, one per
    neighbour of a mutating node (a fifth of them), one per edge."""
    m = 0.5 * n * deg
    size = 4 * n * np
    per_gen = 5 * size + 4 * (n + 1) + 8 * m + 4 * (n + 1) + 4 * m
    return dict(bytes=gens * per_gen, flops=gens * np * (es * n + 0.2 * 2 * m + m))


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        parts = [_run_work(j["n"], j["deg"], case["np"], case["es"], case["gens"]) for j in _jobs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, m = case["n"], 0.5 * case["n"] * case["deg"]
    if kind in ("detect", "request"):
        return _run_work(n, case["deg"], case["np"], case["es"], case["gens"])
    count = case["count"]
    return dict(bytes=4 * n * count + 4 * (n + 1) + 8 * m + 16 * count, flops=count * (m + n))


def _keys(row_ptr, col_idx, labels):
    """Exact (intra [count], S [count], degrees) of [count][n] labels."""
    n = row_ptr.numel() - 1
    degree = row_ptr[1:] - row_ptr[:-1]
    src = torch.repeat_interleave(torch.arange(n, device=row_ptr.device), degree)
    dst = col_idx.long()
    intra, sumsq = [], []
    for lab in labels.long():
        intra.append((lab[src] == lab[dst]).sum() // 2)
        total = torch.zeros(n, dtype=torch.int64, device=lab.device).scatter_add_(0, lab, degree)
        sumsq.append((total * total).sum())
    return torch.stack(intra), torch.stack(sumsq), degree, src, dst


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("evaluate", "noalloc", "stats"):
        return None
    row_ptr, col_idx, member = graph(seed=seed, **_shape(case))
    labels = labellings(member, case["count"], seed)
    intra, sumsq, degree, src, dst = _keys(row_ptr, col_idx, labels)
    if kind != "stats":
        return [intra, sumsq]
    # The front of the population: members that no other dominates in
    # (m - intra, S), in population order.
    n, two_m = case["n"], int(row_ptr[-1])
    k1, k2 = two_m // 2 - intra, sumsq
    le = (k1[:, None] <= k1[None]) & (k2[:, None] <= k2[None])
    lt = (k1[:, None] < k1[None]) | (k2[:, None] < k2[None])
    front = torch.nonzero(~(le & lt).any(0)).flatten().tolist()
    count, sq, mean, top = [], [], [], []
    for i in front:
        lab = labels[i].long()
        zero = torch.zeros(n, dtype=torch.int64, device=lab.device)
        size = zero.scatter_add(0, lab, torch.ones_like(lab))
        vol = zero.scatter_add(0, lab, degree)
        cut = zero.scatter_add(0, lab[src], (lab[src] != lab[dst]).long())
        some = size > 0
        phi = torch.where(cut[some] > 0, cut[some].double() / torch.minimum(vol, two_m - vol)[some].double(), 0.0)
        count.append(int(some.sum()))
        sq.append(int((size * size).sum()))
        mean.append(math.fsum(phi.tolist()) / count[-1])
        top.append(float(phi.max()))
    rest = [0] * (case["count"] - len(front))  # as run() returns them: zero past the front
    return dict(communities=np.array(count + rest), size_sumsq=np.array(sq + rest),
                mean=np.array(mean + rest, dtype=np.float64), max=np.array(top + rest, dtype=np.float64),
                chosen=[None, None])
