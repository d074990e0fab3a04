"""The work that programs have this framework do, as cases to be timed.

A case is a dict of plain values:
  kind      "solve"   : a resident chain; step 0, a solve, the estimate
            "request" : a new chain: create, solve, read the estimate back, destroy
            "steps"   : a resident chain; step 0, single moves with their infos, the estimate
  graph     "tiny"    : out-degree U{1..8} to uniform targets, cycle, self-loops, weights U(0,1]
            "rmat"    : R-MAT (.57,.19,.19,.05), cycle, self-loops; unit weights or (weighted) U(0,1]
            "sym"     : "rmat" with every link both ways (a random walk on an undirected graph)
            "pagerank": the auxiliary-node chain of a unit-weight "rmat" graph on n nodes, damping 17/20,
                        step 0 from the auxiliary node
            "powerlaw", "rmats": `chains` chains of log-spaced sizes in [n_lo, n], block-diagonal
  tol > 0   solve to that residual; else exactly `moves` moves
The other keys are parameters of the library by their own names.
"""
import math

import numpy as np
import torch

from paper_2008_02710_gb300 import rlgl, synth

BATCHES = ("powerlaw", "rmats")
DEFAULTS = {"kind": "solve", "graph": "rmat", "n": 1000, "n_lo": 0, "edge_factor": 16, "weighted": False, "chains": 1,
            "precision": "mixed", "schedule": "link_threshold", "theta_scale": 0.5, "theta_lag": 0,
            "tol": 0.0, "moves": 0}


def _case(**kw):
    return {**DEFAULTS, **kw}


def listed():
    return [
        # the default call (FP64, |C| threshold, tolerance 1e-12) on the smallest configuration: latency alone counts
        _case(name="tiny_fp64", graph="tiny", n=1000, precision="fp64", schedule="threshold", theta_scale=1.0, tol=1e-12),
        # the same call on a web graph of the size of the literature's mid-sized ones, to its tolerance of 1e-11
        _case(name="web_fp64", n=281903, edge_factor=8, precision="fp64", schedule="threshold", theta_scale=1.0, tol=1e-11),
        # moves made one by one by a caller that looks at each (weighted links, FP64)
        _case(name="steps_fp64", kind="steps", n=131072, weighted=True, precision="fp64", moves=16),
        # a solve request that has the GPU to itself: a chain it has not seen, to a tolerance, and gone again
        _case(name="request", kind="request", n=200003, theta_lag=1, tol=1e-6),
        # the small requests that were queued meanwhile, as one batch
        _case(name="request_batch", kind="request", graph="rmats", n_lo=1000, n=131071, chains=8, tol=1e-6),
        # the headline: R-MAT 20 by the per-link threshold, one move stale
        _case(name="rmat20_link", n=1 << 20, theta_lag=1, tol=1e-6),
        # power iteration on the same chain: what the schedules are measured against
        _case(name="rmat20_all_green", n=1 << 20, schedule="all_green", tol=1e-6),
        # PageRank by the auxiliary-node chain: weighted links, one node that all others feed
        _case(name="pagerank", graph="pagerank", n=500000, theta_lag=1, tol=1e-6),
        # a weighted chain beyond the L2 cache in FP64, a fixed number of moves
        _case(name="rmat22_weighted_fp64", n=1 << 22, weighted=True, precision="fp64", moves=12),
        # the largest chains: an undirected graph beyond the L2 cache, by the per-link threshold and by power iteration
        _case(name="rmat24_sym_link", graph="sym", n=1 << 24, theta_lag=1, tol=1e-5),
        _case(name="rmat24_sym_all_green", graph="sym", n=1 << 24, schedule="all_green", moves=60),
        # many independent chains in one launch (a quarter of the 4096-chain mix), at the threshold scale tuned for it
        _case(name="batch_1024", graph="powerlaw", n_lo=100, n=100000, chains=1024, theta_scale=1 / 16, tol=1e-6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "fp64", "request", "batch_request", "link", "link", "all_green", "all_green", "pagerank",
                       "weighted", "sym", "batch", "topfrac", "steps"])
    ef = rng.randint(4, 24)
    tol = rng.choice([1e-4, 1e-5, 1e-6])
    lag = rng.randint(0, 1)
    if kind == "small":
        return _case(graph="tiny", n=_log(rng, 200, 50000), precision=rng.choice(["fp64", "mixed"]), theta_lag=lag,
                     schedule=rng.choice(["threshold", "link_threshold", "all_green"]), theta_scale=1.0, tol=tol)
    if kind == "fp64":
        return _case(n=_log(rng, 20000, 1500000), edge_factor=ef, precision="fp64", theta_lag=lag,
                     schedule=rng.choice(["threshold", "link_threshold", "all_green"]), tol=rng.choice([1e-8, 1e-10, 1e-12]))
    if kind == "request":
        return _case(kind="request", n=_log(rng, 131072, 4000000), edge_factor=ef, theta_lag=1, tol=tol)
    if kind == "batch_request":
        return _case(kind="request", graph="rmats", n_lo=1000, n=131071, chains=rng.randint(2, 48), tol=tol)
    if kind == "link":
        return _case(n=_log(rng, 100000, 4000000), edge_factor=ef, theta_scale=rng.choice([0.25, 0.5, 1.0]), theta_lag=lag,
                     tol=tol)
    if kind == "all_green":
        return _case(graph=rng.choice(["rmat", "rmat", "sym"]), n=_log(rng, 100000, 4000000), edge_factor=ef,
                     schedule="all_green", moves=rng.randint(20, 80))
    if kind == "pagerank":
        return _case(graph="pagerank", n=_log(rng, 50000, 900000), edge_factor=ef, theta_lag=lag, tol=tol)
    if kind == "weighted":
        return _case(n=_log(rng, 200000, 6000000), weighted=True, precision=rng.choice(["fp64", "mixed"]), moves=rng.randint(6, 24),
                     schedule=rng.choice(["link_threshold", "all_green"]))
    if kind == "sym":
        return _case(graph="sym", n=_log(rng, 1000000, 9000000), edge_factor=rng.randint(6, 16), theta_lag=lag, tol=1e-5)
    if kind == "batch":
        return _case(graph="powerlaw", n_lo=100, n=_log(rng, 2000, 100000), chains=_log(rng, 16, 800), theta_scale=1 / 16,
                     schedule=rng.choice(["link_threshold", "all_green"]), tol=tol)
    if kind == "topfrac":
        return _case(n=_log(rng, 50000, 1000000), edge_factor=ef, schedule="topfrac", moves=rng.randint(50, 300))
    return _case(kind="steps", n=_log(rng, 20000, 1000000), edge_factor=ef, weighted=bool(rng.randint(0, 1)),
                 precision="fp64", schedule=rng.choice(["threshold", "link_threshold"]), moves=rng.randint(4, 24))


# ------------------------------------------------------------------ inputs


def _sizes(case):
    """Chain sizes of a batch: log-spaced in [n_lo, n]."""
    k, lo, hi = case["chains"], case["n_lo"], case["n"]
    return [int(round(lo * (hi / lo) ** ((i + 0.5) / k))) for i in range(k)]


def _weights(m, gen):
    return 1.0 - torch.rand(m, generator=gen, device="cuda")


def _both_ways(csr):
    """Every link that is not a self-loop also reversed."""
    src = torch.repeat_interleave(torch.arange(csr.n, dtype=torch.int32, device="cuda"), torch.diff(csr.row_ptr))
    other = src != csr.col
    s, d = torch.cat([src, csr.col[other]]), torch.cat([csr.col, src[other]])
    s, order = torch.sort(s, stable=True)
    row_ptr = torch.zeros(csr.n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(s, minlength=csr.n), 0)
    return synth.CSR(csr.n, row_ptr, d[order], None)


def _powerlaw(case, gen):
    """Per chain a mean out-degree U(4, 32), Poisson out-degrees, targets i = floor(n u^2) (few nodes take most links),
    cycle and self-loop."""
    sizes = torch.tensor(_sizes(case), device="cuda")
    ptr = torch.zeros(len(sizes) + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(sizes, 0)
    n = int(ptr[-1])
    mean = 4 + 28 * torch.rand(len(sizes), generator=gen, device="cuda")
    chain = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), sizes)
    deg = torch.poisson(mean[chain], generator=gen).to(torch.int64) + 2
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(deg, 0)
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    first, size = ptr[:-1][chain], sizes[chain]
    u = torch.rand(src.numel(), generator=gen, device="cuda", dtype=torch.float64)
    col = (first[src] + (u * u * size[src]).to(torch.int64)).to(torch.int32)
    del u, src
    i = torch.arange(n, device="cuda")
    col[row_ptr[:-1]] = (first + (i - first + 1) % size).to(torch.int32)
    col[row_ptr[:-1] + 1] = i.to(torch.int32)
    return synth.CSR(n, row_ptr, col, None), ptr.cpu().numpy()


def _pagerank(csr):
    host = synth.CSR(csr.n, csr.row_ptr.cpu().numpy(), csr.col.cpu().numpy(), None)
    a = synth.pagerank_chain(host)
    return synth.CSR(a.n, *(torch.from_numpy(x).cuda() for x in (a.row_ptr, a.col, a.w)))


def _graph(case, seed):
    """(CSR of device tensors, node_ptr of a batch or None, M_0 or None)."""
    g, n, ef = case["graph"], case["n"], case["edge_factor"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if g == "tiny":
        c = synth.tiny_chain(n, seed)
        return synth.CSR(n, *(torch.from_numpy(x).cuda() for x in (c.row_ptr, c.col, c.w))), None, None
    if g == "powerlaw":
        return (*_powerlaw(case, gen), None)
    if g == "rmats":
        return (*synth.stack_chains_device([synth.rmat_chain_n_device(m, ef, seed * 1000 + k)
                                            for k, m in enumerate(_sizes(case))]), None)
    csr = synth.rmat_chain_n_device(n, ef, seed)
    if g == "sym":
        return _both_ways(csr), None, None
    if g == "pagerank":
        m0 = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
        m0[0] = 1.0
        return _pagerank(csr), None, m0
    if case["weighted"]:
        csr = csr._replace(w=_weights(csr.col.numel(), gen))
    return csr, None, None


class State:
    pass


def _chain(case, s):
    ch = rlgl.Chain(s.csr, m0=s.m0, precision=case["precision"], node_ptr=s.node_ptr)
    ch.set_params(theta_scale=case["theta_scale"],
                  theta_lag=0 if s.node_ptr is not None or case["schedule"] == "topfrac" else case["theta_lag"])
    if s.node_ptr is not None:
        ch.set_chain_tol(np.full(case["chains"], case["tol"]))
    return ch


def prepare(case, seed):
    s = State()
    s.case = case
    s.csr, s.node_ptr, s.m0 = _graph(case, seed)
    s.n = s.csr.n
    s.chain = None
    if case["kind"] != "request":
        s.chain = _chain(case, s)
        s.csr = None  # the context holds its own copy
        first = 1 if case["graph"] == "pagerank" else 0
        s.pi = torch.empty(s.n - first, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return s


# -------------------------------------------------------------------- run


def _solve(case, ch, batch):
    if case["tol"] > 0:
        return ch.solve(case["schedule"], tol=-1.0 if batch else case["tol"])
    return ch.solve(case["schedule"], tol=0.0, max_steps=case["moves"], raise_on_noconv=False)


def run(s):
    case = s.case
    if case["kind"] == "request":
        with _chain(case, s) as ch:
            _solve(case, ch, s.node_ptr is not None)
            moves = ch.chains()[1] if s.node_ptr is not None else None
            pi = ch.estimate()
        rlgl.release_retired()
        return {"pi": pi} if moves is None else {"pi": pi, "moves": moves}
    ch = s.chain
    ch.reset(s.m0)
    if case["kind"] == "steps":
        infos = [ch.step(case["schedule"]) for _ in range(case["moves"])]
        return {"pi": ch.estimate(out=s.pi),
                "green": np.array([i["green"] for i in infos]), "edges": np.array([i["edges_pushed"] for i in infos]),
                "theta": np.array([i["theta"] for i in infos]), "l1_cash": np.array([i["l1_cash"] for i in infos])}
    info = _solve(case, ch, s.node_ptr is not None)
    if case["graph"] == "pagerank":
        return {"pi": ch.estimate_range(1, s.n, out=s.pi), "moves": info["moves"]}
    return {"pi": ch.estimate(out=s.pi), "moves": info["moves"]}


# ------------------------------------------------------------------- work


def _shape(case):
    """(nodes, links) of the case's chain, the links as expected."""
    g, n, ef = case["graph"], case["n"], case["edge_factor"]
    if g == "tiny":
        return n, 6.5 * n
    if g in BATCHES:
        n = sum(_sizes(case))
        return n, n * (20 if g == "powerlaw" else ef + 2)
    if g == "sym":
        return n, n * (2 * ef + 3)
    return (n + 1, n * (ef + 4)) if g == "pagerank" else (n, n * (ef + 2))


def work(case):
    """Every link moved once per full sweep: its index (and weight) read and one multiply-add. An all-green move is one
    sweep; a threshold schedule spends about two sweeps' links per decimal of the tolerance (measured: 11 on R-MAT 20
    and 16 on its symmetrised form to 1e-6), and a fixed number of its moves about a seventh of a sweep each. Per move
    the nodes' cash is read once; the estimate is written once; a request reads its links once more."""
    n, m = _shape(case)
    cash = 4 if case["precision"] == "mixed" else 8
    weighted = case["weighted"] or case["graph"] in ("tiny", "pagerank")
    decimals = -math.log10(case["tol"]) if case["tol"] > 0 else 0.0
    if case["schedule"] == "all_green":
        moves = case["moves"] or 10 * decimals
        sweeps = moves
    else:
        moves = case["moves"] or 13 * decimals
        sweeps = case["moves"] * (0.01 if case["schedule"] == "topfrac" else 1 / 7) if case["moves"] else 2 * decimals
    per_link = 8 if weighted else 4
    bytes_ = sweeps * m * per_link + moves * n * cash + 16 * n
    if case["kind"] == "request":
        bytes_ += m * per_link + 8 * n
    return {"bytes": bytes_, "flops": 2.0 * sweeps * m}


# ------------------------------------------------------------------ exact


class _P:
    """x -> x P in FP64, by adding every link's share to its target."""

    def __init__(self, csr):
        self.n, self.deg = csr.n, torch.diff(csr.row_ptr)
        self.src = torch.repeat_interleave(torch.arange(csr.n, dtype=torch.int32, device="cuda"), self.deg)
        self.col = csr.col
        self.w = None if csr.w is None else csr.w.double()
        self.s = 1.0 / (self.deg.double() if self.w is None
                        else torch.zeros(csr.n, dtype=torch.float64, device="cuda").index_add_(0, self.src, self.w))

    def __call__(self, x):
        v = (x * self.s).index_select(0, self.src)
        if self.w is not None:
            v.mul_(self.w)
        return torch.zeros(self.n, dtype=torch.float64, device="cuda").index_add_(0, self.col, v)


def _law(P, chain, k):
    """The stationary law of every chain (power iteration from the uniform law until it stands still)."""
    ones = torch.ones(P.n, dtype=torch.float64, device="cuda")

    def scaled(x):
        return x / torch.zeros(k, dtype=torch.float64, device="cuda").index_add_(0, chain, x)[chain]

    x = scaled(ones)
    last = math.inf
    for it in range(4000):
        y = scaled(P(x))
        if it % 16 == 15:
            change = float((y - x).abs().sum()) / k
            if change < 1e-15 or (change < 1e-12 and change > 0.9 * last):
                return y
            last = change
        x = y
    return None


def _moves(P, m0, case):
    """Alg. 1 from step 0: (estimate, per move: |G|, its links, theta, ||C||_1 after it)."""
    h = m0.clone()
    c = P(m0) - m0
    infos = []
    link = case["schedule"] == "link_threshold"
    for _ in range(case["moves"]):
        v = c.abs()
        if link:
            v = v / P.deg
        if case["schedule"] == "all_green":
            g, theta = torch.ones_like(c, dtype=torch.bool), 0.0
        elif case["schedule"] == "topfrac":
            k = math.ceil(0.01 * P.n)
            theta = torch.topk(v, k).values[-1]
            g = (v >= theta) & (c != 0)
        else:
            theta = case["theta_scale"] * v.sum() / P.n
            g = (v >= theta) & (c != 0)
        m = torch.where(g, c, torch.zeros_like(c))
        h += m
        c = c - m + P(m)
        if case["kind"] == "steps":
            infos.append((float(theta), float(c.abs().sum())))
    return h / h.sum(), infos


def exact(case, seed):
    csr, node_ptr, m0 = _graph(case, seed)
    if case["graph"] == "sym" and case["tol"] > 0:
        # a walk on an undirected graph: the degrees
        d = torch.diff(csr.row_ptr).double()
        return {"pi": d / d.sum()}
    P = _P(csr)
    if case["tol"] > 0:
        # a solve comes near the stationary law itself, as near as its tolerance
        k = 1 if node_ptr is None else case["chains"]
        chain = (torch.zeros(csr.n, dtype=torch.int64, device="cuda") if node_ptr is None else
                 torch.repeat_interleave(torch.arange(k, device="cuda"), torch.diff(torch.from_numpy(node_ptr).cuda())))
        pi = _law(P, chain, k)
        if pi is not None and case["graph"] == "pagerank":
            pi = pi[1:] / pi[1:].sum()
        return None if pi is None else {"pi": pi}
    if m0 is None:
        m0 = torch.full((csr.n,), 1.0 / csr.n, dtype=torch.float64, device="cuda")
    pi, infos = _moves(P, m0, case)
    if case["kind"] == "steps":
        return {"pi": pi, "theta": np.array([i[0] for i in infos]), "l1_cash": np.array([i[1] for i in infos])}
    return {"pi": pi}
