"""Performance cases of the absorbing-frequency-centrality engine.

A case is one call that a user's program makes: Monte Carlo transition counting (single graph,
batched graphs, row-wise draws), a whole query from host memory, the absorbing-chain solve, the
perturbation sweep and the robust value, each through the package's public Python
entry points, at the sizes of this repository's workloads.  ``prepare`` makes the inputs from the
seed (graphs with numpy, chains with torch on the GPU), ``run`` makes the one call, ``exact``
computes the chain results again in plain torch FP64.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2605_14743_gb300 as afc


# ---- the cases --------------------------------------------------------------------------------

def listed():
    return [
        # The smallest workload: ER G(50, 0.1), survival 0.9, lengths 1..10, FP64.
        dict(name="counts_er50", kind="counts", family="er", n=50, degree=4.9, beta=0.0,
             p_fail=0.1, w_hi=10, realizations=1000, precision="fp64", pool=0.0),
        # The flagship workload: WS(1000, 6, 0.1), failure 0.05, lengths 1..100, a candidate pool
        # of 10% of the nodes, FP64; a tenth of its realization budget.
        dict(name="counts_ws1000", kind="counts", family="ws", n=1000, degree=6.0, beta=0.1,
             p_fail=0.05, w_hi=100, realizations=1000, precision="fp64", pool=0.1),
        # An upper-middle graph of the batched mix alone (ragged size, FP32 with FP64 recheck):
        # too large for a CTA's shared memory.
        dict(name="counts_er2301", kind="counts", family="er", n=2301, degree=8.0, beta=0.0,
             p_fail=0.1, w_hi=50, realizations=128, precision="fp32_recheck", pool=0.0),
        # A large graph of the serving stream (lengths 1..100, FP32 with FP64 recheck).
        dict(name="counts_ws6007", kind="counts", family="ws", n=6007, degree=8.0, beta=0.1,
             p_fail=0.15, w_hi=100, realizations=16, precision="fp32_recheck", pool=0.0),
        # The largest workload: WS(20000, 10, 0.05), failure 0.1, lengths 1..1000, FP64; a few of
        # its realizations (they are processed a few at a time).
        dict(name="counts_ws20000", kind="counts", family="ws", n=20000, degree=10.0, beta=0.05,
             p_fail=0.1, w_hi=1000, realizations=4, precision="fp64", pool=0.0),
        # Graphs of uneven size in one batched call (the batched mix: half ER of mean degree 8,
        # half WS k = 8 beta = 0.2, lengths 1..50, failure 0.01..0.2, FP32 with FP64 recheck).
        dict(name="batch_mix8", kind="batch", graphs=8, n_lo=200, n_hi=2000, realizations=96),
        # The weighted network with 2-hop neighbourhoods: independent draws per row, rounded and
        # clipped normal lengths, every edge present, 77 nodes and 254 edges, 60 draws per row.
        dict(name="rowwise_77", kind="rowwise", n=77, m=254, draws=60, hop_radius=2, w_hi=31),
        # A small query of the serving stream end to end from host memory: copies, counts, solve
        # and results back.
        dict(name="query_er150", kind="query", family="er", n=150, degree=8.0, beta=0.0,
             p_fail=0.1, w_hi=100, realizations=300, precision="fp32_recheck", n_perturb=0),
        # The absorbing-chain solve of a 20,000-node query's chain (many observed states, rows
        # over part of them), on a smaller anchor set.
        dict(name="solve_c1251", kind="solve", n=5000, c=1251, realizations=2048, spread="part"),
        # The perturbation sweep of the flagship workload (every row spreads over all ~100
        # observed states); a fifth of its 10,000 perturbations.
        dict(name="sweep_c97", kind="sweep", n=1000, c=97, realizations=10000, spread="all",
             perturbations=2000),
        # The perturbation sweep of a chain with many observed states.
        dict(name="sweep_c751", kind="sweep", n=3000, c=751, realizations=2048, spread="part",
             perturbations=304),
        # The robust value (policy iteration, worst case expected length) on an estimated chain.
        dict(name="robust_n500", kind="robust", n=500, c=81, realizations=4096, spread="all"),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["counts", "counts", "counts", "counts", "batch", "rowwise", "query",
                       "solve", "sweep", "sweep", "robust"])
    if kind == "counts":
        n = _logu(rng, 50, 12000)
        family = rng.choice(["er", "ws"])
        degree = rng.uniform(5.0, 10.0)
        if family == "ws":
            degree = 2.0 * round(degree / 2.0)
        most = 2000.0 * (1000.0 / n) ** 2.2        # about 0.25 s at most
        return dict(kind="counts", family=family, n=n, degree=degree,
                    beta=rng.choice([0.05, 0.1, 0.2]) if family == "ws" else 0.0,
                    p_fail=round(rng.uniform(0.01, 0.2), 3),
                    w_hi=rng.choice([1, 10, 50, 100, 1000]),
                    realizations=max(2, min(4096, _logu(rng, max(2.0, most / 16.0), max(3.0, most)))),
                    precision=rng.choice(["fp64", "fp32_recheck"]), pool=rng.choice([0.0, 0.1]))
    if kind == "batch":
        return dict(kind="batch", graphs=rng.randint(3, 12), n_lo=rng.randint(100, 300),
                    n_hi=rng.randint(700, 2400), realizations=rng.randint(32, 128))
    if kind == "rowwise":
        n = _logu(rng, 40, 160)
        return dict(kind="rowwise", n=n, m=int(n * rng.uniform(2.0, 4.0)),
                    draws=rng.randint(20, 120), hop_radius=rng.choice([0, 1, 2, 3]),
                    w_hi=rng.choice([9, 31, 63]))
    if kind == "query":
        n = _logu(rng, 100, 800)
        return dict(kind="query", family=rng.choice(["er", "ws"]), n=n,
                    degree=rng.choice([6.0, 8.0, 10.0, 12.0]), beta=0.1,
                    p_fail=round(rng.uniform(0.01, 0.3), 3), w_hi=100,
                    realizations=rng.randint(256, 600), precision="fp32_recheck",
                    n_perturb=rng.choice([0, 500]))
    if kind == "solve":
        n = _logu(rng, 100, 6000)
        c = max(4, min(n // 3, _logu(rng, 16, 1400)))
        return dict(kind="solve", n=n, c=c, realizations=2048,
                    spread="all" if c <= 120 else "part")
    if kind == "sweep":
        if rng.random() < 0.5:
            n = _logu(rng, 100, 2000)
            return dict(kind="sweep", n=n, c=min(n // 2, rng.randint(20, 150)), realizations=10000,
                        spread="all", perturbations=rng.randint(500, 2000))
        n = _logu(rng, 1500, 4000)
        return dict(kind="sweep", n=n, c=rng.randint(200, 900), realizations=2048, spread="part",
                    perturbations=rng.randint(152, 400))
    n = _logu(rng, 60, 700)
    return dict(kind="robust", n=n, c=max(8, min(n // 3, rng.randint(16, 120))), realizations=4096,
                spread="all")


# ---- inputs -----------------------------------------------------------------------------------

def _edges(keys, n):
    keys = np.unique(keys)
    return (keys // n).astype(np.int32), (keys % n).astype(np.int32)


def _graph(rng, family, n, degree, beta):
    """Simple undirected graph: ER of the given mean degree, or a Watts-Strogatz ring lattice
    (degree/2 neighbours per side, each edge rewired with probability beta)."""
    if family == "ws":
        k = max(2, int(round(degree / 2.0)) * 2)
        i = np.repeat(np.arange(n, dtype=np.int64), k // 2)
        j = (i + np.tile(np.arange(1, k // 2 + 1), n)) % n
        j = np.where(rng.random(j.shape[0]) < beta, rng.integers(0, n, j.shape[0]), j)
    else:
        m = int(rng.binomial(n * (n - 1) // 2, min(1.0, degree / (n - 1))))
        i, j = rng.integers(0, n, m), rng.integers(0, n, m)
    ok = i != j
    lo, hi = np.minimum(i, j)[ok], np.maximum(i, j)[ok]
    return _edges(lo * n + hi, n)


def _connected(rng, n, m):
    """Random tree plus uniform extra pairs, about m edges."""
    order = rng.permutation(n)
    par = order[(rng.random(n - 1) * np.arange(1, n)).astype(np.int64)]
    a = np.concatenate([order[1:], rng.integers(0, n, max(0, m - n + 1))])
    b = np.concatenate([par, rng.integers(0, n, max(0, m - n + 1))])
    ok = a != b
    return _edges(np.minimum(a, b)[ok].astype(np.int64) * n + np.maximum(a, b)[ok], n)


def _workload(n, eu, ev, p_survive, w_lo, w_hi, realizations, seed, **more):
    wl = SimpleNamespace(n=n, eu=eu, ev=ev, p_survive=p_survive, w_lo=w_lo, w_hi=w_hi,
                         realizations=realizations, seed=seed, graph_tag=0, alpha=0.15, k_min=5,
                         absorb_floor=1e-6, s_init=None, reward=None, candidates=None, top_k=0,
                         precision="fp64", recheck_margin=1e-4, tie_rel=1e-9, n_perturb=0,
                         l1_radius=0.05, r_min=0.05, perturb_seed=7)
    wl.__dict__.update(more)
    return wl


def _graph_workload(case, rng, seed):
    n = case["n"]
    eu, ev = _graph(rng, case["family"], n, case["degree"], case["beta"])
    pool = case.get("pool", 0.0)
    cand = np.sort(rng.choice(n, max(1, int(pool * n)), replace=False)).astype(np.int32) if pool else None
    return _workload(n, eu, ev, 1.0 - case["p_fail"], 1, case["w_hi"], case["realizations"], seed,
                     candidates=cand, precision=case["precision"], reward=rng.random(n),
                     n_perturb=case.get("n_perturb", 0))


def _batch_graphs(case, rng, seed):
    out = []
    for g in range(case["graphs"]):
        # sizes spread evenly over the logarithm of the range
        n = int(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** ((g + 0.5) / case["graphs"]))
        eu, ev = _graph(rng, "er" if g % 2 == 0 else "ws", n, 8.0, 0.2)
        out.append(_workload(n, eu, ev, 1.0 - rng.uniform(0.01, 0.2), 1, 50, case["realizations"],
                             seed, graph_tag=g, precision="fp32_recheck"))
    return out


def _chain_counts(case, seed):
    """Transition counts [n][n+1] of an estimated chain with c observed states (int32, GPU).
    spread "all": every anchor sees nearly the same centre distribution over all states (one
    giant component); "part": 100-400 targets per row from a popularity-skewed support."""
    n, c, R = case["n"], case["c"], case["realizations"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    opt = dict(device="cuda", dtype=torch.float64)
    C = torch.sort(torch.randperm(n, generator=g, device="cuda")[:c]).values
    pop = 1.0 / torch.arange(1, c + 1, **opt) ** (1.0 if case["spread"] == "all" else 0.8)
    pop = (pop / pop.sum())[torch.randperm(c, generator=g, device="cuda")]
    if case["spread"] == "all":
        w = pop * (1.0 + 0.1 * torch.rand((n, c), generator=g, **opt))
    else:
        k = 100.0 + 300.0 * torch.rand((n, 1), generator=g, **opt)
        w = -torch.log(torch.rand((n, c), generator=g, **opt).clamp_min(1e-12)) * pop
        w = w * (torch.rand((n, c), generator=g, **opt) < k * pop)
    absorbed = 0.02 if case["spread"] == "all" else 0.1
    w = w * ((1.0 - absorbed) * R / w.sum(1, keepdim=True).clamp_min(1e-300))
    cnt = torch.floor(w + torch.rand((n, c), generator=g, **opt)).to(torch.int32)
    j = torch.arange(c, device="cuda")
    cnt[j, j] = cnt[j, j].clamp_min(1)                   # every state is observed
    over = (cnt.sum(1) - R).clamp_min(0)
    cnt[torch.arange(n, device="cuda"), cnt.argmax(1)] -= over.to(torch.int32)
    counts = torch.zeros((n, n + 1), dtype=torch.int32, device="cuda")
    counts[:, C] = cnt
    counts[:, n] = (R - cnt.sum(1)).to(torch.int32)
    return counts


def _chain_query(case, seed):
    """A Query that holds the chain's counts, as after counting on a ring of its n nodes."""
    n = case["n"]
    eu, ev = _edges(np.arange(n - 1, dtype=np.int64) * n + np.arange(1, n), n)
    wl = _workload(n, eu, ev, 1.0, 1, 1, case["realizations"], 1,
                   reward=np.random.default_rng(seed).random(n),
                   n_perturb=case.get("perturbations", 0), perturb_seed=seed)
    q = afc.Query(wl)
    q.counts.copy_(_chain_counts(case, seed))
    return q


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "counts":
        return SimpleNamespace(kind=kind, q=afc.Query(_graph_workload(case, rng, seed)))
    if kind == "batch":
        qs = [afc.Query(wl) for wl in _batch_graphs(case, rng, seed)]
        probs = (afc.McProblem * len(qs))(*[q.prob for q in qs])
        r_count = np.array([q.wl.realizations for q in qs], np.uint32)
        ptrs = np.array([q.counts.data_ptr() for q in qs], np.uint64)
        wsb = afc.afc_transition_counts_batched_workspace(len(qs), probs, r_count)
        return SimpleNamespace(
            kind=kind, qs=qs, probs=probs, r_count=r_count, ptrs=ptrs,
            stats=torch.zeros((len(qs), afc.MC_STATS_WORDS), dtype=torch.int64, device="cuda"),
            ws=torch.empty(max(wsb, 256), dtype=torch.uint8, device="cuda"))
    if kind == "rowwise":
        eu, ev = _connected(rng, case["n"], case["m"])
        w0 = rng.integers(1, case["w_hi"] + 1, size=len(eu)).astype(np.uint32)
        wl = _workload(case["n"], eu, ev, 1.0, w0, case["w_hi"], case["draws"], seed)
        table = afc.afc_weight_table_normal(w0, case["w_hi"], 0.2, 0.1)
        return SimpleNamespace(kind=kind, q=afc.Query(wl, per_row=True, tie_random=True,
                                                      hop_radius=case["hop_radius"],
                                                      length_table=table))
    if kind == "query":
        wl = _graph_workload(case, rng, seed)
        return SimpleNamespace(kind=kind, bufs=afc.engine.HostBuffers(wl))
    q = _chain_query(case, seed)
    if kind == "sweep":
        q.run_solve()
        b_out = torch.empty((case["perturbations"], case["n"]), dtype=torch.float64, device="cuda")
        return SimpleNamespace(kind=kind, q=q, b_out=b_out)
    return SimpleNamespace(kind=kind, q=q)


# ---- the call ---------------------------------------------------------------------------------

def run(state):
    kind = state.kind
    if kind in ("counts", "rowwise"):
        q = state.q
        q.run_counts()
        # the statistics a user reads (the last word only says how the library ran the call)
        return {"counts": q.counts, "stats": q.stats[:7]}
    if kind == "batch":
        for q in state.qs:
            q.counts.zero_()
        state.stats.zero_()
        afc.afc_transition_counts_batched(len(state.qs), state.probs, state.r_count, state.ptrs,
                                          state.stats, state.ws, state.ws.numel(),
                                          torch.cuda.current_stream().cuda_stream)
        return {"counts": [q.counts for q in state.qs], "stats": state.stats[:, :7]}
    if kind == "query":
        res = afc.run_query_host(state.bufs)
        out = {"counts": state.bufs.counts, "b": state.bufs.b, "mu": state.bufs.mu,
               "expected_T": res.expected_T, "b_f": res.b_f, "max_rowsum_N": res.max_rowsum_N,
               "c": res.c, "sources": res.stats.sources, "edge_visits": res.stats.edge_visits}
        if state.bufs.query.n_perturb:
            out["perturb_counters"] = [int(x) for x in res.perturb_counters]
            out["perturb_maxima"] = [float(x) for x in res.perturb_maxima]
        return out
    q = state.q
    if kind == "solve":
        q.run_solve()
        return {"mu": q.mu, "b": q.b, "scalars": q.scalars, "c_list": q.c_list[:q.c],
                "lu": q.lu[:q.c * q.c], "piv": q.piv[:q.c]}
    if kind == "sweep":
        q.run_perturb(b_out=state.b_out)
        return {"counters": q.p_counters, "pairs": q.p_pairs, "hist": q.p_hist, "maxima": q.p_max,
                "b": state.b_out}
    res = q.robust_value(eps=0.01, sense=+1)
    return {k: res[k] for k in ("V", "Qstar", "b_star", "expected_T", "b_f")}


# ---- what one pass cannot do without ----------------------------------------------------------

def _count_flops(n, m_alive, realizations):
    """Two scans of the alive arcs per source (relax forward, accumulate backward), two
    operations per arc."""
    return 8.0 * m_alive * n * realizations


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind in ("counts", "query"):
        m = 0.5 * case["degree"] * n
        w = {"bytes": 12.0 * m + 8.0 * n + 4.0 * n * (n + 1),
             "flops": _count_flops(n, m * (1.0 - case["p_fail"]), case["realizations"])}
        if kind == "query":
            w["bytes"] += 24.0 * n
        return w
    if kind == "batch":
        # mean of n^2 and of n over the log-uniform sizes
        L = math.log(case["n_hi"] / case["n_lo"])
        n2 = (case["n_hi"] ** 2 - case["n_lo"] ** 2) / (2.0 * L)
        n1 = (case["n_hi"] - case["n_lo"]) / L
        return {"bytes": case["graphs"] * (4.0 * n2 + 56.0 * n1),
                "flops": case["graphs"] * case["realizations"] * 8.0 * 4.0 * 0.9 * n2}
    if kind == "rowwise":
        d = 2.0 * case["m"] / n
        ball = n if case["hop_radius"] == 0 else min(n, 1.0 + d * sum(
            (d - 1.0) ** k for k in range(case["hop_radius"])))
        return {"bytes": 12.0 * case["m"] + 4.0 * n * (n + 1),
                "flops": _count_flops(ball, case["m"] * (ball / n) ** 2, case["draws"] * n)}
    if kind == "solve":
        c = case["c"]
        return {"bytes": 4.0 * n * (n + 1) + 8.0 * c * c + 16.0 * n, "flops": 2.0 / 3.0 * c ** 3}
    if kind == "sweep":
        c, P = case["c"], case["perturbations"]
        nnz = n * (c + 1.0 if case["spread"] == "all" else min(c, 250.0))
        # the row draws and the column sums; c^2 triangular work on the nominal factors
        return {"bytes": 12.0 * nnz + 8.0 * P * n, "flops": P * (10.0 * nnz + 4.0 * c * c)}
    return {"bytes": 4.0 * n * (n + 1) + 16.0 * n * n, "flops": 3.0 * 2.0 / 3.0 * n ** 3}


# ---- the chain results in plain FP64 ----------------------------------------------------------

def _assembled(counts, R, alpha=0.15):
    """Q [n][n] and the absorption r [n] (alpha > 0: no row needs the floor)."""
    x = counts.to(torch.float64)
    return (1.0 - alpha) * x[:, :-1] / R, alpha + (1.0 - alpha) * x[:, -1] / R


class _Reduced:
    """The chain on its observed states C: mu_U = s_U, mu_C (I - Q_CC) = s_C + s_U Q_UC."""

    def __init__(self, counts, R):
        self.Q, self.r = _assembled(counts, R)
        n = self.n = counts.shape[0]
        self.C = torch.nonzero((counts[:, :n] > 0).any(0)).flatten()
        self.inC = torch.zeros(n, dtype=torch.bool, device=counts.device)
        self.inC[self.C] = True
        self.QC = self.Q[:, self.C].contiguous()          # [n][c]
        self.s = torch.full((n,), 1.0 / n, dtype=torch.float64, device=counts.device)
        self.eye = torch.eye(len(self.C), dtype=torch.float64, device=counts.device)
        self.lu = torch.linalg.lu_factor(self.eye - self.QC[self.C])
        self.mu, self.t = self.visits(self.QC, self.lu)

    def back(self, lu, y):                                 # x (I - Q_CC) = y
        return torch.linalg.lu_solve(*lu, y[:, None], adjoint=True)[:, 0]

    def visits(self, QC, lu=None):
        lu = torch.linalg.lu_factor(self.eye - QC[self.C]) if lu is None else lu
        y = self.s[self.C] + (self.s * ~self.inC) @ QC
        mu = self.s.clone()
        mu[self.C] = self.back(lu, y)
        tC = torch.linalg.lu_solve(*lu, torch.ones_like(y)[:, None])[:, 0]
        t = 1.0 + QC @ tC
        return mu, t


def _mul32(a, b):
    p = a * b                                              # the low 64 bits, also when negative
    return (p >> 32) & 0xFFFFFFFF, p & 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """First word of Philox4x32-10 (Salmon et al. 2011) on int64 tensors of 32-bit words."""
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mul32(c0, 0xD2511F53)
        h1, l1 = _mul32(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0


def _exact_sweep(case, seed, red, r_min=0.05, radius=0.05):
    n, c, C = red.n, len(red.C), red.C
    q = torch.cat([red.QC, red.r[:, None]], 1)             # [n][c + 1], absorption last
    on = q > 0.0
    on[:, -1] = True
    rows, cols = torch.nonzero(on, as_tuple=True)
    col_id = torch.cat([C, torch.tensor([n], device=C.device)])[cols]
    supp = on.sum(1).to(torch.float64)
    b0, T0 = red.mu / red.mu.sum(), red.mu.sum()
    zero = torch.zeros_like(rows)
    out, mx = torch.empty((case["perturbations"], n), dtype=torch.float64, device=C.device), [0.0] * 3
    dense = torch.zeros_like(q)
    for p in range(case["perturbations"]):
        u = _philox(col_id, rows, zero + p, zero + 1, seed)
        dense[rows, cols] = 2.0 * u.to(torch.float64) / 2.0 ** 32 - 1.0
        d = torch.where(on, dense - dense.sum(1, keepdim=True) / supp[:, None], 0.0)
        d = d * (radius / d.abs().sum(1, keepdim=True).clamp_min(1e-300))
        x = (q + d).clamp_min(0.0) * on
        x = x / x.sum(1, keepdim=True)
        low = x[:, -1:] < r_min
        tr = x[:, :-1].sum(1, keepdim=True)
        x = torch.where(low, x * (1.0 - r_min) / tr, x)
        QC = x[:, :-1].contiguous()
        mu, t = red.visits(QC)
        b = mu / mu.sum()
        ylin = torch.zeros(n, dtype=torch.float64, device=C.device)
        ylin[C] = red.back(red.lu, red.mu @ (QC - red.QC))
        lin = b0 + ylin / T0 - b0 * ylin.sum() / T0
        out[p] = b
        for k, v in enumerate(((b - b0).abs().max(), (b - lin).abs().max(), t.max())):
            mx[k] = max(mx[k], float(v))
    return {"counters": None, "pairs": None, "hist": None, "b": out,
            "maxima": torch.tensor(mx, dtype=torch.float64)}


def _exact_robust(counts, R, f, eps=0.01, r_min=0.05):
    """V = f + max over the box-and-budget set (on each row's support) of q . V, by policy
    iteration; every row fills its upper bounds in descending order of V while the budget
    lasts."""
    Q, _ = _assembled(counts, R)
    n = counts.shape[0]
    low = (Q - eps).clamp_min(0.0)
    cap = torch.where(Q > 0.0, (Q + eps).clamp_max(1.0) - low, 0.0)
    budget = (1.0 - r_min) - low.sum(1, keepdim=True)
    eye = torch.eye(n, dtype=torch.float64, device=Q.device)
    V = torch.zeros(n, dtype=torch.float64, device=Q.device)
    for _ in range(100):
        order = torch.argsort(V, descending=True, stable=True)
        cs = cap[:, order] * (V[order] > 0.0)
        before = torch.cumsum(cs, 1) - cs
        fill = torch.minimum(cs, (budget - before).clamp_min(0.0))
        P = low.clone()
        P[:, order] += fill
        new = torch.linalg.solve(eye - P, f)
        moved = float((new - V).abs().max() / new.abs().max())
        V = new
        if moved <= 1e-13:
            break
    mu = torch.linalg.solve((eye - P).T, torch.full((n,), 1.0 / n, dtype=torch.float64,
                                                    device=Q.device))
    b = mu / mu.sum()
    return {"V": V, "Qstar": P, "b_star": b, "expected_T": float(mu.sum()), "b_f": float(b @ f)}


def exact(case, seed):
    """The chain results in 64 bits; counting returns whole numbers only."""
    kind = case["kind"]
    if kind not in ("solve", "sweep", "robust"):
        return None
    counts, R = _chain_counts(case, seed), case["realizations"]
    f = torch.from_numpy(np.random.default_rng(seed).random(case["n"])).cuda()
    if kind == "robust":
        return _exact_robust(counts, R, f)
    red = _Reduced(counts, R)
    if kind == "sweep":
        return _exact_sweep(case, seed, red)
    b = red.mu / red.mu.sum()
    scalars = torch.tensor([float(red.mu.sum()), float(b @ f), float(red.t.max()),
                            float(len(red.C))], dtype=torch.float64)
    return {"mu": red.mu, "b": b, "scalars": scalars, "c_list": None, "piv": None,
            "lu": red.lu[0].reshape(-1)}
