"""The work that users of this package have it do, as cases that can be timed.

A case is one call sequence of a user's program through the public entry points
(``Matcher``, ``Batch``, ``Server``) on graphs of one family and size:

* ``solve``       cheap matching, then the search, on a graph already on the device
* ``cold``        the search alone, from the empty matching
* ``resolve``     the search from a matching the program holds (``match_from``)
* ``cover``       solve, then one search from the columns left unmatched: the
                  columns it reaches are the horizontal block of the coarse
                  Dulmage-Mendelsohn decomposition and give Koenig's vertex cover
* ``upload``      a new graph arrives in pinned host memory, then solve
* ``exact``       solve with the deterministic option
* ``batch``       many small graphs in one launch, with or without cheap matching
* ``batch_exact`` the same with the deterministic option
* ``serve``       a burst of requests from host memory through the server

Families: ``uniform`` (column degrees U{1..dmax}), ``rmat`` (power law, 0.57 /
0.19 / 0.19 / 0.05), ``stencil`` (5-point mesh with a tenth of the diagonal and
a part ``p_off`` of the other entries dropped; ``rcp``: rows and columns randomly
permuted), and for ``batch`` and ``serve`` the mixes of sizes that the benchmark
draws.  A batch's and a burst's sizes belong to the case (``sizes``), their
edges to the seed.

Which maximum matching the default option returns depends on which thread came
first and changes from run to run, so these cases return what does not: |M| of
every graph, and where the program asks for it the set of columns reached (the
same for every maximum matching).  The deterministic cases return the whole
matching.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1303_1379_gb300 import bmatch, synth


def listed():
    return [
        # the smallest graphs, one after another: a program that solves an assignment-feasibility
        # problem of a hundred rows at each step of an outer loop; latency is all that counts
        {"name": "solve_tiny", "kind": "solve", "family": "uniform", "nr": 100, "nc": 113, "dmax": 4, "graphs": 8},
        # a small sparse system's structural rank, from nothing
        {"name": "cold_uniform10k", "kind": "cold", "family": "uniform", "nr": 10000, "nc": 10000, "dmax": 8,
         "graphs": 1},
        # an ordinary sparse matrix of odd size: matching, then the coarse block structure
        {"name": "cover_uniform300k", "kind": "cover", "family": "uniform", "nr": 300007, "nc": 299993, "dmax": 5,
         "graphs": 1},
        # a large power-law graph (kron_g500-logn21's size), the benchmark's main graph
        {"name": "solve_rmat21", "kind": "solve", "family": "rmat", "n": 1 << 21, "mu": 16, "graphs": 1},
        # the same kind of graph, the search alone from a matching that the program kept
        {"name": "resolve_rmat1M", "kind": "resolve", "family": "rmat", "n": 1000003, "mu": 14, "graphs": 1},
        # the largest: a mesh whose augmenting paths run to thousands of columns (hugetrace, road networks)
        {"name": "cover_stencil2000", "kind": "cover", "family": "stencil", "g": 2000, "p_off": 0.05, "rcp": False,
         "graphs": 1},
        # the structure of the matrix changes between steps of an outer solver: each step uploads it
        {"name": "upload_rmat200k", "kind": "upload", "family": "rmat", "n": 200003, "mu": 12, "graphs": 1},
        # a permuted mesh whose result must be the same on every run
        {"name": "exact_stencil500", "kind": "exact", "family": "stencil", "g": 500, "p_off": 0.05, "rcp": True,
         "graphs": 1},
        # thousands of independent problems at once (scenario sweeps)
        {"name": "batch_4096", "kind": "batch", "graphs": 4096, "greedy": True, "sizes": 3},
        # fewer problems than the chip has multiprocessors, from the empty matching
        {"name": "batch_48_cold", "kind": "batch", "graphs": 48, "greedy": False, "sizes": 3},
        # a batch whose matchings must be the same on every run
        {"name": "batch_exact_512", "kind": "batch_exact", "graphs": 512, "greedy": True, "sizes": 3},
        # a burst of requests of very different sizes on a running server
        {"name": "serve_48", "kind": "serve", "requests": 48, "distinct": 24, "sizes": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, kind):
    """A graph of one family; the deterministic option and the search from the empty matching up to
    a quarter of the size."""
    top = 0.25 if kind in ("exact", "cold") else 1.0
    # (a mesh is nearly always matched whole, so |M| says little of it: cover and exact return more)
    family = rng.choice(["uniform", "uniform", "rmat"] + ["stencil"] * (kind in ("cover", "exact")))
    if family == "uniform":
        nr = _log_int(rng, 100, 1e6 * top)
        return {"family": family, "nr": nr, "nc": max(1, int(round(nr * rng.uniform(0.8, 1.25)))),
                "dmax": rng.randint(3, 8), "graphs": 8 if nr < 3000 else 1}
    if family == "rmat":
        n = _log_int(rng, 1000, 1.5e6 * top)
        return {"family": family, "n": n, "mu": rng.randint(3, 16), "graphs": 8 if n < 3000 else 1}
    g = _log_int(rng, 150, 1200 * math.sqrt(top))
    return {"family": family, "g": g, "p_off": 0.05 if g > 1000 or kind == "exact" else 0.2,
            "rcp": rng.random() < 0.5, "graphs": 1}


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "cold", "cover", "cover", "resolve", "upload", "exact", "batch", "batch",
                       "batch_exact", "serve"])
    if kind == "batch":
        return {"kind": kind, "graphs": _log_int(rng, 5, 4000), "greedy": rng.random() < 0.7,
                "sizes": rng.randint(0, 1000)}
    if kind == "batch_exact":
        return {"kind": kind, "graphs": _log_int(rng, 5, 1000), "greedy": rng.random() < 0.7,
                "sizes": rng.randint(0, 1000)}
    if kind == "serve":
        distinct = _log_int(rng, 3, 30)
        return {"kind": kind, "requests": distinct * rng.randint(1, 3), "distinct": distinct,
                "sizes": rng.randint(0, 1000)}
    return {"kind": kind, **_draw_graph(rng, kind)}


# ---------------------------------------------------------------- inputs
def _graph(case, seed, k):
    s = seed * 64 + k
    if case["family"] == "uniform":
        return synth.uniform_graph(case["nr"], case["nc"], case["dmax"], seed=s)
    if case["family"] == "rmat":
        n = case["n"]
        return synth.rmat_graph(max(1, (n - 1).bit_length()), n * case["mu"], seed=s, n=n)
    n = case["g"] ** 2
    g = synth.stencil_graph(case["g"], n // 10, case["p_off"], seed=s)
    return synth.permute_graph(g, seed=s) if case["rcp"] else g


def _batch(case, seed):
    """Uniform graphs of the benchmark's batch: rows log-uniform in [100, 50,000], columns = rows x U[0.8, 1.25],
    column degree U{1..round(2 mu - 1)} with mu ~ U[2, 12]."""
    rng = np.random.default_rng(case["sizes"])
    graphs = []
    for k in range(case["graphs"]):
        nr = int(np.exp(rng.uniform(np.log(100), np.log(50000))))
        nc = int(round(nr * rng.uniform(0.8, 1.25)))
        graphs.append(synth.uniform_graph(nr, nc, int(round(2 * rng.uniform(2, 12) - 1)), seed=seed, graph=k))
    off = [np.concatenate([[0], np.cumsum([f(g) for g in graphs])]).astype(np.int64)
           for f in (lambda g: g.n_rows, lambda g: g.n_cols, lambda g: g.nnz)]
    return synth.Batch(np.array([g.n_rows for g in graphs], np.int32), np.array([g.n_cols for g in graphs], np.int32),
                       *off, np.concatenate([g.col_ptr for g in graphs]), np.concatenate([g.row_idx for g in graphs]))


def _request_graphs(case, seed):
    """The served mix: uniform and R-MAT graphs in turn, 1,000 to 1,000,000 rows."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for i in range(case["distinct"]):
        nr = int(np.exp(rng.uniform(np.log(1e3), np.log(1e6))))
        nc = max(1, int(round(nr * rng.uniform(0.8, 1.25))))
        mu = rng.uniform(3, 16)
        if i % 2 == 0:
            out.append(synth.uniform_graph(nr, nc, max(1, int(round(2 * mu - 1))), seed=seed * 64 + i))
        else:
            n = max(nr, nc)
            out.append(synth.rmat_graph((n - 1).bit_length(), int(n * mu), seed=seed * 64 + i, n=n))
    return out


def _empty(n):
    return torch.full((n,), -1, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "batch_exact"):
        batch = bmatch.Batch.from_synth(_batch(case, seed), deterministic=int(kind == "batch_exact"))
        return {"case": case, "batch": batch, "rm": _empty(batch.total_rows), "cm": _empty(batch.total_cols),
                "cards": torch.empty(batch.n_graphs, dtype=torch.int32, device="cuda")}
    if kind == "serve":
        host = [(g.n_rows, g.n_cols, torch.from_numpy(g.col_ptr).pin_memory(), torch.from_numpy(g.row_idx).pin_memory())
                for g in _request_graphs(case, seed)]
        # a program that shares the GPU lets idle workers leave soon
        return {"case": case, "server": bmatch.Server(pool_bytes=4 << 30, idle_timeout_ns=200_000), "host": host}
    problems = []
    for k in range(case["graphs"]):
        g = _graph(case, seed, k)
        p = {"rm": _empty(g.n_rows), "cm": _empty(g.n_cols)}
        if kind == "upload":
            p["m"] = bmatch.Matcher(g.n_rows, g.n_cols, g.nnz)
            p["host"] = (torch.from_numpy(g.col_ptr).pin_memory(), torch.from_numpy(g.row_idx).pin_memory())
        else:
            cp, ri = torch.from_numpy(g.col_ptr).cuda(), torch.from_numpy(g.row_idx).cuda()
            p["m"] = bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, deterministic=int(kind == "exact"))
        if kind == "cover":
            p["level"] = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
        if kind == "resolve":  # the kept matching: the deterministic option's cheap matching, the same on every run
            with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, deterministic=1) as first:
                first.greedy()
                p["rm0"], p["cm0"] = torch.empty_like(p["rm"]), torch.empty_like(p["cm"])
                first.get_matching(p["rm0"], p["cm0"])
        problems.append(p)
    return {"case": case, "problems": problems}


# ---------------------------------------------------------------- the calls
def _solve(kind, p):
    m = p["m"]
    if kind == "resolve":
        return m.match_from(p["rm0"], p["cm0"], p["rm"], p["cm"]).card
    if kind == "upload":
        m.upload_csr(*p["host"])
    m.set_matching()  # empty
    if kind != "cold":
        m.greedy()
    card = m.match(p["rm"], p["cm"]).card
    if kind == "cover":
        m.bfs(p["level"])
        return card, p["level"] > 1  # 1: not reached
    if kind == "exact":
        return card, p["rm"], p["cm"]
    return card


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("batch", "batch_exact"):
        rm, cm = state["rm"].fill_(-1), state["cm"].fill_(-1)
        state["batch"].match(rm, cm, greedy=case["greedy"], card_out=state["cards"])
        return (state["cards"], rm, cm) if kind == "batch_exact" else state["cards"]
    if kind == "serve":
        srv, host = state["server"], state["host"]
        ids = [srv.submit(*host[i % len(host)]) for i in range(case["requests"])]
        done = [srv.wait(i) for i in ids]
        for i in ids:
            srv.release(i)
        return np.array([[d["status"], d["card"]] for d in done], dtype=np.int64)
    return [_solve(kind, p) for p in state["problems"]]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: every graph's column CSR read once, every result written once.  No arithmetic counts."""
    kind = case["kind"]
    if kind in ("batch", "batch_exact"):  # the recipe's means: rows, columns, edges of a graph
        rows, edges = 49900 / math.log(500), 49900 / math.log(500) * 1.025 * 7
        return {"bytes": case["graphs"] * 4 * (edges + 2 * 1.025 * rows + rows), "flops": 0}
    if kind == "serve":
        rows = 999000 / math.log(1000)
        return {"bytes": case["requests"] * 4 * (rows * 1.03 * 10 + rows * 1.03), "flops": 0}
    if case["family"] == "uniform":
        nr, nc = case["nr"], case["nc"]
        nnz = nc * (1 + case["dmax"]) / 2
    elif case["family"] == "rmat":
        nr = nc = case["n"]
        nnz = 0.96 * nc * case["mu"]
    else:
        nr = nc = case["g"] ** 2
        nnz = nc * (0.9 + 4 * (1 - case["p_off"]))
    return {"bytes": case["graphs"] * 4 * (nnz + nc + nr + nc), "flops": 0}


def exact(case, seed):
    """Every output is a whole number or a truth value: there is nothing to round."""
    return None
