"""Carried search trees of the persistent kernel: searches of few and of many
phases (cut short, carried, rebuilt from their roots) from starts of every
quality end in a certified maximum matching, for several launch geometries and
again on the same context (claim stamps of an earlier launch)."""
import numpy as np
import pytest

import oracle
from paper_1303_1379_gb300 import bmatch, synth

from helpers import assert_maximum, oracle_max, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRAPHS = {
    "mesh": lambda: synth.stencil_graph(260, 6760, 0.05, seed=11),           # long paths
    "sparse": lambda: synth.uniform_graph(70001, 69997, 4, seed=12),         # many roots that fail
    "rmat": lambda: synth.rmat_graph(16, 1 << 19, seed=13),
    "wide": lambda: synth.uniform_graph(400003, 399989, 5, seed=14),         # levels on both sides of the claim limit
}


@pytest.fixture(scope="module", params=list(GRAPHS))
def graph(request):
    g = GRAPHS[request.param]()
    return g, oracle_max(g)


@pytest.mark.parametrize("block,per_sm", [(0, 0), (96, 1), (1024, 1)])
def test_carried_search_is_maximum(graph, block, per_sm):
    g, want = graph
    cp, ri = to_dev(g)
    rm = torch.empty(g.n_rows, dtype=torch.int32, device="cuda")
    cm = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
    rg, cg, _ = oracle.greedy(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)
    d_rg, d_cg = torch.from_numpy(rg).cuda(), torch.from_numpy(cg).cuda()
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, block_size=block, blocks_per_sm=per_sm) as m:
        for start in ("empty", "oracle", "greedy", "empty"):
            m.set_matching()
            if start == "oracle":
                m.set_matching(d_rg, d_cg)
            elif start == "greedy":
                m.greedy()
            res = m.match(rm, cm)
            assert_maximum(g, rm.cpu().numpy(), cm.cpu().numpy(), res.card, want)
            levels, ends, _, _ = m.phase_profile()
            assert int(levels.sum()) == res.stats["levels"]
            assert int(ends.sum()) == res.stats["endpoints"] == want - res.stats["initial_card"]


def test_a_long_search_passes_both_limits():
    """A mesh from a one-sided start (every column's first free row) takes more
    phases than are carried."""
    g = synth.stencil_graph(500, 25000, 0.05, seed=2)
    cp, ri = to_dev(g)
    rm = torch.empty(g.n_rows, dtype=torch.int32, device="cuda")
    cm = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, deterministic=1) as m:
        m.greedy()
        m.set_options(deterministic=0)
        res = m.match(rm, cm)
    assert_maximum(g, rm.cpu().numpy(), cm.cpu().numpy(), res.card, oracle_max(g))
    assert res.stats["phases"] > 20
