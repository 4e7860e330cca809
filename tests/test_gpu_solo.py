"""Small graphs on one block and on one cluster of blocks: sizes on both sides
of every limit (words of 32 ids, one block / cluster / grid, parts of a long
column, rows beyond a block's memory), every start, and the calls' error cases."""
import numpy as np
import pytest

import oracle
from paper_1303_1379_gb300 import bmatch, synth

from helpers import assert_maximum, csr_from_edges, oracle_max, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def hub_graph():
    """A few columns hold most rows (beyond an even share of the block that owns them), the others 1-3."""
    rng = np.random.default_rng(5)
    nr, edges = 9000, []
    for c in range(6000):
        deg = [9000, 128, 129, 4000, 257][c // 64] if c % 64 == 0 and c // 64 < 5 else int(rng.integers(1, 4))
        edges += [(int(r), c) for r in rng.choice(nr, deg, replace=False)]
    return csr_from_edges(nr, 6000, edges)


CASES = {
    "1x1": lambda: csr_from_edges(1, 1, [(0, 0)]),
    "31x33": lambda: synth.uniform_graph(31, 33, 3, seed=1),
    "8192 entries": lambda: csr_from_edges(1500, 1024, [((7 * c + 31 * k * k) % 1500, c) for c in range(1024) for k in range(8)]),
    "8193 entries": lambda: csr_from_edges(1500, 1025, [((7 * c + 31 * k * k) % 1500, c) for c in range(1024) for k in range(8)] + [(3, 1024)]),
    "few columns": lambda: synth.uniform_graph(30000, 511, 40, seed=2),
    "few rows": lambda: synth.uniform_graph(600, 20000, 5, seed=3),
    "at the side limit": lambda: synth.uniform_graph(32768, 32768, 4, seed=4),
    "over the side limit": lambda: synth.uniform_graph(32769, 30000, 4, seed=4),
    "hubs": hub_graph,
    "mesh": lambda: synth.stencil_graph(120, 1440, 0.1, seed=6),
    "rmat": lambda: synth.rmat_graph(13, 60000, seed=7),
    "repeated rows": lambda: csr_from_edges(700, 900, [(r % 700, r % 900) for r in range(9000)], keep_order=True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_small_graphs_reach_the_maximum(name):
    g = CASES[name]()
    want = oracle_max(g)
    cp, ri = to_dev(g)
    rm = torch.empty(g.n_rows, dtype=torch.int32, device="cuda")
    cm = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
    rg, cg, _ = oracle.greedy(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)
    d_rg, d_cg = torch.from_numpy(rg).cuda(), torch.from_numpy(cg).cuda()

    def check(res, start):
        assert_maximum(g, rm.cpu().numpy(), cm.cpu().numpy(), res.card, want)
        assert res.stats["initial_card"] == start and res.stats["endpoints"] == want - start
        levels, ends, _, _ = m.phase_profile()
        assert int(levels.sum()) == res.stats["levels"] and int(ends.sum()) == want - start

    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri) as m:
        check(m.match(rm, cm), 0)
        m.set_matching()
        card = m.greedy()
        m.get_matching(rm, cm)
        r0, c0 = rm.cpu().numpy(), cm.cpu().numpy()
        assert oracle.validate(g.n_rows, g.n_cols, g.col_ptr, g.row_idx, r0, c0) == (0, card)
        assert np.all(r0[g.row_idx[np.repeat(c0 < 0, np.diff(g.col_ptr))]] >= 0)  # maximal
        check(m.match(rm, cm), card)
        check(m.match_from(d_rg, d_cg, rm, cm), int((cg >= 0).sum()))
        bad = cg.copy()
        bad[int(np.flatnonzero(cg >= 0)[0])] = -1  # a column forgets its row
        with pytest.raises(bmatch.BMError) as e:
            m.match_from(d_rg, torch.from_numpy(bad).cuda())
        assert e.value.status == bmatch.BM_ERR_INVALID_MATCHING
        check(m.match(rm, cm), 0)  # the empty matching is installed, the context usable
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz) as m:
        h_rm, h_cm = rg.copy(), cg.copy()
        res = m.match_host(g.col_ptr, g.row_idx, h_rm, h_cm)
        assert_maximum(g, h_rm, h_cm, res.card, want)
        if g.nnz:
            wrong = g.row_idx.copy()
            wrong[-1] = g.n_rows
            with pytest.raises(bmatch.BMError) as e:
                m.match_host(g.col_ptr, wrong)
            assert e.value.status == bmatch.BM_ERR_INVALID_CSR
        assert m.match_host(g.col_ptr, g.row_idx).card == want
