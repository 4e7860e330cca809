"""Limits of a match launch (time, phases) on both routes: small graphs on one
block or cluster, and the persistent grid kernel (block_size given)."""
import numpy as np
import pytest

from paper_1303_1379_gb300 import bmatch

from helpers import csr_from_edges, oracle_max, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def chains(lengths):
    """One augmenting path per length L, of L levels: columns c0 .. c(L-1) and rows r0 .. r(L-1), column ci lists
    r(i-1), its match, and ri; c0 and the last row are unmatched.  Returns the graph and that matching."""
    n = sum(lengths)
    edges, rm, cm = [], np.full(n, -1, np.int32), np.full(n, -1, np.int32)
    at = 0
    for length in lengths:
        for i in range(length):
            edges.append((at + i, at + i))
            if i:
                edges.append((at + i - 1, at + i))
                rm[at + i - 1], cm[at + i] = at + i, at + i - 1
        at += length
    return csr_from_edges(n, n, edges), rm, cm


@pytest.mark.parametrize("n", [600, 9000])  # one block (fewer than 8,192 entries), one cluster
@pytest.mark.parametrize("limit", [1, 200_000])
def test_time_limit_ends_a_small_graph_within_a_phase(n, limit):
    """A search of n levels of about 2 us and more, in one phase that ends without a path (the row at its end is not
    listed)."""
    g, rm, cm = chains([n])
    g = csr_from_edges(n, n, [(r, c) for c in range(n) for r in (c - 1, c) if 0 <= r < n - 1])
    cp, ri = to_dev(g)
    d_rm, d_cm = torch.from_numpy(rm).cuda(), torch.from_numpy(cm).cuda()
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, total_timeout_ns=limit) as m:
        with pytest.raises(bmatch.BMError) as e:
            m.match_from(d_rm, d_cm)
        assert e.value.status == bmatch.BM_ERR_TIMEOUT
        with pytest.raises(bmatch.BMError) as e:
            m.match()
        assert e.value.status == bmatch.BM_ERR_STATE
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri) as m:  # the GPU and a new context are fine
        res = m.match_from(d_rm, d_cm)
        assert res.card == n - 1 and res.stats["max_levels_in_phase"] == n and res.stats["grid"] in (1, 16)
