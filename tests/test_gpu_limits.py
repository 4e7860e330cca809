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


@pytest.mark.parametrize("block", [0, 512])  # one cluster, the grid
def test_a_limited_phase_is_a_whole_phase(block):
    """3,000 paths of three levels and 40 of twelve, all apart: one whole phase finds every one, however narrow its
    last levels are."""
    g, rm, cm = chains([3] * 3000 + [12] * 40)
    cp, ri = to_dev(g)
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, max_phases=1, block_size=block) as m:
        m.set_matching(torch.from_numpy(rm).cuda(), torch.from_numpy(cm).cuda())
        res = m.match(allow_incomplete=True)
        levels, ends, _, _ = m.phase_profile()
    assert res.card == g.n_cols and res.stats["initial_card"] == g.n_cols - 3040
    assert levels.tolist() == [12] and ends.tolist() == [3040]


@pytest.mark.parametrize("block", [0, 512])
@pytest.mark.parametrize("phases", [1, 2])
def test_limited_phases_from_the_empty_matching(block, phases):
    """The first phase from nothing is one level, with or without the cheap matching's kernels running it: it leaves
    a maximal matching, and no more than that counts as done."""
    rng = np.random.default_rng(phases)
    n = 3000
    g = csr_from_edges(n, n, [(int(r), c) for c in range(n) for r in rng.integers(0, n, 3)])
    cp, ri = to_dev(g)
    rm = torch.empty(n, dtype=torch.int32, device="cuda")
    cm = torch.empty(n, dtype=torch.int32, device="cuda")
    with bmatch.Matcher(n, n, g.nnz, cp, ri, max_phases=phases, block_size=block) as m:
        res = m.match(rm, cm, allow_incomplete=True)
        levels, ends, _, _ = m.phase_profile()
    assert len(levels) == phases and levels[0] == 1 and ends.sum() == res.card < oracle_max(g)
    rm, cm = rm.cpu().numpy(), cm.cpu().numpy()
    assert np.all(rm[g.row_idx[np.repeat(cm < 0, np.diff(g.col_ptr))]] >= 0)
    assert res.status == bmatch.BM_INCOMPLETE


@pytest.mark.parametrize("nnz,per_sm", [(1200 * 1024, 1), (1200 * 1024 + 1, 2)])
def test_default_grid_of_the_deterministic_search(nnz, per_sm):
    """One block an SM up to 1,228,800 entries, two beyond; the matching is the same for every grid."""
    rng = np.random.default_rng(4)
    nr, nc = 300000, 200000
    ptr = np.concatenate([[0], np.sort(rng.integers(0, nnz + 1, nc - 1)), [nnz]]).astype(np.int32)
    cp, ri = torch.from_numpy(ptr).cuda(), torch.from_numpy(rng.integers(0, nr, nnz).astype(np.int32)).cuda()
    out = []
    for options in ({}, {"blocks_per_sm": 3 - per_sm}):
        rm = torch.empty(nr, dtype=torch.int32, device="cuda")
        with bmatch.Matcher(nr, nc, nnz, cp, ri, deterministic=1, **options) as m:
            m.greedy()
            res = m.match(rm)
        out.append((rm, res.stats["grid"]))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert [grid for _, grid in out] == [per_sm * sms, (3 - per_sm) * sms]
    assert torch.equal(out[0][0], out[1][0])
