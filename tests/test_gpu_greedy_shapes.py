"""The cheap matching on graphs of extreme shapes: few columns of many rows and
the reverse, single degree classes, rows that all columns list, rows whose
entry counts share a slot, diagonals, hubs, and both sides of the limits that
send a graph to one block, a cluster of blocks or the grid."""
import numpy as np
import pytest

import oracle
from paper_1303_1379_gb300 import bmatch, synth

from helpers import assert_maximum, oracle_max, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def regular(nr, nc, k, seed=0):
    """nc columns of k different rows each."""
    rng = np.random.default_rng(seed)
    rows = np.array([rng.choice(nr, k, replace=False) for _ in range(nc)], np.int32)
    return synth.Graph(nr, nc, (np.arange(nc + 1) * k).astype(np.int32), rows.reshape(-1).copy(), "regular")


def from_lists(nr, lists):
    ptr = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int32)
    return synth.Graph(nr, len(lists), ptr, np.concatenate(lists).astype(np.int32), "lists")


def greedy(g, start=None, first=None, **options):
    """bm_greedy's (rmatch, cmatch) from `start`; checks that it is valid, maximal and keeps the start."""
    cp, ri = to_dev(g)
    rm = torch.empty(g.n_rows, dtype=torch.int32, device="cuda")
    cm = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, **options) as m:
        if first:
            first(m)
        m.set_matching()
        card = m.greedy()
        m.get_matching(rm, cm)
        res = m.match()
    rm, cm = rm.cpu().numpy(), cm.cpu().numpy()
    assert oracle.validate(g.n_rows, g.n_cols, g.col_ptr, g.row_idx, rm, cm) == (0, card)
    assert np.all(rm[g.row_idx[np.repeat(cm < 0, np.diff(g.col_ptr))]] >= 0)
    assert res.card == oracle_max(g)
    return rm, cm


SHAPES = [(100000, 10, 5000), (40000, 300, 300), (33000, 1, 3000), (10, 40000, 3), (600, 40000, 30), (3000, 3000, 300)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("block", [0, 64])
def test_cheap_matching_of_few_columns_or_few_rows(shape, block):
    greedy(regular(*shape), block_size=block)


@pytest.mark.parametrize("degrees", [[1], [2], [3], [8], [9, 32], [33], [2048], [2049], [2, 2049], [8, 33], [1, 9]], ids=str)
def test_every_degree_class_by_itself_is_matched(degrees):
    """Passes that no column needs are not launched; the others must be."""
    rng = np.random.default_rng(degrees[0])
    lists = [rng.choice(34000, degrees[c % len(degrees)], replace=False) for c in range(70)]
    rm, cm = greedy(from_lists(34000, lists))  # more rows than the small graphs' kernel takes
    assert np.all(cm >= 0)


@pytest.mark.parametrize("first", [None, "deterministic", "host"])
@pytest.mark.parametrize("n", [2000, 40000])  # small graphs' kernel / grid
def test_counted_rows_decide_the_choice(n, first):
    """Column c lists a row that all columns list, one that every 4,096th column lists too and one of its own, which
    it must take, as the row of fewest entries.  The counts are made when the cheap matching first needs them, also
    of a context whose CSR was checked under another option."""
    # (no row has its column's number; the own rows' counting slots are those of the shared ones)
    lists = [np.roll([n, n + 1 + c % 4096, n + 4097 + c], c % 3) for c in range(n)]
    g = from_lists(2 * n + 4097, lists)

    def deterministic(m):
        m.greedy()
        m.match()
        m.set_options(deterministic=0)

    def host(m):
        m.set_options(driver=1)
        m.match()
        m.set_options(driver=0)

    rm, cm = greedy(g, first={"deterministic": deterministic, "host": host}.get(first), deterministic=int(first == "deterministic"))
    shared = np.bincount(1 + np.arange(n) % 4096, minlength=4097)[1 + np.arange(n) % 4096] > 1
    assert np.array_equal(cm[shared], n + 4097 + np.flatnonzero(shared))


def test_counts_follow_the_csr():
    """A new CSR in the same context: its own counts, whichever call brought it."""
    n = 40000
    size = n + n // 2 + n  # rows: n that no column lists, n / 2 that two list, n that one lists
    own = [np.array([n + n // 2 + c, n + c % (n // 2)]) for c in range(n)]
    graphs = [from_lists(size, own), from_lists(size, [x[::-1].copy() for x in own])]
    rm = torch.empty(size, dtype=torch.int32, device="cuda")
    cm = torch.empty(n, dtype=torch.int32, device="cuda")
    with bmatch.Matcher(size, n, 2 * n) as m:
        for k, call in enumerate(["upload", "host", "host given", "upload", "host"]):
            g = graphs[k % 2]
            ri = n + (g.row_idx - n + 777 * k) % (size - n)  # every time another row numbering
            if call == "upload":
                m.upload_csr(g.col_ptr, ri)
            else:
                given = (np.full(size, -1, np.int32), np.full(n, -1, np.int32)) if call == "host given" else ()
                assert m.match_host(g.col_ptr, ri, *given).card == n
            m.set_matching()
            assert m.greedy() == n
            m.get_matching(rm, cm)
            assert np.array_equal(cm.cpu().numpy(), n + (n // 2 + np.arange(n) + 777 * k) % (size - n))


@pytest.mark.parametrize("n,k,cols", [(40, 30, 30), (100, 300, 300), (2, 1200, 400), (2, 2500, 400)])
def test_columns_that_list_the_same_rows(n, k, cols):
    """n blocks of columns that all list the same k rows: every one of them gets one."""
    lists = [b * k + np.roll(np.arange(k), 7 * c) for b in range(n) for c in range(cols)]
    rm, cm = greedy(from_lists(34000, lists))
    assert np.all(cm >= 0)


def banded(n, offsets):
    rows = np.arange(n)[:, None] + np.array(offsets)[None, :]
    ok = (rows >= 0) & (rows < n)
    return synth.Graph(n, n, np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32), rows[ok].astype(np.int32), "banded")


@pytest.mark.parametrize("n", [1000, 20000, 40000])  # one block, cluster, grid
@pytest.mark.parametrize("offsets", [(0, 1), (-1, 0), (-1, 0, 1), tuple(range(-20, 21)), tuple(range(0, 1200))], ids=len)
def test_a_whole_diagonal_is_taken(n, offsets):
    """Bidiagonal matrices have one maximum matching, which no other choice than the diagonal finds."""
    g = banded(n, offsets if len(offsets) < 100 or n > 2000 else offsets[:700])
    if g.nnz > 30_000_000:
        g = banded(n, offsets[:100])
    rm, cm = greedy(g)
    assert np.array_equal(cm, np.arange(n))


def test_a_batch_takes_the_diagonal():
    graphs = [banded(n, o) for n in (50, 3000) for o in ((0, 1), (-1, 0), (-3, -2, -1, 0, 1, 2, 3))]
    off = [np.concatenate([[0], np.cumsum([f(g) for g in graphs])]).astype(np.int64)
           for f in (lambda g: g.n_rows, lambda g: g.n_cols, lambda g: g.nnz)]
    b = synth.Batch(np.array([g.n_rows for g in graphs], np.int32), np.array([g.n_cols for g in graphs], np.int32), *off,
                    np.concatenate([g.col_ptr for g in graphs]), np.concatenate([g.row_idx for g in graphs]))
    with bmatch.Batch.from_synth(b) as bb:
        rm = torch.full((int(off[0][-1]),), -1, dtype=torch.int32, device="cuda")
        cm = torch.full((int(off[1][-1]),), -1, dtype=torch.int32, device="cuda")
        bb.match(rm, cm)
    for k, g in enumerate(graphs):
        assert np.array_equal(cm[off[1][k]:off[1][k + 1]].cpu().numpy(), np.arange(g.n_cols))


@pytest.mark.parametrize("block", [0, 1024])
def test_hub_columns_take_the_row_of_fewest_entries(block):
    """Eight columns of 3,000 rows, all but one of them shared: the one, in the middle of the first step's rows."""
    lists = [100 + np.concatenate([np.arange(1000), [2999 + h], np.arange(1000, 2999)]) for h in range(8)]
    lists += [np.array([5000 + c]) for c in range(33000)]
    rm, cm = greedy(from_lists(40000, lists), block_size=block)
    assert np.array_equal(cm[:8], 100 + 2999 + np.arange(8))


@pytest.mark.parametrize("shape", [(600, 40000, 30), (1500, 40000, 3), (34000, 34000, 3)], ids=str)
def test_first_phase_from_nothing(shape):
    """One level, whether the cheap matching's kernels run it or (many more columns than rows) the search."""
    g = regular(*shape)
    cp, ri = to_dev(g)
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri) as m:
        res = m.match()
        levels, ends, _, _ = m.phase_profile()
    want = oracle_max(g)
    assert res.card == want == ends.sum() == res.stats["endpoints"] and res.stats["initial_card"] == 0
    assert ends[0] > 0.5 * want and levels.sum() == res.stats["levels"]


ROUTES = {  # rows, columns, entries a column -> blocks of the search (0: the grid)
    (64, 64, 10): 1, (1024, 1024, 8): 1, (1100, 1025, 8): 16, (20000, 4096, 2): 1, (20000, 4097, 1): 16,
    (3000, 511, 64): 1, (3000, 511, 65): 0, (3000, 512, 65): 16,
    (32768, 32768, 6): 16, (32768, 32768, 12): 16, (32768, 32768, 13): 0, (32769, 100, 3): 0, (100, 32769, 3): 0,
    (12000, 12288, 17): 16, (12000, 12289, 17): 0, (12000, 12288, 16): 16, (16000, 16384, 12): 16,
}


@pytest.mark.parametrize("shape", list(ROUTES), ids=str)
def test_routes_of_small_graphs(shape):
    """Every call on both sides of the limits, the result checked and the route read from the statistics."""
    nr, nc, k = shape
    rng = np.random.default_rng(k)
    base = rng.permutation(nr)
    lists = [base[(c * 37 + np.arange(k) * (1 + c % 5)) % nr] for c in range(nc)]
    g = from_lists(nr, lists)
    want = oracle_max(g)
    cp, ri = to_dev(g)
    r0, c0, _ = oracle.greedy(nr, nc, g.col_ptr, g.row_idx)
    rm = torch.empty(nr, dtype=torch.int32, device="cuda")
    cm = torch.empty(nc, dtype=torch.int32, device="cuda")

    def check(res, a, b):
        assert_maximum(g, a.cpu().numpy() if torch.is_tensor(a) else a, b.cpu().numpy() if torch.is_tensor(b) else b, res.card, want)
        assert res.stats["grid"] == ROUTES[shape] or (not ROUTES[shape] and res.stats["grid"] > 16)
        assert res.stats["endpoints"] == want - res.stats["initial_card"]

    with bmatch.Matcher(nr, nc, g.nnz, cp, ri) as m:
        check(m.match(rm, cm), rm, cm)  # from nothing
        m.set_matching()
        m.greedy()
        check(m.match(rm, cm), rm, cm)
        check(m.match_from(torch.from_numpy(r0).cuda(), torch.from_numpy(c0).cuda(), rm, cm), rm, cm)
    with bmatch.Matcher(nr, nc, g.nnz) as m:
        h_r, h_c = np.full(nr, -1, np.int32), np.full(nc, -1, np.int32)
        check(m.match_host(g.col_ptr, g.row_idx, h_r, h_c), h_r, h_c)  # given, but empty
        assert m.match_host(g.col_ptr, g.row_idx).card == want
        h_r, h_c = r0.copy(), c0.copy()
        check(m.match_host(g.col_ptr, g.row_idx, h_r, h_c), h_r, h_c)
        # an entry of the columns' array alone is not an empty start, and a bad row is not read
        h_r, h_c = np.full(nr, -1, np.int32), np.full(nc, -1, np.int32)
        h_c[nc // 2] = 0
        with pytest.raises(bmatch.BMError) as e:
            m.match_host(g.col_ptr, g.row_idx, h_r, h_c)
        assert e.value.status == bmatch.BM_ERR_INVALID_MATCHING
        bad = g.row_idx.copy()
        bad[g.nnz // 2] = nr
        for given in ((), (np.full(nr, -1, np.int32), np.full(nc, -1, np.int32))):
            with pytest.raises(bmatch.BMError) as e:
                m.match_host(g.col_ptr, bad, *given)
            assert e.value.status == bmatch.BM_ERR_INVALID_CSR
        assert m.match_host(g.col_ptr, g.row_idx).card == want


@pytest.mark.parametrize("n", [12288, 12289])
@pytest.mark.parametrize("call", ["from", "host", "installed"])
def test_many_unmatched_columns_go_to_the_grid(n, call):
    """A given start that leaves more columns unmatched than the cluster searches from; one more pair is matched."""
    nr = n + 1
    g = from_lists(nr, [[c, (c + 1) % nr] for c in range(n + 1)])
    rm, cm = np.full(nr, -1, np.int32), np.full(n + 1, -1, np.int32)
    rm[0], cm[n] = n, 0
    cp, ri = to_dev(g)
    d_rm, d_cm = torch.from_numpy(rm).cuda(), torch.from_numpy(cm).cuda()
    with bmatch.Matcher(nr, n + 1, g.nnz) as m:
        if call == "host":
            res = m.match_host(g.col_ptr, g.row_idx, rm, cm)
        else:
            m.upload_csr(g.col_ptr, g.row_idx)
            if call == "installed":
                m.set_matching(d_rm, d_cm)
                res = m.match(d_rm, d_cm)
            else:
                res = m.match_from(d_rm, d_cm, d_rm, d_cm)  # in place
            rm, cm = d_rm.cpu().numpy(), d_cm.cpu().numpy()
        assert_maximum(g, rm, cm, res.card, n + 1)
        assert res.stats["initial_card"] == 1 and (res.stats["grid"] == 16) == (n <= 12288)
        again = m.match()
        assert again.card == n + 1 and again.stats["initial_card"] == n + 1
