"""The block routine's cheap matching (entry counts saturating at 255, lists on
both sides of its 8-row window, rows beyond the shared-memory marks, partial
starts) and the batch's default geometry on both sides of its limit."""
import numpy as np
import pytest

import oracle
from paper_1303_1379_gb300 import bmatch, synth

from helpers import csr_from_edges

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def to_batch(graphs):
    off = [np.concatenate([[0], np.cumsum([f(g) for g in graphs])]).astype(np.int64)
           for f in (lambda g: g.n_rows, lambda g: g.n_cols, lambda g: g.nnz)]
    return synth.Batch(np.array([g.n_rows for g in graphs], np.int32), np.array([g.n_cols for g in graphs], np.int32),
                       *off, np.concatenate([g.col_ptr for g in graphs]), np.concatenate([g.row_idx for g in graphs]))


def graphs_at_the_edges():
    rng = np.random.default_rng(9)
    out = [csr_from_edges(1, 1, [(0, 0)]), csr_from_edges(3, 40, [])]
    # every column lists rows 0-6 and one of the others: rows of more than 255 entries, lists of 1, 8 and 9
    out.append(csr_from_edges(400, 390, [(r, c) for c in range(390) for r in (*range(7), 7 + c)]))
    out.append(csr_from_edges(500, 300, [(int(r), c) for c in range(300) for r in rng.choice(500, (1, 7, 8, 9, 16, 17)[c % 6], replace=False)]))
    out.append(synth.uniform_graph(61440, 9000, 3, seed=1))  # the last row count with marks in shared memory
    out.append(synth.uniform_graph(61441, 9000, 3, seed=1))
    out.append(synth.stencil_graph(60, 360, 0.2, seed=2))
    return out


@pytest.mark.parametrize("partial", [False, True])
def test_batch_cheap_matching_at_its_edges(partial):
    graphs = graphs_at_the_edges()
    b = to_batch(graphs)
    want = [oracle.hopcroft_karp(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)[2] for g in graphs]
    rm0, cm0 = np.full(int(b.row_off[-1]), -1, np.int32), np.full(int(b.col_off[-1]), -1, np.int32)
    if partial:
        for k, g in enumerate(graphs):
            _, cg, _ = oracle.greedy(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)
            for c in np.flatnonzero(cg >= 0)[::3]:
                rm0[b.row_off[k] + cg[c]], cm0[b.col_off[k] + c] = c, cg[c]
    with bmatch.Batch.from_synth(b) as bb:
        rm, cm = torch.from_numpy(rm0).cuda(), torch.from_numpy(cm0).cuda()
        card = torch.empty(len(graphs), dtype=torch.int32, device="cuda")
        bb.match(rm, cm, greedy=True, card_out=card)
    assert card.cpu().tolist() == want
    rm, cm = rm.cpu().numpy(), cm.cpu().numpy()
    for k, g in enumerate(graphs):
        assert oracle.validate(g.n_rows, g.n_cols, g.col_ptr, g.row_idx, rm[b.row_off[k]:b.row_off[k + 1]],
                               cm[b.col_off[k]:b.col_off[k + 1]]) == (0, want[k])


@pytest.mark.parametrize("n,block", [(40, 1024), (700, 512)])
def test_batch_default_geometry(n, block):
    graphs = [synth.uniform_graph(200, 210, 4, seed=k) for k in range(n)]
    b = to_batch(graphs)
    with bmatch.Batch.from_synth(b) as bb:
        rm = torch.full((int(b.row_off[-1]),), -1, dtype=torch.int32, device="cuda")
        cm = torch.full((int(b.col_off[-1]),), -1, dtype=torch.int32, device="cuda")
        card = torch.empty(n, dtype=torch.int32, device="cuda")
        _, st = bb.match(rm, cm, card_out=card)
    assert st["block"] == block
    for k in (0, n - 1):
        g = graphs[k]
        assert int(card[k]) == oracle.hopcroft_karp(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)[2]


@pytest.mark.parametrize("first", [{"deterministic": 1}, {"bfs": 0}, {"wr_one_endpoint": 0}], ids=str)
def test_batch_counts_rows_when_an_option_comes_to_read_them(first):
    """Created with options that do not read the rows' entry counts, matched with ones that do: a column lists a row
    of everyone's, one shared with few and one of its own, which the cheap matching must give it."""
    n = 3000  # (no row has its column's number)
    lists = [np.roll([n, n + 1 + c % 100, n + 101 + c], c % 3) for c in range(n)]
    one = synth.Graph(2 * n + 101, n, (3 * np.arange(n + 1)).astype(np.int32), np.concatenate(lists).astype(np.int32), "own rows")
    b = to_batch([one, synth.uniform_graph(70000, 300, 4, seed=1), one])
    with bmatch.Batch.from_synth(b, **first) as bb:
        rm = torch.full((int(b.row_off[-1]),), -1, dtype=torch.int32, device="cuda")
        cm = torch.full((int(b.col_off[-1]),), -1, dtype=torch.int32, device="cuda")
        bb.match(rm, cm)
        assert int((cm >= 0).sum()) == 2 * n + 300
        bb.set_options(deterministic=0, bfs=1, wr_one_endpoint=1)
        rm.fill_(-1)
        cm.fill_(-1)
        bb.match(rm, cm)
    for k in (0, 2):
        assert np.array_equal(cm[b.col_off[k]:b.col_off[k + 1]].cpu().numpy(), n + 101 + np.arange(n))
    assert int((cm >= 0).sum()) == 2 * n + 300


@pytest.mark.parametrize("sizes,det,block", [
    # rows x graphs; one block of 1,024 threads an SM holds 152 graphs at once, two of 512 hold 304
    ([(200, 152)], 0, 1024), ([(200, 153)], 0, 512), ([(200, 303)], 1, 512), ([(1000, 200)], 0, 512),
    ([(1000, 200)], 1, 512), ([(10000, 1), (200, 600)], 0, 1024), ([(40000, 1), (200, 300)], 0, 1024),
    ([(40000, 8), (200, 300)], 1, 1024), ([(3000, 20), (100, 280)], 0, 1024), ([(3000, 20), (2500, 280)], 0, 512), ([(20000, 310)], 1, 1024), ([(20000, 310)], 0, 1024),
], ids=str)
def test_batch_default_geometry_by_the_longest_wait(sizes, det, block):
    pool = {nr: synth.uniform_graph(nr, nr + nr // 20, 7, seed=nr) for nr, _ in sizes}
    graphs = [pool[nr] for nr, n in sizes for _ in range(n)]
    b = to_batch(graphs)
    with bmatch.Batch.from_synth(b, deterministic=det) as bb:
        rm = torch.full((int(b.row_off[-1]),), -1, dtype=torch.int32, device="cuda")
        cm = torch.full((int(b.col_off[-1]),), -1, dtype=torch.int32, device="cuda")
        card = torch.empty(len(graphs), dtype=torch.int32, device="cuda")
        _, st = bb.match(rm, cm, card_out=card)
        want = {nr: oracle.hopcroft_karp(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)[2] for nr, g in pool.items()}
        assert card.cpu().tolist() == [want[nr] for nr, n in sizes for _ in range(n)]
        assert st["block"] == block and st["grid"] == (152 if block == 1024 else 304)
        # a size from the caller counts as before
        bb.set_options(blocks_per_sm=1)
        assert bb.match(rm, cm)[1]["block"] == 512
        bb.set_options(blocks_per_sm=0, block_size=256)
        assert bb.match(rm, cm)[1]["block"] == 256
