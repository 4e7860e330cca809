"""The cheap matching's column order and classes: the tile and lane orders are
permutations (host model), and columns at the edges of every degree class and
of the 32-column tiles end in a valid, maximal matching on the GPU."""
import numpy as np
import pytest

import oracle
from paper_1303_1379_gb300 import bmatch, synth

from helpers import to_dev

M32 = 0xFFFFFFFF


def scatter_bits(x, bits):
    """bmd::scatter_bits of bm_device.cuh."""
    mask, h = (1 << bits) - 1, (bits + 1) >> 1
    for m in (0x9E3779B1, 0x85EBCA77, 0xC2B2AE3D):
        x = (x * m) & mask
        x ^= x >> h
    return x


@pytest.mark.parametrize("bits", range(17))
def test_tile_order_is_a_permutation(bits):
    assert sorted(scatter_bits(k, bits) for k in range(1 << bits)) == list(range(1 << bits))


def test_lane_order_is_a_permutation():
    rng = np.random.default_rng(1)
    for th in [0, M32] + rng.integers(0, 1 << 32, 500).tolist():
        lanes = [(((lane * (th | 1)) & M32) + (th >> 5) & M32 ^ (th >> 10)) & 31 for lane in range(32)]
        assert sorted(lanes) == list(range(32))


def classes_graph(n_cols, seed):
    """Columns whose degrees lie on both sides of every class limit, in random
    order, rows with repetitions allowed, few enough rows to fight over."""
    rng = np.random.default_rng(seed)
    degs = rng.choice([0, 1, 2, 3, 4, 5, 8, 9, 31, 32, 33, 128, 129, 2048, 2049], n_cols,
                      p=[.04, .14, .14, .12, .1, .1, .1, .08, .04, .04, .04, .02, .02, .01, .01])
    nr = max(3, int(0.9 * n_cols))
    ptr = np.zeros(n_cols + 1, np.int32)
    ptr[1:] = np.cumsum(degs)
    return synth.Graph(nr, n_cols, ptr, rng.integers(0, nr, int(ptr[-1])).astype(np.int32), "classes")


@pytest.mark.gpu
@pytest.mark.parametrize("n_cols", [1, 31, 32, 33, 1000, 40001])
@pytest.mark.parametrize("partial", [False, True])
def test_greedy_is_valid_and_maximal_at_the_class_edges(n_cols, partial):
    torch = pytest.importorskip("torch")
    g = classes_graph(n_cols, seed=n_cols)
    cp, ri = to_dev(g)
    rm0, cm0 = oracle.empty_matching(g.n_rows, g.n_cols)
    if partial:
        rg, cg, _ = oracle.greedy(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)
        for c in np.flatnonzero(cg >= 0)[::2]:
            rm0[cg[c]], cm0[c] = c, cg[c]
    rm = torch.empty(g.n_rows, dtype=torch.int32, device="cuda")
    cm = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri) as m:
        m.set_matching(torch.from_numpy(rm0).cuda(), torch.from_numpy(cm0).cuda())
        card = m.greedy()
        m.get_matching(rm, cm)
        res = m.match()
    rm, cm = rm.cpu().numpy(), cm.cpu().numpy()
    assert oracle.validate(g.n_rows, g.n_cols, g.col_ptr, g.row_idx, rm, cm) == (0, card)
    open_edge = np.repeat(cm < 0, np.diff(g.col_ptr))
    assert np.all(rm[g.row_idx[open_edge]] >= 0)
    kept = cm0 >= 0
    assert np.array_equal(cm[kept], cm0[kept])
    assert res.card == oracle.hopcroft_karp(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)[2]
