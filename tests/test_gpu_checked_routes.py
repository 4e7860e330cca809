"""The default option's two searches -- one block or cluster for small graphs,
the persistent grid kernel for the others and wherever a launch geometry or a
barrier limit is given -- on the same small, odd and degenerate graphs, in the
normal library and in the range-checked one.  There the matching is checked
between phases by both, which the library counts."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1303_1379_gb300 import bmatch, synth

from helpers import assert_maximum, csr_from_edges, oracle_max, to_dev

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GRAPHS = {
    "1x1": lambda: csr_from_edges(1, 1, [(0, 0)]),
    "empty columns": lambda: csr_from_edges(5, 40, [(r, 8 * r) for r in range(5)]),
    "no entries": lambda: csr_from_edges(33, 31, []),
    "star": lambda: csr_from_edges(65, 64, [(0, c) for c in range(64)] + [(64, 63)]),
    "repeated": lambda: csr_from_edges(7, 9, [(r % 7, r % 9) for r in range(200)], keep_order=True),
    "33x31": lambda: synth.uniform_graph(33, 31, 4, seed=1),
    "1025x1023": lambda: synth.uniform_graph(1025, 1023, 3, seed=2),
    "uniform": lambda: synth.uniform_graph(7919, 8111, 5, seed=21),
    "wide": lambda: synth.uniform_graph(900, 5003, 6, seed=3),
    "rmat": lambda: synth.rmat_graph(13, 50000, seed=5),
    "mesh": lambda: synth.stencil_graph(90, 810, 0.1, seed=6),
    "permuted mesh": lambda: synth.permute_graph(synth.stencil_graph(110, 1210, 0.1, seed=6), seed=7),
}
OPTIONS = [{}, {"block_size": 512}, {"block_size": 96, "blocks_per_sm": 1}, {"wait_timeout_ns": 2_000_000_000}]


def run(g, options):
    """Every start; returns the phases that found paths."""
    import torch
    want = oracle_max(g)
    cp, ri = to_dev(g)
    rm = torch.empty(g.n_rows, dtype=torch.int32, device="cuda")
    cm = torch.empty(g.n_cols, dtype=torch.int32, device="cuda")
    rg, cg, _ = oracle.greedy(g.n_rows, g.n_cols, g.col_ptr, g.row_idx)
    d_rg, d_cg = torch.from_numpy(rg).cuda(), torch.from_numpy(cg).cuda()
    phases = 0
    with bmatch.Matcher(g.n_rows, g.n_cols, g.nnz, cp, ri, **options) as m:
        for start in ("empty", "oracle", "greedy", "from"):
            m.set_matching()
            if start == "oracle":
                m.set_matching(d_rg, d_cg)
            elif start == "greedy":
                m.greedy()
            res = m.match_from(d_rg, d_cg, rm, cm) if start == "from" else m.match(rm, cm)
            assert_maximum(g, rm.cpu().numpy(), cm.cpu().numpy(), res.card, want)
            assert (res.stats["grid"] in (1, 16)) == (not options)
            levels, ends, _, _ = m.phase_profile()
            assert int(levels.sum()) == res.stats["levels"] and int(ends.sum()) == res.stats["endpoints"]
            found = int(np.count_nonzero(ends))
            # (the first phase from nothing is the cheap matching's, before the search)
            phases += found - (start == "empty" and found > 0)
    return phases


@pytest.mark.parametrize("options", OPTIONS, ids=str)
@pytest.mark.parametrize("name", list(GRAPHS))
def test_both_searches_reach_the_maximum(name, options):
    run(GRAPHS[name](), options)


CHILD = r'''
import ctypes, json, sys
sys.path.insert(0, ROOT); sys.path.insert(0, ROOT + "/tests")
import test_gpu_checked_routes as t
from paper_1303_1379_gb300 import bmatch, build
assert bmatch.library_path() == build.LIB_CHECKED
sweeps = bmatch.load().bm_checked_sweeps
sweeps.restype = ctypes.c_int64
out = []
for name, make in t.GRAPHS.items():
    for options in t.OPTIONS:
        before = sweeps()
        phases = t.run(make(), options)
        out.append([name, options, phases, sweeps() - before])
print("RESULT " + json.dumps(out))
'''


def test_range_checked_library_checks_both_searches_between_phases():
    from paper_1303_1379_gb300 import build
    build.build(checked=True)
    env = dict(os.environ, BMATCH_CHECKED="1")
    res = subprocess.run([sys.executable, "-c", CHILD.replace("ROOT", repr(ROOT))], env=env, capture_output=True, text=True,
                         timeout=600)
    assert res.returncode == 0, res.stdout[-3000:] + res.stderr[-3000:]
    rows = json.loads([l for l in res.stdout.splitlines() if l.startswith("RESULT ")][-1][7:])
    assert len(rows) == len(GRAPHS) * len(OPTIONS) and sum(r[2] for r in rows) > 100
    for name, options, phases, sweeps in rows:
        assert sweeps >= phases, (name, options, phases, sweeps)
