"""Graphs whose edges outgrow shared memory, every output against the oracle: closure rows on both
sides of 4, 8, 16, 32 and 64 words, nodes of more than 8, 16 and 32 predecessors, chains, and
sparse nodes beside dense ones."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import compare_dag, context

pytestmark = pytest.mark.gpu
FIELDS = ("bound", "status", "level", "wanc", "block_of", "group_of", "exec_group", "m", "n_rows")


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


@pytest.mark.parametrize("V", [5, 200, 256, 257, 512, 513, 1024, 1030, 2048, 2049, 2200, 4097])
def test_dense_and_mixed(ctx, V):
    rng = np.random.default_rng(700 + V)
    dags = []
    for deg in (2, 12, 20, 70):
        src, dst = [], []
        for v in range(1, V):
            n = min(v, int(rng.integers(0, deg + 1)) if v % 3 else 1)
            lo = 0 if v % 2 else max(0, v - 4 * deg)  # near and far predecessors
            for u in rng.choice(np.arange(lo, v), size=min(n, v - lo), replace=False):
                src.append(int(u))
                dst.append(v)
        perm = rng.permutation(V) if deg == 12 else np.arange(V)
        rp, col = wl.csr_from_edges(V, perm[np.array(src, np.int64)], perm[np.array(dst, np.int64)])
        dags.append((rp, col, rng.integers(1, 2 ** (31 if deg == 20 else 14), V).astype(np.int64),
                     rng.integers(0, 65, V).astype(np.uint8)))
    b = wl.from_dags(dags, 148)
    lb = ctx.load(b)
    lb.set_tuning(cta_smem=0, warp_max_v=0)  # global workspaces at every size
    res = lb.schedule(0, fields=FIELDS, check=False)
    for d in range(b.n_dags):
        compare_dag(b, res, d, 0, edges=False)
    lb.free()
