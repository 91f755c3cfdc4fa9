"""Batches from host arrays around the sizes at which arrays stop travelling together (64 KB an
array, 256 KB of outputs), one DAG per team and stolen DAGs, one size class and several, against
the oracle; the caller's arrays are overwritten as soon as they are loaded."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import compare_dag, context

pytestmark = pytest.mark.gpu
FIELDS = ("bound", "status", "level", "wanc", "block_of", "group_of", "exec_group", "m", "crit_path")


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _batch(rng, sizes, M):
    dags = []
    for v in sizes:
        src = np.arange(v - 1)
        keep = rng.random(len(src)) < 0.6
        rp, col = wl.csr_from_edges(v, src[keep], src[keep] + 1)
        dags.append((rp, col, rng.integers(1, 200, v).astype(np.int64), rng.integers(0, 65, v).astype(np.uint8)))
    return wl.from_dags(dags, M)


# 8,192 loads are 64 KB; 9 fields of 128 DAGs of 64 nodes are 265 KB, of 127 DAGs 263 KB; 608 CTAs' worth
@pytest.mark.parametrize("sizes,fields", [
    ([20], FIELDS), ([300], FIELDS), ([20, 300], FIELDS), ([64] * 127, FIELDS), ([64] * 128, FIELDS),
    ([64] * 129, ("bound", "status", "m")), ([64] * 100, ("bound", "status")), ([3] * 608, FIELDS), ([3] * 609, ("bound", "status")),
    ([10] * 5000, ("bound", "status", "m")), ([2000], ("bound", "status", "wanc")),
])
def test_host_batches(ctx, sizes, fields):
    rng = np.random.default_rng(len(sizes) + sizes[0])
    b = _batch(rng, sizes, 40)
    given = wl.Batch(*(getattr(b, k).copy() for k in ("node_off", "edge_off", "row_ptr", "col", "wcet", "k64")), b.M)
    stream = torch.cuda.Stream()
    for other in (False, True):
        lb = ctx.load(given)
        for k in ("node_off", "edge_off", "row_ptr", "col", "wcet", "k64"):
            getattr(given, k)[:] = 0  # the library has its own copy
        if other:
            ctx.set_stream(stream.cuda_stream)
        res = lb.schedule(0, fields=fields)
        lb.free()
        ctx.set_stream(None)
        assert res["rc"] == 0
        for d in range(0, b.n_dags, max(1, b.n_dags // 40)):
            compare_dag(b, res, d, 0, edges=False)
        for k in ("node_off", "edge_off", "row_ptr", "col", "wcet", "k64"):
            getattr(given, k)[:] = getattr(b, k)
