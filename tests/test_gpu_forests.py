"""Blocks of more and of at most 32 nodes side by side in warp teams (at most 256 nodes), every
output bit for bit against the oracle: forests with more heads than SMs and with fewer, loads below
and above M and equal ones, bundles of chains that end in joins, ids in and out of topological order."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import compare_dag, context, gpu_schedule
from tests.test_gpu_peel import _forest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _bundles(rng, sizes, width, wmax, permute):
    """Blocks of exactly sizes[i] nodes: chains side by side whose ends meet in a join, one bundle
    after another."""
    src, dst, at, join = [], [], 0, -1
    for n in sizes:
        first = at
        for i in range(n):
            v = at + i
            if i >= width:
                src.append(v - width)
                dst.append(v)
            elif join >= 0:
                src.append(join)
                dst.append(v)
        at += n
        src += range(max(first, at - width), at)
        dst += [at] * min(n, width)
        join = at
        at += 1
    V = at
    perm = rng.permutation(V) if permute else np.arange(V)
    rp, col = wl.csr_from_edges(V, perm[np.array(src, np.int64)], perm[np.array(dst, np.int64)])
    return rp, col, rng.integers(1, wmax + 1, V).astype(np.int64), rng.integers(0, 65, V).astype(np.uint8)


@pytest.mark.parametrize("M", [1, 7, 31, 33, 148, 256, 300])
def test_large_and_small_blocks(ctx, M):
    rng = np.random.default_rng(110 + M)
    dags = []
    for V in (32, 33, 64, 65, 200, 256):
        for roots in (1, 20, V // 2, V):
            for wmax in (1, 3, 2 * M, 40 * M):
                dags.append(_forest(rng, V, roots, wmax, permute=(roots + wmax) % 2 == 0))
    for sizes in ((32, 33, 40), (100, 5, 100), (31, 31, 31), (250,), (34,) * 7):
        for width in (2, 10, 40):
            for wmax in (3, 20 * M):
                dags.append(_bundles(rng, sizes, width, wmax, permute=width == 10))
    b = wl.from_dags(dags, M)
    lb, res = gpu_schedule(ctx, b, 0)
    for d in range(b.n_dags):
        compare_dag(b, res, d, 0)
    lb.free()
