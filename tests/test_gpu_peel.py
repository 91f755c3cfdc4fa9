"""Alg.1 and the closure in CTA teams, every output bit for bit against the oracle: forests
(one block whose heads outnumber the SMs, so that Top_M evicts and refills), with loads below
and above M and equal W^anc, blocks around a warp's 32 nodes, ids in and out of topological
order, workspaces in shared memory (both classes) and in global memory."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import compare_dag, context, gpu_schedule

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _forest(rng, V, roots, wmax, permute):
    """A random out-forest: node v >= roots hangs below a random earlier node."""
    par = np.array([rng.integers(max(0, v - 60), v) for v in range(roots, V)], dtype=np.int64)
    perm = rng.permutation(V) if permute else np.arange(V)
    rp, col = wl.csr_from_edges(V, perm[par], perm[np.arange(roots, V)])
    return rp, col, rng.integers(1, wmax + 1, V).astype(np.int64), rng.integers(0, 65, V).astype(np.uint8)


def _stars(rng, V, leaves):
    """Groups of `leaves` sources that share one join: blocks of exactly that many nodes."""
    src, dst, n = [], [], 0
    while n + leaves + 1 <= V:
        src += list(range(n, n + leaves))
        dst += [n + leaves] * leaves
        n += leaves + 1
    rp, col = wl.csr_from_edges(V, src, dst)
    return rp, col, rng.integers(1, 300, V).astype(np.int64), np.full(V, 40, np.uint8)


@pytest.mark.parametrize("M", [1, 5, 40, 148, 4096])
def test_forests_and_block_sizes(ctx, M):
    rng = np.random.default_rng(90 + M)
    dags = []
    for V in (257, 600, 1100):
        for roots in (1, 30, V // 2, V):
            dags.append(_forest(rng, V, roots, 3 if roots == 30 else max(2, 2 * M), permute=roots % 2 == 0))
        for leaves in (31, 32, 33, 80):
            dags.append(_stars(rng, V, leaves))
    b = wl.from_dags(dags, M)
    for smem in (2, 0):
        lb, res = gpu_schedule(ctx, b, 0)
        if smem == 0:
            lb.set_tuning(cta_smem=0)
            res = lb.schedule(0, fields=("bound", "group_of", "block_of", "wanc", "level", "m", "status"), check=False)
        for d in range(b.n_dags):
            compare_dag(b, res, d, 0, edges=smem == 2)
        lb.free()
