"""Candidate kernels by the length of a plan, bit for bit against the oracle: tables of a row's choices
that the lanes of a warp share in other ways for 1, 2, 4, 8, 16 and more rows, and exhaustive
enumerations of plans of 63, 64 (all that the kernel's row records hold) and 65 rows, the row of
node 0 in a group of its own, among others, first and last."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context
from tests.oracle_checks import random_small_dag
from tests.test_gpu_search import _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


@pytest.mark.parametrize("mode", [oracle.SEARCH_RANDOM, oracle.SEARCH_PERTURB])
@pytest.mark.parametrize("n_alloc", [15, 64])
def test_choices_of_short_plans(ctx, mode, n_alloc):
    rng = np.random.default_rng(120)
    b = wl.from_dags([random_small_dag(rng, V, 0.3, 5000) for V in (1, 2, 3, 4, 5, 7, 8, 9, 12, 15, 16, 17)], 8)
    levels = [0, 1, 2, 3, 4] if mode == oracle.SEARCH_PERTURB else list(range(1, 32, 2))
    _check(ctx, b, [0, 1], n_alloc, levels, 11, range(b.n_dags), mode=mode)


@pytest.mark.parametrize("V", [63, 64, 65])
def test_exhaustive_at_the_row_limit(ctx, V):
    rng = np.random.default_rng(130 + V)
    chain = (np.arange(V - 1), np.arange(1, V))
    edges = [((), ()), chain, (chain[1], chain[0]),                       # alone; first; last
             (np.full(V - 1, V - 1), np.arange(V - 1)),                   # among the last
             (np.arange(1, V), np.zeros(V - 1, np.int64))]                # the join of all others
    dags = []
    for src, dst in edges:
        rp, col = wl.csr_from_edges(V, np.array(src, np.int64), np.array(dst, np.int64))
        dags.append((rp, col, rng.integers(1, 40, V).astype(np.int64), rng.integers(0, 65, V).astype(np.uint8)))
    b = wl.from_dags(dags, 6)
    lb = ctx.load(b)
    assert (lb.schedule(1, fields=("n_rows",))["n_rows"] == V).all()  # (no parallel launches: a row per node)
    lb.free()
    for levels, n_alloc in (([1, 2], 3 ** 6), (list(range(1, 16)), 16 ** 2)):
        _check(ctx, b, [1], n_alloc, levels, 0, range(b.n_dags), mode=oracle.SEARCH_EXHAUSTIVE)
        _check(ctx, b, [0, 1], n_alloc, levels, 0, range(b.n_dags), mode=oracle.SEARCH_EXHAUSTIVE)
