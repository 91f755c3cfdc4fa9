"""Candidate kernels that take one DAG per CTA or cluster, at their edges and bit for bit
against the oracle: candidate counts around a warp's 32 and 64 and beyond one pass (2,048),
plans around the 32-row windows, bytes that divide by every 64 m, sums that need 64 bits, and
exhaustive enumerations whose base, plan length (64 rows) or arithmetic takes each path."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context
from tests.oracle_checks import random_small_dag
from tests.test_gpu_bound import _run
from tests.test_gpu_search import _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _dags(seed, sizes, wmax, M, p=0.1):
    rng = np.random.default_rng(seed)
    return wl.from_dags([random_small_dag(rng, V, p, wmax) for V in sizes], M)


@pytest.mark.parametrize("n_alloc", [1, 31, 32, 33, 63, 65, 96, 1100])
def test_byte_candidates(ctx, n_alloc):
    b = _dags(40 + n_alloc, (1, 2, 15, 31, 32, 33, 64, 90, 300), 2 ** 17 - 1, 255)
    alloc, stride = wl.candidate_allocations(b, 2, n_alloc, list(range(0, 256)), seed=n_alloc)
    _run(ctx, b, [0, 3], n_alloc, alloc, stride)


@pytest.mark.parametrize("mode", [oracle.SEARCH_RANDOM, oracle.SEARCH_PERTURB])
@pytest.mark.parametrize("n_alloc", [1, 32, 33, 100, 1500])
@pytest.mark.parametrize("wmax", [5000, 2 ** 32 - 1])
def test_generated_candidates(ctx, mode, n_alloc, wmax):
    b = _dags(50, (1, 30, 32, 33, 70, 280), wmax, 148)
    levels = [0, 0, 1, 2, 3, 4] if mode == oracle.SEARCH_PERTURB else [1, 3, 7, 64, 200]
    _check(ctx, b, [0, 2], n_alloc, levels, 7, range(b.n_dags), mode=mode)


@pytest.mark.parametrize("levels,n_alloc", [([3], 2 ** 12), ([1, 2], 3 ** 7), (list(range(1, 16)), 16 ** 3), ([5, 2, 9], 1)])
@pytest.mark.parametrize("wmax", [30, 2 ** 32 - 1])
def test_exhaustive_paths(ctx, levels, n_alloc, wmax):
    b = _dags(60, (1, 2, 3, 7, 13, 31, 40), wmax, 6, 0.3)
    _check(ctx, b, [0, 1, 3], n_alloc, levels, 0, range(b.n_dags), mode=oracle.SEARCH_EXHAUSTIVE)
    # only the winners: repeated candidates are skipped, ties still go to the smallest
    lb = ctx.load(b)
    for v in (0, 1, 3):
        lb.schedule(v, fields=("status",))
    full = lb.search([0, 1, 3], n_alloc, levels, want_all=True, mode=oracle.SEARCH_EXHAUSTIVE)
    best = lb.search([0, 1, 3], n_alloc, levels, mode=oracle.SEARCH_EXHAUSTIVE)
    for f in ("best_bound", "best_cand"):
        assert np.array_equal(full[f], best[f]), f
    lb.free()
