"""Alg.2's group step at its branch points, every output bit for bit against the oracle and
the same with the few outputs most callers ask for: groups of 1 to 148 members (one member,
one lane per member, more than a warp), loads on both sides of the 32-bit arithmetic rule
(64 M max C^ below 2^32 or not), and released sets on both sides of the summary-word rule
(1,024 nodes)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import compare_dag, context, gpu_schedule
from tests.oracle_checks import random_small_dag

pytestmark = pytest.mark.gpu

FEW = ("bound", "status", "n_groups", "n_seg", "n_rows", "exec_group", "m", "crit_path")


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _check(ctx, batch, variant):
    lb, res = gpu_schedule(ctx, batch, variant)
    few = lb.schedule(variant, fields=FEW, check=False)
    for d in range(batch.n_dags):
        compare_dag(batch, res, d, variant)
    for f in FEW:
        assert np.array_equal(few[f], res[f]), f
    lb.free()


def _wide(rng, n, load_hi):
    """n isolated nodes (groups of up to M of them) feeding a sparse second layer."""
    V = n + 10
    src = rng.integers(0, n, 30)
    dst = n + rng.integers(0, 10, 30)
    key = np.unique(src * V + dst)
    rp, col = wl.csr_from_edges(V, key // V, key % V)
    return rp, col, rng.integers(1, load_hi + 1, V).astype(np.int64), rng.integers(0, 65, V).astype(np.uint8)


@pytest.mark.parametrize("variant", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("M", [33, 148, 300])
def test_group_sizes(ctx, variant, M):
    rng = np.random.default_rng(70 + variant)
    dags = [_wide(rng, n, hi) for n in (1, 2, 31, 32, 33, 64, 65, 148, 200) for hi in (1, 9, M - 1, 4 * M)]
    _check(ctx, wl.from_dags(dags, M), variant)


@pytest.mark.parametrize("M", [1, 8, 148, 4096])
def test_load_width_rule(ctx, M):
    """Largest load at 2^32 / (64 M) - 1, at it and one above, and at 2^32 - 1."""
    rng = np.random.default_rng(71)
    edge = 2 ** 26 // M
    dags = []
    for top in (edge - 1, edge, edge + 1, 2 ** 32 - 1):
        for V in (40, 300):
            rp, col, w, k = random_small_dag(rng, V, 6.0 / V, 10)
            w = rng.integers(max(1, top // 1000), top + 1, V).astype(np.int64)
            w[rng.integers(0, V)] = top
            dags.append((rp, col, w, k))
    for variant in range(5):
        _check(ctx, wl.from_dags(dags, M), variant)


@pytest.mark.parametrize("V", [1023, 1024, 1025, 2100])
def test_released_set_width(ctx, V):
    rng = np.random.default_rng(72)
    rp, col, w, k = random_small_dag(rng, V, 3.0 / V, 3000)
    for variant in (0, 2, 3):
        _check(ctx, wl.from_dags([(rp, col, w, k)], 148), variant)


@pytest.mark.parametrize("V", [2, 17, 33, 64, 100, 128, 129, 200, 256, 300])
def test_ids_in_and_out_of_topological_order(ctx, V):
    """The same graphs with ids in topological order (a path of its own in the warp teams) and
    permuted, with many equal W^anc (equal loads) and with distinct ones."""
    rng = np.random.default_rng(73 + V)
    dags = []
    for wmax in (2, 5000):
        rp, col, w, k = random_small_dag(rng, V, min(0.5, 6.0 / V), wmax)
        dags.append((rp, col, w, k))
        src, perm = np.repeat(np.arange(V), np.diff(rp)), rng.permutation(V)
        prp, pcol = wl.csr_from_edges(V, perm[src], perm[col])
        pw, pk = np.empty_like(w), np.empty_like(k)
        pw[perm], pk[perm] = w, k
        dags.append((prp, pcol, pw, pk))
    for M in (4, 148):
        _check(ctx, wl.from_dags(dags, M), 0)
