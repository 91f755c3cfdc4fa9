"""Batches with DAGs the scheduler rejects, at the start, between others, at the end, and without
nodes but with edges: their edges belong to no node's list, so logits and gradient are those of the
other DAGs alone and every parameter stays finite.

What a node adds to a gradient is the same to the bit in both batches, but sums over nodes run in
another order: each of the two sums of up to N terms t is within N 2^-23 sum |t| (single-precision
accumulation without rounding to nearest), and sum |t| within 4 (mag + flip) of the oracle's
magnitudes (every gate it may set the other way counted)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import gnn as G
from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context
from tests.oracle_checks import random_small_dag
from tests.test_gpu_gnn import _oracle_inputs

pytestmark = pytest.mark.gpu
N_LEVELS = 7


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _cycle(V):
    """A ring: every node has an edge, none is a source."""
    return (np.arange(V + 1, dtype=np.int32), np.roll(np.arange(V, dtype=np.int32), -1),
            np.ones(V, np.int64), np.full(V, 40, np.uint8))


def _edges_only(E):
    """No node, yet E edges in its part of the successor array."""
    return np.zeros(1, np.int32), np.zeros(E, np.int32), np.zeros(0, np.int64), np.zeros(0, np.uint8)


@pytest.mark.parametrize("sizes", [(40, 60), (2100, 30)])
def test_gradient_without_the_rejected(ctx, sizes):
    from paper_2602_20826_gb300.dagrt import Model
    rng = np.random.default_rng(95)
    good = [random_small_dag(rng, V, min(0.3, 6.0 / V), 5000, kmin=1) for V in sizes]
    order = [_cycle(5), good[0], _edges_only(70), good[1], _cycle(300), _edges_only(3)]
    mixed, alone = wl.from_dags(order, 148), wl.from_dags(good, 148)
    at = np.concatenate([np.arange(mixed.node_off[d], mixed.node_off[d + 1]) for d in (1, 3)])
    labels = rng.integers(0, N_LEVELS, alone.total_nodes()).astype(np.int8)
    labels_mixed = np.full(mixed.total_nodes(), -1, np.int8)
    labels_mixed[at] = labels
    model = Model(ctx, list(range(1, N_LEVELS + 1)), seed=3)
    lm, la = ctx.load(mixed), ctx.load(alone)
    st = lm.schedule(0, fields=("status",), check=False)["status"]
    assert [bool(x) for x in st] == [True, False, True, False, True, True]
    assert np.array_equal(model.logits(lm)[at], model.logits(la))
    preds, succs, x, _ = _oracle_inputs(alone)
    p = model.params().astype(np.float64)
    mag, flip = G.grad_magnitude(p, x, preds, succs, labels, N_LEVELS, bf=True, gate_slack=2.0 ** -6)
    loss_m, gm = model.grad(lm, labels_mixed)
    loss_a, ga = model.grad(la, labels)
    assert abs(loss_m - loss_a) <= 1e-6 * loss_a
    tol = 2 * len(labels) * 2.0 ** -23 * 4 * (mag + flip)
    assert (np.abs(gm.astype(np.float64) - ga) <= tol).all()
    for _ in range(2):
        assert np.isfinite(model.train_step(lm, labels_mixed, 1e-3))
    assert np.isfinite(model.params()).all()
    model.free()
    lm.free()
    la.free()
