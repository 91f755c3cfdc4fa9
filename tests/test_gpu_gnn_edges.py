"""The proposer's kernels at their edges: node counts around the 128-row tiles and fewer nodes
than CTAs, graphs on both sides of the shared-memory limit of the predecessor lists (2,048
nodes), 1 to 16 levels in the top-k and the head. Tolerances as in tests/test_gpu_gnn.py."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import gnn as G
from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context
from tests.oracle_checks import random_small_dag
from tests.test_gpu_gnn import _oracle_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


@pytest.mark.parametrize("sizes,n_levels", [((1,), 1), ((127,), 2), ((128,), 15), ((100, 29), 16), ((3, 0, 253, 1), 5),
                                            ((2100,), 7)])
def test_logits_gradient_and_topk(ctx, sizes, n_levels):
    from paper_2602_20826_gb300.dagrt import Model
    rng = np.random.default_rng(80 + sum(sizes))
    b = wl.from_dags([random_small_dag(rng, V, min(0.3, 6.0 / max(V, 1)), 5000, kmin=1) for V in sizes], 148)
    lb = ctx.load(b)
    levels = list(range(1, n_levels + 1))
    model = Model(ctx, levels, seed=3)
    preds, succs, x, _ = _oracle_inputs(b)
    p = model.params().astype(np.float64)
    ref, _ = G.forward(p, x, preds, succs, n_levels, bf=True)
    z = model.logits(lb)
    assert np.abs(z - ref).max() <= 2e-2 * (1 + np.sqrt(np.mean(ref ** 2)))
    labels = rng.integers(-1, n_levels, size=b.total_nodes()).astype(np.int8)
    loss, g = model.grad(lb, labels)
    rl, rg = G.loss_and_grad(p, x, preds, succs, labels, n_levels, bf=True)
    assert abs(loss - rl) <= 1e-3 * max(1.0, rl)
    mag, flip = G.grad_magnitude(p, x, preds, succs, labels, n_levels, bf=True, gate_slack=2.0 ** -6)
    assert (np.abs(g.astype(np.float64) - rg) <= 2.0 ** -6 * mag + flip + 1e-9).all()
    loss2, g2 = model.grad(lb, labels)
    assert loss2 == loss and np.array_equal(g, g2)
    for k in (1, 16):
        res = model.propose(lb, k, want_all=True)
        for d in range(b.n_dags):
            a, e = int(b.node_off[d]), int(b.node_off[d + 1])
            if a == e:
                continue
            plan = _oracle_inputs(b.subset([d]))[3][0]
            rows, V = res["cand_m"][2 * a: 2 * a + plan["n_rows"]], e - a
            rid = plan["row_id"]
            assign = np.zeros((k, V), np.int64)
            for r in range(plan["n_rows"]):
                if rid[r] < V:
                    assign[:, rid[r]] = rows[r, 1:] - 1
            n = min(k, n_levels ** min(V, 5))
            assert len({tuple(t) for t in assign}) == n
            zd = z[a:e].astype(np.float64)
            got = sorted(G.cost_of(zd, assign[j]) for j in range(n))
            want = [c for c, _ in G.k_best(zd, n)]
            assert np.allclose(got, want, atol=1e-4 * (1 + max(want)))
    model.free()
    lb.free()


@pytest.mark.parametrize("extra", [0, 1, 200])
def test_forward_around_four_tiles_per_sm(ctx, extra):
    """Up to 512 nodes per SM the forward pass takes its small-batch form. A node's logits do not
    depend on the rest of the batch, so a batch on either side of the line gives bit for bit what
    its parts give (which the test above compares with the oracle)."""
    import torch
    from paper_2602_20826_gb300.dagrt import Model
    total = 512 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    rng = np.random.default_rng(90 + extra)
    sizes = [400] * (total // 400) + [total % 400]
    dags = [random_small_dag(rng, V, 0.02, 5000, kmin=1) for V in sizes if V]
    model = Model(ctx, list(range(1, 16)), seed=3)
    z = []
    for part in (dags, dags[:9], dags[9:]):
        lb = ctx.load(wl.from_dags(part, 148))
        z.append(model.logits(lb).copy())
        lb.free()
    model.free()
    assert len(z[0]) == total and np.array_equal(z[0], np.concatenate(z[1:]))
