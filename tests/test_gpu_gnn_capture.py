"""The proposer's calls in a captured graph, replayed with other parameters: batches whose layers'
kernels overlap (programmatic launches, up to 512 nodes per SM) and a larger one give bit for bit
what the same calls give outside a capture."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context
from tests.oracle_checks import random_small_dag

pytestmark = pytest.mark.gpu
LEVELS = [1, 2, 4, 8, 16]


@pytest.mark.parametrize("n_dags,V", [(1, 5), (30, 90), (300, 300)])
def test_replay_with_other_parameters(n_dags, V):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_2602_20826_gb300.dagrt import Model
    ctx = context()
    rng = np.random.default_rng(140 + V)
    dag = [random_small_dag(rng, V, 0.05, 5000) for _ in range(3)]
    b = wl.from_dags([dag[i % 3] for i in range(n_dags)], 148)
    lb, model = ctx.load(b), Model(ctx, LEVELS, seed=1)
    N = b.total_nodes()

    def buffers():
        return (torch.zeros(N * len(LEVELS), dtype=torch.float32, device="cuda"),
                {"out_bound": torch.zeros(n_dags * 9, dtype=torch.int64, device="cuda"),
                 "best_bound": torch.zeros(n_dags, dtype=torch.int64, device="cuda"),
                 "best_cand": torch.zeros(n_dags, dtype=torch.int32, device="cuda")})

    def calls(z, out):
        model.logits(lb, out=z)
        model.propose(lb, 8, out=out)

    z, out = buffers()
    calls(z, out)  # allocates what a capture may not
    ctx.graph_begin()
    calls(z, out)
    graph = ctx.graph_end()
    other = Model(ctx, LEVELS, seed=2)
    params = [model.params(), other.params(), model.params()]
    for p in params:
        model.params(set_to=p)
        z.fill_(0)
        torch.cuda.synchronize()
        graph.launch()
        ctx.sync()
        want_z, want = buffers()
        calls(want_z, want)
        ctx.sync()
        assert torch.equal(z, want_z)
        for k in out:
            assert torch.equal(out[k], want[k]), k
    for x in (graph, model, other, lb):
        x.free()
