"""Device memory that a batch holds for the proposer, per node: lists, features, logits, candidates and
the paper schedule's plan (229 bytes) and three activations of 256 bytes, in which a forward pass
also keeps its aggregated inputs; for training 3,137 more (gradients of the logits, of the three
activations and of a layer's input in single precision, labels)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context

pytestmark = pytest.mark.gpu


def test_bytes_per_node():
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_2602_20826_gb300.dagrt import Model
    n, V = 2000, 1000
    rp, col = wl.csr_from_edges(V, range(0, V - 1, 2), range(1, V, 2))
    b = wl.from_dags([(rp, col, np.arange(1, V + 1), np.full(V, 40, np.uint8))] * n, 148)
    ctx = context()
    model = Model(ctx, [1, 2, 4], seed=0)
    warm = ctx.load(b.subset(range(3)))  # the kernels' own memory
    labels = np.zeros(n * V, np.int8)
    model.train_step(warm, labels[:3 * V], 1e-3)
    model.logits(warm)
    warm.free()
    params = model.params()
    lb = ctx.load(b)
    z = torch.zeros(n * V * 3, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    free = [torch.cuda.mem_get_info()[0]]
    model.logits(lb, out=z)
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
    model.train_step(lb, labels, 1e-3)
    free.append(torch.cuda.mem_get_info()[0])
    slack = 25 * (2 << 20)  # an allocation takes whole pages of 2 MB
    fwd, train = free[0] - free[1], free[1] - free[2]
    assert fwd <= n * V * (229 + 3 * 256) + slack, fwd / (n * V)
    assert train <= n * V * 3137 + slack, train / (n * V)
    # a forward pass beside the training state gives what it gave before
    model2 = Model(ctx, [1, 2, 4], seed=0)
    model2.params(set_to=params)
    z2 = torch.zeros_like(z)
    model2.logits(lb, out=z2)
    assert torch.equal(z, z2)
    for x in (model, model2, lb):
        x.free()
