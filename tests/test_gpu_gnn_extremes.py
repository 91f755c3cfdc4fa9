"""The proposer's gradient where values overflow: an infinity stays an infinity where it did not meet
a zero, and levels that the model does not have get no gradient."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2602_20826_gb300 import workloads as wl
from tests.gpu_helpers import context

pytestmark = pytest.mark.gpu
H, F, LEVELS = 128, 16, 16
W1, W2, W3 = 0, 3 * F * H + H, 3 * F * H + 2 * H + 3 * H * H
B2, WH = W2 + 3 * H * H, W3 + 3 * H * H + H
BH = WH + H * LEVELS


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    return context()


def _grad(ctx, h2):
    """Two kernels, 0 -> 1; every parameter zero but one feature of layer 2 (`h2` at both), its weight
    3e38 in the predecessors' third of layer 3, and the first level's weights of the head: kernel
    1's h3 is 3e38 h2, its label is the other level."""
    from paper_2602_20826_gb300.dagrt import Model
    f = 5
    rp, col = wl.csr_from_edges(2, [0], [1])
    b = wl.from_dags([(rp, col, np.array([3, 4]), np.array([64, 64]))], 8)
    model = Model(ctx, [1, 2], seed=0)
    p = np.zeros(model.n_params, np.float32)
    p[B2 + f] = h2
    p[W3 + (H + f) * H:W3 + (H + f + 1) * H] = 3e38
    p[WH:WH + H * LEVELS:LEVELS] = 1
    model.params(set_to=p)
    lb = ctx.load(b)
    loss, g = model.grad(lb, np.array([-1, 1], np.int8))
    model.free()
    lb.free()
    return loss, g, f


def test_infinite_input_gradient(ctx):
    """h2 = 1e-37: the forward pass is finite (h3 = 30), dA of kernel 1 is 128 * 3e38; kernel 0 gets
    it divided by one predecessor, and the bias of the feature with it."""
    loss, g, f = _grad(ctx, 1e-37)
    assert np.isfinite(loss)
    assert np.isinf(g[B2 + f])


def test_levels_beyond_the_models(ctx):
    """h2 = 2: h3 is infinite, the gradient of the model's two levels not a number; the other 14
    columns of the head stay zero."""
    _, g, _ = _grad(ctx, 2.0)
    assert not np.isfinite(g[WH:BH].reshape(H, LEVELS)[:, :2]).any()
    assert (g[WH:BH].reshape(H, LEVELS)[:, 2:] == 0).all() and (g[BH + 2:BH + LEVELS] == 0).all()
