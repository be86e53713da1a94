"""The cut scorer's tiled kernels at the edges of their tiles (needs a GPU).

Nodes are taken in tiles of 64, gradients in at most two partial sums per SM:
batches of one node, just below, at and above a tile, graphs that straddle
tiles, isolated nodes, and more tiles than partial sums, against the FP64
oracle at the same FP16-rounded weights.

Tolerances: every prediction is a chain of FP32 sums of at most 2 x 64 terms
through three layers and a mean, rounding below 400 x 2^-24 = 2.4e-5 of the
terms' magnitude; a gradient entry sums at most a tile per partial and then
the partials, with terms that carry the forward rounding: 2e-4 of the largest
entry covers both with the cancellation of the signed sums.
"""
import numpy as np
import pytest
from scipy.sparse import csr_matrix

from paper_2303_10788_gb300 import ccs
from oracle import mpnn as om

pytestmark = pytest.mark.gpu


def random_graph(rng, n):
    """A random sparse symmetric interaction graph (some nodes isolated)."""
    i = rng.integers(0, n, 2 * n)
    j = np.minimum(n - 1, i + rng.integers(1, 6, 2 * n))
    keep = i != j
    w = csr_matrix((rng.integers(1, 9, keep.sum()).astype(float), (i[keep], j[keep])), shape=(n, n))
    w = (w + w.T).tocsr()
    w.sort_indices()
    deg = np.asarray(w.sum(axis=1)).ravel()
    row = np.repeat(np.arange(n), np.diff(w.indptr))
    return ccs.Graph(rng.random((n, 8)).astype(np.float32), w.indptr.astype(np.int32), w.indices.astype(np.int32),
                     (w.data / deg[row]).astype(np.float32), (w.data / deg[w.indices]).astype(np.float32),
                     rng.random(8).astype(np.float32))


@pytest.mark.parametrize("sizes", [[1], [63], [64], [65], [1, 130, 64, 7, 62], [200] * 40, [310] * 70],
                         ids=lambda s: f"{len(s)}x{max(s)}")
def test_tiles_match_oracle(sizes):
    rng = np.random.default_rng(sum(sizes) + len(sizes))
    ctx = ccs.ccs_create(0)
    b = ccs.make_batch([random_graph(rng, n) for n in sizes])
    a = b._arrays
    n = int(b.n_nodes)
    A = csr_matrix((a["val"].astype(np.float64), a["col"], a["rowptr"]), shape=(n, n))
    net = ccs.ccs_mpnn_create(ctx, seed=len(sizes))
    theta = ccs.ccs_mpnn_params(ctx, net)
    theta[om.SHAPES["b0"][0]:om.SHAPES["b0"][0] + 64] = rng.normal(0, 0.1, 64)
    ccs.ccs_mpnn_set_params(ctx, net, theta)
    t16 = theta.astype(np.float16).astype(np.float64)
    t = rng.normal(size=len(sizes)).astype(np.float32)
    want, _ = om.forward(t16, a["x"].astype(np.float64), A, a["graph_off"], a["glob"].astype(np.float64))
    got = ccs.ccs_mpnn_forward(ctx, net, b)
    assert np.abs(got - want).max() <= 1e-4 * max(1.0, np.abs(want).max())
    loss, grad = ccs.ccs_mpnn_gradient(ctx, net, b, t)
    loss_o, grad_o = om.loss_and_grad(t16, a["x"].astype(np.float64), A, a["graph_off"],
                                      a["glob"].astype(np.float64), t.astype(np.float64))
    assert loss == pytest.approx(loss_o, rel=1e-4)
    err = np.abs(grad - grad_o).max() / np.abs(grad_o).max()
    print(f"{n} nodes: gradient max rel err {err:.1e}")
    assert err < 2e-4
    # the training step's Adam update of the same gradient (first step: lr g / (|g| + eps))
    loss_t = ccs.ccs_mpnn_train_step(ctx, net, b, t, lr=1e-2)
    step = ccs.ccs_mpnn_params(ctx, net) - theta
    assert loss_t == loss
    assert np.abs(step + 1e-2 * grad / (np.abs(grad) + 1e-8)).max() < 1e-2 * 1e-3
