"""The warm-start network at the edges of its tiles: node counts around a warp's 8 nodes and
the backward tile's 32, output widths around the 4 of a lane, a hub whose row takes several
batches of entries and a degree past the table, isolated nodes, and a predicted factor whose
rows are wider than the network's outputs or not of whole 16-byte units.

Float activations against the FP64 oracle.  A pre-activation is a sum of at most 65 products of
values of order 1 in float (error below 65 * 6e-8 = 4e-6), three layers deep and divided by a
norm of order 1: 1e-4 bounds the rows.  The gradient adds the backward pass's sums (normwise
1e-3, the bound of the other gradient tests, for graphs where no pre-activation changes sign).
"""
import numpy as np
import pytest

import workloads as W
from oracle import gnn_oracle as G
from tests._util import rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2407_15049_gb300 as L  # noqa: E402
from paper_2407_15049_gb300 import warmstart as WS  # noqa: E402


def _graph(n, hub):
    """A ring with chords on the first nodes, node 0 joined to `hub` others; the last node alone."""
    rng = np.random.default_rng(n)
    last = max(n - 1, 2)
    i = np.concatenate([np.arange(last - 1), np.zeros(hub, dtype=np.int64), rng.integers(0, last, n)])
    j = np.concatenate([np.arange(1, last), 1 + np.arange(hub) % max(last - 1, 1), rng.integers(0, last, n)])
    lo, hi = np.minimum(i, j), np.maximum(i, j)
    keys = np.unique(lo[lo != hi] * n + hi[lo != hi])
    return W.maxcut_instance(n, (keys // n, keys % n, rng.choice([-1.0, 1.0, 0.5], len(keys))))


@pytest.mark.parametrize("n,hub", [(3, 0), (7, 0), (9, 5), (31, 8), (33, 20), (65, 60), (130, 100)])
@pytest.mark.parametrize("r", [1, 3, 4, 24, 29, 32])
def test_network_shapes(n, hub, r):
    inst = _graph(n, hub)
    g = G.Graph(inst)
    theta = G.init_params(r, 7).astype(np.float32)
    # no pre-activation within 2e-5 of the kink of the leaky ReLU (checked with the oracle)
    seed = 4 if n == 65 else 3
    x = G.node_features(g, seed)
    want, _ = G.forward(g, x, theta.astype(np.float64), r)
    net = WS.WarmStart(r, act="fp32", theta=theta)
    try:
        dg = WS.device_graph(inst)
        for ld in (L.padded_ld(r), r, r + 35):
            got = net.predict(dg, seed, ld).cpu().numpy()
            assert rel_err(got[:, :r], want) <= 1e-4 and np.all(got[:, r:] == 0.0)
        Rs = np.random.default_rng(1).standard_normal((n, r)) / np.sqrt(r)
        loss, grad_ref, _ = G.loss_and_grad(g, x, theta.astype(np.float64), r, G.edge_targets(g, Rs))
        Rd = torch.zeros((n, L.padded_ld(r)), dtype=torch.float64, device="cuda")
        Rd[:, :r] = torch.as_tensor(Rs, device="cuda")
        grad = torch.empty(theta.size, dtype=torch.float32, device="cuda")
        got_loss = net.train_step(dg, WS.edge_targets(dg, Rd, r), 0.0, feature_seed=seed, grad_out=grad)
        assert abs(got_loss - loss) <= 1e-4 * max(loss, 1e-6)
        # with one output the normalised row is +-1 and its gradient only rounding
        if r > 1:
            assert rel_err(grad.cpu().numpy(), grad_ref) <= 1e-3
        # bf16 activations: the rows stay within what bf16 storage moves them
        half = WS.WarmStart(r, act="bf16", theta=theta)
        if r > 3:
            assert rel_err(half.predict(dg, seed).cpu().numpy()[:, :r], want) <= 0.1
        half.close()
    finally:
        net.close()
