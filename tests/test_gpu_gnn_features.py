"""The node features of the warm-start network, seen through the network itself.

theta is chosen so that the outputs are features: layer 1 passes +x_k and -x_k through the ReLU, layers 2
and 3 pass both on, the output layer subtracts them, so o_i is a row of features.  Output 0 is the constant
feature 1, so a feature is the ratio of its output to output 0 (the normalisation cancels), within a few
float roundoffs: exact after rounding to bf16, in which the features are stored.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import gnn_oracle as G
from paper_2407_15049_gb300 import warmstart as WS

pytestmark = pytest.mark.gpu

F, H = G.FEATURES, G.HIDDEN


def _theta():
    """Parameters of a network whose 16 outputs are the 16 features."""
    first = np.zeros((H, F))
    first[:F], first[F:] = np.eye(F), -np.eye(F)
    out = np.concatenate([np.eye(F), -np.eye(F)], axis=1)
    parts = [first, np.zeros((H, F)), np.zeros(H)]
    for _ in range(G.LAYERS - 1):
        parts += [np.eye(H), np.zeros((H, H)), np.zeros(H)]
    return np.concatenate([p.ravel() for p in parts + [out, np.zeros(F)]]).astype(np.float32)


def _features(graph, act, seed):
    net = WS.WarmStart(F, act=act, theta=_theta())
    try:
        R = net.predict(graph, seed)
    finally:
        net.close()
    return R[:, 1:F] / R[:, :1]


@pytest.mark.parametrize("seed", [3, 2024])
def test_bf16_normals_are_the_rounded_fp64_normals(seed):
    """1.2e6 normals: some 600 lie within the rounding test's 16 ulp of a tie and are formed in FP64.
    Reference: the FP64 draw rounded to float, then to bf16, as the kernel documents."""
    n = 100003
    inst = W.maxcut_instance(n, W.er_graph(n, 2 * n, 1, "pm1"))
    got = _features(WS.device_graph(inst), "bf16", seed).to(torch.bfloat16)[:, 3:]
    want = G.node_features(G.Graph(inst), seed)[:, G.N_STRUCT:]
    want = torch.as_tensor(want).float().to(torch.bfloat16).cuda()
    assert int((got != want).sum()) == 0


@pytest.mark.parametrize("act", ["fp32", "bf16"])
def test_diagonal_entries_of_a_row_add_up(act):
    """A row whose diagonal is stored as two entries has the features of their sum."""
    n = 70
    inst = W.maxcut_instance(n, W.er_graph(n, 3 * n, 4, "pm1"))
    rows = np.repeat(np.arange(n), np.diff(inst.rowptr))
    diag = rows == inst.colind
    rep = np.where(diag, 2, 1)
    split = dict(WS.device_graph(inst))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, weights=rep, minlength=n))]).astype(np.int64)
    val = np.repeat(np.where(diag, 0.5 * inst.val, inst.val), rep)
    split.update(rowptr=torch.as_tensor(rowptr, device="cuda"), colind=torch.as_tensor(np.repeat(inst.colind, rep), device="cuda"),
                 val=torch.as_tensor(val, device="cuda"))
    want, got = _features(WS.device_graph(inst), act, 5), _features(split, act, 5)
    assert torch.equal(got, want)
