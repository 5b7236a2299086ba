"""Loss and gradient of the learned initial partition at the edges of its
tiles: row counts around 32, 128 and 256, class counts that do not divide by 4
or 16, and features that do not start on a 16-byte boundary.  Against the
oracle's float64 evaluation with the same bf16 operand rounding, with the
bounds of test_gpu_learned: an operand on the other side of a rounding boundary
moves by 2^-8 of itself, about 5e-4 of a 64-wide row's norm; a wrong row, column
or mask is of the order of the norm."""
import numpy as np
import pytest
import torch

import graphgen
from oracle import mpnn
from test_gpu_learned import FWD_RTOL, GRAD_RTOL, _d, _theta, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

jet = pytest.importorskip("paper_2304_13194_gb300")


@pytest.mark.parametrize("n,k,shift", [(1, 2, 0), (31, 7, 1), (33, 256, 0), (128, 18, 0), (255, 33, 2), (257, 255, 1),
                                       (513, 64, 0)])
def test_gradient_at_tile_edges(ctx, n, k, shift):
    g = graphgen.gnp(n, min(1.0, 6.0 / n), seed=n)
    theta = _theta(k, n + k)
    r = np.random.default_rng(n)
    X = r.normal(0, 1, (n, 16)).astype(np.float32)
    y = r.integers(0, k, n).astype(np.int32)
    m = jet.LearnedPartitioner(ctx, k, theta)
    flat = torch.zeros(16 * n + shift, device="cuda")
    Xd = flat[shift:].view(n, 16)
    Xd.copy_(_d(X, torch.float32))
    xadj, adj = _d(g.xadj, torch.int64), _d(g.adjncy, torch.int32)
    logits = m.forward(xadj, adj, Xd).cpu().numpy()
    ref, _, _ = mpnn.forward(g, X, theta.astype(np.float64), k, emulate_bf16=True)
    assert np.linalg.norm(logits - ref) <= FWD_RTOL * np.linalg.norm(ref)
    loss, grad = m.loss_grad(xadj, adj, Xd, _d(y, torch.int32))
    grad = grad.cpu().numpy().astype(np.float64)
    l_ref, g_ref = mpnn.loss_and_grad(g, X, theta.astype(np.float64), k, y, emulate_bf16=True)
    assert abs(loss - l_ref) <= 1e-4 * abs(l_ref)
    o = 0
    for shape in mpnn.param_shapes(k):
        c = int(np.prod(shape))
        assert np.linalg.norm(grad[o:o + c] - g_ref[o:o + c]) <= GRAD_RTOL * np.linalg.norm(g_ref[o:o + c]) + 1e-7, shape
        o += c
    m.close()
