"""FP32 sums of the weight gradients stay short however many rows they have: every sample and vertex
contributes the same product here, so an entry of dW2 is that product times the rows, and the error
is that of the sums alone.  At most 32 products and 32 sums of 32 are added in FP32 before FP64
takes over; with the roundings of the factors and of the result 68 roundings of 2^-24."""

import numpy as np
import pytest

from workloads import square_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,batch", [(16, 0, 1), (32, 2, 3), (128, 3, 8)])
def test_equal_contributions_add_up(lib, base, levels, batch):
    import torch
    from paper_1812_00185_gb300 import binding as cg
    b = square_mesh(base)
    mesh = cg.Mesh(b.xy, b.tri, b.tag, levels)
    n = mesh.level(levels)["rowptr"].size - 1
    net = cg.cgp_mlp_create(mesh.handle, levels, batch)
    g = np.random.default_rng(0)
    w1, w3 = g.integers(128, 256, 64) / 256, g.integers(1, 257, 64) / 256   # exact in bfloat16
    W1, W3, one = np.zeros((64, 8)), np.zeros(128), np.ones(64)
    W1[:, 0], W3[:64] = w1, w3                 # a1 = w1 (r / rms(r) = 1), a2 = 1, a3 = sum of w3
    cg.cgp_mlp_set_params(net, np.concatenate([W1.ravel(), 0 * one, np.zeros(64 * 128), one, W3, [0.0]]).astype(np.float32))
    r = torch.ones(batch * n, dtype=torch.float64, device="cuda")
    loss, grad = cg.cgp_mlp_grad(net, r, r, 3.0 * r, batch)      # clipped target (3 - 1) / 1 = 2
    d = w3.sum() - 2.0
    assert abs(loss / d ** 2 - 1.0) < 1e-6
    rows = batch * n
    g2 = w3 * float(np.float32(2.0 * d / rows))
    o = 64 * 8 + 64
    dW2 = grad[o:o + 64 * 128].reshape(64, 128).astype(float)
    want = rows * np.outer(g2, w1)
    tol = 68 * 2.0 ** -24
    assert np.abs(dW2[:, :64] / want - 1.0).max() <= tol
    assert np.abs(dW2[:, 64:] / want - 1.0).max() <= tol + 5 * 2.0 ** -24   # (the ring's mean: up to 6 roundings)
    assert np.abs(grad[o + 64 * 128:o + 64 * 129] / (rows * g2) - 1.0).max() <= tol
    cg.cgp_mlp_destroy(net)
    mesh.close()
