"""Gradient kernel of the learned weights at the edges of its tiles: a warp takes 16 samples, a block
64 at a time, and the grid 608 blocks, so that a batch ends inside a tile, on the edge of a tile, on
the edge of a block's 64, and in a second pass of the grid.

Reference: the oracle's formulas in float64 with the operand roundings of the tensor cores (weights,
activations and dz to bfloat16).  Kernel and reference may still round an operand to neighbouring
bfloat16 values where they stand at a tie: a product's two operands are then off by 2^-8 each, and
dz passes three products on its way to the first layer, at most 6 * 2^-8 = 2.4e-2 of a term.  The
bound of the whole tensor is that of the existing gradient test, 2e-2 relative in L2; a sample left out
or counted twice changes the gradient of a batch of n by about 1/n or more, so the largest batches
also hold one sample far from the rest (in the last row) that carries a tenth of the gradient.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import _theta, smooth_stencils

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(th, S, T):
    W1, b1, W2, b2, W3, b3, W4, b4 = M.unpack(M.bf16(th))
    x, amp = M.normalise(S.astype(np.float64))
    tn = (T.astype(np.float64) - S[:, 2]) / amp
    om, (a0, z1, h1, z2, h2, z3, h3, _) = M.forward(M.bf16(th), x, round_activations=True)
    q = M.candidates(x)
    res = np.sum(om * q, axis=1) - tn
    dom = (2.0 * res / len(S))[:, None] * q
    dz4 = om * (dom - np.sum(om * dom, axis=1, keepdims=True))
    dz3 = (M.bf16(dz4) @ W4) * M.gelu_grad(z3)
    dz2 = (M.bf16(dz3) @ W3) * M.gelu_grad(z2)
    dz1 = (M.bf16(dz2) @ W2) * M.gelu_grad(z1)
    return np.mean(res * res), [M.bf16(dz1).T @ a0, dz1.sum(0), M.bf16(dz2).T @ h1, dz2.sum(0),
                                M.bf16(dz3).T @ h2, dz3.sum(0), M.bf16(dz4).T @ h3, dz4.sum(0)]


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 129, 608 * 64, 608 * 64 + 1,
                               2 * 608 * 64 + 17])
def test_gradient_of_ragged_batches(n):
    from paper_1905_00182_gb300 import ibfsa as ib
    th = _theta(5).astype(np.float32)
    S, T = smooth_stencils(n, 6)
    amp = np.max(np.abs(S - S[:, 2:3]), axis=1)
    T = (T + 0.3 * amp).astype(np.float32)  # a residual that does not cancel
    T[-1] += np.float32(0.05 * n) * amp[-1]
    loss, g = ib.MLP(th).gradient(torch.from_numpy(S).cuda(), torch.from_numpy(T).cuda())
    lo, parts = _reference(th.astype(np.float64), S, T)
    assert abs(loss - lo) <= 2e-2 * lo, (loss, lo)
    for k, (a, b) in enumerate(zip(M.unpack(g.astype(np.float64)), parts)):
        rel = np.linalg.norm(a - b) / np.linalg.norm(b)
        assert rel <= 2e-2, (n, k, rel)
