"""Closure gradients at the sizes where the whole-network kernel and the joint weight gradients can go wrong, against
the FP64 oracle: samples of one tile and less, one position beyond a tile, its longest and one position more (which
takes the kernels per layer), two layers, its deepest and one layer more, more layers than one weight-gradient launch
takes, and more samples than the GPU has SMs.  Tolerances as in the other gradient tests (BF16 operands)."""
import numpy as np
import pytest

from oracle import closure_oracle as CO

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("X,layers,B", [(16, 5, 3), (127, 5, 2), (129, 5, 3), (257, 4, 2), (512, 5, 2), (513, 5, 2),
                                        (64, 2, 3), (200, 3, 3), (130, 6, 3), (64, 9, 2), (20, 3, 400)])
def test_gradients_match_oracle_at_edge_sizes(gpu, X, layers, B):
    import torch
    rng = np.random.default_rng(X + layers)
    net = gpu.Closure(7, 5, X, B, seed=X, layers=layers)
    shapes = CO.layer_shapes(7, 5, layers)
    p = net.get_params().astype(np.float64)
    for l, (W, b) in enumerate(CO.unpack(p, shapes)):
        b[:5 if l == layers - 1 else 64] = rng.normal(0, 0.05, 5 if l == layers - 1 else 64)
    net.set_params(p.astype(np.float32))
    x = rng.normal(0, 1, (B, X, 7)).astype(np.float32)
    y = rng.normal(0, 0.5, (B, X, 5)).astype(np.float32)
    per = (np.arange(B) % 2).astype(np.int32)
    loss, g = net.gradients(*[torch.tensor(a, device="cuda") for a in (x, y, per)])
    bf16 = lambda a: torch.tensor(a, dtype=torch.float32).bfloat16().double().numpy()
    po = p.astype(np.float32).astype(np.float64)
    for W, b in CO.unpack(po, shapes):
        W[...] = bf16(W)
    xin = np.zeros((B, X, 16))
    xin[:, :, :7] = bf16(x)
    lo, go = CO.loss_and_grad(po, shapes, xin, y.astype(np.float64), per, 5)
    assert loss == pytest.approx(lo, rel=2e-2)
    assert np.linalg.norm(g - go) <= 5e-2 * np.linalg.norm(go)
