"""Loss and gradient where a training block takes one, part of one or several chunks of
samples, with and without a mask, against the FP64 oracle; tolerances as in
tests/test_mlp_gpu.py (1e-4 of the largest gradient entry, 1e-5 of the loss)."""
import numpy as np
import pytest

from oracle import mlp as om
from tests.test_mlp_gpu import data, dev, params

pytestmark = pytest.mark.gpu


# 16 samples a chunk, 256 blocks: one chunk each up to 4,096 samples, two from 4,097 on.
@pytest.mark.parametrize("n", [15, 16, 17, 4096, 4097, 9001])
@pytest.mark.parametrize("masked", [True, False])
def test_loss_and_gradient_over_chunks(lib, n, masked):
    import torch
    X, T, mask, _ = data(n, 5)
    th = params(6).astype(np.float32).astype(np.float64)
    X32, T32 = X.astype(np.float32).astype(np.float64), T.astype(np.float32).astype(np.float64)
    if not masked:
        mask = None
    loss, grad = om.loss_and_grad(th, X32, T32, mask)
    g, got = torch.full((om.N_PARAMS,), float("nan"), device="cuda"), torch.full((1,), float("nan"), device="cuda")
    lib.mlp_loss_grad(dev(torch, th), dev(torch, X), dev(torch, T), None if mask is None else dev(torch, mask), g, got)
    assert got.item() == pytest.approx(loss, rel=1e-5)
    assert np.max(np.abs(g.cpu().numpy() - grad)) <= 1e-4 * np.max(np.abs(grad))
