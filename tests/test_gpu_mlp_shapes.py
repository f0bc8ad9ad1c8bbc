"""Network gradients at the edges of the tiles: batches around the 32, 64 and 128
row tiles, one and several column tiles, and a smaller batch after a larger one
(whose padded columns must read as zeros): against the bfloat16 oracle."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,width,batches", [(64, 64, (1, 130, 33)), (320, 192, (129, 64)), (576, 256, (257, 31))])
def test_gradients_at_tile_edges(n_in, width, batches):
    import torch

    from paper_2406_08314_gb300 import cv
    net = cv.MLP(n_in, width, seed=1)
    p = net.params().astype(np.float64)
    sizes = [width * n_in, width, width * width, width, width * width, width, width, 1]
    for B in batches:
        rng = np.random.default_rng(B)
        x = rng.standard_normal((B, n_in)).astype(np.float32)
        t = rng.standard_normal(B).astype(np.float32)
        loss, g = net.grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
        loss_ref, g_ref = mo.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), n_in, width, bf16=True)
        assert abs(float(loss.item()) - loss_ref) <= 2e-3 * loss_ref
        g, off = g.cpu().numpy(), 0
        # bfloat16 roundings of activations flip where FP32 and FP64 sums differ by
        # a rounding: 2^-8 of an entry, as in the network's gradient test
        for k, n in enumerate(sizes):
            a, b = g[off:off + n], g_ref[off:off + n]
            assert np.max(np.abs(a - b)) <= 1e-2 * max(np.max(np.abs(b)), 1e-30), (B, k)
            off += n
