"""The selector's gradients at the edges of their kernels' tiles: batches around
the 8 samples of a block and the 64 staged at a time, output counts that fill
and do not fill a group of four neurons, a fractional and an empty mask; against
the oracle's backward pass (2e-4 of a layer's largest gradient: float sums of up
to 200 products, as in test_gpu_learned)."""
import numpy as np
import pytest
import torch

from oracle import learned as L
from paper_2012_06925_gb300 import binding as B
from test_gpu_learned import pack, random_params, unpack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nout", [3, 9, 24])
@pytest.mark.parametrize("batch", [1, 8, 9, 63, 64, 65, 200])
def test_gradients_match_the_oracle(batch, nout):
    p = random_params(nout, batch)
    rng = np.random.default_rng(batch + nout)
    X = rng.uniform(0, 1, (batch, 6))
    T = rng.standard_normal((batch, nout)).astype(np.float32)
    mask = (rng.integers(0, 3, (batch, nout)) / 2).astype(np.float32)
    y, cache = L.forward_bf16(p, X)
    loss, gy = L.loss_and_grad_out(y, T, mask)
    g = L.backward(cache, gy)
    grads, gl = B.mlp_gradients(torch.from_numpy(pack(p)).cuda(), nout,
                                torch.from_numpy(X.astype(np.float32)).cuda(), torch.from_numpy(T).cuda(),
                                torch.from_numpy(mask).cuda())
    gg = unpack(grads.cpu().numpy().astype(np.float64), nout)
    assert abs(gl.item() - loss) <= 1e-5 * abs(loss)
    for k in g:
        assert np.abs(gg[k] - g[k]).max() <= 2e-4 * np.abs(g[k]).max(), k


def test_empty_mask_gives_zero_gradients():
    nout, batch = 9, 70
    p = torch.from_numpy(pack(random_params(nout, 1))).cuda()
    x = torch.rand(batch, 6, device="cuda")
    grads, loss = B.mlp_gradients(p, nout, x, torch.randn(batch, nout, device="cuda"),
                                  torch.zeros(batch, nout, device="cuda"))
    assert loss.item() == 0.0 and torch.count_nonzero(grads).item() == 0
