"""The weight gradient on more tiles than blocks: with a power-of-two batch the output gradients of a batch are
those of its samples scaled exactly, so the batch's parameter gradients are the mean of the samples' up to the order
of the FP32 sums.  A value is a sum of T tile sums of random signs (sum of magnitudes about sqrt(T) of the total), added
at a depth of at most 60: the bound in the 2-norm is 60 * 2^-24 * sqrt(T)."""
import numpy as np
import pytest
import torch

from paper_1606_00541_gb300 import learn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,zs,batch", [(40, 9, 48, 8), (32, 32, 32, 8), (5, 3, 2, 4), (33, 4, 1, 1)])
def test_batch_gradient_is_the_mean_of_its_samples(nx, ny, zs, batch):
    from paper_1606_00541_gb300 import hec
    gen = torch.Generator(device="cuda").manual_seed(3)
    n = nx * ny * zs
    X = torch.zeros(batch * n, learn.C, dtype=torch.bfloat16, device="cuda")
    X[:, :2] = torch.randn(batch * n, 2, device="cuda", generator=gen).to(torch.bfloat16)
    T = torch.randn(batch * n, device="cuda", generator=gen)
    net = hec.Net(learn.init_params(1, last_scale=1.0))
    net.backward(X, T, (nx, ny, zs * batch), zs=zs)
    g = net.params(grads=True)[1].astype(np.float64)
    one = np.zeros_like(g)
    for b in range(batch):
        net.backward(X[b * n:(b + 1) * n].contiguous(), T[b * n:(b + 1) * n].contiguous(), (nx, ny, zs), zs=zs)
        one += net.params(grads=True)[1].astype(np.float64) / batch
    tiles = -(-nx // 32) * -(-ny // 4) * zs * batch
    assert np.linalg.norm(g - one) <= 60 * 2.0 ** -24 * np.sqrt(tiles) * np.linalg.norm(one)
