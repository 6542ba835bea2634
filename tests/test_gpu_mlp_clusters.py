"""MLP gradients over the shapes where the forward kernel splits the hidden
units over 1, 2, 4 or 8 CTAs of a cluster, with ragged batches, against
float64 on the operands the kernels round (W1 in BF16)."""
import numpy as np
import pytest
import torch

from paper_2112_10408_gb300 import tnn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,dh", [(48, 64), (96, 128), (192, 256), (384, 512), (64, 192)])
@pytest.mark.parametrize("B", [1, 127, 129, 2048, 9731, 20001])
def test_gradients_at_every_cluster_size(d_in, dh, B):
    g = torch.Generator(device="cuda").manual_seed(d_in + B)
    x = torch.randn((B, d_in), generator=g, device="cuda").to(torch.bfloat16)
    y = torch.randn((B, 2), generator=g, device="cuda") * 5.0 + 3.0
    mlp = tnn.MLP(d_in, dh, seed=B)
    loss, grad = mlp.gradients(x, y)
    loss2, grad2 = mlp.gradients(x, y)
    torch.cuda.synchronize()
    assert torch.equal(grad, grad2)  # fixed order of every sum
    w = torch.from_numpy(mlp.get_params()).cuda()
    P = d_in * dh
    W1 = w[:P].view(d_in, dh).to(torch.bfloat16).double().requires_grad_()
    b1, W2, b2 = (v.double().requires_grad_() for v in (w[P:P + dh], w[P + dh:P + 3 * dh].view(dh, 2), w[P + 3 * dh:]))
    z = x.double() @ W1 + b1
    out = z * 0.5 * (1.0 + torch.erf(z / 2.0 ** 0.5)) @ W2 + b2
    ref = ((out - y.double()) ** 2).mean()
    gr = torch.cat([v.reshape(-1) for v in torch.autograd.grad(ref, (W1, b1, W2, b2))])
    # H and dZ are rounded to BF16 (2^-9 of each term); the sums' errors grow
    # at most like their terms
    assert abs(loss.item() - ref.item()) <= 2.0 ** -8 * ref.item()
    for a, b in ((0, P), (P, P + dh), (P + dh, P + 3 * dh), (P + 3 * dh, P + 3 * dh + 2)):
        err, size = (grad[a:b].double() - gr[a:b]).norm().item(), gr[a:b].norm().item()
        assert err <= 2.0 ** -7 * size, (a, err, size)
