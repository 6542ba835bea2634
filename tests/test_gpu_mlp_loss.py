"""The training loss: the same bits on every call, and the mean of the squared
errors to within the roundings of a sum in a fixed order."""
import pytest
import torch

from paper_2112_10408_gb300 import tnn

pytestmark = pytest.mark.gpu


def _mlp(d_in, dh, seed):
    mlp = tnn.MLP(d_in, dh, seed=seed)
    w = mlp.get_params()
    w[d_in * dh + dh:] = 0.0  # W2 = 0: the head is b2 = (0.75, -1.25) whatever the input
    w[-2:] = (0.75, -1.25)
    mlp.set_params(w)
    return mlp


@pytest.mark.parametrize("d_in,dh", [(192, 256), (96, 128), (384, 512), (64, 192)])
@pytest.mark.parametrize("B", [1, 129, 4096, 20001])
def test_loss_repeats_and_is_the_mean(d_in, dh, B):
    g = torch.Generator(device="cuda").manual_seed(7 * d_in + B)
    x = torch.randn((B, d_in), generator=g, device="cuda").to(torch.bfloat16)
    y = torch.randn((B, 2), generator=g, device="cuda") * 5.0 + 3.0
    mlp = _mlp(d_in, dh, B)
    losses = torch.stack([mlp.gradients(x, y)[0].reshape(()) for _ in range(40)])
    torch.cuda.synchronize()
    assert bool((losses == losses[0]).all())
    e = torch.tensor([0.75, -1.25], dtype=torch.float64) - y.cpu().double()
    ref = float((e * e).mean())
    # roundings of any one term on its way: its difference (twice, squared), two
    # products, 5 + 3 sums inside a row tile, the chain of a column's partials
    # (eight chains of tiles / 8, then 3), the mean's factor and product
    depth = 4 + 8 + -(-B // 128) // 8 + 8 + 3 + 3
    assert abs(float(losses[0]) - ref) <= depth * 2.0 ** -24 * ref


def test_training_step_gives_the_same_loss_as_the_gradients():
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((4096, 192), generator=g, device="cuda").to(torch.bfloat16)
    y = torch.randn((4096, 2), generator=g, device="cuda")
    mlp = tnn.MLP(192, 256, seed=1)
    loss, _ = mlp.gradients(x, y)
    step = mlp.train_step(x, y, tnn.AdamW(lr=1e-3), loss=torch.empty_like(loss))
    torch.cuda.synchronize()
    assert float(step) == float(loss)
