"""A network's precision set after it was made: the other precision's products
with the same parameters, in room of its own."""
import pytest

from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("made,used", [("bf16", "f32"), ("f32", "bf16")])
def test_precision_set_later(made, used):
    import torch
    from paper_2203_01462_gb300.surrogate import UNet
    params = I.unet_params(8, 5)
    gen = torch.Generator(device="cuda").manual_seed(9)
    x = torch.rand(2, 2, 24, 40, generator=gen, device="cuda")
    t = torch.rand(1, 2, 24, 40, generator=gen, device="cuda")
    ref = UNet(base=8, batch=2, H=24, W=40, params=params, precision=used)
    net = UNet(base=8, batch=2, H=24, W=40, params=params, precision=made)
    net.forward(x)
    net.precision = used
    assert torch.equal(net.forward(x), ref.forward(x))
    net.train_step(x, t, 1e-3)
    ref.train_step(x, t, 1e-3)
    torch.cuda.synchronize()
    for n in ref.w:
        assert torch.equal(net.gw[n], ref.gw[n]) and torch.equal(net.w[n], ref.w[n])
