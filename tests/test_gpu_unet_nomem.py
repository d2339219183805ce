"""A box too large for the device is refused, and the network then works as
before: buffers that gave way to the refused box's are allocated again."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("channels", [(16,), (16, 32, 48)])
def test_forward_and_backward_after_a_refused_box(om, channels):
    rng = np.random.default_rng(9)
    net = om.UNet(2, 1, channels, seed=5)
    w = torch.from_numpy(rng.uniform(-0.1, 0.1, net.n_params).astype(np.float32)).cuda()
    net.set_params(w)
    x = torch.from_numpy(rng.uniform(0, 1, (1, 8, 12, 16, 2)).astype(np.float32)).cuda()
    t = torch.zeros((1, 8, 12, 16, 1), device="cuda")
    m = torch.ones((1, 8, 12, 16), dtype=torch.uint8, device="cuda")

    def both():
        y = torch.full((8 * 12 * 16,), -1.0, device="cuda")
        net.forward(x, y)
        return y, net.backward(x, t, m)

    y0, loss0 = both()
    with pytest.raises(om.OmError) as e:  # 4.4 TB for the first activation alone
        om._call("om_unet_forward", net.h, om._ptr(x), 16, 2048, 2048, 2048, om._ptr(x), om._stream(None))
    assert e.value.status == om.OM_ENOMEM
    y1, loss1 = both()
    assert torch.equal(y1, y0) and loss1 == pytest.approx(loss0, rel=1e-12)
