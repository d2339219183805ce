"""The plane-marching convolution where its tiling can go wrong, against the FP64
reference: grids below, at and above the 8 x 16 tile, one voxel, one plane,
more planes than its accumulator ring, shares that start inside a column, and
every count of 32-channel input chunks and output parts it takes.

Reference and kernel hold the same BF16 inputs, weights and stored activations;
a stored activation moves to its neighbouring BF16 value (2^-8 relative) only
where the FP32 sum falls on a rounding boundary.  An output sums at most a few
such moves through the 1x1 head: below 2^-8 times the terms' magnitudes, taken
as 2 % of the output's scale element-wise and 0.2 % of its mean on average."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ch,shape", [
    ((16,), (1, 1, 1, 1)), ((16,), (1, 1, 16, 8)), ((16,), (2, 2, 17, 9)), ((16,), (1, 70, 3, 7)),
    ((32,), (1, 41, 15, 8)), ((32,), (3, 5, 33, 31)), ((80,), (1, 9, 17, 10)), ((96,), (1, 12, 16, 16)),
    ((48,), (1, 40, 130, 40)), ((64,), (2, 13, 16, 24)),
    ((16, 32), (1, 34, 18, 10)), ((32, 64), (1, 6, 34, 18)), ((16, 80), (2, 4, 16, 16))])
def test_planes_match_reference(om, ch, shape):
    from oracle import unet as R
    net = om.UNet(2, 2, ch, seed=5)
    n = net.n_params
    flat = torch.empty(n, dtype=torch.float32, device="cuda")
    net.get_params(flat)
    g = torch.Generator().manual_seed(21)
    nh = ch[0] * 2 + 2
    flat[n - nh:] = (0.3 * torch.randn(nh, generator=g)).cuda()
    net.set_params(flat)
    x = torch.rand(*shape, 2, generator=g)
    y = torch.full((*shape, 2), float("nan"), dtype=torch.float32, device="cuda")
    net.forward(x.cuda(), y)
    ref = R.forward(R.unflatten(flat.cpu().double(), 2, 2, ch), x.double(), 2, 2, ch, round_bf16=True)
    err = (y.cpu().double() - ref).abs()
    assert torch.isfinite(err).all()
    assert err.max().item() <= 2e-2 * ref.abs().max().item()
    assert err.mean().item() <= 2e-3 * ref.abs().mean().item()
