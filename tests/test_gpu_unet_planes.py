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


@pytest.mark.parametrize("ch,shape,out_ch", [((16,), (1, 3, 5, 7), 1), ((48, 16), (1, 2, 6, 10), 3), ((16, 32), (2, 4, 6, 8), 6)])
def test_gradients_of_the_fused_passes(om, ch, shape, out_ch):
    """Bias and head gradients where the fused passes' cases meet: one level (the head's gradient enters the
    encoder), channel counts that do not divide a block, more outputs than the fused head takes.  Bounds of
    test_gpu_unet.py (BF16 operands of the gradients on both sides)."""
    from oracle import unet as R
    net = om.UNet(2, out_ch, ch, seed=9)
    n = net.n_params
    flat = torch.empty(n, dtype=torch.float32, device="cuda")
    net.get_params(flat)
    g = torch.Generator().manual_seed(4)
    nh = ch[0] * out_ch + out_ch
    flat[n - nh:] = (0.3 * torch.randn(nh, generator=g)).cuda()
    net.set_params(flat)
    x, t = torch.rand(*shape, 2, generator=g), torch.rand(*shape, out_ch, generator=g)
    m = (torch.rand(*shape, generator=g) < 0.7).to(torch.uint8)
    loss = net.backward(x.cuda(), t.cuda(), m.cuda())
    got = torch.empty(n, dtype=torch.float32, device="cuda")
    net.get_grads(got)
    ref_loss, ref, _ = R.loss_and_grads(flat.cpu().double(), x.double(), t.double(), m, 2, out_ch, ch, round_bf16=True)
    assert loss == pytest.approx(ref_loss, rel=2e-2)
    off = 0
    for name, shp in R.layout(2, out_ch, ch):
        k = 1
        for v in shp:
            k *= v
        a, b = got[off:off + k].cpu().double(), ref[off:off + k]
        off += k
        if b.norm() > 1e-12 * ref.norm():
            assert ((a - b).norm() / b.norm()).item() <= 4e-2, name
    # new weights reach the operands
    net.set_params(0.5 * flat)
    y = torch.empty(*shape, out_ch, dtype=torch.float32, device="cuda")
    net.forward(x.cuda(), y)
    ry = R.forward(R.unflatten(0.5 * flat.cpu().double(), 2, out_ch, ch), x.double(), 2, out_ch, ch, round_bf16=True)
    assert (y.cpu().double() - ry).abs().max().item() <= 2e-2 * ry.abs().max().item()


@pytest.mark.parametrize("ch,shape", [((16,), (1, 457, 17, 33)), ((32,), (2, 130, 17, 65))])
def test_planes_shared_multiprocessor(om, ch, shape):
    """Enough planes that three (16 channels) or two (32) blocks share a multiprocessor, with shares that start
    inside a column and tiles cut at the far edges; same bounds."""
    test_planes_match_reference(om, ch, shape)
