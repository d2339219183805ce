"""The odd sweeps with parked slot offsets (flow variants 13 and 14, diffusion
variant 9, batch variant 1) against the plain ones, bit for bit: every launch
variant does the same arithmetic per node.  Boxes of faces only, ragged ones, one
whose last block is nearly empty; every storage format, both drives, both
diffusion lattices, and FP32 flow in its rebased mode (through a solve)."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu

SHAPES = [(4, 2, 3), (5, 3, 2), (4, 9, 33), (11, 20, 70)]


def _nodes(om, shape, p=0.7):
    m = S.random_mask(shape, p, 3)
    m[:, 0, 0] = 1
    tr = torch.from_numpy(m.reshape(-1)).cuda()
    return om.domain(shape), tr, om.NodeSet(tr, om.domain(shape))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("drive", [0, 1])
def test_flow_parked_bits(om, shape, prec, drive):
    dom, tr, ns = _nodes(om, shape)
    N = tr.numel()
    u0 = torch.from_numpy(S.random_field(N, 5, -1e-2, 1e-2, np.float32)).cuda()
    ref = None
    for variant in (0, 13, 14):
        fl = om.Flow(ns, om.flow_params(tau=0.8, precision=prec, variant=variant, drive=drive, check_every=4))
        fl.init_velocity(u0)
        fl.step(9)
        fl.step(4)
        f = torch.empty(19 * N, dtype=torch.float64, device="cuda")
        fl.get_populations(f)
        if ref is None:
            ref = f
        assert torch.equal(f, ref), variant


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("lattice", [7, 19])
def test_diffusion_parked_bits(om, shape, prec, lattice):
    dom, tr, ns = _nodes(om, shape)
    N = tr.numel()
    d = torch.from_numpy(S.random_field(N, 6, 5.0, 60.0, np.float32)).cuda()
    c0 = torch.from_numpy(S.random_field(N, 7, 0.0, 1.0, np.float32)).cuda()
    ref = None
    for variant in (0, 9):
        df = om.Diffusion(ns, d, om.diff_params(precision=prec, variant=variant, lattice=lattice, check_every=4))
        df.init_concentration(c0)
        df.step(9)
        df.step(4)
        g = torch.empty(lattice * N, dtype=torch.float64, device="cuda")
        df.get_populations(g)
        if ref is None:
            ref = g
        assert torch.equal(g, ref), variant


def test_rebased_fp32_solve_parked(om):
    dom, tr, ns = _nodes(om, (11, 20, 70), 0.9)
    out = []
    for variant in (0, 13, 14):
        fl = om.Flow(ns, om.flow_params(precision=om.OM_F32, variant=variant, conv_tol=1e-7, max_steps=4000))
        st, k, info = fl.solve()
        out.append((st, k, info.steps))
    assert out[0][2] > 100 and out[1] == out[0] and out[2] == out[0]


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_batch_parked_bits(om, prec):
    doms, trs, ds = [], [], []
    for k, shape in enumerate(SHAPES):
        dom, tr, ns = _nodes(om, shape)
        doms.append(dom)
        trs.append(tr)
        ds.append(torch.from_numpy(S.random_field(tr.numel(), 6 + k, 5.0, 60.0, np.float32)).cuda())
    ref = {}
    for variant in (0, 1):
        b = om.Batch(doms, trs, ds, flow=om.flow_params(precision=prec, variant=variant),
                     diff=om.diff_params(precision=prec, variant=variant))
        for model, q in ((0, 19), (1, 7)):
            for k, tr in enumerate(trs):
                f0 = torch.from_numpy(S.random_field(tr.numel(), 20 + k, 0.0, 1e-2, np.float32)).cuda()
                b.init_fields(model, k, f0)
            b.step(model, 13)
            for k, tr in enumerate(trs):
                f = torch.empty(q * tr.numel(), dtype=torch.float64, device="cuda")
                b.get_populations(model, k, f)
                assert torch.equal(f, ref.setdefault((model, k), f)), (variant, model, k)
        b.close()
