"""Forms that only some calls reach: every launch variant of the odd sweeps
against the oracle and, on a box beyond the neighbour records' fields, against
variant 0 bit for bit; more balls in one batch than the shared-memory counters
hold; inscribed spheres around a solid voxel, whose brick lists more bricks
than fit at a time; CHORD13 where the scratch for its packed lines cannot be
had."""
import ctypes as C
import math

import numpy as np
import pytest
import torch

import synthetic as S
from conftest import recon_args, recon_params
from test_gpu_lbm import GEOMS, _diff_run, _flow_run, _rand_d, _rand_diff, _rand_pops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [13, 14])
def test_parked_flow_matches_oracle(orc, om, variant):
    node = GEOMS["blobs"]()
    f0 = _rand_pops(orc, node, 7)
    got = _flow_run(om, node, f0, 0.8, 1e-5, 7, om.OM_F64, variant)
    assert np.abs(got - orc.flow_step(node, f0, 0.8, 1e-5, 7)).max() <= 1e-13 * 7


@pytest.mark.parametrize("q", [7, 19])
def test_parked_diffusion_matches_oracle(orc, om, q):
    node = GEOMS["ragged"]()
    g0, d = _rand_diff(node, 8, q=q), _rand_d(node, 9)
    got = _diff_run(om, node, d, g0, 7, om.OM_F64, 0.9, 0.2, 9)
    assert np.abs(got - orc.diff_step(node, g0, orc.omega_field(node, d), 0.9, 0.2, 7)).max() <= 1e-13 * 7


@pytest.mark.parametrize("prec", ["OM_F64", "OM_F32", "OM_F16DEV"])
def test_variants_without_records(orc, om, prec):
    node = S.random_mask((5, 6, 1030), 0.7, 21)  # records hold z edges up to 1023
    P = getattr(om, prec)
    f0 = _rand_pops(orc, node, 22, amp=0.05)
    first = _flow_run(om, node, f0, 1.0, 1e-5, 5, P, 0)
    for v in range(7, 15):
        assert np.array_equal(_flow_run(om, node, f0, 1.0, 1e-5, 5, P, v), first), v
    d = _rand_d(node, 24)
    for q in (7, 19):
        g0 = _rand_diff(node, 23, q=q)
        first = _diff_run(om, node, d, g0, 5, P, 1.0, 0.0, 0)
        for v in range(6, 10):
            assert np.array_equal(_diff_run(om, node, d, g0, 5, P, 1.0, 0.0, v), first), (q, v)


def test_raster_global_counters(orc, om):
    cfg = S.Recon(6, (56, 56, 56), 1.0, 2.0, 0.2, 1.5, 2.5, 0.48, 0.9)
    # the first batch places 1.15 times what the mean volume asks for, and 16
    first = math.ceil(1.15 * cfg.porosity * 56 ** 3 / (4 * math.pi / 3 * (0.5 * cfg.mean_nm) ** 3)) + 16
    assert first > 16384  # counters of a block
    rc, mask_o, sph, eps_o, _ = orc.reconstruct(*recon_args(cfg))
    st, mask_g, eps_g, n_g = om.om_reconstruct(cfg.seed, om.domain(cfg.shape, cfg.dx_nm), recon_params(om, cfg))
    assert rc == 0 and st == om.OM_OK
    assert np.array_equal(mask_o, mask_g)
    assert len(sph) == n_g and eps_o == eps_g


@pytest.mark.parametrize("shape", [(40, 36, 33), (33, 38, 43)])
@pytest.mark.parametrize("solids", [1, 3])
def test_inscribed_more_bricks_than_the_list(om, shape, solids):
    mask = np.ones(shape, np.uint8)
    at = np.random.default_rng(solids).choice(mask.size, solids, replace=False)
    at[0] = np.ravel_multi_index([s // 2 for s in shape], shape)
    mask.flat[at] = 0
    n = torch.tensor(shape, device="cuda")
    v = torch.stack(torch.meshgrid(*[torch.arange(s, device="cuda") for s in shape], indexing="ij"), -1).reshape(-1, 3)

    def dist2(a, b):
        g = (a[:, None] - b[None]).abs()
        g = torch.cat([g[..., :1], torch.minimum(g[..., 1:], n[1:] - g[..., 1:])], -1)
        return (g * g).sum(-1)

    r2 = dist2(v, v[torch.from_numpy(at).cuda()]).amin(1)
    best = torch.cat([torch.where(dist2(p, v) < r2[None], r2[None], 0).amax(1) for p in v.split(512)])
    # the brick of the first solid voxel: no ball holds all of it, its smallest radius is 1, and
    # the balls of more than 480 bricks reach it
    b = torch.tensor([s // 2 // 4 * 4 for s in shape], device="cuda")
    home = dist2(v, torch.stack([torch.clamp(b + torch.tensor([i, j, k], device="cuda"), max=n - 1) for i in range(4)
                                 for j in range(4) for k in range(4)])).amin(1)
    reach = v[(home < r2) & (r2 > 1)] // 4
    assert len(torch.unique(reach, dim=0)) > 480
    d, w = om.om_local_pore_diameter(mask, om.domain(shape, 1.5), om.OM_PORE_MIS, witness=True)
    assert np.array_equal(w.ravel(), r2.cpu().numpy())
    best = best.cpu().numpy()
    want = np.where(mask.ravel() > 0, (1.5 * (2.0 * np.sqrt(best.astype(np.float64)) - 1.0)).astype(np.float32), 0)
    assert np.array_equal(d.ravel(), want.astype(np.float32))


class _PoolProps(C.Structure):  # CUmemPoolProps
    _fields_ = [("alloc", C.c_int), ("handles", C.c_int), ("where", C.c_int), ("device", C.c_int), ("security", C.c_void_p),
                ("most", C.c_size_t), ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]


def test_chord13_without_scratch(om):
    shape = (336, 352, 352)  # the packed lines take 68 MB
    mask = torch.from_numpy(S.random_mask(shape, 0.6, 5).reshape(-1)).cuda()
    dom = om.domain(shape, 1.5)
    packed, walked = (torch.full((mask.numel(),), -1.0, device="cuda") for _ in range(2))
    om.om_local_pore_diameter_dev(mask, dom, om.OM_PORE_CHORD13, packed)
    torch.cuda.synchronize()
    cu, dev = C.CDLL("libcuda.so.1"), torch.cuda.current_device()
    old, small = C.c_void_p(), C.c_void_p()
    assert cu.cuDeviceGetMemPool(C.byref(old), dev) == 0
    props = _PoolProps(1, 0, 1, dev, None, 1 << 21)  # pinned memory of this device, 2 MB of it
    assert cu.cuMemPoolCreate(C.byref(small), C.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(dev, small) == 0
    try:
        p = C.c_void_p()
        assert cu.cuMemAllocAsync(C.byref(p), C.c_size_t(60 << 20), None) != 0  # so the packed form has no scratch
        om.om_local_pore_diameter_dev(mask, dom, om.OM_PORE_CHORD13, walked)
        torch.cuda.synchronize()
    finally:
        assert cu.cuDeviceSetMemPool(dev, old) == 0
        cu.cuMemPoolDestroy(small)
    assert torch.equal(walked, packed)
