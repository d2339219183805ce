"""The rasteriser's forms against the oracle, bit for bit: balls just below and
above the size from which a voxel may lie in two periodic images (the box
edge less 8 voxels), balls wider than the box, and more balls in one batch
than the shared-memory counters hold (16384)."""
import numpy as np
import pytest

import synthetic as S
from conftest import recon_args, recon_params

pytestmark = pytest.mark.gpu

CFGS = [
    S.Recon(3, (21, 20, 20), 1.0, 12.0, 0.5, 11.0, 13.0, 0.5, 0.4, dist=1),
    S.Recon(4, (18, 31, 17), 1.5, 14.0, 3.0, 6.0, 24.0, 0.45, 0.6),
    S.Recon(5, (30, 12, 70), 1.0, 18.0, 2.0, 12.0, 24.0, 0.5, 0.7),
    S.Recon(6, (48, 48, 48), 1.0, 2.0, 0.2, 1.5, 2.5, 0.48, 0.9),
]


@pytest.mark.parametrize("cfg", CFGS)
def test_raster_forms(orc, om, cfg):
    rc, mask_o, sph, eps_o, _ = orc.reconstruct(*recon_args(cfg))
    st, mask_g, eps_g, n_g = om.om_reconstruct(cfg.seed, om.domain(cfg.shape, cfg.dx_nm), recon_params(om, cfg))
    assert rc == 0 and st == om.OM_OK
    assert np.array_equal(mask_o, mask_g)
    assert len(sph) == n_g and eps_o == eps_g
