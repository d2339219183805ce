"""The pore-size kernels at the sizes where their packing can go wrong, against
the oracle: boxes whose edges are one below, at and above the 32-bit words and
the 4-voxel bricks they work on, edges of one voxel, and masks so full that
lines run through many words or close on themselves.  Counts are integers and
the sizes fixed sequences of double operations, so the comparison is exact."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

SHAPES = [(33, 32, 31), (31, 33, 65), (64, 1, 7), (3, 7, 1), (1, 40, 33), (34, 63, 97), (5, 6, 129)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("p", [0.5, 0.97, 0.9995, 1.0])
def test_chord13_words_and_loops(orc, om, shape, p):
    mask = S.random_mask(shape, p, 11)
    d_o, w_o = orc.chord13(mask, 1.5, counts=True)
    d, w = om.om_local_pore_diameter(mask, om.domain(shape, 1.5), om.OM_PORE_CHORD13, witness=True)
    assert np.array_equal(w, w_o)
    assert np.array_equal(d, d_o)


# small boxes: the oracle tests every pair of voxels
@pytest.mark.parametrize("shape", [(64, 1, 7), (3, 7, 1), (1, 40, 33), (5, 6, 129), (9, 5, 4), (17, 13, 19), (21, 15, 18)])
@pytest.mark.parametrize("p", [0.5, 0.97, 0.9995])
def test_inscribed_bricks(orc, om, shape, p):
    mask = S.random_mask(shape, p, 12)
    mask.flat[mask.size // 2] = 0
    rc, d_o, r2_o = orc.mis(mask, 1.5)
    d, r2 = om.om_local_pore_diameter(mask, om.domain(shape, 1.5), om.OM_PORE_MIS, witness=True)
    assert rc == 0 and np.array_equal(r2, r2_o)
    assert np.array_equal(d, d_o)


@pytest.mark.parametrize("shape", [(90, 85, 83), (140, 137, 131)])
def test_chord13_listed_voxels(orc, om, shape):
    """Boxes where a block lists the pores of two and of eight voxels a thread, the last block cut short."""
    mask = S.random_mask(shape, 0.6, 13)
    mask[: shape[0] // 3] = 0  # blocks without a pore
    d_o, w_o = orc.chord13(mask, 1.5, counts=True)
    d, w = om.om_local_pore_diameter(mask, om.domain(shape, 1.5), om.OM_PORE_CHORD13, witness=True)
    assert np.array_equal(w, w_o)
    assert np.array_equal(d, d_o)


@pytest.mark.parametrize("shape", [(32, 16, 11), (40, 9, 15), (13, 22, 20)])
@pytest.mark.parametrize("solids", [1, 5])
def test_inscribed_large_balls(orc, om, shape, solids):
    """Balls larger than several bricks, and wider than the box is in y and z."""
    mask = np.ones(shape, np.uint8)
    mask.flat[np.random.default_rng(solids).choice(mask.size, solids, replace=False)] = 0
    rc, d_o, r2_o = orc.mis(mask, 1.5)
    d, r2 = om.om_local_pore_diameter(mask, om.domain(shape, 1.5), om.OM_PORE_MIS, witness=True)
    assert rc == 0 and np.array_equal(r2, r2_o)
    assert np.array_equal(d, d_o)
