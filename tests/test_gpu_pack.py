"""Mask bytes packed to bits 16 at a time (rows that are multiples of 16 voxels
and start on a 16-byte boundary) and by warp ballots (any other): labels,
transport set, node numbering and chord counts against the oracle, for masks
whose pores are not all the byte 1."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(9, 4, 16), (6, 5, 48), (5, 3, 64), (4, 4, 80), (5, 4, 17), (3, 6, 8)])
@pytest.mark.parametrize("offset", [0, 8])
def test_packing(orc, om, shape, offset):
    m = S.random_mask(shape, 0.6, 8)
    lab_o, tr_o, conn_o = orc.label18(m)
    d_o, _ = orc.chord13(m, 1.5, counts=False)
    N = m.size
    raw = torch.zeros(N + 32, dtype=torch.uint8, device="cuda")
    values = np.array([1, 2, 0x80, 0xff], np.uint8)[np.arange(N) % 4] * m.reshape(-1)
    mask = raw[offset:offset + N]
    mask.copy_(torch.from_numpy(values))
    dom = om.domain(shape, 1.5)
    lab = torch.empty(N, dtype=torch.int32, device="cuda")
    tr = torch.empty(N, dtype=torch.uint8, device="cuda")
    assert om.om_label_connectivity_dev(mask, dom, lab, tr) == conn_o
    assert np.array_equal(lab.cpu().numpy().reshape(shape), lab_o)
    assert np.array_equal(tr.cpu().numpy().reshape(shape), tr_o)
    d = torch.empty(N, dtype=torch.float32, device="cuda")
    om.om_local_pore_diameter_dev(mask, dom, om.OM_PORE_CHORD13, d)
    assert np.array_equal(d.cpu().numpy().reshape(shape), d_o)
    ns = om.NodeSet(mask, dom)
    vox = torch.empty(ns.n_nodes, dtype=torch.int64, device="cuda")
    ns.voxels(vox)
    assert np.array_equal(vox.cpu().numpy(), np.flatnonzero(m))
