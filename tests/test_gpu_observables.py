"""The observables' sums against exact sums of the stored populations: equal
sizes, fourteen decades at once, cancelling pairs, few non-zeros, none.  The
device sums a node's populations to 2^-57 of the largest, then nodes in double:
the bound is 2^-50 of the sum of the nodes' largest terms, taken per value."""
import math

import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu

EX = [0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0]
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.mark.parametrize("kind", ["even", "decades", "cancel", "few", "none"])
@pytest.mark.parametrize("shape", [(5, 4, 3), (12, 20, 70)])
def test_flow_sums(om, kind, shape):
    rng = np.random.default_rng(3)
    N = int(np.prod(shape))
    dev = rng.uniform(-1e-3, 1e-3, (19, N))
    if kind == "decades":
        dev *= 10.0 ** rng.uniform(-12, 0, dev.shape)
    elif kind == "cancel":
        dev[2] = -dev[1] * (1 + 1e-6)
        dev[8::2] = -dev[7:-1:2]
    elif kind == "few":
        dev *= rng.random(dev.shape) < 0.05
    elif kind == "none":
        dev *= 0.0
    fd = W[:, None] + dev
    f = (fd - W[:, None]).astype(np.float32).astype(np.float64)  # what the solver stores
    g = 1e-6
    dom = om.domain(shape)
    ns = om.NodeSet(torch.ones(N, dtype=torch.uint8, device="cuda"), dom)
    fl = om.Flow(ns, om.flow_params(body_force=g, precision=om.OM_F32, variant=0))
    fl.set_populations(torch.from_numpy(fd.reshape(-1)).cuda())
    ux, dux, aux, mass = fl.observe()
    jx = [math.fsum(e * v for e, v in zip(EX, f[:, n]) if e) + 0.5 * float(np.float32(g)) for n in range(N)]
    bound = 2.0 ** -50 * (math.fsum(np.abs(f).max(0)) + 0.5 * g * N)
    assert abs(ux - math.fsum(jx)) <= bound
    assert abs(aux - math.fsum(map(abs, jx))) <= bound
    assert abs(mass - math.fsum(f.ravel())) <= bound * 2
    assert dux == 0.0  # set_populations observed this state


def test_flow_sums_show_divergence(om):
    shape = (4, 4, 40)
    N = int(np.prod(shape))
    fd = np.repeat(W[:, None], N, 1)
    for bad in (np.inf, np.nan, 3e38):
        f = fd.copy()
        f[1, 17] = bad
        ns = om.NodeSet(torch.ones(N, dtype=torch.uint8, device="cuda"), om.domain(shape))
        fl = om.Flow(ns, om.flow_params(precision=om.OM_F32, variant=0))
        fl.set_populations(torch.from_numpy(f.reshape(-1)).cuda())
        ux, _, aux, mass = fl.observe()
        if bad == 3e38:
            assert ux == pytest.approx(3e38, rel=1e-6) and mass == pytest.approx(3e38, rel=1e-6)
        else:
            assert not math.isfinite(ux) and not math.isfinite(mass)
