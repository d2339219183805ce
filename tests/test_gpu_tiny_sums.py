"""Sums over populations as small as single precision holds, subnormal ones
among them: a flux that dies away (a structure whose pores meet only along
links the diffusion lattice does not have) ends there, and a solver that read
it as exactly 0 would report convergence.  Observables and exported fields
against sums of the stored populations; the bound is that of the larger ones,
2^-50 of the sum of the nodes' largest terms."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPE = (12, 20, 70)
N = SHAPE[0] * SHAPE[1] * SHAPE[2]
EX = np.array([0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0.0])
W19 = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
W7 = np.array([1 / 4] + [1 / 8] * 6)
SCALES = [1e-3, 1e-23, 1e-25, 1e-30, 1e-38, 1e-42, None]  # None: every node its own


def _scale(rng, scale):
    return 10.0 ** rng.uniform(-42, -1, N) if scale is None else np.full(N, scale)


def _nodes(om):
    return om.NodeSet(torch.ones(N, dtype=torch.uint8, device="cuda"), om.domain(SHAPE))


@pytest.mark.parametrize("lattice", [7, 19])
@pytest.mark.parametrize("scale", SCALES)
def test_diffusion_tiny_sums(om, lattice, scale):
    rng = np.random.default_rng(4)
    w = W7 if lattice == 7 else W19
    gd = rng.uniform(0.5, 1.0, (lattice, N)) * _scale(rng, scale)
    total = np.zeros(N)
    for row in gd:
        total = total + row
    ref = total.astype(np.float32).astype(np.float64)
    g = (gd - w[:, None] * ref).astype(np.float32).astype(np.float64)  # what the solver stores
    d = torch.full((N,), 60.0, device="cuda")  # relaxation rate 1
    df = om.Diffusion(_nodes(om), d, om.diff_params(precision=om.OM_F32, variant=0, lattice=lattice))
    df.set_populations(torch.from_numpy(gd.reshape(-1)).cuda())
    sj, dc, _, sc, _ = df.observe()
    flux = 0.5 * (EX[:lattice, None] * g)
    bound = 2.0 ** -50 * math.fsum(np.abs(g).max(0))
    assert abs(sj - math.fsum(flux.ravel())) <= bound
    assert abs(sc - math.fsum(g.ravel()) - math.fsum(ref)) <= bound + 2.0 ** -50 * math.fsum(ref)
    assert dc == 0.0
    jx = torch.empty(N, device="cuda")
    df.get_fields(None, jx)
    one = flux.sum(0)
    assert np.all(np.abs(jx.cpu().numpy() - one) <= 2.0 ** -24 * np.abs(one) + 2.0 ** -150 + 2.0 ** -50 * np.abs(g).max(0))


@pytest.mark.parametrize("scale", SCALES)
def test_flow_tiny_sums(om, scale):
    rng = np.random.default_rng(5)
    u = (rng.uniform(0.5, 1.0, N) * _scale(rng, scale)).astype(np.float32)
    fl = om.Flow(_nodes(om), om.flow_params(body_force=0.0, precision=om.OM_F32, variant=0))
    fl.init_velocity(torch.from_numpy(u).cuda())
    ux = fl.observe()[0]
    # each population of the equilibrium is stored to 2^-24 of itself or half of 2^-149, ten of them carry u
    bound = (2.0 ** -24 + 2.0 ** -50) * u.astype(np.float64) * 2 + 10 * 2.0 ** -150
    assert abs(ux - math.fsum(u.astype(np.float64))) <= math.fsum(bound)
    v = torch.empty(3 * N, device="cuda")
    fl.get_velocity(v)
    v = v.cpu().numpy()
    assert np.all(np.abs(v[:N] - u.astype(np.float64)) <= bound + 2.0 ** -24 * u + 2.0 ** -150)
    assert not v[N:].any()
