"""The horizon sums on shared-memory tiles (boundary field of a node weight,
Eq. 47 energy density) at the edges of their tiles: a 2D grid lower than one
tile, the smallest 3D box, tiles that wrap around the box, a reach of 20 cells, and a horizon whose
tile does not fit (the sums that read global memory), against the oracle.

Tolerances are those of the force tests: 1e-11 relative L2 in FP64 (rounding
of a reordered sum), 1e-5 in FP32; breaking decisions are exact in FP64."""
import numpy as np
import pytest
import torch

from paper_2105_06055_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
SHAPES = [((16, 32), 2.0), ((64, 32), 6.0), ((16, 16, 32), 2.0), ((32, 16, 64), 3.0), ((32, 32, 32), 7.0)]


@pytest.fixture(scope="module")
def pdm():
    from paper_2105_06055_gb300 import build, pd
    build.build()
    pd.load()
    return pd


def _body(shape, delta, g):
    m = int(np.ceil(delta))
    chi = inputs.box_mask(shape, (m,) * len(shape), tuple(n - m for n in shape[::-1]))
    chi[g.random(shape) < 0.1] = 0
    return chi


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape,delta", SHAPES)
def test_weighted_force(pdm, oracle, shape, delta, fp64):
    g = inputs.rng(5)
    chi = _body(shape, delta, g)
    d = len(shape)
    dt = torch.float64 if fp64 else torch.float32
    u = torch.tensor(g.normal(size=(d,) + shape), dtype=dt, device=DEV)
    s = torch.tensor(0.5 + g.random(shape), dtype=dt, device=DEV)
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=delta, fp64=fp64), torch.tensor(chi, device=DEV))
    L = plan.force(u, s=s).double().cpu().numpy()
    plan.close()
    ref = oracle.force_bond(u.double().cpu().numpy(), chi, 1.0, delta, oracle.alpha_bond(d, 1.0, delta),
                            s=s.double().cpu().numpy())
    assert np.linalg.norm(L - ref) / np.linalg.norm(ref) < (1e-11 if fp64 else 1e-5)


@pytest.mark.parametrize("shape,delta", SHAPES[:4])
def test_breaking_by_the_energy_sum(pdm, oracle, shape, delta):
    """Three steps through the breaking of many nodes."""
    g = inputs.rng(6)
    chi = _body(shape, delta, g)
    d = len(shape)
    lam = chi.copy()
    lam[g.random(shape) < 0.05] = 0
    u = 1e-3 * g.normal(size=(d,) + shape) * chi
    alpha = oracle.alpha_bond(d, 1.0, delta)
    W = oracle.energy_bond(u, chi, 1.0, delta, alpha, lam=lam)
    wc = float(np.quantile(W[(chi & lam) == 1], 0.8))
    om = np.stack([chi] * d)
    z = np.zeros_like(u)
    uo, vo, lo, nb = oracle.verlet_damage(u, z, lam, chi, om, z, z, 1.0, delta, alpha, 1.0, 0.1, wc, 3)
    assert 0 < nb < int((chi & lam).sum())
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=delta, rho=1.0, Wc=wc, fp64=True), torch.tensor(chi, device=DEV))
    plan.set_energy_mode(True)
    ud, vd, bd = (torch.tensor(a, device=DEV) for a in (u, z, z))
    ld = torch.tensor(lam, device=DEV)
    assert plan.step_verlet(ud, vd, ld, bd, None, dt=0.1, nsteps=3, count_broken=True) == nb
    plan.close()
    assert np.array_equal(ld.cpu().numpy(), lo)
    assert np.linalg.norm(ud.cpu().numpy() - uo) / np.linalg.norm(uo) < 1e-11


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape,dx,delta", [((32, 128), (0.1, 1.0), 2.0), ((16, 16, 64), (0.1, 1.0, 1.0), 2.0)])
def test_long_reach_along_x1(pdm, oracle, shape, dx, delta, fp64):
    """A horizon of 20 cells along x1 (uneven spacings): rows of the tile longer than two columns per lane."""
    g = inputs.rng(7)
    d = len(shape)
    chi = np.zeros(shape, np.uint8)
    chi[(slice(2, -2),) * (d - 1) + (slice(20, -20),)] = 1
    chi[g.random(shape) < 0.1] = 0
    dt = torch.float64 if fp64 else torch.float32
    u = torch.tensor(g.normal(size=(d,) + shape), dtype=dt, device=DEV)
    s = torch.tensor(0.5 + g.random(shape), dtype=dt, device=DEV)
    plan = pdm.Plan(pdm.Problem(shape=shape, dx=dx, delta=delta, fp64=fp64), torch.tensor(chi, device=DEV))
    L = plan.force(u, s=s).double().cpu().numpy()
    plan.close()
    ref = oracle.force_bond(u.double().cpu().numpy(), chi, dx, delta, oracle.alpha_bond(d, 1.0, delta),
                            s=s.double().cpu().numpy())
    assert np.linalg.norm(L - ref) / np.linalg.norm(ref) < (1e-11 if fp64 else 1e-5)
