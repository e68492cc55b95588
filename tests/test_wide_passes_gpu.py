"""The passes of many fields on long axes, whose transforms run in field groups with
radix-16 stages, and 3D rows of 2048 nodes (two warps a row, in the kernel that reads
its length): thin boxes against the FP64 direct-sum oracle.

Fields are white noise, whose FP32 transform error is a few 1e-7 of the result.
Tolerances as in the force, nonlinear and adjoint tests: 1e-11 relative L2 in FP64, in
FP32 1e-5, and 2e-5 for the adjoint."""
import numpy as np
import pytest
import torch

from paper_2105_06055_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


@pytest.fixture(scope="module")
def pdm():
    from paper_2105_06055_gb300 import build, pd
    build.build()
    pd.load()
    return pd


def _case(shape, fp64, amp):
    g = inputs.rng(sum(shape) + int(fp64))
    chi = inputs.box_mask(shape, (3,) * len(shape), tuple(n - 3 for n in shape[::-1]))
    chi[g.random(shape) < 0.1] = 0
    dt = torch.float64 if fp64 else torch.float32
    u = torch.tensor(amp * g.normal(size=(len(shape),) + shape), dtype=dt, device=DEV)
    return g, chi, u


def _rel(a, b):
    return np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b)


@pytest.mark.parametrize("fp64", [True, False])
def test_3d_rows_of_2048_nodes(pdm, oracle, fp64):
    shape = (16, 16, 2048)
    _, chi, u = _case(shape, fp64, 1.0)
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=2.5, fp64=fp64), torch.tensor(chi, device=DEV))
    L, W = plan.force(u, want_energy=True)
    L2 = plan.force(u)
    plan.close()
    un, alpha = u.double().cpu().numpy(), oracle.alpha_bond(3, 1.0, 2.5)
    ref, wref = oracle.force_bond(un, chi, 1.0, 2.5, alpha), oracle.energy_bond(un, chi, 1.0, 2.5, alpha)
    tol = 1e-11 if fp64 else 1e-5
    assert _rel(L, ref) < tol and _rel(L2, ref) < tol and _rel(W, wref) < tol


@pytest.mark.parametrize("shape,fp64", [((256, 16, 32), False), ((512, 16, 32), False), ((256, 16, 32), True),
                                        ((512, 64), False), ((1024, 32), False), ((512, 64), True)])
def test_nonlinear_on_a_long_last_axis(pdm, oracle, shape, fp64):
    _, chi, u = _case(shape, fp64, 0.1)
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=2.5, model=pdm.PD_NONLIN_BOND, fp64=fp64),
                    torch.tensor(chi, device=DEV))
    L = plan.force(u)
    plan.close()
    ref = oracle.force_nonlinear(u.double().cpu().numpy(), chi, 1.0, 2.5, oracle.alpha_bond(len(shape), 1.0, 2.5))
    assert _rel(L, ref) < (1e-11 if fp64 else 1e-5)


@pytest.mark.parametrize("shape,fp64", [((512, 16, 32), False), ((512, 16, 32), True), ((1024, 16, 32), False),
                                        ((1024, 32), False), ((1024, 32), True)])
def test_adjoint_on_a_long_last_axis(pdm, oracle, shape, fp64):
    g, chi, u = _case(shape, fp64, 1.0)
    s = torch.tensor(0.5 + g.random(shape), dtype=u.dtype, device=DEV)
    p = torch.tensor(g.normal(size=u.shape), dtype=u.dtype, device=DEV)
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=2.5, fp64=fp64), torch.tensor(chi, device=DEV))
    gu, gs = plan.force_adjoint(u, p, s=s)
    plan.close()
    un, sn, pn = (t.double().cpu().numpy() for t in (u, s, p))
    alpha = oracle.alpha_bond(len(shape), 1.0, 2.5)
    tol = 1e-11 if fp64 else 2e-5
    assert _rel(gu, oracle.force_bond(pn, chi, 1.0, 2.5, alpha, s=sn)) < tol
    assert _rel(gs, oracle.force_bond_grad_s(un, pn, chi, 1.0, 2.5, alpha, s=sn)) < tol
