"""Force passes over every axis length and shape of their kernels: row lengths
32 to 2048 (and grids with fewer rows than a warp transforms at once), column
lengths 16 to 1024 as x2 and as last axis, both precisions, against the FP64
direct-sum oracle; the adjoint on fields that start on odd elements.

Tolerances as in the force tests: 1e-11 relative L2 in FP64, 1e-5 in FP32
(white-noise fields: the transform error is a few 1e-7)."""
import numpy as np
import pytest
import torch

from paper_2105_06055_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")

SHAPES = [(16, 32), (32, 64), (64, 128), (128, 32), (256, 256), (512, 64), (1024, 32), (16, 512), (32, 1024),
          (16, 2048), (16, 16, 32), (16, 32, 64), (32, 16, 128), (64, 32, 32), (128, 16, 32), (16, 64, 256),
          (256, 16, 32), (16, 256, 32), (512, 16, 32), (16, 16, 512), (16, 16, 1024), (1024, 16, 32)]


@pytest.fixture(scope="module")
def pdm():
    from paper_2105_06055_gb300 import build, pd
    build.build()
    pd.load()
    return pd


def _body(shape, g):
    chi = inputs.box_mask(shape, (3,) * len(shape), tuple(n - 3 for n in shape[::-1]))
    chi[g.random(shape) < 0.1] = 0
    return chi


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_force_every_length(pdm, oracle, shape, fp64):
    g = inputs.rng(sum(shape))
    d = len(shape)
    chi = _body(shape, g)
    dt = torch.float64 if fp64 else torch.float32
    u = torch.tensor(g.normal(size=(d,) + shape), dtype=dt, device=DEV)
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=2.5, fp64=fp64), torch.tensor(chi, device=DEV))
    L2 = plan.force(u)
    if fp64 and d == 3 and shape[0] == 1024:
        # nine fields of 1024 doubles do not fit a block's shared memory: refused
        with pytest.raises(pdm.PDError):
            plan.force(u, want_energy=True)
        L, W = L2, None
    else:
        L, W = plan.force(u, want_energy=True)
        W = W.double().cpu().numpy()
    L, L2 = (a.double().cpu().numpy() for a in (L, L2))
    plan.close()
    un = u.double().cpu().numpy()
    alpha = oracle.alpha_bond(d, 1.0, 2.5)
    ref, wref = oracle.force_bond(un, chi, 1.0, 2.5, alpha), oracle.energy_bond(un, chi, 1.0, 2.5, alpha)
    tol = 1e-11 if fp64 else 1e-5
    for a, r in ((L, ref), (L2, ref), (W if W is not None else wref, wref)):
        assert np.linalg.norm(a - r) / np.linalg.norm(r) < tol


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape", [(32, 64), (16, 32, 32)])
def test_adjoint_on_odd_elements(pdm, shape, fp64):
    """pd_force_adjoint takes fields that start on any element of a buffer."""
    g = inputs.rng(3)
    d = len(shape)
    dt = torch.float64 if fp64 else torch.float32
    plan = pdm.Plan(pdm.Problem(shape=shape, delta=2.5, fp64=fp64), torch.tensor(_body(shape, g), device=DEV))

    def odd(x):
        buf = torch.empty(x.numel() + 1, dtype=dt, device=DEV)
        buf[1:] = x.reshape(-1)
        return buf[1:].view(x.shape)

    u, p = (torch.tensor(g.normal(size=(d,) + shape), dtype=dt, device=DEV) for _ in range(2))
    gu, gs = plan.force_adjoint(u, p)
    gu2, gs2 = plan.force_adjoint(odd(u), odd(p))
    assert torch.equal(gu, gu2) and torch.equal(gs, gs2)
    plan.close()
