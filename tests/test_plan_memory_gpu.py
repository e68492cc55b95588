"""Device memory of a plan: nothing beyond the passes' own packed spectra, which are
transformed in place, and the fields, masks and tables.

Bytes per node of an FP32 plan with a horizon of 2.5: spectra 4 per slot (bond model: 7
slots in 2D, 12 in 3D; nonlinear model in 3D: 21) and 8 per FP64 slot (2 in 2D, 5 in
3D); masks 2 + d; boundary field 12 per component; solver vectors 16 d, weight field 4 per
component, FP64 residual 8 d, dilatations 12; kernel spectra 12 per component (nonlinear:
+ 12 + 36) on the folded box, (n1/2 + 1)(n2/2 + 1)... modes of N. A boundary node has its
list entry in FP64 and FP32 (88 bytes), the moments of the affine split and the
nonlinear model's 16. Twiddles, bond tables and reduction buffer: below 2 MB, rounding
up of allocations 2%."""
import pytest
import torch

from paper_2105_06055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,nonlinear", [((512, 1024), False), ((64, 64, 128), False), ((64, 64, 128), True)])
def test_plan_holds_no_spare_spectra(shape, nonlinear):
    from paper_2105_06055_gb300 import build, pd
    build.build()
    pd.load()
    d, N, modes = len(shape), 1, 1
    for n in shape:
        N, modes = N * n, modes * (n // 2 + 1)
    nsym = d * (d + 1) // 2
    chi = torch.tensor(inputs.box_mask(shape, (3,) * d, tuple(n - 3 for n in shape[::-1])), device="cuda")
    plan = pd.Plan(pd.Problem(shape=shape, delta=2.5, model=pd.PD_NONLIN_BOND if nonlinear else pd.PD_LIN_BOND), chi)
    slots = 21 if nonlinear else 2 * d + nsym
    node = 4 * slots + 8 * (2 if d == 2 else 5) + 2 + d + 12 * nsym + 16 * d + 4 * nsym + 8 * d + 12
    rest = node * N + (12 * nsym + (48 if nonlinear else 0)) * modes
    rest += plan.boundary_nodes * (88 + 4 * nsym * d + (16 if nonlinear else 0))
    assert rest <= plan.workspace_bytes <= 1.02 * rest + (2 << 20)
    plan.close()
