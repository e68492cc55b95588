"""The tuning record after an autotuner: the tile shapes that the plan's force passes run
with, whatever was stored before.

Columns: 2D passes take 32 bytes of a row (2 complex values in FP64, 4 in FP32), 3D
passes of these lengths 128 bytes; there is no x2 pass in 2D. Rows: as many as a warp
transforms at once (H = n1/2 packed values on H/16 lanes, on H/8 in FP64 and up to 512
nodes in 2D, at most 32; two warps a row from H = 1024)."""
import numpy as np
import pytest
import torch

from paper_2105_06055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pdm():
    from paper_2105_06055_gb300 import build, pd
    build.build()
    pd.load()
    return pd


def _plan(pdm, shape, fp64, **kw):
    chi = inputs.box_mask(shape, (4,) * len(shape), tuple(n - 4 for n in shape[::-1]))
    return pdm.Plan(pdm.Problem(shape=shape, delta=2.5, fp64=fp64, **kw), torch.tensor(chi, device="cuda"))


@pytest.mark.parametrize("shape,fp64,rows,w2,wl", [
    ((128, 128), True, 4, 0, 2), ((512, 256), False, 2, 0, 4), ((64, 64, 64), False, 16, 16, 16),
    ((32, 32, 64), True, 8, 8, 8), ((16, 16, 128), False, 8, 16, 16)])
def test_autotune_records_the_shapes_that_run(pdm, shape, fp64, rows, w2, wl):
    plan = _plan(pdm, shape, fp64)
    assert not any(plan.tuning.values())
    want = {"rows": rows, "w_x2": w2, "w_last": wl, "sched": 0, "stages": 1, "stages_inv": 1}
    plan.set_tuning(32, 32, 32, 1, 2, 2)
    assert plan.autotune() == want
    plan.set_tuning(32, 32, 32, 1, 2, 2)
    assert plan.autotune(solve=True) == want
    plan.close()


def test_batch_autotune_records_each_plan(pdm):
    shapes = [(64, 64), (128, 128)]
    chis = [inputs.box_mask(s, (4, 4), (s[1] - 4, s[0] - 4)) for s in shapes]
    batch = pdm.Batch([pdm.Problem(shape=s, delta=2.5) for s in shapes],
                      [torch.tensor(np.ascontiguousarray(c), device="cuda") for c in chis])
    assert [(t["rows"], t["w_x2"], t["w_last"]) for t in batch.autotune()] == [(8, 0, 4), (4, 0, 4)]
    batch.close()
