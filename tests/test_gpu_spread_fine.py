"""Spreading with 12 points and more in the TF32x3 form: a neutral drop of water in vacuum, as for the FP32 form.

Tolerance: the grid method itself (stencil cut-off, aliasing), evaluated in 64 bits, is off by 1.0e-6 of the far
potential's norm here; three times that leaves rounding twice the method's error.  (Brick sums that the tensor cores
truncate: 5e-6.)
"""
import numpy as np
import pytest

import oracle as O
from paper_1911_01377_gb300 import build as B
from paper_1911_01377_gb300 import usr
from paper_1911_01377_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points, ratio, r_c, multilevel", [(12, 1.0, 9.0, 0), (12, 1.0, 9.0, 1), (16, 1.1, 8.5, 0)])
def test_drop_in_vacuum(points, ratio, r_c, multilevel):
    import torch
    from tests.golden import paper_tables
    B.build()
    box, n = (90.0, 90.0, 90.0), 6000
    _, rows = W.lattice_water_box(31, n, 0.1)
    rows[:, :3] += np.float32(20.0)
    ref = O.evaluate(O.Series(*paper_tables()["table2_C1"]), r_c, box, rows[:, :3], rows[:, 3])
    ctx = usr.USeries(box, (88, 88, 88), r_c, "C1_B2", max_atoms=n, conv=1, spread_points=points,
                      spread_sigma_over_h=ratio, multilevel=multilevel)
    usr.usr_set_keep_parts(ctx.ctx, True)
    ctx.eval(torch.from_numpy(rows).cuda())
    _, far = ctx.parts(n)
    assert usr.usr_last_device_status(ctx.ctx) == 0
    assert O.rms_rel(far.cpu().numpy().astype(np.float64)[:, 3], ref.phi_far) < 3e-6
