"""Systems with a net charge (all charges of one sign) in the tensor-core forms: the k = 0 mode of rho, which Eq. 4
drops, is then as large as rho itself, and must neither be left in nor cost the operand splits their digits.

Far part against the FP64 oracle, rms relative to the far part itself.  Tolerances: TF32x3 at 12 points 2e-6 in the
potential and 5e-6 in the force, within a factor of four of the FP32 form's errors on such systems (5e-7, 1.5e-6) as
its operands keep two binary digits less (with the mean left in the operands the potential was off by 2.8e-6 to 1.1e-5,
multilevel 9.8e-7 to 1.8e-6); BF16x3, whose operands keep 16 digits (1.5e-5), 5e-5 and 2e-4.
"""
import numpy as np
import pytest

import oracle as O
from paper_1911_01377_gb300 import build as B
from paper_1911_01377_gb300 import usr
from paper_1911_01377_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BOX, GRID, N = (60.0, 40.0, 40.0), (64, 40, 40), 5000
TOL = {1: (2e-6, 5e-6), 2: (5e-5, 2e-4)}


def rows_of(kind):
    rows = W.random_neutral(9, N, BOX, min_dist=1.2)
    if kind == "unit":
        rows[:, 3] = 1.0
    elif kind == "spread":
        rows[:, 3] = 0.5 + 0.5 * np.abs(rows[:, 3])
    elif kind == "large":          # a few charges far above the others
        rows[:, 3] = np.where(np.arange(N) % 16 == 0, 400.0, 0.5)
    else:                          # charges in a far larger unit
        rows[:, 3] = -1e-9
    return rows


@pytest.mark.parametrize("kind", ["unit", "spread", "large", "tiny"])
@pytest.mark.parametrize("conv, multilevel", [(1, 0), (2, 0), (1, 1), (2, 1)])
def test_far_part_with_net_charge(kind, conv, multilevel):
    import torch
    from tests.golden import paper_tables
    B.build()
    rows = rows_of(kind)
    ref = O.evaluate(O.Series(*paper_tables()["table2_C1"]), 8.5, BOX, rows[:, :3], rows[:, 3])
    ctx = usr.USeries(BOX, GRID, 8.5, "C1_B2", max_atoms=N, conv=conv, spread_points=12, spread_sigma_over_h=1.0,
                      multilevel=multilevel)
    usr.usr_set_keep_parts(ctx.ctx, True)
    x = torch.from_numpy(rows).cuda()
    out, _ = ctx.eval(x)
    _, far = ctx.parts(N)
    far = far.cpu().numpy().astype(np.float64)
    assert usr.usr_last_device_status(ctx.ctx) == 0
    tol_phi, tol_f = TOL[conv]
    assert O.rms_rel(far[:, 3], ref.phi_far) < tol_phi
    assert O.rms_rel(far[:, :3], ref.F_far) < tol_f
    again, _ = ctx.eval(x)         # the charges' sum starts from zero in each evaluation
    assert torch.equal(out, again)
