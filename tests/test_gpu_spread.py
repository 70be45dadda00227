"""The spreading kernel at the edges of its bricks (16 x 8 x 8 grid points) and lists: far part against the FP64
oracle.  Grids that are not multiples of the brick, stencils that reach a brick through two periodic images (n =
P + 8), each number of warps per brick, every stencil width, a net charge.

Tolerances: rms relative to the far part itself, potential 2e-5 and force 1e-4 for the 12- to 16-point stencils
(the far-part tolerances of the parity tests); 2e-4 for the 8-point one, whose cut-off leaves about 1.2e-4 of the
potential, and 5e-5 for the 10-point one (about 2e-5).
"""
import numpy as np
import pytest

import oracle as O
from paper_1911_01377_gb300 import build as B
from paper_1911_01377_gb300 import usr
from paper_1911_01377_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# box, grid, r_c, points, width / spacing, convolution, net charge per atom
CASES = {
    "two_images": ((26.0, 26.0, 26.0), (24, 24, 24), 8.5, 16, 1.1, 0, 0.0),
    "ragged_14": ((27.3, 31.7, 36.1), (25, 31, 37), 8.5, 14, 1.05, 0, 0.01),
    "one_point_over": ((25.5, 33.0, 41.0), (33, 25, 41), 8.2, 12, 1.0, 0, 0.0),
    "bf16_8": ((40.0, 32.0, 24.0), (40, 32, 24), 7.8, 8, 0.83, 2, 0.0),
    "four_warps": ((64.0, 64.0, 80.0), (64, 64, 80), 9.0, 12, 1.0, 0, 0.0),
    "two_warps": ((96.0, 80.0, 80.0), (96, 80, 80), 9.0, 10, 0.9, 1, 0.0),
    "one_warp": ((128.0, 128.0, 64.0), (128, 128, 64), 9.0, 12, 1.0, 1, 0.0),
}
TOL = {8: (2e-4, 2e-4), 10: (5e-5, 1e-4), 12: (2e-5, 1e-4), 14: (2e-5, 1e-4), 16: (2e-5, 1e-4)}


@pytest.mark.parametrize("name", sorted(CASES))
def test_far_part_at_brick_edges(name):
    import torch
    from tests.golden import paper_tables
    B.build()
    box, grid, r_c, points, ratio, conv, extra = CASES[name]
    xyzq = W.random_neutral(5, 1200, box, min_dist=1.3)
    xyzq[:, 3] += np.float32(extra)
    # atoms on the box faces, on a brick's face and just below it
    h = np.array(box) / np.array(grid)
    xyzq[0, :3] = box
    xyzq[1, :3] = 0.0
    xyzq[2, :3] = (np.array([16, 8, 8]) * h).astype(np.float32)
    xyzq[3, :3] = np.nextafter(xyzq[2, :3] + np.float32(2 * h), np.float32(0))
    xyzq[0, 3] = 0.0                                            # rows 0 and 1 are one point
    ctx = usr.USeries(box, grid, r_c, "C1_B2", max_atoms=1200, conv=conv, spread_points=points,
                      spread_sigma_over_h=ratio)
    usr.usr_set_keep_parts(ctx.ctx, True)
    ctx.eval(torch.from_numpy(xyzq).cuda())
    _, far = ctx.parts(1200)
    far = far.cpu().numpy().astype(np.float64)
    ref = O.evaluate(O.Series(*paper_tables()["table2_C1"]), r_c, box, xyzq[:, :3], xyzq[:, 3])
    tol_phi, tol_f = TOL[points]
    assert O.rms_rel(far[:, 3], ref.phi_far) < tol_phi
    assert O.rms_rel(far[:, :3], ref.F_far) < tol_f
