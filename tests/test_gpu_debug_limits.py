"""The bounds-checking debug build records an index beyond the sizes it was told and skips the access.  The sizes are
lowered below the buffers' own, so that every index stays inside the buffers whatever the checks do.

- max_groups = 1 of several: the pair kernel stops at the second group and the status says so.
- max_slots = 8: the spreading, the gather and the combination see the first cluster only; rows of other slots keep
  what the caller's buffer held.
"""
import os
import subprocess
import sys

import pytest

from paper_1911_01377_gb300 import build as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import torch
from paper_1911_01377_gb300 import usr, workloads as W
conv, grid, points, ratio, what = int(sys.argv[1]), int(sys.argv[2]), int(sys.argv[3]), float(sys.argv[4]), sys.argv[5]
x = torch.from_numpy(W.random_neutral(11, 600, (20.0, 20.0, 20.0), min_dist=1.0)).cuda()
ctx = usr.USeries((20.0, 20.0, 20.0), (grid,) * 3, 6.0, "C1_B2", max_atoms=600, conv=conv, spread_points=points,
                  spread_sigma_over_h=ratio)
n_slots, n_groups = (8, 1 << 30) if what == "slots" else (1 << 30, 1)
assert usr.lib().usr_debug_limit_bounds(ctx.ctx, n_slots, n_groups) == 0
out = torch.full((600, 4), -7.0, device="cuda")
usr.usr_eval(ctx.ctx, 600, x.data_ptr(), out.data_ptr(), None)
torch.cuda.synchronize()
st = usr.usr_last_device_status(ctx.ctx)
assert st == 8, f"status {st}"
kept = int((out == -7.0).all(dim=1).sum().item())
if what == "slots":
    assert 592 <= kept < 600, f"{kept} rows kept"
else:
    assert kept == 0, f"{kept} rows kept"
ctx.close()
print("DEBUG_LIMITS_OK")
"""


@pytest.mark.parametrize("what", ["slots", "groups"])
@pytest.mark.parametrize("conv, grid, points, ratio", [(0, 24, 8, 0.83), (1, 32, 12, 1.0)])
def test_lowered_limits_are_flagged(conv, grid, points, ratio, what):
    lib = B.build(debug_bounds=True)
    env = dict(os.environ, USR_LIBRARY=lib, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD, str(conv), str(grid), str(points), str(ratio), what], cwd=ROOT,
                       env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "DEBUG_LIMITS_OK" in r.stdout, r.stdout + r.stderr
