"""Charged atoms at the edges of the spreading kernel's bricks (16 x 8 x 8 grid points) and of the box: one float below
each box side and each brick face, on them, and one float to either side of the coordinates where a stencil begins and
ceases to reach a brick.  Far part against the FP64 oracle; no status bit.

Tolerances: the far-part tolerances of the spreading tests (potential and force, rms relative to the far part).
"""
import itertools

import numpy as np
import pytest

import oracle as O
from paper_1911_01377_gb300 import build as B
from paper_1911_01377_gb300 import usr
from paper_1911_01377_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {8: (2e-4, 2e-4), 10: (5e-5, 1e-4), 12: (2e-5, 1e-4), 16: (2e-5, 1e-4)}


def edge_rows(box, grid, points):
    """Atoms on a diagonal of edges: entry j of each axis's list of edge coordinates, with the lists turned against each
    other so that no two atoms are close."""
    f = np.float32
    H = points // 2
    lists = []
    for a, (L, n, brick) in enumerate(zip(box, grid, (16, 8, 8))):
        h = L / n
        at = [0.0, L, brick * h, 2 * brick * h, (brick - H) * h, (2 * brick + H - 1) % n * h]
        c = []
        for v in at:
            v = f(v)
            c += [np.nextafter(v, f(0)), v, np.nextafter(v, f(2 * L))]
        c = [v for v in c if 0 <= v <= f(L)]
        lists.append(c)
    m = max(len(c) for c in lists)
    rows = []
    for j, turn in itertools.product(range(m), (0, 5, 11)):
        p = [lists[a][(j + (a * turn)) % len(lists[a])] for a in range(3)]
        d = np.array(p, dtype=np.float64)
        if all(np.linalg.norm((d - q + np.array(box) / 2) % np.array(box) - np.array(box) / 2) > 1.0 for q in rows):
            rows.append(d)
    return np.array(rows, dtype=np.float32)


@pytest.mark.parametrize("box, grid, r_c, points, ratio, conv", [
    ((32.0, 32.0, 32.0), (32, 32, 32), 8.5, 12, 1.0, 0),
    ((47.9, 36.1, 52.7), (47, 35, 53), 8.5, 12, 1.0, 0),
    ((26.0, 26.0, 26.0), (24, 24, 24), 8.5, 16, 1.1, 0),
    ((32.0, 40.0, 48.0), (32, 40, 48), 8.5, 10, 0.9, 1),
    ((40.0, 32.0, 32.0), (40, 32, 32), 8.5, 8, 0.83, 2),
])
def test_atoms_on_edges(box, grid, r_c, points, ratio, conv):
    import torch
    from tests.golden import paper_tables
    B.build()
    xyz = edge_rows(box, grid, points)
    assert len(xyz) >= 8
    rng = np.random.default_rng(3)
    fill = W.random_neutral(4, 400, box, min_dist=1.3)[:, :3]
    d = fill[:, None, :].astype(np.float64) - xyz[None, :, :]
    d -= np.array(box) * np.round(d / np.array(box))
    fill = fill[(d * d).sum(axis=2).min(axis=1) > 1.0]
    xyz = np.concatenate([xyz, fill])
    q = rng.normal(0.0, 1.0, len(xyz))
    rows = np.concatenate([xyz, (q - q.mean())[:, None]], axis=1).astype(np.float32)
    ctx = usr.USeries(box, grid, r_c, "C1_B2", max_atoms=len(rows), conv=conv, spread_points=points,
                      spread_sigma_over_h=ratio)
    usr.usr_set_keep_parts(ctx.ctx, True)
    ctx.eval(torch.from_numpy(rows).cuda())
    _, far = ctx.parts(len(rows))
    far = far.cpu().numpy().astype(np.float64)
    assert usr.usr_last_device_status(ctx.ctx) == 0
    ref = O.evaluate(O.Series(*paper_tables()["table2_C1"]), r_c, box, rows[:, :3], rows[:, 3])
    tol_phi, tol_f = TOL[points]
    assert O.rms_rel(far[:, 3], ref.phi_far) < tol_phi
    assert O.rms_rel(far[:, :3], ref.F_far) < tol_f
