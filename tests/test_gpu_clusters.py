"""Clusters of crowded cells: 1,024 atoms are the most that are packed in slabs, columns and runs; beyond, the Morton
order is ranked against tiles of 1,024 keys, four atoms to a thread.  All of a system's charges but eight lie in one
cell, at the edges of both.

Tolerance: the FP32 path's, 1e-5 rms relative in force and potential against the FP64 oracle (the inputs are the same
rounded rows on both sides, and differences of coordinates below 16 are exact to 2^-20 of the 0.3 Angstrom that the
closest charges are apart).
"""
import numpy as np
import pytest

import oracle as O
from paper_1911_01377_gb300 import build as B
from paper_1911_01377_gb300 import usr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crowd", [1016, 1024, 1025, 2047, 2049, 4608])
def test_crowded_cell(crowd):
    import torch
    from tests.golden import paper_tables
    B.build()
    rng = np.random.default_rng(crowd)
    m = int(np.ceil(crowd ** (1.0 / 3.0)))
    site = rng.permutation(m ** 3)[:crowd]
    ijk = np.stack([site % m, site // m % m, site // (m * m)], axis=1)
    xyz = 1.0 + (ijk + 0.5 + rng.uniform(-0.15, 0.15, (crowd, 3))) * (8.0 / m)
    xyz = np.concatenate([xyz, rng.uniform(12.0, 30.0, (8, 3))])
    q = rng.normal(0.0, 0.1, crowd + 8)
    rows = np.concatenate([xyz, (q - q.mean())[:, None]], axis=1).astype(np.float32)
    rows = rows[rng.permutation(crowd + 8)]
    box = (31.0, 31.0, 31.0)
    ctx = usr.USeries(box, (32, 32, 32), 9.0, "C1_B2", max_atoms=crowd + 8)
    out, _ = ctx.eval(torch.from_numpy(rows).cuda())
    again, _ = ctx.eval(torch.from_numpy(rows).cuda())
    assert torch.equal(out, again)
    out = out.cpu().numpy().astype(np.float64)
    ref = O.evaluate(O.Series(*paper_tables()["table2_C1"]), 9.0, box, rows[:, :3], rows[:, 3])
    assert O.rms_rel(out[:, :3], ref.F) < 1e-5
    assert O.rms_rel(out[:, 3], ref.phi) < 1e-5
