"""Boson panel product: how a sector is cut into units does not show in y.

Single panels, panels in pairs (with an odd one out) and pieces of one, two and four 32-row chunks are
chosen by the sector's size; the sectors below meet each of them, with blocks of fewer than 32 rows and
blocks whose last chunk is short. Every row is one exact sum rounded once, so FP64 y equals the general
kernel's (which serves two right-hand sides) bit for bit.
"""

import numpy as np
import pytest
import torch

from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("L,Q,N", [(4, 3, 1), (6, 4, 3), (9, 4, 8), (13, 4, 7), (12, 4, 11), (13, 3, 13),
                                   (14, 3, 13), (13, 4, 12), (14, 4, 13)])
def test_units(L, Q, N):
    rng = np.random.default_rng(L * 100 + N)
    terms = [("HOP", int(i), int(j), float(c)) for (i, j), c in zip(wl.chain_bonds(L), rng.uniform(0.5, 1.5, L))]
    terms += [("U", i, -1, float(u)) for i, u in enumerate(rng.uniform(2.0, 6.0, L))]
    s = b.make_sector(L, Q, N, 2)
    t = b.make_terms(s, terms)
    assert t.path == "panel_q"
    x = torch.from_numpy(rng.uniform(-1, 1, s.dim)).to(DEV)
    y = b.matvec(s, t, x)
    both = b.matvec(s, t, torch.stack([x, x], 1).contiguous())
    assert torch.equal(y, both[:, 0])
    s.check_device()
