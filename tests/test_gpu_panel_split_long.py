"""The split order where the sector's own panels are shorter, two subsystems among them.

P_1 of the split order takes 13, 14 or 15 sites here against 11 to 14 of the sector's own form, across
the border of the last subsystem (pieces) or inside it. Both this kernel and the general ones (two
right-hand sides take them) sum in fixed point with the same scaling of x, and the coefficients lie on
both grids, so the rounded results must be equal.
"""

import pytest
import torch

from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def chain(L):
    return wl.heisenberg_terms(wl.chain_bonds(L), 1.0) + wl.heisenberg_terms([(i, (i + 2) % L) for i in range(L)], 0.5)


def lattice(Lx, Ly):
    nn, nnn = wl.square_bonds(Lx, Ly)
    return wl.heisenberg_terms(nn, 1.0) + wl.heisenberg_terms(nnn, 0.5)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("L,N,n_sub,terms", [
    (22, 11, 2, chain(22)),       # 11 -> 13 sites
    (23, 12, 2, chain(23)),       # 11 -> 14
    (24, 15, 2, lattice(6, 4)),   # 12 -> 15
    (25, 9, 2, lattice(5, 5)),
    (27, 13, 2, lattice(9, 3)),   # 13 -> 15
    (28, 7, 4, chain(28)),        # a tail of 14 sites -> 15
    (29, 7, 2, chain(29)),        # 14 -> 15
    (31, 6, 2, chain(31)),        # P_1 has 15 sites already: the own form
])
def test_longer_panels_equal_the_general_kernels(L, N, n_sub, terms, dtype):
    s = b.make_sector(L, 2, N, n_sub)
    assert s.dim >= 1 << 19
    t = b.make_terms(s, terms)
    assert t.path == "panel"
    g = torch.Generator(device="cuda").manual_seed(L)
    x = (torch.rand(s.dim, generator=g, device="cuda", dtype=torch.float64) - 0.5).to(dtype)
    x[::7] *= 2.0 ** -20
    y = b.matvec(s, t, x, torch.full_like(x, float("nan")))
    two = b.matvec(s, t, torch.stack([x, x], dim=1).contiguous())
    s.check_device()
    assert torch.equal(y, two[:, 0])
