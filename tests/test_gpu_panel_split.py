"""The panel product on the split order (three or more subsystems, at least 2^19 rows), against the
general kernels (two right-hand sides take them) on the same sector.

Both sum in fixed point with the same scaling of x, and the coefficients used here (1 and 1/2, halves
and quarters of them) lie exactly on both kernels' grids, so the rounded results must be equal."""

import pytest
import torch

from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def j1j2_chain(L):
    return wl.heisenberg_terms(wl.chain_bonds(L), 1.0) + wl.heisenberg_terms([(i, (i + 2) % L) for i in range(L)], 0.5)


def lattice(Lx, Ly):
    nn, nnn = wl.square_bonds(Lx, Ly)
    return wl.heisenberg_terms(nn, 1.0) + wl.heisenberg_terms(nnn, 0.5)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("L,N,n_sub,terms,path", [
    (22, 11, 5, j1j2_chain(22), "panel"),       # tail of 8 sites -> 11 sites
    (24, 8, 3, j1j2_chain(24), "panel_w"),      # warp panels; pieces of an 8-site subsystem
    (24, 8, 6, lattice(6, 4), "panel"),         # 12 sites = three whole subsystems, one piece
    (25, 8, 7, lattice(5, 5), "panel"),         # subsystems of 4 and 3 sites, eight pieces
    (27, 7, 3, lattice(9, 3), "general"),       # the sector's own form does not fit the operator
    (31, 6, 3, j1j2_chain(31), "panel_w"),      # 16 + 15 sites, the longest of both
])
def test_split_order_equals_the_general_kernels(L, N, n_sub, terms, path, dtype):
    s = b.make_sector(L, 2, N, n_sub)
    assert s.dim >= 1 << 19
    t = b.make_terms(s, terms)
    assert t.path == path
    g = torch.Generator(device="cuda").manual_seed(L)
    x = (torch.rand(s.dim, generator=g, device="cuda", dtype=torch.float64) - 0.5).to(dtype)
    x[::5] *= 2.0 ** -20
    y = b.matvec(s, t, x, torch.full_like(x, float("nan")))
    two = b.matvec(s, t, torch.stack([x, x], dim=1).contiguous())
    s.check_device()
    assert torch.equal(y, two[:, 0])


def test_split_order_reports_a_non_finite_vector():
    s = b.make_sector(24, 2, 8, 3)
    t = b.make_terms(s, j1j2_chain(24))
    x = torch.ones(s.dim, dtype=torch.float64, device="cuda")
    x[s.dim // 3] = float("inf")
    y = b.matvec(s, t, x)
    assert torch.isnan(y).all()
    with pytest.raises(b.DQError) as e:
        s.check_device()
    assert e.value.code == b.DQ_EDEVICE
