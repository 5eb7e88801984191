"""Which kernel a product runs, as the library reports it (decided on the host, no GPU needed)."""

import ctypes

import pytest
import torch

from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl


def chain(L):
    return wl.heisenberg_terms(wl.chain_bonds(L), 1.0) + wl.heisenberg_terms([(i, (i + 2) % L) for i in range(L)], 0.5)


def xxz(L):
    return wl.heisenberg_terms(wl.chain_bonds(L), [1.0 + 0.01 * i for i in range(L)])


def lattice(Lx, Ly):
    nn, nnn = wl.square_bonds(Lx, Ly)
    return wl.heisenberg_terms(nn, 1.0) + wl.heisenberg_terms(nnn, 0.5)


@pytest.mark.parametrize("L,N,n_sub,terms,path,kernel,two", [
    (16, 8, 2, chain(16), "panel_w", "panel_w", "general"),      # short sector: its own panels
    (22, 11, 2, chain(22), "panel", "panel_split", "general"),   # 11 -> 13 sites
    (22, 11, 5, chain(22), "panel", "panel_split", "general"),
    (30, 15, 2, lattice(6, 5), "panel", "panel", "general"),     # P_1 of 15 sites already
    (30, 15, 3, lattice(6, 5), "panel_w", "panel_split", "general"),
    (27, 13, 3, lattice(9, 3), "general", "panel_split", "general"),
    (24, 12, 2, xxz(24), "panel_pb", "panel_pb", "panel_pb"),
    (20, 10, 2, xxz(20), "panel_pb", "panel_pb", "general"),     # two columns of a short sector
    (24, 12, 3, xxz(24), "general", "general", "general"),
])
def test_kernel_of_a_product(L, N, n_sub, terms, path, kernel, two):
    t = b.make_terms(b.make_sector(L, 2, N, n_sub), terms)
    assert t.path == path
    for dtype in (torch.float64, torch.float32):
        assert t.kernel(dtype) == kernel
        assert t.kernel(dtype, 2) == two
        assert t.kernel(dtype, 64) == "general"


def test_cluster_terms_and_bad_arguments():
    s = b.make_sector(12, 2, 6, 2)
    t = b.make_cluster_terms(s, chain(12), 4)
    assert t.kernel(torch.float64) == t.kernel(torch.float32, 5) == "cluster"
    for nrhs in (0, 65):
        with pytest.raises(b.DQError) as e:
            t.kernel(torch.float64, nrhs)
        assert e.value.code == b.DQ_EINVAL
    assert b.lib().dq_matvec_kernel(None, b.DQ_F64, 1, ctypes.byref(ctypes.c_int())) == b.DQ_EINVAL
    assert b.lib().dq_matvec_kernel(t.handle, 7, 1, ctypes.byref(ctypes.c_int())) == b.DQ_EINVAL
    assert b.lib().dq_matvec_kernel(t.handle, b.DQ_F64, 1, None) == b.DQ_EINVAL


@pytest.mark.parametrize("L,N,n_sub,terms,kernel", [
    # the split order's panels are mostly short: 49, 60, 204, 257 and 269 rows on average
    (31, 6, 3, chain(31), "panel_w"),
    (30, 6, 3, chain(30), "panel_w"),
    (28, 7, 3, chain(28), "panel_w"),
    (30, 8, 3, chain(30), "panel_w"),
    (27, 7, 3, lattice(9, 3), "general"),
    # 362 and 438 rows
    (26, 7, 3, chain(26), "panel_split"),
    (28, 8, 3, chain(28), "panel_split"),
    # against a tail or two subsystems of fewer sites it wins at any length: 49 and 158 rows
    (31, 6, 5, chain(31), "panel_split"),
    (29, 7, 2, chain(29), "panel_split"),
])
def test_split_order_only_where_its_panels_are_long(L, N, n_sub, terms, kernel):
    s = b.make_sector(L, 2, N, n_sub)
    assert s.dim >= 1 << 19
    assert b.make_terms(s, terms).kernel(torch.float64) == kernel


@pytest.mark.parametrize("L,N,f64,f32", [
    # columns up to which a product of a disordered chain takes the per-bond panels
    (26, 7, 1, 1),    # 113 rows a panel on average
    (27, 8, 1, 1),    # 172
    (23, 9, 2, 2),    # 203
    (25, 9, 3, 2),    # 262
    (23, 10, 3, 2),   # 280
    (27, 9, 3, 2),    # 314, 4.7 M rows
    (23, 11, 3, 3),   # 330
    (25, 10, 4, 3),   # 404, 3.3 M rows
    (24, 10, 3, 3),   # 480, but 2.0 M rows
    (24, 12, 8, 3),   # 660
])
def test_columns_of_the_per_bond_panels(L, N, f64, f32):
    t = b.make_terms(b.make_sector(L, 2, N, 2), xxz(L))
    for dtype, most in ((torch.float64, f64), (torch.float32, f32)):
        got = [c for c in range(1, 65) if t.kernel(dtype, c) == "panel_pb"]
        assert got == list(range(1, most + 1)), dtype
