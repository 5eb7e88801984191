"""Coefficient gradients keep their grid for any number of columns and any size of sector.

A product dy * x is rounded to units of 2^(lg cols - 48) of a power of two above the largest one. Here
the largest product is 1 (bounded by 4 in the scaling), every other entry is a small power of two, and
each product dy_i x_j is a whole number of those units: nothing may be rounded away, and the sums have
fewer than 53 bits, so the gradient equals the reference sum in 64 bits exactly."""

import math

import pytest
import torch

from paper_2407_14591_gb300 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,cols", [(20, 10, 64), (24, 12, 3), (24, 12, 64), (26, 13, 8), (27, 13, 1)])
def test_no_product_is_rounded_away(L, N, cols):
    s = b.make_sector(L, 2, N, 2)
    L1 = s.partition[1]
    assert L1 <= 13
    lg = math.ceil(math.log2(cols))
    e = 46 - lg  # the unit is 4 * 2^(lg - 48)
    ex = e // 2
    shape = (s.dim, cols) if cols > 1 else (s.dim,)
    x = torch.full(shape, 2.0 ** -ex, dtype=torch.float64, device="cuda")
    dy = torch.full(shape, 2.0 ** (ex - e), dtype=torch.float64, device="cuda")
    row = s.dim // 2
    x[row] = 1.0
    dy[row] = 1.0
    u = L - L1  # first site of P_1
    places = [(0, 1), (0, u - 1), (u, u + 1), (u, L - 1), (u - 1, u), (0, L - 1), (1, L - 2)]
    terms = [(k, i, j) for i, j in places for k in ("XY", "ZZ", "HOP", "NN")]
    terms += [(k, i, -1) for i in (0, u - 1, u, L - 1) for k in ("Z", "N")]
    g = b.term_grads(s, terms, x, dy).cpu()
    # the columns are equal, so one product stands for all of them
    x1, dy1 = (x[:, 0].contiguous(), dy[:, 0].contiguous()) if cols > 1 else (x, dy)
    for q, (k, i, j) in enumerate(terms):
        t = b.make_terms(s, [(k, i, j, 1.0)])
        assert float(g[q]) == cols * float((dy1 * b.matvec(s, t, x1)).sum()), (k, i, j)
    s.check_device()
