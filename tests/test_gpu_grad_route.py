"""Coefficient gradients on both sides of the rule that picks the pass over panels (four kernels) or the
general kernels (six or more: the columns of x and dy are scaled apart, each 32 terms take two launches).

Both round a row's product dy * x, or the sum of a few, to 2^-48 of the largest one over the columns, so
the two differ from the FP64 sums of single-term products by at most n 2^-47 max|dy| max|x| for a sum of n
products, and by about the square root of n of that in practice."""

import pytest
import torch

from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,cols,few,many", [
    # panels run with `few` terms (8), with all of them
    (26, 6, 1, True, True),      # one column: always
    (26, 6, 3, False, False),    # 56 rows a panel on average
    (20, 6, 4, True, True),      # little work: 3,392 panels over all columns
    (20, 6, 16, False, False),
    (20, 10, 8, True, True),     # 8,192 panels of 180 rows
    (20, 10, 16, False, False),
    (22, 11, 16, False, True),   # 344 rows: with many terms up to 16 columns
    (22, 11, 17, False, False),
    (24, 12, 4, True, True),     # 660 rows: four columns with any number of terms
    (24, 12, 5, False, True),
])
def test_route_and_values(L, N, cols, few, many):
    s = b.make_sector(L, 2, N, 2)
    terms = [t[:3] for t in wl.heisenberg_terms(wl.chain_bonds(L), 1.0) + wl.field_terms([1.0] * L)]
    g = torch.Generator(device="cuda").manual_seed(L + cols)
    shape = (s.dim, cols) if cols > 1 else (s.dim,)
    x = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 0.5
    dy = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 0.5
    bound = s.dim * cols * 2.0 ** -47 * float(x.abs().max() * dy.abs().max())
    for part, panels in ((terms[::len(terms) // 7][:8], few), (terms, many)):
        b.timing_enable(True)
        got = b.term_grads(s, part, x, dy)
        launched = b.timing_read()[2]
        b.timing_enable(False)
        assert launched == 4 if panels else launched >= 6
        for q in range(0, len(part), max(1, len(part) // 8)):
            k, i, j = part[q]
            t = b.make_terms(s, [(k, i, j, 1.0)])
            tx = b.matvec(s, t, x) if cols == 1 else torch.stack([b.matvec(s, t, c.contiguous()) for c in x.unbind(1)], 1)
            assert abs(float(got[q]) - float((dy * tx).sum())) <= bound, part[q]
    s.check_device()
