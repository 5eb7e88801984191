"""Panel products of operators with more than 127 hops of one amplitude in a row.

The hops of one amplitude are summed in 64-bit integers of up to 2^56 each, so 128 entries of x of one
sign next to a power of two would leave the range. XY bonds between the even and the odd sites make a
Neel row hop along every bond: with x = 1.9 everywhere y is 0.95 times the row's number of hops, one
rounding of an exact product, and every row must agree with the general kernel (two right-hand sides
take it), whose sums run over one bond distance at a time."""

import pytest
import torch

from paper_2407_14591_gb300 import binding as b

pytestmark = pytest.mark.gpu


def even_odd(L):
    return [(i, j) for i in range(L) for j in range(i + 1, L) if (j - i) % 2]


def without(bonds, keep_out, count):
    """The bonds less the first `count` of those that keep_out picks."""
    out = [p for p in bonds if keep_out(p)][:count]
    assert len(out) == count
    return [p for p in bonds if p not in out]


def ring(L):
    return sorted({(min(i, (i + d) % L), max(i, (i + d) % L)) for i in range(L) for d in (1, 3, 5, 7, 9)})


CASES = {
    # at most 64 bonds may cross 12 | 12: drop eight that lie inside the 15 lowest sites, whose split then
    # has 68 across the cut and does not fit, so the sector's own panels are used
    "own": (24, 12, 2, "panel", without(even_odd(24), lambda p: 9 <= p[0] < 12 <= p[1], 8)),
    # drop eight that cross 9 | 15 as well: the split into 9 and 15 sites fits
    "split_two": (24, 12, 2, "panel", without(even_odd(24), lambda p: p[0] < 9 and p[1] >= 12, 8)),
    # 64 inside the upper 16 sites, 16 inside the lower eight, 64 across
    "warp": (24, 12, 3, "panel_w", even_odd(24)),
    # the same on a sector that takes the split order
    "split_three": (24, 12, 3, "panel_w", without(even_odd(24), lambda p: p[0] < 9 <= p[1], 8)),
    "ring_two": (28, 14, 2, "panel", ring(28)),
    "ring_three": (28, 14, 3, "general", ring(28)),  # the sector's own form does not fit
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("case", CASES)
def test_every_bond_active(case, dtype):
    L, N, n_sub, path, bonds = CASES[case]
    assert len(bonds) > 127
    s = b.make_sector(L, 2, N, n_sub)
    t = b.make_terms(s, [("XY", i, j, 1.0) for i, j in bonds])
    assert t.path == path
    x = torch.full((s.dim,), 1.9, dtype=dtype, device="cuda")
    y = b.matvec(s, t, x)
    two = b.matvec(s, t, torch.stack([x, x], dim=1))[:, 0].contiguous()
    s.check_device()
    top = (0.5 * (x[:1].double() * len(bonds))).to(dtype)
    assert torch.equal(y.max(), top[0])
    assert torch.equal(y, two)


@pytest.mark.parametrize("case,other", [("own", 4), ("split_two", 7), ("warp", 10), ("split_three", 3)])
def test_two_amplitudes_and_both_signs(case, other):
    """A second amplitude on a few bonds, x of one sign on half of the rows and of both on the rest; the
    allocation-free call runs the same kernels."""
    L, N, n_sub, path, bonds = CASES[case]
    assert len(bonds) - other > 127
    s = b.make_sector(L, 2, N, n_sub)
    t = b.make_terms(s, [("XY", i, j, 1.0 if q >= other else -0.375) for q, (i, j) in enumerate(bonds)] +
                     [("ZZ", 0, 1, 0.25)])
    assert t.path == path
    g = torch.Generator(device="cuda").manual_seed(other)
    x = 1.98 + 0.02 * torch.rand(s.dim, generator=g, device="cuda", dtype=torch.float64)
    x[s.dim // 2:] *= torch.where(torch.rand(s.dim - s.dim // 2, generator=g, device="cuda") < 0.5, -1.0, 1.0)
    two = b.matvec(s, t, torch.stack([x, x], dim=1))[:, 0].contiguous()
    assert torch.equal(b.matvec(s, t, x), two)
    assert torch.equal(b.matvec_noalloc(s, t, x, torch.empty_like(x)), two)
    assert torch.equal(b.matvec(s, t, -x), -two)
    s.check_device()
