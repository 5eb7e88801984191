"""Batched product on sectors long enough for a warp to take several chunks of rows.

A batch with few rows is cut into tiles of 32 rows per warp; these keep at least two chunks (of 256 rows)
per warp in the coarse shapes, so that the walk from row to row, every step of the ordering by hop count
and the second chunk run. The dimensions are no multiples of 32, and the last subsystems of three and four
sites make the walk start over every few rows. Every shape must give the bits of the first; that one is
compared with the single-sector products in exact fixed point: a row sums at most 64 products, each
rounded once, so 64 roundings of 2^-53 (2^-24 with compensated FP32 sums) of sum |H_ij||x_j| cover it."""

import pytest
import torch

from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
ITEMS = [(23, 11, 2), (24, 9, 7), (25, 10, 3), (23, 10, 6), (12, 6, 2)]


@pytest.fixture(scope="module")
def batch_items():
    out = []
    for k, (L, N, n_sub) in enumerate(ITEMS):
        s = b.make_sector(L, 2, N, n_sub)
        coef = 1.0 if k % 2 else [1.0 + 0.01 * i for i in range(L)]
        t = b.make_terms(s, wl.heisenberg_terms(wl.chain_bonds(L), coef) + wl.field_terms([0.3 * i - 2 for i in range(L)]))
        out.append((s, t))
    return out


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 5, 8])
def test_every_shape_on_long_sectors(batch_items, nrhs, dtype):
    secs, terms = [s for s, _ in batch_items], [t for _, t in batch_items]
    batch = b.make_batch(secs, terms, nrhs, dtype)
    g = torch.Generator(device="cuda").manual_seed(nrhs)
    xs = [(torch.rand((s.dim, nrhs), generator=g, device="cuda", dtype=torch.float64) * 2 - 1).to(dtype) for s in secs]
    ys = [torch.full_like(x, float("nan")) for x in xs]
    first = None
    for shape in range(batch.n_shapes()):
        batch.set_shape(shape)
        for y in ys:
            y.fill_(float("nan"))
        batch.matvec(xs, ys)
        if first is None:
            first = [y.clone() for y in ys]
        else:
            assert all(torch.equal(a, c) for a, c in zip(first, ys)), shape
    eps = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    for s, t, x, y in zip(secs, terms, xs, first):
        # |H| applied to |x| is below the row sum: L bonds of 5/4 L / 4 on the diagonal and 1/2 * 5/4 off it, fields
        bound = (s.L * 1.25 * 0.75 + s.L * 2.8) * 1.0
        tol = 64 * eps * bound
        for c in range(nrhs):
            ref = b.matvec(s, t, x[:, c].contiguous().double())
            assert float((y[:, c].double() - ref).abs().max()) <= tol
