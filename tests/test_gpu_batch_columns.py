"""Batched product: every number of columns, with vectors at any element of their storage.

The columns of a row are shared out over lanes by 4, 8 or 16-byte loads, whichever divides the row
and fits the vectors' alignment. Sectors of one row, of fewer rows than a warp and of one to four
subsystems go through both row mappings, and nothing outside y may be written. Bounds: a row sums at
most 40 products, so 64 roundings of 2^-53 (2^-24 with compensated FP32 sums, products rounded once)
of sum |H_ij||x_j| cover it.
"""

import numpy as np
import pytest
import torch

from oracle import OracleSector, matvec as o_matvec
from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"
PAD = 8


def _items():
    rng = np.random.default_rng(7)
    out = []
    for L, N, n_sub in [(6, 0, 2), (7, 1, 1), (9, 4, 2), (12, 6, 2), (13, 6, 3), (14, 5, 4)]:
        coef = rng.uniform(0.5, 1.5, L) if L % 2 else 1.0
        out.append((L, N, n_sub, wl.heisenberg_terms(wl.chain_bonds(L), coef) + wl.field_terms(rng.uniform(-5, 5, L))))
    return out


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("nrhs", range(1, 9))
def test_columns_and_alignment(nrhs, dtype):
    items = _items()
    secs = [b.make_sector(L, 2, N, n_sub) for L, N, n_sub, _ in items]
    terms = [b.make_terms(s, t) for s, (_, _, _, t) in zip(secs, items)]
    oracles = [OracleSector(L, 2, N, partition=s.partition) for s, (L, N, _, _) in zip(secs, items)]
    rng = np.random.default_rng(nrhs)
    batch = b.make_batch(secs, terms, nrhs, dtype)
    eps = 2.0**-53 if dtype == torch.float64 else 2.0**-24
    for shift in (0, 1, 2):
        xs, ys, bufs, refs, tols = [], [], [], [], []
        for s, o, (_, _, _, t) in zip(secs, oracles, items):
            n = s.dim * nrhs
            store = torch.zeros(n + PAD, device=DEV, dtype=dtype)
            x = store[shift:shift + n].view(s.dim, nrhs)
            x.copy_(torch.from_numpy(rng.uniform(-1, 1, (s.dim, nrhs))))
            buf = torch.full((n + PAD,), 7.0, device=DEV, dtype=dtype)
            bufs.append(buf)
            xs.append(x)
            ys.append(buf[shift:shift + n].view(s.dim, nrhs))
            xd = x.double().cpu().numpy()
            refs.append(o_matvec(o, t, xd))
            tols.append(64 * eps * 40 * 6.0 * np.max(np.abs(xd)))  # |H_ij| <= 5 L / 2 + L / 4 on the diagonal
        for shape in (1, 7):  # rows, walk
            batch.set_shape(shape)
            for buf in bufs:
                buf.fill_(7.0)
            batch.matvec(xs, ys)
            torch.cuda.synchronize()
            for buf, y, ref, tol in zip(bufs, ys, refs, tols):
                assert np.max(np.abs(y.double().cpu().numpy() - ref)) <= tol
                edge = torch.cat([buf[:shift], buf[shift + y.numel():]])
                assert torch.all(edge == 7.0)
