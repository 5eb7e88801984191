"""Coefficient gradients on panels (Q = 2, two subsystems) against single-term products.

d_grads[q] = <dy, T_q x>: the reference applies each term alone (dq_matvec) and sums dy * (T_q x) in
64 bits. A product dy * x is rounded to 2^-48 of the largest one (fewer bits only on sectors far beyond
these), so a sum of n products is off by at most n 2^-48 max|dy| max|x| (and FP64 rounding of the
reference, n 2^-53 of the same), and by about the square root of n of that in practice."""

import numpy as np
import pytest
import torch

from paper_2407_14591_gb300 import binding as b

pytestmark = pytest.mark.gpu
KINDS = ("XY", "ZZ", "Z", "HOP", "NN", "N", "U")


def all_places(L, L1, rng):
    """Every kind on pairs inside P_0, inside P_1 and across the cut (sites 0 .. L - L1 - 1 are P_0),
    each twice with the sites swapped, the single-site kinds on both sides."""
    L0 = L - L1
    pairs = []
    for lo, hi in ((0, L0), (L0, L)):
        if hi - lo >= 2:
            pairs += [tuple(int(v) for v in rng.choice(np.arange(lo, hi), 2, replace=False)) for _ in range(3)]
            pairs.append((lo, hi - 1))
    pairs += [(int(rng.integers(0, L0)), int(rng.integers(L0, L))) for _ in range(4)] + [(0, L - 1), (L0 - 1, L0)]
    terms = []
    for i, j in pairs:
        for k in ("XY", "ZZ", "HOP", "NN"):
            terms += [(k, i, j), (k, j, i)]
    for i in (0, L0 - 1, L0, L - 1):
        terms += [(k, i, -1) for k in ("Z", "N", "U")]
    return terms


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("L,N,cols", [(6, 3, 1), (9, 2, 2), (13, 6, 1), (14, 13, 1), (17, 8, 3), (20, 10, 1), (22, 3, 1),
                                      (26, 5, 1)])
def test_all_terms_against_single_products(L, N, cols, dtype):
    rng = np.random.default_rng(L * 100 + N)
    s = b.make_sector(L, 2, N, 2)
    shape = (s.dim, cols) if cols > 1 else (s.dim,)
    scale = 10.0 ** np.arange(cols) if cols > 1 else 1.0
    x = torch.from_numpy(rng.uniform(-1, 1, shape) * scale).to("cuda", dtype)
    dy = torch.from_numpy(rng.uniform(-1, 1, shape)).to("cuda", dtype)
    terms = all_places(L, s.partition[1], rng)
    g = b.term_grads(s, terms, x, dy).cpu().numpy()
    bound = s.dim * cols * 2.0 ** -47 * float(x.double().abs().max() * dy.double().abs().max())
    for q, (k, i, j) in enumerate(terms):
        tx = torch.stack([b.matvec(s, b.make_terms(s, [(k, i, j, 1.0)]), x[:, c].contiguous().double())
                          for c in range(cols)], dim=1) if cols > 1 else b.matvec(s, b.make_terms(s, [(k, i, j, 1.0)]), x.double())
        ref = float((dy.double() * tx).sum())
        assert abs(g[q] - ref) <= bound, (k, i, j, g[q], ref)


def test_same_result_every_time_and_many_terms():
    """Integer sums: repeated calls agree bit for bit; 200 terms take the same route as one."""
    rng = np.random.default_rng(1)
    s = b.make_sector(18, 2, 9, 2)
    x = torch.rand(s.dim, dtype=torch.float64, device="cuda") - 0.5
    dy = torch.rand(s.dim, dtype=torch.float64, device="cuda") - 0.5
    terms = [(KINDS[q % 6], int(q % 18), int((q * 5 + 1) % 18)) for q in range(200) if q % 18 != (q * 5 + 1) % 18]
    g = b.term_grads(s, terms, x, dy)
    assert torch.equal(g, b.term_grads(s, terms, x, dy))
    for q in (0, 7, len(terms) - 1):
        assert torch.equal(g[q:q + 1], b.term_grads(s, [terms[q]], x, dy))


def test_non_finite_input():
    s = b.make_sector(14, 2, 7, 2)
    x = torch.ones(s.dim, dtype=torch.float64, device="cuda")
    dy = torch.ones_like(x)
    dy[3] = float("nan")
    assert torch.isnan(b.term_grads(s, [("XY", 0, 1), ("Z", 3, -1)], x, dy)).all()
    with pytest.raises(b.DQError) as e:
        s.check_device()
    assert e.value.code == b.DQ_EDEVICE
