"""Rank and unrank of long lists (tables in shared memory) against the general kernels.

A list that starts at an odd element of its storage takes the general kernels, so the same list at an
even and at an odd element must give the same words and indices, invalid entries (all ones, one error
each) among them. The sectors have one to four subsystems, digits of one to three bits, dimensions below
and above 2^32 and tables of up to 16 bits; a few entries are also compared with the host functions.
"""

import numpy as np
import pytest
import torch

from paper_2407_14591_gb300 import binding as b

pytestmark = pytest.mark.gpu
DEV = "cuda"
SECTORS = [
    (14, 2, 7, 1), (32, 2, 16, 2), (29, 2, 11, 3), (36, 2, 18, 3), (40, 2, 13, 4), (33, 2, 0, 3),
    (18, 4, 27, 3), (16, 3, 15, 2), (12, 5, 24, 3), (21, 7, 60, 5),
]


def _errors(s):
    with pytest.raises(b.DQError) as e:
        s.check_device()
    return str(e.value)


def _at(values, shift):
    store = torch.zeros(values.numel() + 2, dtype=torch.int64, device=DEV)
    v = store[shift:shift + values.numel()]
    v.copy_(values)
    return v


@pytest.mark.parametrize("L,Q,N,n_sub", SECTORS)
def test_long_lists_equal_the_general_kernels(L, Q, N, n_sub):
    s = b.make_sector(L, Q, N, n_sub)
    rng = np.random.default_rng(L * 100 + N)
    for n in (1 << 21, (1 << 21) + 1):
        idx = rng.integers(0, s.dim, n)
        idx[:4] = [0, s.dim - 1, s.dim // 2, 0]
        idx[n - 1] = s.dim - 1
        bad = rng.choice(np.arange(8, n - 1), 5, replace=False)
        idx[bad] = np.array([s.dim, s.dim + 1, 1 << 62, -1, s.dim])
        t = torch.from_numpy(idx)
        got = s.state_at_batch(_at(t, 0))
        found = _errors(s)
        store = torch.zeros(n + 2, dtype=torch.int64, device=DEV)
        ref = s.state_at_batch(_at(t, 1), out=store[1:n + 1])
        assert _errors(s) == found
        assert torch.equal(got, ref)
        for q in (0, 1, 2, n - 1):
            assert int(got[q].item()) == s.state_at(int(idx[q]))
        # words: valid ones, all ones (from the entries above), one digit too many and one bit beyond the top
        words = got.clone()
        words[5] += 1
        words[6] ^= 1
        words[7] |= 1 << 62
        back = s.index_of_batch(_at(words, 0))
        found = _errors(s)
        ref = s.index_of_batch(_at(words, 1), out=store[1:n + 1])
        assert torch.equal(back, ref)
        assert _errors(s) == found
        good = np.ones(n, bool)
        good[bad] = False
        good[5:8] = False
        assert np.array_equal(back.cpu().numpy()[good], idx[good])
