"""Performance cases of the sector library: what its users run, through the public entry points.

A case is a dict of plain values. ``listed()`` gives the standing ones, ``draw(rng)`` one more of
the same ranges. ``prepare`` builds what a user's program holds before the call (sector, compiled
operator, vectors on the GPU), ``run`` makes one call, ``work`` counts the bytes and operations a
pass cannot do without, and ``exact`` computes the same outputs in 64 bits with plain torch.

Operators: "lattice" is the spin-1/2 J1-J2 model on a periodic Lx x Ly square lattice (J1 = 1,
J2 = 0.5), "chain" the uniform periodic Heisenberg chain, "xxz" the periodic XXZ chain with a
random coupling per bond and a random field per site, "bose" the periodic Bose-Hubbard chain with
random on-site U. Vectors are U[-1, 1], normalised per column in 64 bits and then cast.
"""

import math
import random

import numpy as np
import torch

from paper_2407_14591_gb300 import autograd as ag
from paper_2407_14591_gb300 import binding as b
from paper_2407_14591_gb300 import workloads as wl

DTYPES = {"f64": torch.float64, "f32": torch.float32}


def listed():
    return [
        # a 16-site cluster: the smallest sector people diagonalise, where launches and latency count
        {"name": "cluster_4x4_f64", "kind": "product", "model": "lattice", "Lx": 4, "Ly": 4, "Q": 2, "N": 8,
         "n_sub": 2, "nrhs": 1, "dtype": "f64"},
        # the frustrated magnet at the size one GPU is bought for: one product of an FP64 iteration
        {"name": "j1j2_6x5_f64", "kind": "product", "model": "lattice", "Lx": 6, "Ly": 5, "Q": 2, "N": 15,
         "n_sub": 2, "nrhs": 1, "dtype": "f64"},
        # the same sector split into three, FP32 vectors (half the memory)
        {"name": "j1j2_6x5_nsub3_f32", "kind": "product", "model": "lattice", "Lx": 6, "Ly": 5, "Q": 2, "N": 15,
         "n_sub": 3, "nrhs": 1, "dtype": "f32"},
        # the same sector split into five (the smallest tables), FP64 vectors
        {"name": "j1j2_6x5_nsub5_f64", "kind": "product", "model": "lattice", "Lx": 6, "Ly": 5, "Q": 2, "N": 15,
         "n_sub": 5, "nrhs": 1, "dtype": "f64"},
        # a disordered chain (many-body localisation studies): a coefficient per bond and site
        {"name": "xxz_L24_f64", "kind": "product", "model": "xxz", "L": 24, "Q": 2, "N": 12, "n_sub": 2, "nrhs": 1,
         "dtype": "f64"},
        # a complex wavefunction of an odd chain, stored as two real columns (time evolution)
        {"name": "xxz_L23_complex_f64", "kind": "product", "model": "xxz", "L": 23, "Q": 2, "N": 11, "n_sub": 2,
         "nrhs": 2, "dtype": "f64"},
        # bosons with up to three particles per site, FP32 vectors
        {"name": "bose_Q4_L14_f32", "kind": "product", "model": "bose", "L": 14, "Q": 4, "N": 14, "n_sub": 2,
         "nrhs": 1, "dtype": "f32"},
        # a training step on the couplings and fields: product, its adjoint, and one gradient per coefficient
        {"name": "xxz_L24_grad_f64", "kind": "grad", "L": 24, "N": 12, "dtype": "f64"},
        # disorder averaging: many chains of uneven size, eight vectors each, in one launch
        {"name": "batch_64_chains_f64", "kind": "batch", "count": 64, "L_min": 16, "L_max": 26, "sizes": 4, "nrhs": 8,
         "dtype": "f64"},
        # basis functions in bulk (observables, embeddings): unrank 2^24 indices, rank the states again
        {"name": "rank_L32_16M", "kind": "rank", "L": 32, "Q": 2, "N": 16, "n_sub": 3, "count": 1 << 24},
        # a whole ground-state run on a small chain, with the Ritz vector
        {"name": "lanczos_chain_L20_f64", "kind": "lanczos", "model": "chain", "L": 20, "Q": 2, "N": 10, "n_sub": 2,
         "steps": 60, "dtype": "f64"},
        # a ground-state run on an odd cluster with FP32 vectors
        {"name": "lanczos_5x5_f32", "kind": "lanczos", "model": "lattice", "Lx": 5, "Ly": 5, "Q": 2, "N": 12,
         "n_sub": 2, "steps": 40, "dtype": "f32"},
    ]


def draw(rng):
    dtype = rng.choice(["f64", "f32"])
    kind = rng.choice(["product", "product", "product", "product", "grad", "batch", "rank", "lanczos"])
    if kind == "product":
        model = rng.choice(["lattice", "lattice", "chain", "xxz", "bose"])
        case = {"kind": kind, "model": model, "Q": 2, "nrhs": 1, "dtype": dtype}
        if model == "lattice":
            case["Lx"], case["Ly"] = rng.choice([(4, 4), (5, 4), (7, 3), (6, 4), (5, 5), (9, 3), (7, 4), (6, 5)])
        elif model == "chain":
            case["L"] = rng.randint(14, 28)
        elif model == "xxz":
            case["L"] = rng.randint(14, 26)
            case["nrhs"] = rng.choice([1, 1, 2, 3, 8])
        else:
            case["Q"] = rng.randint(3, 5)
            case["L"] = rng.randint(6, {3: 14, 4: 14, 5: 11}[case["Q"]])
        L = _sites(case)
        case["N"] = rng.randint(L // 2, L) if model == "bose" else rng.randint(L // 2 - 3, L // 2)
        case["n_sub"] = rng.choice([2, 2, 3, 5]) if model in ("lattice", "chain") else 2
        return case
    if kind == "grad":
        L = rng.randint(12, 24)
        return {"kind": kind, "L": L, "N": rng.randint(L // 2 - 3, L // 2), "dtype": dtype}
    if kind == "batch":
        low = rng.randint(12, 18)
        return {"kind": kind, "count": round(math.exp(rng.uniform(math.log(3), math.log(64)))), "L_min": low,
                "L_max": rng.randint(low + 2, 26), "sizes": rng.randrange(1 << 20), "nrhs": rng.choice([1, 2, 5, 8]),
                "dtype": dtype}
    if kind == "rank":
        Q = rng.choice([2, 2, 4])
        L = rng.randint(16, 36) if Q == 2 else rng.randint(8, 18)
        return {"kind": kind, "L": L, "Q": Q, "N": rng.randint(L // 4, (Q - 1) * L // 2), "n_sub": rng.randint(2, 4),
                "count": round(math.exp(rng.uniform(math.log(1 << 12), math.log(1 << 24))))}
    model = rng.choice(["chain", "lattice"])
    case = {"kind": kind, "model": model, "Q": 2, "n_sub": rng.choice([2, 3]), "steps": rng.randint(20, 40),
            "dtype": dtype}
    if model == "chain":
        case["L"] = rng.randint(16, 24)
    else:
        case["Lx"], case["Ly"] = rng.choice([(5, 4), (7, 3), (6, 4), (5, 5)])
    L = _sites(case)
    case["N"] = rng.randint(L // 2 - 2, L // 2)
    return case


def _sites(case):
    return case["L"] if "L" in case else case["Lx"] * case["Ly"]


def _terms(case, rng):
    """Term list of a case's operator; rng (numpy) draws the disorder."""
    model, L = case["model"], _sites(case)
    if model == "lattice":
        nn, nnn = wl.square_bonds(case["Lx"], case["Ly"])
        return wl.heisenberg_terms(nn, 1.0) + wl.heisenberg_terms(nnn, 0.5)
    bonds = wl.chain_bonds(L)
    if model == "chain":
        return wl.heisenberg_terms(bonds, 1.0)
    if model == "xxz":
        return wl.heisenberg_terms(bonds, rng.uniform(0.5, 1.5, L)) + wl.field_terms(rng.uniform(-3.0, 3.0, L))
    return [("HOP", i, j, 1.0) for i, j in bonds] + [("U", i, -1, float(u)) for i, u in enumerate(rng.uniform(2.0, 6.0, L))]


def _batch_sizes(case):
    r = random.Random(case["sizes"])
    out = []
    for _ in range(case["count"]):
        L = r.randint(case["L_min"], case["L_max"])
        out.append((L, r.randint(L // 2 - 3, L // 2)))
    return out


def _batch_terms(L, rng):
    """A uniform chain in random fields U[-5, 5]."""
    return wl.heisenberg_terms(wl.chain_bonds(L), 1.0) + wl.field_terms(rng.uniform(-5.0, 5.0, L))


def _grad_params(L):
    """theta = (couplings, fields): (kind, i, j, parameter, scale)."""
    out = []
    for k, (i, j) in enumerate(wl.chain_bonds(L)):
        out += [("XY", i, j, k, 1.0), ("ZZ", i, j, k, 1.0)]
    return out + [("Z", i, -1, L + i, 1.0) for i in range(L)]


def _theta(L, rng):
    return torch.from_numpy(np.concatenate([rng.uniform(0.5, 1.5, L), rng.uniform(-3.0, 3.0, L)]))


def _vector(gen, D, nrhs, dtype):
    x = torch.rand((D, nrhs), generator=gen, device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0)
    x /= torch.linalg.vector_norm(x, dim=0, keepdim=True)
    x = x.to(DTYPES[dtype])
    return x[:, 0].contiguous() if nrhs == 1 else x


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "batch":
        sizes = _batch_sizes(case)
        secs = [b.make_sector(L, 2, N, 0) for L, N in sizes]
        terms = [b.make_terms(s, _batch_terms(L, rng)) for s, (L, N) in zip(secs, sizes)]
        batch = b.make_batch(secs, terms, case["nrhs"], DTYPES[case["dtype"]])
        xs = [_vector(gen, s.dim, case["nrhs"], case["dtype"]) for s in secs]
        return {"kind": kind, "batch": batch, "xs": xs, "ys": [torch.empty_like(x) for x in xs]}
    if kind == "rank":
        s = b.make_sector(case["L"], case["Q"], case["N"], case["n_sub"])
        return {"kind": kind, "sector": s, "index": _indices(gen, s.dim, case["count"])}
    if kind == "grad":
        s = b.make_sector(case["L"], 2, case["N"], 2)
        op = ag.ParamOperator(s, _grad_params(case["L"]), n_params=2 * case["L"])
        theta = _theta(case["L"], rng).requires_grad_(True)
        x = _vector(gen, s.dim, 1, case["dtype"]).requires_grad_(True)
        return {"kind": kind, "op": op, "theta": theta, "x": x, "dy": _vector(gen, s.dim, 1, case["dtype"])}
    s = b.make_sector(_sites(case), case["Q"], case["N"], case["n_sub"])
    t = b.make_terms(s, _terms(case, rng))
    x = _vector(gen, s.dim, case.get("nrhs", 1), case["dtype"])
    state = {"kind": kind, "sector": s, "terms": t, "x": x}
    if kind == "lanczos":
        state["steps"] = case["steps"]
    else:
        state["y"] = torch.empty_like(x)
    return state


def _indices(gen, D, n):
    return (torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * D).long().clamp_(max=D - 1)


def run(state):
    kind = state["kind"]
    if kind == "product":
        return b.matvec(state["sector"], state["terms"], state["x"], state["y"])
    if kind == "batch":
        return state["batch"].matvec(state["xs"], state["ys"])
    if kind == "rank":
        states = state["sector"].state_at_batch(state["index"])
        return [states, state["sector"].index_of_batch(states)]
    if kind == "grad":
        y = ag.matvec(state["op"], state["x"], state["theta"])
        dx, dtheta = torch.autograd.grad(y, (state["x"], state["theta"]), state["dy"])
        return [y.detach(), dx, dtheta]
    r = b.lanczos(state["sector"], state["terms"], state["x"], state["steps"], want_vector=True)
    return [r["E0"], r["alpha"], r["beta"], r["psi"]]


# ---- work ---------------------------------------------------------------------------------------

def _dim(L, Q, N):
    """Number of digit strings of L digits below Q with digit sum N."""
    c = [1] + [0] * N
    for _ in range(L):
        c = [sum(c[n - d] for d in range(min(Q - 1, n) + 1)) for n in range(N + 1)]
    return c[N]


def _hops(case, L, Q, N):
    """Nonzero off-diagonal elements of H, all rows together (every bond of the model hops)."""
    bonds = {"lattice": 4 * L, "chain": L, "xxz": L, "bose": L}[case["model"]]
    if Q == 2:
        return bonds * 2 * _dim(L - 2, 2, N - 1)
    pairs = sum(_dim(L - 2, Q, N - nu - nd) for nu in range(Q - 1) for nd in range(1, Q) if N >= nu + nd)
    return bonds * 2 * pairs


def work(case):
    kind = case["kind"]
    es = 4 if case.get("dtype") == "f32" else 8
    if kind == "rank":  # indices in, states out, indices out
        return {"bytes": 24 * case["count"], "flops": 8 * case["n_sub"] * case["count"]}
    if kind == "batch":
        nr, by, fl = case["nrhs"], 0, 0
        for L, N in _batch_sizes(case):
            D = _dim(L, 2, N)
            by += 2 * D * nr * es
            fl += 2 * nr * (D + _hops({"model": "chain"}, L, 2, N))
        return {"bytes": by, "flops": fl}
    if kind == "grad":  # x, dy in; y, dx out; two products and a multiply-add per term and row
        L, N = case["L"], case["N"]
        D, h = _dim(L, 2, N), _hops({"model": "xxz"}, L, 2, N)
        return {"bytes": 4 * D * es, "flops": 4 * (D + h) + 2 * (h + 2 * L * D)}
    L, Q, N = _sites(case), case["Q"], case["N"]
    D, h = _dim(L, Q, N), _hops(case, L, Q, N)
    if kind == "product":
        return {"bytes": 2 * D * case["nrhs"] * es, "flops": 2 * case["nrhs"] * (D + h)}
    # Lanczos: start vector in, Ritz vector out; per step the product, the projection on the basis
    # so far and its update
    m = case["steps"]
    return {"bytes": 2 * D * es, "flops": m * 2 * (D + h) + 4 * D * (m * (m + 1) // 2)}


# ---- the same outputs in 64 bits with plain torch -------------------------------------------------

class _Exact:
    """A sector's basis in canonical order (sorted by particle number and pattern of each subsystem
    in turn) and the position of every state, by enumeration of all digit strings."""

    def __init__(self, L, Q, N, n_sub):
        self.L, self.Q, self.nb = L, Q, (Q - 1).bit_length()
        n_sub = n_sub or -(-self.nb * L // 16)
        bits, dm = self.nb * L, (1 << self.nb) - 1
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        found = []
        for lo in range(0, 1 << bits, 1 << 26):
            s = torch.arange(lo, min(lo + (1 << 26), 1 << bits), device=dev)
            n, ok = torch.zeros_like(s), torch.ones_like(s, dtype=torch.bool)
            for i in range(L):
                d = (s >> (self.nb * i)) & dm
                n += d
                if Q != dm + 1:
                    ok &= d < Q
            found.append(s[ok & (n == N)])
        s = torch.cat(found)
        key = torch.zeros_like(s)
        at = L
        for k in range(n_sub):
            length = L // n_sub + (1 if k < L % n_sub else 0)
            at -= length
            f = (s >> (self.nb * at)) & ((1 << (self.nb * length)) - 1)
            n = torch.zeros_like(s)
            for i in range(length):
                n += (f >> (self.nb * i)) & dm
            key = (((key << ((Q - 1) * length).bit_length()) | n) << (self.nb * length)) | f
        self.s = s[torch.argsort(key)]
        self.position = torch.zeros(1 << bits, dtype=torch.int32, device=dev)
        self.position[self.s] = torch.arange(len(s), dtype=torch.int32, device=dev)

    def digit(self, i):
        return (self.s >> (self.nb * (self.L - 1 - i))) & ((1 << self.nb) - 1)

    def rows(self, states):
        return self.position[states].long()

    def apply(self, kind, i, j, x):
        """T x for one term with coefficient 1; x is (D, nrhs) in 64 bits."""
        ni = self.digit(i)
        if kind == "Z":
            return (ni.double() - 0.5)[:, None] * x
        if kind == "U":
            return (0.5 * (ni * (ni - 1)).double())[:, None] * x
        nj = self.digit(j)
        if kind == "ZZ":
            return ((ni.double() - 0.5) * (nj.double() - 0.5))[:, None] * x
        bi, bj = 1 << (self.nb * (self.L - 1 - i)), 1 << (self.nb * (self.L - 1 - j))
        if kind == "XY":
            go = ni != nj
            to = self.rows(torch.where(go, self.s ^ (bi | bj), self.s))
            return torch.where(go, 0.5, 0.0).double()[:, None] * x[to]
        out = torch.zeros_like(x)  # HOP: -(b+_i b_j + b+_j b_i)
        for up, dn, nu, nd in ((bi, bj, ni, nj), (bj, bi, nj, ni)):
            go = (nu < self.Q - 1) & (nd > 0)
            to = self.rows(torch.where(go, self.s + up - dn, self.s))
            out -= (torch.sqrt(((nu + 1) * nd).double()) * go)[:, None] * x[to]
        return out

    def product(self, terms, x):
        y = torch.zeros_like(x)
        for kind, i, j, c in terms:
            y += c * self.apply(kind, i, j, x)
        return y


def _columns(x):
    x = x.detach().double()
    return x[:, None] if x.dim() == 1 else x


def _exact_lanczos(H, terms, v0, steps):
    """Lanczos with full re-orthogonalisation (two passes) and the Ritz vector of the lowest value."""
    v = _columns(v0)
    V = [v / torch.linalg.vector_norm(v)]
    alpha, beta = [], []
    for k in range(steps):
        w = H.product(terms, V[k])
        a = (V[k] * w).sum()
        w -= a * V[k]
        if k:
            w -= beta[-1] * V[k - 1]
        B = torch.cat(V, dim=1)
        for _ in range(2):
            w -= B @ (B.T @ w)
        alpha.append(a.item())
        beta.append(torch.linalg.vector_norm(w).item())
        V.append(w / beta[-1])
    T = torch.diag(torch.tensor(alpha, dtype=torch.float64))
    off = torch.tensor(beta[:-1], dtype=torch.float64)
    e, U = torch.linalg.eigh(T + torch.diag(off, 1) + torch.diag(off, -1))
    u = U[:, 0] * torch.sign(U[torch.argmax(U[:, 0].abs()), 0])
    psi = torch.cat(V[:steps], dim=1) @ u.to(v.device)
    return [e[0].item(), np.array(alpha), np.array(beta), psi]


def exact(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "rank":  # whole numbers, compared as they are
        return None
    if kind == "batch":
        sizes = _batch_sizes(case)
        if sum(_dim(L, 2, N) * L for L, N in sizes) * case["nrhs"] > 3e10:
            return None
        terms = [_batch_terms(L, rng) for L, N in sizes]
        xs = [_vector(gen, _dim(L, 2, N), case["nrhs"], case["dtype"]) for L, N in sizes]
        out = []
        for (L, N), t, x in zip(sizes, terms, xs):
            out.append(_Exact(L, 2, N, 0).product(t, _columns(x)).reshape(x.shape))
        return out
    if kind == "grad":
        L, N = case["L"], case["N"]
        theta = _theta(L, rng)
        H = _Exact(L, 2, N, 2)
        x = _vector(gen, len(H.s), 1, case["dtype"])
        dy = _vector(gen, len(H.s), 1, case["dtype"])
        params = _grad_params(L)
        terms = [(k, i, j, c * theta[p].item()) for k, i, j, p, c in params]
        g = torch.zeros(2 * L, dtype=torch.float64)
        for k, i, j, p, c in params:
            g[p] += c * (_columns(dy) * H.apply(k, i, j, _columns(x))).sum().item()
        return [H.product(terms, _columns(x))[:, 0], H.product(terms, _columns(dy))[:, 0], g]
    terms = _terms(case, rng)
    H = _Exact(_sites(case), case["Q"], case["N"], case["n_sub"])
    x = _vector(gen, len(H.s), case.get("nrhs", 1), case["dtype"])
    if kind == "lanczos":
        return _exact_lanczos(H, terms, x, case["steps"])
    return H.product(terms, _columns(x)).reshape(x.shape)
