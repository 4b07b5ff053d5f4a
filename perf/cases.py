"""The calls that a user of this framework spends time in, over the sizes that they use.

A study of the random-field Heisenberg chain applies H to vectors, solves
shift-invert systems with MINRES (in 64 bits, in 32 bits, and in 32 bits with
64-bit refinement), finds the eigenpairs nearest an energy, sweeps over disorder
realisations, and takes twist overlaps and their derivatives from the eigenvectors.
Chains run from L = 8 (tests, scans of many realisations) to L = 28.

A case is a dict: "kind" says which call, "L" the chain length (dimension
n = C(L, L/2)), the rest the call's options. MINRES runs at long chains stop
after a fixed number of iterations: the system of a long chain takes 1e5 and
more of them, all alike, and after some fifty of them two orders of summation
no longer give the same iterate.
"""
import math

import numpy as np
import torch

from paper_2203_09732_gb300 import hs

SIGMA = 0.05      # an energy near the middle of the spectrum
FIELD = 3.7       # disorder strength: h_j uniform on [-FIELD, FIELD]

LISTED = [
    # one small product: a call's latency is all there is
    {"name": "product_l12_f64", "kind": "product", "L": 12, "dtype": "f64", "shifted": 1},
    # 64-bit products at a long chain: the extremal Lanczos run that finds sigma, residuals
    {"name": "product_l24_f64", "kind": "product", "L": 24, "dtype": "f64", "shifted": 0},
    # the longest chain: the product that every inner iteration does
    {"name": "product_l28_f32", "kind": "product", "L": 28, "dtype": "f32", "shifted": 1},
    # a whole shift-invert solve at the size of disorder studies (default tolerance)
    {"name": "solve_l16_f64", "kind": "solve", "L": 16, "precond": "row", "mixed": 0},
    # a whole solve in 32 bits with 64-bit refinement
    {"name": "solve_l14_mixed", "kind": "solve", "L": 14, "precond": "row", "mixed": 1},
    # iterations at the longest chain whose vectors stay on chip
    {"name": "iterate_l20_f64", "kind": "iterate", "L": 20, "dtype": "f64", "precond": "row", "iters": 45},
    # iterations at long chains: 64 bits, and the 32-bit inner solver at the longest
    {"name": "iterate_l24_f64", "kind": "iterate", "L": 24, "dtype": "f64", "precond": "row", "iters": 33},
    {"name": "iterate_l28_f32", "kind": "iterate", "L": 28, "dtype": "f32", "precond": "row", "iters": 24},
    # the eigenpairs of one realisation, from host fields to host vectors, with their twist overlaps
    {"name": "eigs_l12_k10", "kind": "eigs", "L": 12, "K": 10, "mixed": 0},
    # many realisations of two lengths in one call
    {"name": "sweep_l10_l12", "kind": "sweep", "La": 10, "Ba": 24, "Lb": 12, "Bb": 8, "K": 4},
    # twist overlaps of a set of eigenvectors of a long chain
    {"name": "twist_l24_k10", "kind": "twist", "L": 24, "K": 10},
    # the backward direction: derivatives of overlaps and energies by the fields
    {"name": "adjoint_l12_k3", "kind": "adjoint", "L": 12, "K": 3},
]


def listed():
    return [dict(c) for c in LISTED]


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in LISTED]
    while (case := _any(rng)) in known:
        pass
    return case


def _any(rng):
    kind = rng.choice(["product", "product", "solve", "iterate", "iterate", "iterate", "eigs", "sweep", "twist",
                       "adjoint"])
    pc = rng.choice(["row", "row", "id"])
    if kind == "product":
        dtype = rng.choice(["f32", "f64"])
        return {"kind": kind, "L": rng.randrange(8, 29 if dtype == "f32" else 27, 2), "dtype": dtype,
                "shifted": rng.randrange(2)}
    if kind == "solve":
        return {"kind": kind, "L": rng.randrange(8, 17 if pc == "row" else 15, 2), "precond": pc,
                "mixed": rng.randrange(2)}
    if kind == "iterate":
        dtype = rng.choice(["f32", "f64"])
        return {"kind": kind, "L": rng.randrange(14, 29 if dtype == "f32" else 27, 2), "dtype": dtype,
                "precond": pc, "iters": rng.randint(9, 24 if dtype == "f32" else 45)}
    if kind == "eigs":
        return {"kind": kind, "L": rng.choice([8, 10, 12]), "K": rng.randint(3, 10),
                "mixed": rng.randrange(2)}
    if kind == "sweep":
        La = rng.choice([8, 10])
        return {"kind": kind, "La": La, "Ba": rng.randint(5, 32), "Lb": rng.choice([La, 12]),
                "Bb": rng.randint(1, 8), "K": rng.randint(2, 5)}
    if kind == "twist":
        return {"kind": kind, "L": rng.randrange(12, 27, 2), "K": rng.randint(1, 12)}
    return {"kind": "adjoint", "L": rng.choice([8, 10, 12]), "K": rng.randint(1, 6)}


# ---------------------------------------------------------------------------
# inputs


def _dim(L):
    return math.comb(L, L // 2)


def _fields(L, seed):
    return np.random.default_rng([seed, L]).uniform(-FIELD, FIELD, L)


def _gaussian(n, seed, dtype=torch.float64, count=None):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (n,) if count is None else (count, n)
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _rhs(n, seed, dtype=torch.float64):
    b = _gaussian(n, seed)
    return (b / b.norm()).to(dtype)


def _sweep_fields(case, seed):
    """The lengths and fields of a sweep: strengths uniform on [0.5, 6]."""
    rng = np.random.default_rng([seed, 77])
    Ls = [case["La"]] * case["Ba"] + [case["Lb"]] * case["Bb"]
    return Ls, [rng.uniform(-1, 1, L) * rng.uniform(0.5, 6.0) for L in Ls]


def _wave_vectors(L, K, seed):
    """K vectors with the wide spread of amplitudes of localised eigenvectors."""
    g = _gaussian(_dim(L), seed, count=2 * K)
    psi = g[:K] * torch.exp(1.5 * g[K:])
    return (psi / psi.norm(dim=1, keepdim=True)).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        Ls, fields = _sweep_fields(case, seed)
        return {"kind": kind, "Ls": Ls, "fields": fields, "K": case["K"], "seed": seed}
    L = case["L"]
    n = _dim(L)
    h = _fields(L, seed)
    if kind == "eigs":
        return {"kind": kind, "L": L, "h": h, "K": case["K"], "mixed": bool(case["mixed"]), "seed": seed,
                "out": np.zeros((case["K"], n))}
    s = {"kind": kind, "chain": hs.Chain(L, h, sigma=SIGMA)}
    if kind == "product":
        s["x"] = _gaussian(n, seed, torch.float32 if case["dtype"] == "f32" else torch.float64)
        s["y"] = torch.empty_like(s["x"])
        s["shifted"] = bool(case["shifted"])
    elif kind == "solve":
        s.update(b=_rhs(n, seed), precond=case["precond"], mixed=bool(case["mixed"]))
        s["x"] = torch.empty_like(s["b"])
    elif kind == "iterate":
        s.update(b=_rhs(n, seed, torch.float32 if case["dtype"] == "f32" else torch.float64),
                 precond=case["precond"], iters=case["iters"])
        s["x"] = torch.empty_like(s["b"])
    elif kind == "twist":
        s["psi"] = _wave_vectors(L, case["K"], seed)
    else:
        w, psi = _eigenpairs(L, h, case["K"])
        s["psi"] = psi.T.contiguous().cuda()
        s["E"] = w.numpy()
    return s


def run(s):
    kind = s["kind"]
    if kind == "product":
        return s["chain"].matvec(s["x"], s["y"], shifted=s["shifted"])
    if kind == "solve":
        return s["chain"].minres(s["b"], s["x"], precond=s["precond"], mixed=s["mixed"])[0]
    if kind == "iterate":
        solve = s["chain"].minres_f32 if s["b"].dtype == torch.float32 else s["chain"].minres
        return solve(s["b"], s["x"], tol=0.0, kmax=s["iters"], precond=s["precond"],
                     allow_not_converged=True)[0]
    if kind == "eigs":
        ev, vec, res, z, info = hs.eigs_host(s["L"], s["h"], s["K"], tol=1e-12, seed=s["seed"],
                                             mixed=s["mixed"], out=s["out"])
        return ev, _signed(vec), z
    if kind == "sweep":
        ev, res, z, zz, info = hs.sweep(s["Ls"], s["fields"], s["K"], tol=1e-12, seed=s["seed"])
        return ev, z, zz
    if kind == "twist":
        return s["chain"].twist(s["psi"])
    z, dz2, dE, info = s["chain"].twist_grad(s["psi"], s["E"], tol=1e-12)
    return z, dz2, dE


def _signed(vec):
    """The vectors with their largest entry positive (an eigenvector's sign is free)."""
    top = np.abs(vec).argmax(axis=1)
    return vec * np.sign(vec[np.arange(len(vec)), top])[:, None]


def work(case):
    """Bytes that go in and come out, and the operations of the products that the
    call needs (per row: one addition per antiparallel bond, L/2 on average and a
    little more, the diagonal, and about 12 for a MINRES iteration's vectors)."""
    kind = case["kind"]
    if kind == "sweep":
        flops = 0.0
        for L, B in ((case["La"], case["Ba"]), (case["Lb"], case["Bb"])):
            flops += B * _dim(L) * (L / 2 + 15) * _solve_iters(L) * (3 * case["K"] + 15)
        return {"bytes": 8.0 * (case["Ba"] * (case["La"] + 4 * case["K"]) + case["Bb"] * (case["Lb"] + 4 * case["K"])),
                "flops": flops}
    L = case["L"]
    n = _dim(L)
    size = 4 if case.get("dtype") == "f32" else 8
    it = n * (L / 2 + 15.0)
    if kind == "product":
        return {"bytes": 2.0 * n * size, "flops": n * (L / 2 + 3.0)}
    if kind == "solve":
        return {"bytes": 16.0 * n, "flops": it * _solve_iters(L) * (2.8 if case["mixed"] else 1.0)}
    if kind == "iterate":
        return {"bytes": 2.0 * n * size, "flops": it * case["iters"]}
    if kind == "eigs":
        return {"bytes": 8.0 * n * case["K"], "flops": it * _solve_iters(L) * (3 * case["K"] + 15)}
    if kind == "twist":
        return {"bytes": 8.0 * n * case["K"], "flops": 2.0 * n * case["K"]}
    return {"bytes": 8.0 * n * case["K"], "flops": 2.0 * case["K"] * it * _solve_iters(L)}


def _solve_iters(L):
    """About how many iterations a whole 64-bit solve takes."""
    return 0.9 * _dim(L) ** 1.05


# ---------------------------------------------------------------------------
# the same in 64 bits, without the library


class _Plain:
    """H of Eq. (1) in the Sz = 0 sector from the definition: states in ascending
    order, bit j = site j + 1 up; a state's rank from two tables, of its high and
    of its low half."""

    def __init__(self, L, h, device):
        self.L, self.half = L, L // 2
        lo = np.arange(1 << self.half)
        hi = np.arange(1 << (L - self.half))
        pc = lambda a: np.array([bin(int(v)).count("1") for v in a])  # noqa: E731
        pl, ph = pc(lo), pc(hi)
        low_rank = np.zeros(len(lo), np.int64)
        by = {w: lo[pl == w] for w in range(self.half + 1)}
        for w, p in by.items():
            low_rank[p] = np.arange(len(p))
        first = np.zeros(len(hi), np.int64)
        parts, at = [], 0
        for H in hi:
            first[H] = at
            p = by.get(L // 2 - ph[H])
            if p is not None and len(p):
                parts.append((int(H) << self.half) | p)
                at += len(p)
        self.states = torch.from_numpy(np.concatenate(parts)).to(device)
        self.low_rank = torch.from_numpy(low_rank).to(device)
        self.first = torch.from_numpy(first).to(device)
        self.mask = (1 << self.half) - 1
        self.h = h
        self.n = len(self.states)
        self.bonds = [(1 << j) | (1 << ((j + 1) % L)) for j in range(L)]
        d = torch.zeros(self.n, dtype=torch.float64, device=device)
        self.anti = torch.zeros(self.n, dtype=torch.int64, device=device)
        for m in self.bonds:
            a = self._anti(m)
            self.anti += a
            d += torch.where(a, -0.25, 0.25)
        for j in range(L):
            d -= float(h[j]) * (((self.states >> j) & 1).to(torch.float64) - 0.5)
        self.diag = d

    def _anti(self, m):
        both = self.states & m
        return (both != 0) & (both != m)

    def rank(self, s):
        return self.first[s >> self.half] + self.low_rank[s & self.mask]

    def __call__(self, x, sigma=0.0):
        y = (self.diag - sigma) * x
        for m in self.bonds:
            a = self._anti(m)
            t = self.rank(torch.where(a, self.states ^ m, self.states))
            y += torch.where(a, 0.5 * x[t], 0.0)
        return y

    def dense(self):
        A = torch.diag(self.diag)
        rows = torch.arange(self.n, device=A.device)
        for m in self.bonds:
            a = self._anti(m)
            A[rows[a], self.rank(self.states[a] ^ m)] = 0.5
        return A

    def precond(self, kind, sigma):
        if kind == "id":
            return torch.ones_like(self.diag)
        return torch.sqrt((self.diag - sigma) ** 2 + 0.25 * self.anti)

    def twist_phases(self):
        t = torch.zeros(self.n, dtype=torch.float64, device=self.diag.device)
        for j in range(self.L):
            t += (j + 1) * (((self.states >> j) & 1).to(torch.float64) - 0.5)
        return torch.polar(torch.ones_like(t), 2 * math.pi / self.L * t)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _eigenpairs(L, h, K, sigma=SIGMA):
    """The K eigenpairs nearest sigma (None: the middle of the spectrum), by distance; columns."""
    w, V = torch.linalg.eigh(_Plain(L, h, "cpu").dense())
    if sigma is None:
        sigma = 0.5 * float(w[0] + w[-1])
    at = torch.argsort((w - sigma).abs(), stable=True)[:K]
    return w[at], V[:, at]


def _minres(A, M, b, iters, sigma):
    """x after `iters` steps of preconditioned MINRES (x_0 = 0)."""
    zero = torch.zeros_like(b)
    z, z_prev, d, d_prev, x = b.clone(), zero, zero, zero, zero.clone()
    beta_prev, beta = 1.0, float((b * b / M).sum().sqrt())
    c, s, dh, eps, phi = 1.0, 0.0, 0.0, 0.0, beta
    for _ in range(iters):
        q = z / M
        p = A(q, sigma)
        alpha = float((q * p).sum()) / beta**2
        z_next = p / beta - alpha / beta * z - beta / beta_prev * z_prev
        beta_next = float((z_next * z_next / M).sum().sqrt())
        delta, gh = c * dh + s * alpha, -s * dh + c * alpha
        eps_next, dh = s * beta_next, c * beta_next
        gamma = math.hypot(gh, beta_next)
        c, s = gh / gamma, beta_next / gamma
        d, d_prev = (q / beta - delta * d - eps * d_prev) / gamma, d
        x += c * phi * d
        phi, eps = -s * phi, eps_next
        z, z_prev, beta, beta_prev = z_next, z, beta_next, beta
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        Ls, fields = _sweep_fields(case, seed)
        ev, z, zz = [], [], []
        for L, h in zip(Ls, fields):
            w, V = _eigenpairs(L, h, case["K"], None)
            o = (_Plain(L, h, "cpu").twist_phases() @ (V * V).to(torch.complex128)).numpy()
            ev.append(w.numpy())
            z.append(o)
            zz.append((np.abs(o) ** 2).mean())
        return np.array(ev), np.array(z), np.array(zz)
    L = case["L"]
    n = _dim(L)
    h = _fields(L, seed)
    if kind == "eigs":
        w, V = _eigenpairs(L, h, case["K"], None)
        z = (_Plain(L, h, "cpu").twist_phases() @ (V * V).to(torch.complex128)).numpy()
        return w.numpy(), _signed(V.T.numpy().copy()), z
    if kind == "adjoint":
        P = _Plain(L, h, "cpu")
        w, V = torch.linalg.eigh(P.dense())
        at = torch.argsort((w - SIGMA).abs(), stable=True)[: case["K"]]
        u = P.twist_phases()
        sz = torch.stack([((P.states >> j) & 1).to(torch.float64) - 0.5 for j in range(L)])
        zs, dz2, dE = [], [], []
        for i in at.tolist():
            psi = V[:, i]
            z = (u * psi * psi).sum()
            g = w[i] - w
            g[i] = math.inf
            coef = (V.T @ (sz * psi).T) / g[:, None]          # <m|Sz_j|psi> / (E - E_m)
            dpsi = -(V @ coef)                                 # d psi / d h_j
            dz = 2 * ((u * psi)[:, None] * dpsi).sum(0)
            zs.append(complex(z))
            dz2.append((2 * (z.conj() * dz).real).numpy())
            dE.append(-(sz @ (psi * psi)).numpy())
        return np.array(zs), np.array(dz2), np.array(dE)
    P = _Plain(L, h, _device())
    if kind == "product":
        x = _gaussian(n, seed, torch.float32 if case["dtype"] == "f32" else torch.float64)
        return P(x.double(), SIGMA if case["shifted"] else 0.0)
    if kind == "solve":
        if L > 16:
            return None
        A = P.dense()
        A.diagonal().sub_(SIGMA)
        return torch.linalg.solve(A, _rhs(n, seed))
    if kind == "iterate":
        b = _rhs(n, seed, torch.float32 if case["dtype"] == "f32" else torch.float64).double()
        return _minres(P, P.precond(case["precond"], SIGMA), b, case["iters"], SIGMA)
    psi = _wave_vectors(L, case["K"], seed)
    u = P.twist_phases()
    return ((psi * psi).to(torch.complex128) @ u).cpu().numpy()
