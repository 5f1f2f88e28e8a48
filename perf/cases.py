"""Performance cases: the work that a program using this library has it do, through its public entry points.

A case is a dict of plain values.  Common keys: ``kind`` (which entry points), ``geom`` with its sizes (which
spin system), ``dtype`` ("c64" or "c128"), ``R`` vectors and, for Lanczos runs, ``M`` steps.  Systems follow the
library's benchmark workloads (rings, open lattices, ladders, chains, the centred cube of spins 5/2 and 2) with
couplings and fields drawn from the seed.  Runs are cut to M steps over which rounding has not yet been amplified
by the loss of orthogonality, so that the coefficients of two correct programs can be compared; a step costs the
same at any M.

Complex64 runs return their numbers as float32: the library hands them out in doubles, but they come from
single-precision vectors.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_25585_gb300 as F

TEMPERATURES = 50.0 ** (np.arange(40) / 39.0)   # 40 log-spaced points, 1 .. 50 K: what a few steps resolve
MU_B, C_DIP, G = 0.6717, 0.6228, 2.0            # K/T, K A^3, g factor


def listed():
    return [
        # the smallest run: a spin-1 ring of 729 states in double precision (latency: every kernel is tiny)
        dict(name="run ring6 s1 c128", kind="run", geom="ring", n=6, two_s=2, dtype="c128", R=10, M=24, start="random"),
        # plain FTLM in double precision on a middle-sized spin-1/2 lattice
        dict(name="run lattice4x4 c128", kind="run", geom="lattice", lx=4, ly=4, two_s=1, dtype="c128", R=50, M=16,
             start="random"),
        # the benchmark's headline: 64 vectors of the 4x5 spin-1/2 lattice in single precision
        dict(name="run lattice4x5 c64", kind="run", geom="lattice", lx=4, ly=5, two_s=1, dtype="c64", R=64, M=12,
             start="random"),
        # the largest single system: the 2x13 spin-1/2 ladder, 67 million states
        dict(name="run ladder2x13 c64", kind="run", geom="lattice", lx=13, ly=2, two_s=1, dtype="c64", R=4, M=5,
             start="random"),
        # many uneven systems at once: spin-1 chains of 10 to 12 sites, each in 8 field directions
        dict(name="batch chains s1 c64", kind="batch", geom="chain", n=10, n_last=12, two_s=2, fields=8, dtype="c64",
             R=16, M=8, start="random"),
        # powder average of the centred-cube molecule from pairs of time-reversed vectors
        dict(name="batch cube9 c64", kind="batch", geom="cube", n=9, two_s=4, fields=10, dtype="c64", R=8, M=6,
             start="pairs"),
        # the symmetric estimator of the same molecule (stored Lanczos vectors and their overlaps)
        dict(name="sym cube9 c64", kind="sym", geom="cube", n=9, two_s=4, dtype="c64", R=8, M=12, start="random"),
        # one product H x on a caller's block: a program with its own eigensolver, 64 vectors
        dict(name="apply lattice4x5 c64", kind="apply", geom="lattice", lx=4, ly=5, two_s=1, dtype="c64", R=64),
        # the same for one vector in double precision
        dict(name="apply lattice4x5 c128", kind="apply", geom="lattice", lx=4, ly=5, two_s=1, dtype="c128", R=1),
        # H x on a row-major block of a spin-1 chain
        dict(name="apply chain12 s1 c64", kind="apply", geom="chain", n=12, two_s=2, dtype="c64", R=16),
        # the smallest call: H x of a small mixed-spin molecule, odd sizes
        dict(name="apply mixed5 c128", kind="apply", geom="mixed", n=5, two_s=3, dtype="c128", R=3),
        # start vectors and the observable's first product for a caller's own recurrence
        dict(name="start lattice4x5 c64", kind="start", geom="lattice", lx=4, ly=5, two_s=1, dtype="c64", R=32),
    ]


def _steps(case):
    """state-vectors that a pass applies H (or u.S) to"""
    d = sum(math.prod(t + 1 for t in s["two_s"]) for s in _systems(case, 0, sizes_only=True))
    return d * case["R"] * case.get("M", 1)


def draw(rng):
    """One more case of the listed ranges: any kind, geometry, precision and size, odd ones among them."""
    while True:
        kind = rng.choice(["run", "run", "run", "run", "batch", "sym", "apply", "apply", "apply", "start"])
        geom = rng.choice(["ring", "lattice", "lattice", "lattice", "chain", "cube", "mixed"])
        c = dict(kind=kind, geom=geom, dtype=rng.choice(["c64", "c64", "c128"]))
        if geom == "lattice":
            c.update(lx=rng.randint(2, 13), ly=rng.randint(2, 5), two_s=1, buckle=rng.choice([0.0, 0.0, 0.0, 0.5]))
        elif geom == "cube":
            c.update(n=rng.randint(4, 9), two_s=rng.choice([3, 4]))
        elif geom == "mixed":
            c.update(n=rng.randint(3, 11), two_s=rng.randint(2, 5))
        else:
            c.update(n=rng.randint(4, 22), two_s=rng.choice([1, 2, 2, 3]))
        c["R"] = int(round(math.exp(rng.uniform(0, math.log(64)))))
        if kind in ("run", "batch", "sym"):
            c["M"] = rng.randint(4, 24 if c["dtype"] == "c128" else 12)
            c["start"] = rng.choice(["random", "random", "pairs"])
        if kind == "batch":
            if geom not in ("chain", "cube", "ring"):
                continue
            c["fields"] = rng.randint(2, 10)
            c["n_last"] = c["n"] + (rng.randint(0, 2) if geom != "cube" else 0)
        if geom == "lattice" and c["lx"] * c["ly"] > 24:
            continue
        d = max(math.prod(t + 1.0 for t in s["two_s"]) for s in _systems(c, 0, sizes_only=True))
        low = 2.0 ** rng.uniform(6, 24)             # spread the dimensions over their logarithm
        if not low / 4 <= d <= low * 4 or d > 1.7e7:
            continue
        cost = float(_steps(c)) * (25 if c["dtype"] == "c128" else 1) * (1 if c["two_s"] == 1 else 5)
        if cost > 1.3e9 or c.get("M", 4) >= d / 4 or (kind == "sym" and d * c["R"] * c["M"] > 2e8):
            continue
        return c


# --- systems ---------------------------------------------------------------------------------------------------

def _unit(rng, k):
    v = rng.normal(size=(k, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _lattice(case, rng, sizes_only):
    lx, ly = case["lx"], case["ly"]
    n = lx * ly
    s = dict(two_s=[case["two_s"]] * n)
    if not sizes_only:
        J = np.zeros((n, n))
        for y in range(ly):
            for x in range(lx):
                i = x + lx * y
                if x + 1 < lx:
                    J[i, i + 1] = rng.uniform(0.5, 1.5)
                if y + 1 < ly:
                    J[i, i + lx] = rng.uniform(0.5, 1.5)
        z = case.get("buckle", 0.0)                  # sites alternately above and below the plane
        pos = [(3.5 * (i % lx), 3.5 * (i // lx), z * (1 if (i % lx + i // lx) % 2 else -1)) for i in range(n)]
        s.update(J=J, pos=np.array(pos, dtype=float), B=rng.uniform(0.2, 2.0) * _unit(rng, 1)[0])
    return [s]


def _ring(case, rng, sizes_only, n):
    s = dict(two_s=[case["two_s"]] * n)
    if not sizes_only:
        a = 2 * np.pi * np.arange(n) / n
        t = np.deg2rad(30)
        J = np.zeros((n, n))
        for i in range(n):
            j = (i + 1) % n
            J[min(i, j), max(i, j)] = rng.uniform(0.6, 1.4)
        r = 3.0 * max(1.0, n / 6)
        s.update(J=J, pos=np.stack([r * np.cos(a), r * np.sin(a), 0 * a], axis=1), B=_unit(rng, 1)[0])
        if case["two_s"] > 1:
            s.update(d_ion=np.full(n, -5.0) * rng.uniform(0.8, 1.2),
                     e_axes=np.stack([np.sin(t) * np.cos(a), np.sin(t) * np.sin(a), np.cos(t) + 0 * a], axis=1))
    return s


def _chain(case, rng, sizes_only, n):
    s = dict(two_s=[case["two_s"]] * n)
    if not sizes_only:
        J = np.zeros((n, n))
        for i in range(n - 1):
            J[i, i + 1] = 0.8
        s.update(J=J, pos=np.stack([4.0 * np.arange(n), np.zeros(n), np.zeros(n)], axis=1), B=_unit(rng, 1)[0])
        if case["two_s"] > 1:
            s.update(d_ion=np.full(n, -3.0), e_axes=_unit(rng, n))
    return s


def _cube(case, rng, sizes_only, n):
    """a centre of spin s + 1/2 and n - 1 vertices of a cube with spin s and tilted easy axes"""
    s = dict(two_s=[case["two_s"] + 1] + [case["two_s"]] * (n - 1))
    if not sizes_only:
        v = 1.8 * np.array([(0, 0, 0)] + [(x, y, z) for z in (1, -1) for x, y in ((1, 1), (-1, 1), (-1, -1), (1, -1))])
        J = np.zeros((n, n))
        for k in range(1, n):
            J[0, k] = -1.2
            for l in range(k + 1, n):
                if np.count_nonzero(np.abs(v[k] - v[l]) > 0.1) == 1:
                    J[k, l] = rng.uniform(0.2, 0.5)
        th = np.deg2rad(30)
        ph = np.where(v[:n, 2] > 0, np.deg2rad(10), np.deg2rad(-10))
        ax = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th) + 0 * ph], axis=1)
        s.update(J=J, pos=v[:n].astype(float), B=_unit(rng, 1)[0], d_ion=np.array([0.0] + [-1.5] * (n - 1)), e_axes=ax)
    return s


def _mixed(case, rng, sizes_only, n):
    """a molecule of different spins at general positions"""
    s = dict(two_s=[1 + (i * 2) % case["two_s"] for i in range(n)])
    if not sizes_only:
        pos = 3.0 * np.stack([np.arange(n), np.arange(n) % 2, np.arange(n) % 3], axis=1) + rng.uniform(-0.5, 0.5, (n, 3))
        s.update(J=np.triu(rng.uniform(-0.5, 1.0, (n, n)), 1), pos=pos, B=_unit(rng, 1)[0],
                 d_ion=rng.uniform(-2, 0, n), e_axes=_unit(rng, n))
    return s


def _systems(case, seed, sizes_only=False):
    """The case's systems, as dicts of the System arguments."""
    rng = np.random.default_rng(seed)
    if case["geom"] == "lattice":
        return _lattice(case, rng, sizes_only)
    make = {"ring": _ring, "chain": _chain, "cube": _cube, "mixed": _mixed}[case["geom"]]
    out = []
    for n in range(case["n"], case.get("n_last", case["n"]) + 1):
        one = make(case, rng, sizes_only, n)
        for b in ([None] if sizes_only else _unit(rng, case["fields"])) if case["kind"] == "batch" and not sizes_only else \
                [None] * (case["fields"] if case["kind"] == "batch" else 1):
            out.append(dict(one) if b is None else dict(one, B=b))
    return out


def _make(s):
    return F.System(s["two_s"], s["J"], s.get("d_ion"), s.get("e_axes"), G, s["B"], s["pos"])


def _dtype(case):
    return torch.complex64 if case["dtype"] == "c64" else torch.complex128


# --- the passes ------------------------------------------------------------------------------------------------

def _block(case, seed, dim):
    """A caller's block of normalised Gaussian vectors [dim][R], the same numbers in either precision."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    x = torch.randn((dim, case["R"], 2), generator=g, device="cuda", dtype=torch.float32) / math.sqrt(2.0 * dim)
    return torch.view_as_complex(x).to(_dtype(case))


def prepare(case, seed):
    systems = [_make(s) for s in _systems(case, seed)]
    state = dict(case=case, seed=seed, systems=systems)
    dim = systems[0].dim
    if case["kind"] == "apply":
        state["x"] = _block(case, seed, dim)
        state["y"] = torch.empty_like(state["x"])
    elif case["kind"] == "start":
        state["x"] = torch.empty((dim, case["R"]), dtype=_dtype(case), device="cuda")
        state["y"] = torch.empty_like(state["x"])
    return state


def _numbers(case, r):
    """The results of one run: thermodynamics per temperature and the tridiagonal data."""
    f, c = (np.float32, np.complex64) if case["dtype"] == "c64" else (np.float64, np.complex128)
    keys = ["lnZ", "E", "C", "alpha", "beta"] + (["M_B_sym"] if case["kind"] == "sym" else [])
    out = {k: r[k].astype(f) for k in keys}
    out["M_B"] = (r["M_B"] + 1j * r["M_B_imag"]).astype(c)      # its imaginary part vanishes with R
    out["p"] = r["p"].astype(c)
    out["M_eff"] = r["M_eff"]
    if case["kind"] == "sym":
        out["O"] = r["O"].astype(c)
    return out


def run(state):
    c, systems = state["case"], state["systems"]
    if c["kind"] == "apply":
        F.apply_h(systems[0], state["x"], state["y"], c["R"], c["dtype"])
        return state["y"]
    if c["kind"] == "start":
        F.start_block(systems[0], state["x"], c["R"], state["seed"], dtype=c["dtype"])
        F.apply_sdir(systems[0], state["x"], state["y"], c["R"], c["dtype"])
        return [state["x"], state["y"]]
    kw = dict(R=c["R"], M=c["M"], T=TEMPERATURES, seed=state["seed"], dtype=c["dtype"], start=c["start"])
    if c["kind"] == "batch":
        rs = F.run_batch(systems, **kw)
        out = [_numbers(c, r) for r in rs]
        return {k: np.stack([o[k] for o in out]) for k in out[0]}
    return _numbers(c, F.run(systems[0], symmetric=c["kind"] == "sym", **kw))


def work(case):
    """Bytes: per step read q_j, q_{j-1} and the observable's block and write the new vector (H x: read x, write
    y).  Flops: the matrix elements of H that every row has, a complex multiply-add each."""
    size = 8 if case["dtype"] == "c64" else 16
    nbytes = flops = 0.0
    for s in _systems(case, 0, sizes_only=True):
        q = np.asarray(s["two_s"], dtype=np.float64) + 1
        d, n = float(np.prod(q)), len(q)
        keep = 1 - 1 / q                              # share of rows with a +1 (or -1) step at a site
        flips = 2 * keep.sum()
        pairs = 4 * sum(keep[i] * keep[i + 1:].sum() for i in range(n))
        sv = d * case["R"]
        if case["kind"] == "start":
            nbytes += sv * size * 3
            flops += sv * 8 * flips
        elif case["kind"] == "apply":
            nbytes += sv * size * 2
            flops += sv * (8 * (flips + pairs) + 2)
        else:
            nbytes += sv * size * 4 * case["M"]
            flops += sv * (8 * (flips + pairs) + 14) * case["M"]
            if case["kind"] == "sym":
                flops += sv * 8 * (flips + case["M"]) * case["M"]
    return {"bytes": float(nbytes), "flops": float(flops)}


# --- the same results in plain 64-bit torch ----------------------------------------------------------------------

def _spin(two_s):
    """(s^x, s^y, s^z) of one site, digit a = m + s."""
    s = two_s / 2
    m = np.arange(two_s + 1) - s
    up = np.diag(np.sqrt(s * (s + 1) - m[:-1] * (m[:-1] + 1)), -1)      # <a+1| s+ |a>
    return (up + up.T) / 2, (up - up.T) / 2j, np.diag(m)


class _Plain:
    """H and u.S as sums of one- and two-site operators over blocks [dim][R]; site 0 is the fastest digit."""

    def __init__(self, s):
        self.q = [t + 1 for t in s["two_s"]]
        n = self.n = len(self.q)
        self.dim = math.prod(self.q)
        ops = [_spin(t) for t in s["two_s"]]
        self.diag = torch.zeros(self.dim, dtype=torch.float64, device="cuda")
        self.moves = []                                                   # (sites, out digits, in digits, factor)
        for i in range(n):
            one = sum(MU_B * G * s["B"][c] * ops[i][c] for c in range(3)).astype(complex)
            if s.get("d_ion") is not None and s["d_ion"][i]:
                e = s["e_axes"][i] / np.linalg.norm(s["e_axes"][i])
                p = sum(e[c] * ops[i][c] for c in range(3))
                one = one + s["d_ion"][i] * (p @ p)
            self._add((i,), one)
            for j in range(i + 1, n):
                r = s["pos"][j] - s["pos"][i]
                r2 = r @ r
                A = 2 * s["J"][i, j] * np.eye(3) + C_DIP * G * G / r2 ** 1.5 * (np.eye(3) - 3 * np.outer(r, r) / r2)
                self._add((i, j), sum(A[a, b] * np.kron(ops[j][b], ops[i][a]) for a in range(3) for b in range(3)))
        b = np.asarray(s["B"]) / np.linalg.norm(s["B"])
        self.sdir = [sum(b[c] * ops[i][c] for c in range(3)) for i in range(n)]

    def _view(self, x, sites):
        """x as [.., digit of the last site, .., digit of the first site, ..]"""
        shape, rest = [], self.n
        for i in reversed(sites):
            shape += [math.prod(self.q[i + 1:rest]), self.q[i]]
            rest = i
        return x.reshape(shape + [-1])

    @staticmethod
    def _at(view, digits):
        for k, a in enumerate(reversed(digits)):
            view = view.narrow(1 + 2 * k, a, 1)
        return view

    def _add(self, sites, matrix):
        q = [self.q[i] for i in sites]
        dig = lambda k: (k,) if len(q) == 1 else (k % q[0], k // q[0])  # noqa: E731
        for k in range(matrix.shape[0]):
            self._at(self._view(self.diag, sites), dig(k)).add_(float(matrix[k, k].real))
            for l in range(matrix.shape[1]):
                if k != l and abs(matrix[k, l]) > 1e-15:
                    self.moves.append((sites, dig(k), dig(l), complex(matrix[k, l])))

    def h(self, x):
        y = self.diag[:, None] * x
        for sites, out, inn, f in self.moves:
            self._at(self._view(y, sites), out).add_(self._at(self._view(x, sites), inn), alpha=f)
        return y

    def s(self, x):
        y = torch.zeros_like(x)
        for i, m in enumerate(self.sdir):
            for k in range(m.shape[0]):
                for l in range(m.shape[1]):
                    if abs(m[k, l]) > 1e-15:
                        self._at(self._view(y, (i,)), (k,)).add_(self._at(self._view(x, (i,)), (l,)), alpha=complex(m[k, l]))
        return y

    def reversed(self, x):
        """Time reversal: (-1)^(digit sum) conj(x[dim - 1 - nu])."""
        y = x.flip(0).conj().resolve_conj().clone()
        for i in range(self.n):
            v = self._view(y, (i,))
            for a in range(1, self.q[i], 2):
                self._at(v, (a,)).neg_()
        return y


def _philox(nu, vec, seed):
    """Philox4x32-10 of counter (nu, vec), key seed: four words of 32 bits in int64 tensors."""
    mask = 0xFFFFFFFF
    c = [nu & mask, nu >> 32, torch.full_like(nu, vec & mask), torch.full_like(nu, vec >> 32)]
    k0, k1 = seed & mask, seed >> 32

    def mul(a, b):                                                        # 32 x 32 bits -> (high, low)
        lo, hi = (a & 0xFFFF) * b, (a >> 16) * b
        return (hi + (lo >> 16)) >> 16, ((hi << 16) + lo) & mask

    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _start(plain, R, seed, pairs):
    x = torch.empty((plain.dim, R), dtype=torch.complex128, device="cuda")
    nu = torch.arange(plain.dim, device="cuda")
    for k in range(R):
        if pairs and k % 2:
            x[:, k] = plain.reversed(x[:, k - 1].clone()[:, None])[:, 0]
            continue
        c = _philox(nu, k // 2 if pairs else k, seed)
        u1, u2 = (((c[a] << 21 | c[a + 1] >> 11).double() + 1.0) * 2.0 ** -53 for a in (0, 2))
        rho = torch.sqrt(-2.0 * torch.log(u1))
        x[:, k] = torch.complex(rho * torch.cos(2 * np.pi * u2), rho * torch.sin(2 * np.pi * u2))
    return x / torch.linalg.vector_norm(x, dim=0)


def _dot(a, b):
    return torch.stack([torch.vdot(a[:, k], b[:, k]) for k in range(a.shape[1])])


def _lanczos(case, plain, seed):
    R, M = case["R"], case["M"]
    v = _start(plain, R, seed, case["start"] == "pairs")
    u = plain.s(v)
    before, beta = None, torch.zeros(R, dtype=torch.float64, device="cuda")
    al, be, p, kept, su = [], [], [], [], []
    for _ in range(M):
        if case["kind"] == "sym":
            kept.append(v)
            su.append(plain.s(v))
        w = plain.h(v)
        a = _dot(v, w).real
        w -= a * v
        if before is not None:
            w -= beta * before
        p.append(_dot(v, u))
        beta = torch.linalg.vector_norm(w, dim=0)
        al.append(a)
        be.append(beta)
        before, v = v, w / beta
    al, be, p = (torch.stack(t, dim=1).cpu().numpy() for t in (al, be, p))
    O = None
    if case["kind"] == "sym":
        O = np.array([[[complex(torch.vdot(kept[i][:, r], su[j][:, r])) for j in range(M)] for i in range(M)] for r in range(R)])
    eps, U = [], []
    for r in range(R):
        e, w = np.linalg.eigh(np.diag(al[r]) + np.diag(be[r, :-1], 1) + np.diag(be[r, :-1], -1))
        eps.append(e)
        U.append(w)
    e0 = min(e[0] for e in eps)
    out = {k: np.zeros(len(TEMPERATURES)) for k in ("lnZ", "E", "C", "M_B_sym")}
    out["M_B"] = np.zeros(len(TEMPERATURES), dtype=np.complex128)
    for k, T in enumerate(TEMPERATURES):
        z = z1 = z2 = num = sym = 0.0
        for r in range(R):
            w = np.exp(-(eps[r] - e0) / T)
            w0 = U[r][0] ** 2 * w
            z, z1, z2 = z + w0.sum(), z1 + (w0 * eps[r]).sum(), z2 + (w0 * eps[r] ** 2).sum()
            num += (w * U[r][0] * (np.conj(p[r]) @ U[r])).sum()
            if O is not None:
                y = U[r] @ (np.sqrt(w) * U[r][0])
                sym += (y @ O[r] @ y).real
        out["lnZ"][k] = math.log(plain.dim / R * z) - e0 / T
        out["E"][k] = z1 / z
        out["C"][k] = (z2 / z - (z1 / z) ** 2) / T ** 2
        out["M_B"][k] = -G * num / z
        out["M_B_sym"][k] = -G * sym / z
    if O is None:
        del out["M_B_sym"]
    else:
        out["O"] = O
    return dict(out, alpha=al, beta=be, p=p, M_eff=np.full(R, M, dtype=np.int32))


def exact(case, seed):
    systems = _systems(case, seed)
    if case["kind"] == "apply":
        plain = _Plain(systems[0])
        return plain.h(_block(case, seed, plain.dim).to(torch.complex128))
    if case["kind"] == "start":
        plain = _Plain(systems[0])
        x = _start(plain, case["R"], seed, False)
        return [x, plain.s(x)]
    outs = [_lanczos(case, _Plain(s), seed) for s in systems]
    if case["kind"] == "batch":
        return {k: np.stack([o[k] for o in outs]) for k in outs[0]}
    return outs[0]
