"""Timing cases of the library: products y = H x over the model spaces, block
sizes and precisions the framework is used with, and the other calls a
calculation makes (adjoint, densities, block Gram-Schmidt, Lanczos).

listed() names the cases, draw() gives more of the same ranges, prepare()
builds what a program has before the call, run() makes one call, work() counts
the bytes and operations of that call, exact() computes its result in 64 bits
with plain torch (own Slater determinants, own Clebsch-Gordan coefficients).
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300.inputs import Orbit

# (n, l, 2j, particle-hole weight) and single-particle energies of the valence spaces
SPACES = {
    "p": ([(0, 1, 3, 0), (0, 1, 1, 1)], [0.0, 1.0]),
    "sd": ([(0, 2, 5, 0), (1, 0, 1, 1), (0, 2, 3, 1)], [-3.95, -3.16, 1.65]),
    "pf": ([(0, 3, 7, 0), (1, 1, 3, 1), (0, 3, 5, 1), (1, 1, 1, 1)], [0.0, 2.0, 6.5, 4.0]),
}
DTYPES = {"f64": (N.BS_F64, torch.float64), "f32": (N.BS_F32, torch.float32)}


def _hx(name, space, Z, Nn, twoM, k, dtype, mode=0, excite=-1):
    return {"name": name, "call": "hx", "space": space, "Z": Z, "N": Nn, "twoM": twoM, "k": k, "dtype": dtype,
            "mode": mode, "excite": excite}


def listed():
    return [
        # the first thing a user runs, and every step of a small Lanczos run: one 640-component product, all latency
        _hx("hx sd 2p2n f64 k1", "sd", 2, 2, 0, 1, "f64"),
        # an odd nucleus of the sd shell, M = 1/2: ragged sectors, a block that fits in cache many times over
        _hx("hx sd 5p6n f32 k8", "sd", 5, 6, 1, 8, "f32"),
        # 48Cr in double precision, one vector: plain Lanczos and the FP64 refinement of every mixed run
        _hx("hx pf 4p4n f64 k1", "pf", 4, 4, 0, 1, "f64"),
        # 48Cr, the benchmark's block product in single precision
        _hx("hx pf 4p4n f32 k8", "pf", 4, 4, 0, 8, "f32"),
        # 48Cr with a small block: single-precision Lanczos on one or two pivots
        _hx("hx pf 4p4n f32 k2", "pf", 4, 4, 0, 2, "f32"),
        # 52Fe, 110 million components: the largest space; the kernel mode measured for it is replayed, as the benchmark does
        _hx("hx pf 6p6n f32 k4", "pf", 6, 6, 0, 4, "f32", mode=18),
        # a particle-hole truncated basis (at most four particles out of 0f7/2), its only kernel
        _hx("hx pf 5p4n 4p-4h f32 k4", "pf", 5, 4, 1, 4, "f32", excite=4),
        # gradient of a loss of y = H(theta) x on 48Cr, interaction fitting with FP32 vectors
        {"name": "backward pf 4p4n f32 k4", "call": "backward", "space": "pf", "Z": 4, "N": 4, "twoM": 0, "k": 4,
         "dtype": "f32", "same": False},
        # Hellmann-Feynman derivatives of one level in FP64 (and orbit occupations): x = gy
        {"name": "backward sd 6p6n f64 k1", "call": "backward", "space": "sd", "Z": 6, "N": 6, "twoM": 0, "k": 1,
         "dtype": "f64", "same": True},
        # transition densities between two pairs of 48Cr states
        {"name": "density pf 4p4n k2", "call": "density", "space": "pf", "Z": 4, "N": 4, "twoM": 0, "k": 2},
        # one Gram-Schmidt pass of block Lanczos on 48Cr against 24 stored blocks, and the block's own overlaps
        {"name": "reorth pf 4p4n f32 k8 nb24", "call": "reorth", "space": "pf", "Z": 4, "N": 4, "twoM": 0, "k": 8,
         "dtype": "f32", "nb": 24},
        # a whole mixed-precision calculation: 24Mg-size block Lanczos, the five lowest levels refined in FP64
        {"name": "lanczos sd 4p4n f32 k4", "call": "lanczos", "space": "sd", "Z": 4, "N": 4, "twoM": 0, "k": 4,
         "dtype": "f32", "niter": 48, "nkeep": 5},
    ]


# ---------------------------------------------------------------- sizes without building a basis
def _states(space):
    """(orbit, 2m, l mod 2, weight) of every single-particle state, orbit after orbit, 2m ascending."""
    return [(a, tm, l % 2, w) for a, (_, l, tj, w) in enumerate(SPACES[space][0]) for tm in range(-tj, tj + 1, 2)]


def _counts(space, n):
    """{(2M, parity, weight): number of n-particle determinants}."""
    c = {(0, (0, 0, 0)): 1}
    for (_, tm, par, w) in _states(space):
        d = dict(c)
        for (m, (M, P, W)), v in c.items():
            if m < n:
                key = (m + 1, (M + tm, P ^ par, W + w))
                d[key] = d.get(key, 0) + v
        c = d
    return {key: v for (m, key), v in c.items() if m == n}


def _dim(space, Z, Nn, twoM, excite=-1):
    p, q = _counts(space, Z), _counts(space, Nn)
    par = (Z + Nn) * (SPACES[space][0][0][1] % 2) % 2
    wmin = min(w for _, _, w in p) + min(w for _, _, w in q)   # of all determinants, whatever their M
    d = 0
    for (M1, P1, W1), v1 in p.items():
        for (M2, P2, W2), v2 in q.items():
            if M1 + M2 == twoM and P1 ^ P2 == par and (excite < 0 or W1 + W2 <= wmin + excite):
                d += v1 * v2
    return d


def _candidates(lo, hi, most):
    out = []
    for space in ("p", "sd", "pf"):
        ns = len(_states(space))
        for Z in range(1, min(most, ns - 1) + 1):
            for Nn in range(1, min(most, ns - 1) + 1):
                for twoM in ((0, 2) if (Z + Nn) % 2 == 0 else (1, 3)):
                    d = _dim(space, Z, Nn, twoM)
                    if lo <= d <= hi:
                        out.append((d, space, Z, Nn, twoM))
    return out


_sized = {}


def _pick(rng, lo, hi, most=6):
    """A space with a dimension near a log-uniform target in [lo, hi]."""
    if (lo, hi, most) not in _sized:
        _sized[lo, hi, most] = _candidates(lo, hi, most)
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    near = sorted(_sized[lo, hi, most], key=lambda c: abs(math.log(c[0] / t)))[:6]
    return rng.choice(near)[1:]


def draw(rng):
    """One more case: a product (most often), a truncated product, an adjoint, densities, a Gram-Schmidt pass or a
    Lanczos run, in a space whose dimension is spread over the logarithm of the range."""
    what = rng.choice(["hx"] * 6 + ["trunc", "backward", "density", "reorth", "lanczos"])
    k = rng.choice([1, 2, 4, 8])
    dt = rng.choice(["f32", "f32", "f64"])
    if what == "hx":
        space, Z, Nn, twoM = _pick(rng, 100, 2.0e6)
        c = _hx("", space, Z, Nn, twoM, k, dt)
    elif what == "trunc":
        while True:
            Z, Nn, excite = rng.randint(2, 6), rng.randint(2, 6), rng.randint(1, 4)
            twoM = (Z + Nn) % 2
            if 1000 <= _dim("pf", Z, Nn, twoM, excite) <= 2.0e6:
                break
        c = _hx("", "pf", Z, Nn, twoM, k, dt, excite=excite)
    elif what == "backward":
        space, Z, Nn, twoM = _pick(rng, 500, 2.0e6)
        c = {"call": "backward", "space": space, "Z": Z, "N": Nn, "twoM": twoM, "k": min(k, 4), "dtype": dt,
             "same": rng.random() < 0.5}
    elif what == "density":
        space, Z, Nn, twoM = _pick(rng, 500, 2.0e6)
        c = {"call": "density", "space": space, "Z": Z, "N": Nn, "twoM": twoM, "k": min(k, 4)}
    elif what == "reorth":
        space, Z, Nn, twoM = _pick(rng, 2.0e4, 2.0e6)
        c = {"call": "reorth", "space": space, "Z": Z, "N": Nn, "twoM": twoM, "k": k, "dtype": dt,
             "nb": rng.randint(3, 40)}
    else:
        space, Z, Nn, twoM = _pick(rng, 3.0e3, 3.0e4)
        c = {"call": "lanczos", "space": space, "Z": Z, "N": Nn, "twoM": twoM, "k": k, "dtype": dt,
             "niter": {1: 120, 2: 80, 4: 48, 8: 36}[k], "nkeep": rng.randint(1, 4)}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _labels(space):
    """Pauli-allowed, parity-conserving (a, b, c, d, J, T), 1-based, (ab) <= (cd)."""
    orb = SPACES[space][0]
    pairs = [(a, b) for a in range(len(orb)) for b in range(a, len(orb))]
    out = []
    for T in (0, 1):
        for J in range(max(o[2] for o in orb) + 1):
            ok = [(a, b) for a, b in pairs if abs(orb[a][2] - orb[b][2]) <= 2 * J <= orb[a][2] + orb[b][2]
                  and (a != b or (J + T) % 2 == 1)]
            for x, (a, b) in enumerate(ok):
                for c, d in ok[x:]:
                    if (orb[a][1] + orb[b][1] + orb[c][1] + orb[d][1]) % 2 == 0:
                        out.append((a + 1, b + 1, c + 1, d + 1, J, T))
    return out


def _interaction(space, seed):
    """Single-particle energies and Gaussian matrix elements: 2 MeV wide on the diagonal, 1 MeV off it."""
    rng = np.random.default_rng(1000003 * seed + 17)
    labels = _labels(space)
    v = rng.standard_normal(len(labels))
    return list(SPACES[space][1]), [(*t, float(x) * (2.0 if t[:2] == t[2:4] else 1.0)) for t, x in zip(labels, v)]


def _block(dim, k, seed, which, dtype):
    """A [dim][k] block of normal components, columns normalized: the values of Lanczos vectors."""
    g = torch.Generator(device="cuda").manual_seed(7919 * seed + which)
    x = torch.randn((dim, k), device="cuda", dtype=torch.float64 if dtype == torch.float64 else torch.float32, generator=g)
    return x / torch.linalg.vector_norm(x, dim=0, keepdim=True)


def _pair(c, dim, seed, tdt):
    """x and gy of a backward pass: gy = x, or x plus as much again that is not along it."""
    x = _block(dim, c["k"], seed, 1, tdt)
    return x, x if c["same"] else x + _block(dim, c["k"], seed, 2, tdt)


def _context(c, seed):
    spe, tb = _interaction(c["space"], seed)
    orbits = [Orbit(*o) for o in SPACES[c["space"]][0]]
    excite = c.get("excite", -1)
    par = +1 if _parity(c) == 0 else -1
    return N.make(orbits, spe, tb, c["Z"], c["N"], c["twoM"], par, max_excite=None if excite < 0 else excite)


def _parity(c):
    """Natural parity of the space: 1 (negative) for an odd number of particles in odd-l orbits."""
    return (c["Z"] + c["N"]) * (SPACES[c["space"]][0][0][1] % 2) % 2


def prepare(case, seed):
    ctx = _context(case, seed)
    dim, k = ctx.dim, case.get("k", 1)
    bs, tdt = DTYPES[case.get("dtype", "f64")]
    s = {"case": case, "ctx": ctx, "k": k, "bs": bs, "stream": torch.cuda.current_stream().cuda_stream}
    if case["call"] == "hx":
        s["x"] = _block(dim, k, seed, 1, tdt)
        s["y"] = torch.empty_like(s["x"])
        if case["mode"]:
            ctx.set_tuned(k, bs, case["mode"])
        elif case["excite"] < 0:
            ctx.autotune(k, bs, s["stream"])
    elif case["call"] == "backward":
        s["x"], s["gy"] = _pair(case, dim, seed, tdt)
        s["gx"] = torch.empty_like(s["x"])
    elif case["call"] == "density":
        s["F"], s["X"] = _block(dim, k, seed, 1, tdt), _block(dim, k, seed, 2, tdt)
        s["ns"] = len(_states(case["space"]))
    elif case["call"] == "reorth":
        nb = case["nb"]
        s["V"] = torch.stack([_block(dim, k, seed, 10 + b, tdt) for b in range(nb)])
        s["W0"] = _block(dim, k, seed, 1, tdt)
        s["W"] = torch.empty_like(s["W0"])
        s["C"] = torch.zeros(nb * k * k, device="cuda", dtype=torch.float64)
        s["O"] = torch.zeros(k * k, device="cuda", dtype=torch.float64)
    else:
        s["pivot"] = _block(dim, k, seed, 1, tdt)
    return s


def run(s):
    c, ctx, k, bs, st = s["case"], s["ctx"], s["k"], s["bs"], s["stream"]
    if c["call"] == "hx":
        ctx.apply_H(s["x"], s["y"], k, bs, st)
        return s["y"]
    if c["call"] == "backward":
        g = ctx.apply_H_backward(s["x"], s["gy"], s["gx"], k, bs, n_theta=ctx.n_spe + ctx.n_tbme, stream=st)
        return {"gx": s["gx"], "gtheta": g}
    if c["call"] == "density":
        return ctx.density(s["F"], s["X"], k, s["ns"], st)
    if c["call"] == "reorth":
        # the pass works in place: it starts from a fresh copy of the block each time
        s["W"].copy_(s["W0"])
        ctx.block_dots(s["V"], c["nb"], s["W"], k, bs, s["C"], st)
        ctx.block_update(s["V"], c["nb"], s["C"], s["W"], k, bs, st)
        ctx.block_dots(s["W"], 1, s["W"], k, bs, s["O"], st)
        return {"C": s["C"], "W": s["W"], "O": s["O"]}
    ev, _ = ctx.lanczos(s["pivot"], k, bs, c["niter"], c["nkeep"], refine=True, stream=st)
    return ev


# ---------------------------------------------------------------- work
def _ops(c):
    """Multiply-adds of one H x per vector: for the basis of case c, the pairs (proton jump, neutron jump) and the
    like-particle moves between determinants, counted from the numbers of determinants that hold given states."""
    st = _states(c["space"])
    ns = len(st)
    total = 0.0
    dens = {}
    for n in {c["Z"], c["N"]}:
        # determinants of n - 1 particles by (2M, parity): the cores one-body jumps pass through
        d = {}
        for (M, P, _), v in _counts(c["space"], n - 1).items() if n else ():
            d[M, P] = d.get((M, P), 0) + v
        dens[n] = d
    # pn: a pair of cores (Z-1, N-1) with a free proton-neutron pair of states on either side
    pairs = {}
    for (_, m1, p1, _) in st:
        for (_, m2, p2, _) in st:
            pairs[m1 + m2, p1 ^ p2] = pairs.get((m1 + m2, p1 ^ p2), 0) + 1
    fz, fn = (ns - c["Z"] + 1) / ns, (ns - c["N"] + 1) / ns
    for (M1, P1), v1 in dens[c["Z"]].items():
        for (M2, P2), v2 in dens[c["N"]].items():
            q = pairs.get((c["twoM"] - M1 - M2, P1 ^ P2 ^ _parity(c)), 0)
            total += v1 * v2 * (q * fz * fn) ** 2
    dim = _dim(c["space"], c["Z"], c["N"], c["twoM"])
    # like particles: the distinct determinants two moves away, about a tenth of the pn work each
    for n in (c["Z"], c["N"]):
        free = ns - n
        total += dim * (1 + n * free / 8.0 + n * (n - 1) * free * (free - 1) / 64.0)
    if c.get("excite", -1) >= 0:
        total *= _dim(c["space"], c["Z"], c["N"], c["twoM"], c["excite"]) / max(1, dim)
    return total


def work(case):
    es = 8 if case.get("dtype", "f64") == "f64" else 4
    k = case.get("k", 1)
    dim = _dim(case["space"], case["Z"], case["N"], case["twoM"], case.get("excite", -1))
    vec = float(dim) * k * es
    if case["call"] == "hx":
        return {"bytes": 2 * vec, "flops": 2 * _ops(case) * k}
    if case["call"] == "backward":
        return {"bytes": 3 * vec, "flops": 4 * _ops(case) * k}
    if case["call"] == "density":
        ns = len(_states(case["space"]))
        jumps = sum(n * (1 + (ns - n) / 8.0) for n in (case["Z"], case["N"]))
        return {"bytes": 2 * vec, "flops": 2.0 * dim * jumps * k * k}
    if case["call"] == "reorth":
        nb = case["nb"]
        return {"bytes": (2 * nb + 3) * vec, "flops": (4.0 * nb + 2) * dim * k * k}
    n = case["niter"]
    return {"bytes": 2 * vec * n + 2 * vec * n * n, "flops": 2 * _ops(case) * k * n + 4.0 * dim * k * k * n * n}


# ---------------------------------------------------------------- 64 bits
def _cg(j1, m1, j2, m2, J, M):
    """<j1 m1 j2 m2 | J M>, arguments doubled (Racah's sum)."""
    if m1 + m2 != M or abs(m1) > j1 or abs(m2) > j2 or abs(M) > J or not abs(j1 - j2) <= J <= j1 + j2:
        return 0.0
    f = math.factorial
    a, b, c = (j1 + j2 - J) // 2, (j1 - m1) // 2, (j2 + m2) // 2
    d, e = (J - j2 + m1) // 2, (J - j1 - m2) // 2
    s = sum((-1) ** t / (f(t) * f(a - t) * f(b - t) * f(c - t) * f(d + t) * f(e + t))
            for t in range(max(0, -d, -e), min(a, b, c) + 1))
    n = (J + 1) * f(a) * f((j1 - j2 + J) // 2) * f((j2 - j1 + J) // 2) / f((j1 + j2 + J) // 2 + 1)
    n *= f((j1 + m1) // 2) * f(b) * f(c) * f((j2 - m2) // 2) * f((J + M) // 2) * f((J - M) // 2)
    return math.sqrt(n) * s


def _decouple(space):
    """The linear maps from the matrix elements to the M-scheme ones: rows (t, ij, kl, coefficient), states numbered
    orbit after orbit; like particles with i < j and k < l, proton-neutron for all."""
    orb = SPACES[space][0]
    first = np.cumsum([0] + [o[2] + 1 for o in orb])
    ns = int(first[-1])
    like, pn = [], []

    def coupled(a, b, J):
        """(i, j, M, coefficient) of a state a(m1) b(m2) in |a b; J M>."""
        ja, jb = orb[a][2], orb[b][2]
        return [(int(first[a]) + (m1 + ja) // 2, int(first[b]) + (m2 + jb) // 2, m1 + m2, _cg(ja, m1, jb, m2, 2 * J, m1 + m2))
                for m1 in range(-ja, ja + 1, 2) for m2 in range(-jb, jb + 1, 2) if abs(m1 + m2) <= 2 * J]

    for t, (a, b, c, d, J, T) in enumerate(_labels(space)):
        a, b, c, d = a - 1, b - 1, c - 1, d - 1
        z = math.sqrt((2.0 if a == b else 1.0) * (2.0 if c == d else 1.0))
        for (a1, b1, c1, d1) in ((a, b, c, d), (c, d, a, b)) if (a, b) != (c, d) else ((a, b, c, d),):
            if T == 1:
                ket = coupled(c1, d1, J)
                for i, j, M, x in coupled(a1, b1, J):
                    if i < j:
                        like += [(t, i * ns + j, k * ns + l, z * x * y) for k, l, M2, y in ket if k < l and M2 == M]
            for p, q in itertools.product({(a1, b1), (b1, a1)}, {(c1, d1), (d1, c1)}):
                ph = 1.0
                for (u, v), (u0, v0) in ((p, (a1, b1)), (q, (c1, d1))):
                    if (u, v) != (u0, v0):
                        ph *= (-1.0) ** ((orb[u][2] + orb[v][2]) // 2 + J + T)
                ket = coupled(q[0], q[1], J)
                for i, j, M, x in coupled(p[0], p[1], J):
                    pn += [(t, i * ns + j, k * ns + l, 0.5 * ph * z * x * y) for k, l, M2, y in ket if M2 == M]
    return ns, like, pn


def _dev(a, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=dtype)


class _Side:
    """The determinants of one species by (2M, parity), and their one- and two-body moves."""

    def __init__(self, space, n):
        st = _states(space)
        ns = len(st)
        rows = []
        for occ in itertools.combinations(range(ns), n):
            rows.append((sum(st[s][1] for s in occ), sum(st[s][2] for s in occ) % 2, sum(1 << s for s in occ),
                         sum(st[s][3] for s in occ)))
        rows.sort()   # (2M, parity, bits): a truncated basis orders by weight inside this, see _Exact
        self.key = [(r[0], r[1]) for r in rows]
        self.bits = np.array([r[2] for r in rows], dtype=np.int64)
        self.w = np.array([r[3] for r in rows], dtype=np.int64)
        self.sec = {}
        for g, key in enumerate(self.key):
            lo, _ = self.sec.get(key, (g, g))
            self.sec[key] = (lo, g + 1)
        self.order = np.argsort(self.bits, kind="stable")
        self.sorted = self.bits[self.order]
        self.ns, self.n, self.st = ns, n, st

    def find(self, b):
        return self.order[np.searchsorted(self.sorted, b)]

    @staticmethod
    def below(b, s):
        m = b & ((1 << s) - 1)
        c = np.zeros_like(b)
        while np.any(m):
            c += m & 1
            m = m >> 1
        return 1.0 - 2.0 * (c & 1)

    def one(self, i, k):
        """(source, destination, sign) of a+_i a_k."""
        src = np.nonzero((self.bits >> k) & 1)[0]
        b = self.bits[src]
        s = self.below(b, k)
        b = b & ~(1 << k)
        ok = ((b >> i) & 1) == 0
        src, b, s = src[ok], b[ok], s[ok]
        return src, self.find(b | (1 << i)), s * self.below(b, i)

    def two(self):
        """(pair ij, pair kl, source, destination, sign) of a+_i a+_j a_l a_k, i < j, k < l, of equal 2m and parity."""
        if self.n < 2:
            return [np.zeros(0, dtype=np.int64)] * 4 + [np.zeros(0)]
        groups = {}
        for i in range(self.ns):
            for j in range(i + 1, self.ns):
                groups.setdefault((self.st[i][1] + self.st[j][1], self.st[i][2] ^ self.st[j][2]), []).append((i, j))
        out = [[], [], [], [], []]
        for pairs in groups.values():
            for k, l in pairs:
                src = np.nonzero(((self.bits >> k) & 1) & ((self.bits >> l) & 1))[0]
                b = self.bits[src]
                s = self.below(b, k)
                b = b & ~(1 << k)
                s = s * self.below(b, l)
                b = b & ~(1 << l)
                for i, j in pairs:
                    ok = (((b >> i) & 1) == 0) & (((b >> j) & 1) == 0)
                    c, sg = b[ok], s[ok]
                    sg = sg * self.below(c, j)
                    c = c | (1 << j)
                    sg = sg * self.below(c, i)
                    c = c | (1 << i)
                    for o, v in zip(out, (np.full(len(c), i * self.ns + j), np.full(len(c), k * self.ns + l), src[ok],
                                          self.find(c), sg)):
                        o.append(v)
        return [np.concatenate(o) for o in out]


class _Exact:
    """H of a case in 64 bits, block by block: dense like-particle matrices, and per proton operator a+_i a_k the
    neutron matrix sum_jl W(ij,kl) a+_j a_l."""

    def __init__(self, c, seed):
        self.c = c
        spe, tb = _interaction(c["space"], seed)
        v = np.array([t[6] for t in tb])
        self.ns, self.like, self.pn = _decouple(c["space"])
        ns = self.ns
        self.nt, self.no = len(tb), len(spe)
        wl, wp = np.zeros((ns * ns, ns * ns)), np.zeros((ns * ns, ns * ns))
        for tab, w in ((self.like, wl), (self.pn, wp)):
            t, ij, kl, x = (np.array(q) for q in zip(*tab))
            np.add.at(w, (ij.astype(int), kl.astype(int)), x * v[t.astype(int)])
        self.P, self.Q = _Side(c["space"], c["Z"]), _Side(c["space"], c["N"])
        P, Q = self.P, self.Q
        self.orb = np.array([s[0] for s in P.st])
        # blocks of equal (2M, parity), and the place of each of their elements in the library's order
        self.blocks = []
        par = _parity(c)
        for key, (lo, hi) in sorted(P.sec.items()):
            o = (c["twoM"] - key[0], key[1] ^ par)
            if o in Q.sec:
                self.blocks.append((key, lo, hi, *Q.sec[o]))
        self.of = {b[0]: n for n, b in enumerate(self.blocks)}
        excite = c.get("excite", -1)
        wmax = P.w.min() + Q.w.min() + excite if excite >= 0 else 1 << 30
        at, sub = 0, []
        self.where = [np.full((b[2] - b[1], b[4] - b[3]), -1, dtype=np.int64) for b in self.blocks]
        for n, (key, p0, p1, q0, q1) in enumerate(self.blocks):
            for wp_ in sorted(set(P.w[p0:p1])) if excite >= 0 else [None]:
                rp = np.nonzero(P.w[p0:p1] == wp_)[0] if excite >= 0 else np.arange(p1 - p0)
                for wq in sorted(set(Q.w[q0:q1])) if excite >= 0 else [None]:
                    rq = np.nonzero(Q.w[q0:q1] == wq)[0] if excite >= 0 else np.arange(q1 - q0)
                    if excite >= 0 and wp_ + wq > wmax:
                        continue
                    self.where[n][np.ix_(rp, rq)] = at + np.arange(len(rp) * len(rq)).reshape(len(rp), len(rq))
                    at += len(rp) * len(rq)
        self.dim = at
        self.at = [_dev(w) for w in self.where]
        # like-particle moves and matrices
        self.moves, self.H = [], []
        for S in (P, Q):
            ij, kl, src, dst, sg = S.two()
            self.moves.append([_dev(ij), _dev(kl), _dev(src), _dev(dst), _dev(sg)])
            h = torch.zeros((len(S.bits), len(S.bits)), device="cuda", dtype=torch.float64)
            W = _dev(wl)
            if len(ij):
                m = self.moves[-1]
                h.index_put_((m[3], m[2]), W[m[0], m[1]] * m[4], accumulate=True)
            e = sum(spe[S.st[s][0]] * ((S.bits >> s) & 1) for s in range(ns))
            h.diagonal().add_(_dev(e, torch.float64))
            self.H.append(h)
        self.wp = wp
        # neutron moves by (change of 2m, parity): operator ij -> entries
        self.nops = {}
        for j in range(ns):
            for l in range(ns):
                key = (Q.st[j][1] - Q.st[l][1], Q.st[j][2] ^ Q.st[l][2])
                src, dst, sg = Q.one(j, l)
                self.nops.setdefault(key, []).append((j, l, src, dst, sg))
        for key, ops in self.nops.items():
            num = np.concatenate([np.full(len(o[2]), n) for n, o in enumerate(ops)])
            self.nops[key] = ([(o[0], o[1]) for o in ops], _dev(num),
                              *(_dev(np.concatenate([o[x] for o in ops])) for x in (2, 3, 4)))

    def split(self, x):
        """[dim][k] to one [protons][neutrons][k] array per block (zeros where the truncation leaves states out)."""
        x = x.double()
        pad = torch.cat([x, torch.zeros((1, x.shape[1]), device=x.device, dtype=x.dtype)])
        return [pad[a] for a in self.at]

    def join(self, X):
        out = torch.zeros((self.dim + 1, X[0].shape[2]), device="cuda", dtype=torch.float64)
        for a, b in zip(self.at, X):
            out[a.reshape(-1)] = b.reshape(-1, b.shape[2])
        return out[:-1]

    def proton_ops(self):
        """For every a+_i a_k: (i, k, its neutron operators' key, [(source block, destination block, rows, rows, signs)])."""
        P = self.P
        for i in range(self.ns):
            for k in range(self.ns):
                src, dst, sg = P.one(i, k)
                dm, dp = P.st[i][1] - P.st[k][1], P.st[i][2] ^ P.st[k][2]
                if (-dm, dp) not in self.nops or not len(src):
                    continue
                parts = []
                for n, (key, p0, p1, q0, q1) in enumerate(self.blocks):
                    m = self.of.get((key[0] + dm, key[1] ^ dp))
                    if m is None:
                        continue
                    at = (src >= p0) & (src < p1)
                    if at.any():
                        parts.append((n, m, _dev(src[at] - p0), _dev(dst[at] - self.blocks[m][1]), _dev(sg[at])))
                yield i, k, (-dm, dp), parts

    def apply(self, X):
        Y = [torch.einsum("pr,rnk->pnk", self.H[0][p0:p1, p0:p1], b) + torch.einsum("nr,prk->pnk", self.H[1][q0:q1, q0:q1], b)
             for (_, p0, p1, q0, q1), b in zip(self.blocks, X)]
        nq = len(self.Q.bits)
        B = torch.zeros((nq, nq), device="cuda", dtype=torch.float64)
        ns, w = self.ns, self.wp
        for i, k, key, parts in self.proton_ops():
            ops, num, src, dst, sg = self.nops[key]
            wv = _dev([w[i * ns + j, k * ns + l] for j, l in ops])
            B.zero_()
            B.index_put_((dst, src), wv[num] * sg, accumulate=True)
            for n, m, rs, rd, s in parts:
                q0, q1 = self.blocks[n][3:5]
                d0, d1 = self.blocks[m][3:5]
                kk = X[n].shape[2]
                xs = (X[n][rs] * s[:, None, None]).permute(1, 0, 2).reshape(q1 - q0, -1)
                y = (B[d0:d1, q0:q1] @ xs).reshape(d1 - d0, len(rs), kk).permute(1, 0, 2)
                Y[m].index_add_(0, rd, y)
        return Y

    def gtheta(self, X, G):
        """sum over the columns of g^T (dH/dtheta) x."""
        ns = self.ns
        out = np.zeros(self.no + self.nt)
        rho2 = torch.zeros(ns ** 4, device="cuda", dtype=torch.float64)
        for S, mv, proton in ((self.P, self.moves[0], True), (self.Q, self.moves[1], False)):
            D = torch.zeros((len(S.bits), len(S.bits)), device="cuda", dtype=torch.float64)
            for (_, p0, p1, q0, q1), x, g in zip(self.blocks, X, G):
                if proton:
                    D[p0:p1, p0:p1] += g.reshape(p1 - p0, -1) @ x.reshape(p1 - p0, -1).T
                else:
                    D[q0:q1, q0:q1] += g.permute(1, 0, 2).reshape(q1 - q0, -1) @ x.permute(1, 0, 2).reshape(q1 - q0, -1).T
            d = D.diagonal().cpu().numpy()
            for s in range(ns):
                out[self.orb[s]] += d[((S.bits >> s) & 1) == 1].sum()
            rho2.index_add_(0, mv[0] * ns * ns + mv[1], D[mv[3], mv[2]] * mv[4])
        rho = np.zeros((ns * ns, ns * ns))
        nq = len(self.Q.bits)
        D = torch.zeros((nq, nq), device="cuda", dtype=torch.float64)
        for i, k, key, parts in self.proton_ops():
            ops, num, src, dst, sg = self.nops[key]
            D.zero_()
            for n, m, rs, rd, s in parts:
                q0, q1 = self.blocks[n][3:5]
                d0, d1 = self.blocks[m][3:5]
                xs = (X[n][rs] * s[:, None, None]).permute(1, 0, 2).reshape(q1 - q0, -1)
                gs = G[m][rd].permute(1, 0, 2).reshape(d1 - d0, -1)
                D[d0:d1, q0:q1] += gs @ xs.T
            v = torch.zeros(len(ops), device="cuda", dtype=torch.float64)
            v.index_add_(0, num, D[dst, src] * sg)
            for (j, l), u in zip(ops, v.cpu().numpy()):
                rho[i * ns + j, k * ns + l] = u
        for tab, r in ((self.like, rho2.cpu().numpy().reshape(ns * ns, ns * ns)), (self.pn, rho)):
            t, ij, kl, x = (np.array(q) for q in zip(*tab))
            np.add.at(out, self.no + t.astype(int), x * r[ij.astype(int), kl.astype(int)])
        return out

    def density(self, F, X):
        ns, k = self.ns, X[0].shape[2]
        out = np.zeros((2, ns, ns, k, k))
        for t, S in ((0, self.P), (1, self.Q)):
            D = torch.zeros((len(S.bits), len(S.bits), k, k), device="cuda", dtype=torch.float64)
            for (_, p0, p1, q0, q1), f, x in zip(self.blocks, F, X):
                if t == 0:
                    D[p0:p1, p0:p1] += torch.einsum("pnf,qnj->pqfj", f, x)
                else:
                    D[q0:q1, q0:q1] += torch.einsum("npf,nqj->pqfj", f, x)
            for i in range(ns):
                for l in range(ns):
                    if S.st[i][1:3] == S.st[l][1:3]:
                        src, dst, sg = S.one(i, l)
                        out[t, i, l] = (D[_dev(dst), _dev(src)] * _dev(sg)[:, None, None]).sum(dim=0).cpu().numpy()
        return out


def exact(case, seed):
    dim = _dim(case["space"], case["Z"], case["N"], case["twoM"], case.get("excite", -1))
    if dim > 3.0e6:
        return None   # 52Fe: minutes and more memory than the card has
    k = case.get("k", 1)
    _, tdt = DTYPES[case.get("dtype", "f64")]
    if case["call"] == "reorth":
        V = torch.stack([_block(dim, k, seed, 10 + b, tdt) for b in range(case["nb"])]).double()
        W = _block(dim, k, seed, 1, tdt).double()
        C = torch.einsum("bai,aj->bij", V, W)
        W = W - torch.einsum("bai,bij->aj", V, C)
        return {"C": C.reshape(-1), "W": W, "O": (W.T @ W).reshape(-1)}
    E = _Exact(case, seed)
    if case["call"] == "hx":
        return E.join(E.apply(E.split(_block(dim, k, seed, 1, tdt))))
    if case["call"] == "backward":
        x, g = (E.split(v) for v in _pair(case, dim, seed, tdt))
        return {"gx": E.join(E.apply(g)), "gtheta": E.gtheta(x, g)}
    if case["call"] == "density":
        return E.density(E.split(_block(dim, k, seed, 1, tdt)), E.split(_block(dim, k, seed, 2, tdt)))
    # Lanczos: the Ritz values of the same block Krylov space, orthonormalized in full
    if case["niter"] * k * dim > 1.0e7:
        return None
    v, _ = torch.linalg.qr(_block(dim, k, seed, 1, tdt).double())
    V, HV = [v], []
    for n in range(min(case["niter"], dim // k)):
        HV.append(E.join(E.apply(E.split(V[-1]))))
        A = torch.cat(V, dim=1)
        w = HV[-1]
        for _ in range(2):
            w = w - A @ (A.T @ w)
        V.append(torch.linalg.qr(w)[0])
    A = torch.cat(V[:-1], dim=1)
    T = A.T @ torch.cat(HV, dim=1)
    return torch.linalg.eigvalsh(0.5 * (T + T.T))[:case["nkeep"]].cpu().numpy()
