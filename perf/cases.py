"""Workloads of the exact-diagonalization library, each through its public calls.

A case names a cluster (with its couplings), a symmetry sector and what is done
with it:

  apply    y = H x for nvec vectors, from the stored structure (the inner loop of
           every Lanczos run) or matrix-free (one-off applications, sectors whose
           structure is not kept)
  batch    y = H x for all (k, rho_k) sectors of a cluster in one launch
  setup    a sector from nothing: basis, Hamiltonian, stored structure, first H x
  lanczos  a ground state by ed_lanczos with its eigenvector
  evolve   one Krylov step exp(-i H dt) psi
  observe  spin correlations of a state, all site pairs

`exact` restates H x in plain torch: the basis by brute force over the group, the
columns through a table over all 2^N configurations.
"""
import math
from functools import lru_cache

import numpy as np
import torch

import paper_2210_03511_gb300 as ed
from edinputs import configs as C
from paper_2210_03511_gb300 import observables

# Clusters: lattice, periodicity, couplings, sublattice blocks (0: chosen by the
# input generator).  The couplings are those of the repository's workloads.
CLUSTERS = {
    "chain16": ("chain", 16, 1.0, 0.0, 0.0, 0),
    "chain19": ("chain", 19, 1.0, 0.3, 0.0, 0),
    "chain24": ("chain", 24, 1.0, 0.3, 0.0, 0),
    "chain28": ("chain", 28, 1.0, 0.4, 0.0, 0),
    "square16": ("square", ((4, 0), (0, 4)), 1.0, 0.5, 0.0, 0),
    "square20": ("square", ((4, 2), (-2, 4)), 1.0, 0.5, 0.0, 4),
    "square26": ("square", ((5, 1), (-1, 5)), 1.0, 0.5, 0.0, 0),
    "square32": ("square", ((4, 4), (4, -4)), 1.0, 0.5, 0.0, 2),
    "square36": ("square", ((6, 0), (0, 6)), 1.0, 0.5, 0.0, 0),
    "triangular24": ("triangular", ((5, 1), (4, -4)), 1.0, 0.125, 0.0, 2),
    "triangular27": ("triangular", ((3, 3), (-3, 6)), 1.0, 0.125, 0.0, 0),
    "kagome18": ("kagome", ((3, 0), (0, 2)), 1.0, 0.2, 0.3, 0),
    "kagome24": ("kagome", ((4, 0), (0, 2)), 1.0, 0.2, 0.3, 0),
    "kagome27": ("kagome", ((3, 0), (0, 3)), 1.0, 0.2, 0.3, 0),
    "kagome36": ("kagome", ((2, 2), (-2, 4)), 1.0, 0.2, 0.3, 0),
}
SITES = {"kagome36": 36, "square36": 36}


def _case(name, kind, cluster, **kw):
    c = dict(kind=kind, cluster=cluster, n_up=0, momentum=0, irrep="A1", point="full", flip=0, translations=True,
             bits=64, cplx=False, nvec=1, stored=True, name=name)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest workload: 12,870 states without symmetry, an H x of a few microseconds
        _case("chain16 apply f64", "apply", "chain16", irrep="A", point="none", translations=False),
        # the bench's mid-size sector (2.4 million states): the H x of its FP64 Lanczos run, L2-resident
        _case("square32 apply f64", "apply", "square32"),
        # the same cluster's complex sector (C4 character i, 4.7 million states), FP64
        _case("square32 E1 apply c128", "apply", "square32", irrep="E1", point="rot", cplx=True),
        # several FP32 vectors at once (refinement of several levels, block methods), an odd number
        _case("square32 apply f32 x5", "apply", "square32", bits=32, nvec=5),
        # a real sector of 63 million states: vectors beyond L2, several column segments, 64-bit words
        _case("square36 apply f64", "apply", "square36", irrep="A", point="rot"),
        # the bench's chiral spin-liquid model, 63 million states: FP32 vectors of the mixed-precision run
        _case("kagome36 apply c64", "apply", "kagome36", irrep="A", point="rot", flip=1, bits=32, cplx=True),
        # and the FP64 vectors of its full-precision run
        _case("kagome36 apply c128", "apply", "kagome36", irrep="A", point="rot", flip=1, cplx=True),
        # one-off H x without a stored structure
        _case("square32 free f64", "apply", "square32", stored=False),
        # every sector of the 24-site triangular torus in one launch (complex because of the momenta)
        _case("triangular24 batch c128", "batch", "triangular24", cplx=True),
        # time to the first H x of a large sector: enumeration, structure build
        _case("kagome36 setup c64", "setup", "kagome36", irrep="A", point="rot", flip=1, bits=32, cplx=True),
        # a ground state with its eigenvector at the library's defaults (full reorthogonalisation)
        _case("square32 lanczos f64", "lanczos", "square32"),
        # spin correlations of a state: one small Hamiltonian and one expectation per pair orbit
        _case("triangular24 observe f64", "observe", "triangular24"),
    ]


# Sectors a draw may take: cluster, then (momentum index, irrep, point group) choices
# and whether the sector may carry a spin flip at S^z = 0.
_SECTORS = {
    "chain16": [(0, "A", "none"), (3, "A", "none"), (0, "A1", "full")],
    "chain19": [(0, "A1", "full"), (2, "A", "none")],
    "chain24": [(0, "A1", "full"), (0, "A2", "full"), (5, "A", "none")],
    "chain28": [(0, "A1", "full"), (3, "A", "none")],
    "square16": [(0, "A1", "full"), (0, "B1", "full"), (0, "E1", "rot")],
    "square20": [(0, "A", "rot"), (0, "B", "rot"), (0, "E1", "rot")],
    "square26": [(0, "A", "rot"), (0, "B", "rot"), (0, "E1", "rot")],
    "square32": [(0, "A1", "full"), (0, "A2", "full"), (0, "B1", "full"), (0, "E1", "rot"), (0, "A", "rot")],
    "square36": [(0, "A1", "full"), (0, "B2", "full"), (0, "E1", "rot")],
    "triangular24": [(0, "A1", "full"), (0, "A", "none"), (5, "A", "none")],
    "triangular27": [(0, "A1", "full"), (0, "A", "rot"), (0, "E1", "rot")],
    "kagome18": [(0, "A", "none"), (1, "A", "none")],
    "kagome24": [(0, "A", "none"), (3, "A", "none")],
    "kagome27": [(0, "A", "rot"), (0, "E1", "rot")],
    "kagome36": [(0, "A", "rot"), (0, "B", "rot"), (0, "E1", "rot")],
}
_BY_SIZE = [("chain16", "chain19", "square16", "square20", "kagome18"),
            ("chain24", "square26", "triangular24", "triangular27", "kagome24"),
            ("chain28", "square32", "square32", "kagome27"),
            ("square36", "kagome36")]


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["setup", "batch", "lanczos", "evolve", "observe"])
    tiers = {"apply": 4, "setup": 4, "batch": 2, "lanczos": 3, "evolve": 3, "observe": 2}[kind]
    while True:
        if kind == "batch":
            cl = rng.choice(["square16", "square20", "triangular24"])
            N = _n_sites(cl)
            c = _case("", kind, cl, n_up=rng.randint(N // 4, N // 2), cplx=True, bits=rng.choice([32, 64]),
                      nvec=rng.choice([1, 1, 2, 3, 5, 8]), stored=rng.random() < 0.8)
            del c["name"]
            return c
        cl = rng.choice(_BY_SIZE[rng.randrange(tiers)])
        N = _n_sites(cl)
        mom, irrep, point = rng.choice(_SECTORS[cl])
        n_up = rng.randint(max(3, N // 3), N // 2)
        flip = rng.choice([0, 1, -1]) if 2 * n_up == N and N < 36 else (1 if 2 * n_up == N else 0)
        c = _case("", kind, cl, n_up=n_up, momentum=mom, irrep=irrep, point=point, flip=flip,
                  bits=rng.choice([32, 64]), cplx=rng.random() < 0.3)
        del c["name"]
        p = _problem(_key(c))
        c["cplx"] = c["cplx"] or not _is_real(p) or kind == "evolve"
        D = _dim(p.sector)
        if kind == "apply":
            c["stored"] = rng.random() < 0.7
            if N < 36:
                c["nvec"] = rng.choice([1, 1, 1, 2, 3, 5, 7, 8])
        if kind == "lanczos":
            c["bits"] = 64
        top = {"apply": 64e6 if c["stored"] else 20e6, "setup": 64e6}.get(kind, 5e6)
        if 200 <= D * c["nvec"] <= top:
            return c


# ---------------------------------------------------------------- inputs
def _n_sites(cl):
    return SITES.get(cl) or int("".join(ch for ch in cl if ch.isdigit()))


def _key(c):
    return (c["cluster"], c["n_up"], c["momentum"], c["irrep"], c["point"], c["flip"], c["translations"])


@lru_cache(maxsize=64)
def _problem(key):
    cluster, n_up, mom, irrep, point, flip, translations = key
    lat, P, J1, J2, Jchi, n_sub = CLUSTERS[cluster]
    kw = dict(irrep=irrep, spinflip=flip or None, n_up=n_up or None, n_sublat=n_sub or None)
    if lat == "chain":
        return C.chain(P, J1, J2, translations=translations, reflection=point == "full", k=mom, **kw)
    from edinputs.lattice import Cluster, allowed_momenta, kagome_lattice, square_lattice, triangular_lattice
    Pm = [list(r) for r in P]
    if mom:
        L = {"square": square_lattice, "triangular": triangular_lattice, "kagome": kagome_lattice}[lat]()
        kw["k"] = tuple(allowed_momenta(Cluster(L, Pm))[mom])
    kw.update(point=point, translations=translations, max_table_bytes=4 << 20 if n_sub else 96 * 1024)
    if lat == "kagome":
        return C.kagome(Pm, J1, J2, Jchi, **kw)
    return (C.square if lat == "square" else C.triangular)(Pm, J1, J2, **kw)


@lru_cache(maxsize=16)
def _all_sectors(cluster, n_up):
    lat, P, J1, J2, _, n_sub = CLUSTERS[cluster]
    return tuple(C.all_sectors(lat, [list(r) for r in P], J1, J2, n_sublat=n_sub or 2, n_up=n_up or None))


def _is_real(p):
    return bool(p.sector.is_real and p.terms.is_real)


def _tdtype(c):
    if c["cplx"]:
        return torch.complex128 if c["bits"] == 64 else torch.complex64
    return torch.float64 if c["bits"] == 64 else torch.float32


def _vector(shape, dtype, seed):
    """Normalised amplitudes of random sign or phase whose sizes spread over a few orders of
    magnitude, as a low-lying state's do."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    real = torch.float64 if dtype in (torch.float64, torch.complex128) else torch.float32
    x = torch.empty(shape, dtype=dtype, device="cuda")
    xr = torch.view_as_real(x) if dtype.is_complex else x
    xr.copy_(torch.randn(xr.shape, dtype=real, device="cuda", generator=g))
    size = torch.exp(torch.randn(shape, dtype=real, device="cuda", generator=g))
    x.mul_(size)
    x.div_(torch.linalg.vector_norm(x, dim=-1, keepdim=True))
    return x


_DT = {torch.float64: ed.ED_F64, torch.float32: ed.ED_F32, torch.complex128: ed.ED_C128, torch.complex64: ed.ED_C64}


def prepare(case, seed):
    kind, dt = case["kind"], _tdtype(case)
    if kind == "batch":
        hs = []
        for p in _all_sectors(case["cluster"], case["n_up"]):
            try:
                h = ed.Hamiltonian(ed.Basis(p.sector), p.terms)
            except ed.EdError as e:
                if e.name != "ED_ERR_EMPTY_SECTOR":
                    raise
                continue
            if case["stored"]:
                h.store(_DT[dt])
            hs.append(h)
        b = ed.Batch(hs)
        x = _vector((b.total * case["nvec"],), dt, seed)
        return dict(kind=kind, batch=b, nvec=case["nvec"], x=x, y=torch.empty_like(x))
    p = _problem(_key(case))
    if kind == "setup":
        x = _vector((_dim(p.sector),), dt, seed)
        return dict(kind=kind, problem=p, dtype=_DT[dt], x=x, y=torch.empty_like(x))
    basis = ed.Basis(p.sector)
    if kind == "observe":
        return dict(kind=kind, basis=basis, sector=p.sector, psi=_vector((basis.dim,), dt, seed))
    h = ed.Hamiltonian(basis, p.terms)
    if case["stored"]:
        h.store(_DT[dt])
    if kind == "apply":
        shape = (basis.dim,) if case["nvec"] == 1 else (case["nvec"], basis.dim)
        x = _vector(shape, dt, seed)
        return dict(kind=kind, h=h, x=x, y=torch.empty_like(x))
    if kind == "lanczos":
        ev = torch.empty((1, basis.dim), dtype=dt, device="cuda")
        return dict(kind=kind, h=h, dtype=_DT[dt], evecs=ev, seed=int(seed))
    return dict(kind=kind, h=h, psi=_vector((basis.dim,), dt, seed))


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["h"].apply(state["x"], state["y"])
    if kind == "batch":
        return state["batch"].apply(state["x"], state["y"], nvec=state["nvec"])
    if kind == "setup":
        p = state["problem"]
        h = ed.Hamiltonian(ed.Basis(p.sector), p.terms)
        h.store(state["dtype"])
        return h.apply(state["x"], state["y"])
    if kind == "lanczos":
        ev, rep = state["h"].lanczos(n_eig=1, tol=1e-10, dtype=state["dtype"], seed=state["seed"],
                                     evecs=state["evecs"])
        return ev, state["evecs"]
    if kind == "evolve":
        err, m = state["h"].evolve(state["psi"], 0.1, m=30)
        return state["psi"]
    return observables.correlations(state["basis"], state["sector"], state["psi"])


# ---------------------------------------------------------------- work
@lru_cache(maxsize=256)
def _dim_of(perm, flip, chi, N, n_up):
    perm = np.frombuffer(perm, np.int64).reshape(-1, N)
    flip = np.frombuffer(flip, np.uint8)
    chi = np.frombuffer(chi, complex)
    total = 0j
    for p, f, c in zip(perm, flip, chi):
        seen, cyc = np.zeros(N, bool), []
        for i in range(N):
            n, j = 0, i
            while not seen[j]:
                seen[j] = True
                j = p[j]
                n += 1
            if n:
                cyc.append(n)
        if f:
            fixed = 2 ** len(cyc) if all(n % 2 == 0 for n in cyc) else 0
        else:
            ways = [1] + [0] * n_up
            for n in cyc:
                for k in range(n_up, n - 1, -1):
                    ways[k] += ways[k - n]
            fixed = ways[n_up]
        total += c * fixed
    return int(round(total.real / len(perm)))


def _dim(s):
    """Dimension of a sector: (1/|G|) sum_g chi(g) (number of configurations g leaves unchanged)."""
    return _dim_of(np.ascontiguousarray(s.perm, np.int64).tobytes(), np.ascontiguousarray(s.spinflip, np.uint8).tobytes(),
                   np.ascontiguousarray(s.chi, complex).tobytes(), int(s.n_sites), int(s.n_up))


def _pairs(p):
    """Site pairs with an exchange or chirality term, each flipping an antiparallel pair."""
    prs = {tuple(sorted(map(int, b))) for b in np.asarray(p.terms.bonds).reshape(-1, 2)}
    for t in np.asarray(p.terms.tris).reshape(-1, 3):
        prs |= {tuple(sorted((int(t[a]), int(t[(a + 1) % 3])))) for a in range(3)}
    return len(prs)


def _elements(p, D):
    """Off-diagonal elements: rows times pairs times the share of antiparallel pairs."""
    s = p.sector
    N, u = int(s.n_sites), int(s.n_up)
    return D * _pairs(p) * 2.0 * u * (N - u) / (N * (N - 1.0))


def work(case):
    """One pass: vectors read and written once; of a stored structure one 4-byte word per element,
    |Stab| and the diagonal per row; matrix-free, the representatives and |Stab|."""
    kind = case["kind"]
    sx = (16 if case["cplx"] else 8) * case["bits"] // 64
    fl = 8.0 if case["cplx"] else 2.0
    if kind == "batch":
        ps = _all_sectors(case["cluster"], case["n_up"])
    else:
        ps = [_problem(_key(case))]
    by = fp = 0.0
    for p in ps:
        D = _dim(p.sector)
        G = _elements(p, D)
        word = 4 if p.sector.n_sites <= 32 else 8
        held = 10.0 * D + 4.0 * G if case["stored"] else (word + 2.0) * D
        nv = case["nvec"]
        if kind in ("apply", "batch"):
            by += held + 2.0 * nv * sx * D
            fp += fl * nv * G
        elif kind == "setup":
            by += 2.0 * (word + 2.0) * D + 2.0 * held + 2.0 * sx * D
            fp += fl * G
        elif kind == "lanczos":
            n = 55  # steps to a residual of 1e-10 on the mid-size sectors
            by += n * (held + 2.0 * sx * D) + sx * D * n * (n + 1.0) + sx * D
            fp += n * fl * G + 2.0 * fl * D * n * (n + 1.0)
        elif kind == "evolve":
            n = 30
            by += n * (held + 2.0 * sx * D) + sx * D * n * (n + 1.0) + sx * D
            fp += n * fl * G + 2.0 * fl * D * n * (n + 1.0)
        else:
            orbits = len(observables.pair_orbits(p.sector))
            N, u = int(p.sector.n_sites), int(p.sector.n_up)
            by += orbits * ((word + 2.0) * D + 2.0 * sx * D)
            fp += fl * D * (N * (N - 1) / 2.0) * 2.0 * u * (N - u) / (N * (N - 1.0))
    return {"bytes": by, "flops": fp}


# ---------------------------------------------------------------- exact
class _Plain:
    """H of one sector in plain torch, 64 bits: representatives by brute force over the group, and
    for every configuration the index of its representative and the element that leads to it."""

    def __init__(self, p):
        s = p.sector
        self.N, self.n_up = int(s.n_sites), int(s.n_up)
        N, dev = self.N, "cuda"
        perm = np.asarray(s.perm, np.int64)
        self.flip = np.asarray(s.spinflip, np.uint8)
        self.chi = np.asarray(s.chi, complex)
        nb = (N + 7) // 8
        lut = np.zeros((len(perm), nb, 256), np.int64)
        v = np.arange(256)
        for bit in range(N):
            to = N - 1 - perm[:, N - 1 - bit]
            lut[:, bit >> 3, :] |= (((v >> (bit & 7)) & 1)[None, :] << to[:, None])
        self.lut = torch.tensor(lut, device=dev)
        self.full = (1 << N) - 1
        reps = []
        step = min(1 << N, 1 << 26)
        for lo in range(0, 1 << N, step):
            c = torch.arange(lo, lo + step, device=dev)
            c = c[_popcount(c) == self.n_up]
            for g in range(1, len(perm)):
                if not len(c):
                    break
                c = c[self.act(g, c) >= c]
            reps.append(c)
        r = torch.cat(reps)
        stab = torch.zeros(len(r), dtype=torch.float64, device=dev)
        proj = torch.zeros(len(r), dtype=torch.complex128, device=dev)
        for g in range(len(perm)):
            same = self.act(g, r) == r
            stab += same
            proj += same * complex(self.chi[g])
        keep = proj.abs() > 0.5
        self.reps, self.stab = r[keep], stab[keep]
        D = len(self.reps)
        # configuration -> its representative's index (-1: none in the sector) and group element
        self.index = torch.full((1 << N,), -1, dtype=torch.int32, device=dev)
        self.elem = torch.zeros(1 << N, dtype=torch.int16, device=dev)
        ids = torch.arange(D, device=dev, dtype=torch.int32)
        for g in range(len(perm)):
            t = self.act(g, self.reps)
            self.index[t] = ids
            self.elem[t] = g
        self.real = bool(np.all(np.abs(self.chi.imag) < 1e-12))
        self.conj = torch.tensor(np.conj(self.chi), device=dev)

    def act(self, g, s):
        r = self.lut[g, 0][s & 255]
        for b in range(1, self.lut.shape[1]):
            r = r | self.lut[g, b][(s >> (8 * b)) & 255]
        return r ^ self.full if self.flip[g] else r

    def spin(self, site):
        return (self.reps >> (self.N - 1 - int(site))) & 1

    def pull(self, x, mask, amp):
        """amp (per row) times psi at the configurations reps ^ mask, over psi's factor at the rows."""
        t = self.reps ^ mask
        j = self.index[t].long()
        ok = j >= 0
        j = j.clamp(min=0)
        w = torch.sqrt(self.stab[j] / self.stab) * ok * amp
        ph = self.conj[self.elem[t].long()]
        c = w * (ph.real if not x.is_complex() else ph)
        return c * x[..., j]

    def apply(self, bonds, J, tris, Jchi, x):
        y = torch.zeros_like(x)
        for (a, b), Jv in zip(np.asarray(bonds).reshape(-1, 2), np.asarray(J)):
            anti = (self.spin(a) != self.spin(b)).double()
            y += 0.25 * float(Jv) * (1.0 - 2.0 * anti) * x
            mask = (1 << (self.N - 1 - int(a))) | (1 << (self.N - 1 - int(b)))
            y += self.pull(x, mask, 0.5 * float(Jv) * anti)
        for t, Jv in zip(np.asarray(tris).reshape(-1, 3), np.asarray(Jchi)):
            for r in range(3):
                a, b, c = (int(t[(r + q) % 3]) for q in range(3))
                mask = (1 << (self.N - 1 - a)) | (1 << (self.N - 1 - b))
                sgn = (self.spin(a) - self.spin(b)).double()
                y += self.pull(x, mask, sgn * (self.spin(c).double() - 0.5)) * (0.5j * float(Jv))
        return y


def _popcount(v):
    v = v - ((v >> 1) & 0x5555555555555555)
    v = (v & 0x3333333333333333) + ((v >> 2) & 0x3333333333333333)
    v = (v + (v >> 4)) & 0x0F0F0F0F0F0F0F0F
    return ((v * 0x0101010101010101) >> 56) & 0xFF


def _wide(x):
    return x.to(torch.complex128 if x.is_complex() else torch.float64)


def exact(case, seed):
    kind, dt = case["kind"], _tdtype(case)
    if _n_sites(case["cluster"]) > 32 or kind == "lanczos":
        return None
    if kind == "batch":
        ps = [p for p in _all_sectors(case["cluster"], case["n_up"]) if _dim(p.sector) > 0]
        dims = [_dim(p.sector) for p in ps]
        x = _wide(_vector((sum(dims) * case["nvec"],), dt, seed))
        parts = x.split([d * case["nvec"] for d in dims])
        out = []
        for p, d, v in zip(ps, dims, parts):
            t = p.terms
            out.append(_Plain(p).apply(t.bonds, t.J, t.tris, t.Jchi, v.reshape(case["nvec"], d)).reshape(-1))
        return torch.cat(out)
    p = _problem(_key(case))
    t, D = p.terms, _dim(p.sector)
    h = _Plain(p)
    if kind == "observe":
        psi = _wide(_vector((D,), dt, seed))
        N, n2 = h.N, torch.linalg.vector_norm(psi) ** 2
        corr = np.full((N, N), 0.75)
        for orb in observables.pair_orbits(p.sector):
            y = h.apply(orb, np.full(len(orb), 1.0 / len(orb)), [], [], psi)
            v = float((torch.vdot(psi, y) / n2).real)
            corr[orb[:, 0], orb[:, 1]] = corr[orb[:, 1], orb[:, 0]] = v
        return corr
    if kind == "evolve":
        psi = _wide(_vector((D,), dt, seed))
        out, term = psi.clone(), psi
        if D * len(t.bonds) > 1e8:
            return None
        for n in range(1, 40):  # Taylor series of exp(-0.1 i H)
            term = h.apply(t.bonds, t.J, t.tris, t.Jchi, term) * (-0.1j / n)
            out += term
        return out
    shape = (D,) if case["nvec"] == 1 else (case["nvec"], D)
    return h.apply(t.bonds, t.J, t.tris, t.Jchi, _wide(_vector(shape, dt, seed)))
