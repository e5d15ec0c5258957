"""Performance cases of the library: the calls a campaign, a serving stream or a notebook makes.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges, ``prepare(case, seed)`` builds what a program
holds before the call, ``run(state)`` is one pass through the C ABI, ``work(case)`` what a pass cannot do without, and
``exact(case, seed)`` the same outputs in 64 bits from the definitions of include/ftlm.h, written here in plain torch.

Kinds of case:
  hv       one H·v: ftlm_hv_packed on a packed set (every irrep of the group, or one block), or ftlm_hv on one block's
           [dim][B] vectors; flips searched in the call or read from the sector's entry table;
  lanczos  FTLM chains: ftlm_lanczos on one block (a serving job) or ftlm_lanczos_sets over S^z sectors (a batch);
  prepare  a new sector: enumeration, entry table, packed set and the first H·v on it;
  thermo   the thermal sums of a campaign from its chains' coefficients.

The irreps are tabulated ones (ftlm_group_set_irreps), made here from the regular representation, so that ``exact``
works in the same irrep basis.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2607_17429_gb300 import ftlm as F
from workloads import cluster

DTYPES = {"f64": (F.F64, torch.float64), "f32": (F.F32, torch.float32), "f16": (F.F16, torch.float16)}
DEV = "cuda" if torch.cuda.is_available() else "cpu"
SETS = ("icosahedron", "dodecahedron", "icosidodecahedron", "cuboctahedron", "tetrahedron")  # clusters with set kernels


def listed():
    hv = dict(kind="hv", two_M=0, irrep=-1, api="packed", table=False, flip=False)
    return [
        # The smallest call: the plain FP64 check system (s = 1/2 icosahedron against full diagonalisation), R = 4.
        dict(hv, name="hv_icosahedron_f64_b4", cluster="icosahedron", two_s=1, dtype="f64", B=4),
        # A sector of the batched s = 1 cuboctahedron campaign: R = 24 chains, a width that is no power of two.
        dict(hv, name="hv_cuboctahedron_f32_b24", cluster="cuboctahedron", two_s=2, dtype="f32", B=24),
        # The benchmark sector with its entry table: icosidodecahedron, M = 0, all ten irreps, eight chains.
        dict(hv, name="hv_icosidodecahedron_f32_b8_table", cluster="icosidodecahedron", two_s=1, dtype="f32", B=8,
             table=True),
        # The same sector as the campaign driver and the serving loop run it: flips searched in every H·v.
        dict(hv, name="hv_icosidodecahedron_f32_b8_search", cluster="icosidodecahedron", two_s=1, dtype="f32", B=8),
        # The half-precision storage mode on the benchmark sector.
        dict(hv, name="hv_icosidodecahedron_f16_b8_table", cluster="icosidodecahedron", two_s=1, dtype="f16", B=8,
             table=True),
        # Plain FP64, one block at a time on its own [dim][B] vectors (the comparison runs); a 3-dimensional irrep,
        # the most frequent dimension of I_h.
        dict(hv, name="hv_block_f64_b8", cluster="icosidodecahedron", two_s=1, irrep=2, dtype="f64", B=8, api="block"),
        # A large single block at one right-hand side from the table (s = 3/2 dodecahedron, H_g), in the sector whose
        # tables leave room for several of them.
        dict(hv, name="hv_dodecahedron_f32_b1_table", cluster="dodecahedron", two_s=3, two_M=28, irrep=8, dtype="f32",
             B=1, table=True),
        # Spin-flip symmetry at M = 0 (Gamma- of a 4-dimensional irrep) with five chains: rows of 20 bytes.
        dict(hv, name="hv_flip_block_f32_b5", cluster="icosidodecahedron", two_s=1, irrep=13, dtype="f32", B=5,
             flip=True),
        # The batched campaign: S^z sectors of the s = 3/2 icosahedron, all irreps, 24 Rademacher chains.
        dict(kind="lanczos", name="lanczos_batch_icosahedron", cluster="icosahedron", two_s=3, two_M=0, sectors=6,
             irrep=-1, dtype="f32", R=24, steps=14, rng="rademacher", table=False),
        # One job of the serving stream: a block of the periodic 4x6 square lattice, R = 4.
        dict(kind="lanczos", name="lanczos_job_square", cluster="square:4x6:c2v", two_s=1, two_M=0, sectors=1, irrep=0,
             dtype="f32", R=4, steps=14, rng="gauss", table=False),
        # What every new sector costs before its chains run: enumeration, entry table, packed set, first H·v.
        dict(kind="prepare", name="prepare_icosidodecahedron", cluster="icosidodecahedron", two_s=1, two_M=0, irrep=-1,
             dtype="f32", B=8, flip=False),
        # The end of the s = 3/2 icosahedron campaign: 19 sectors x 10 irreps x 24 chains of 60 steps, 200 temperatures.
        dict(kind="thermo", name="thermo_campaign", blocks=190, R=24, steps=60, n_T=200),
    ]


def draw(rng):
    kind = rng.choices(("hv", "lanczos", "prepare", "thermo"), (6, 2, 1, 1))[0]
    if kind == "thermo":
        return dict(kind="thermo", blocks=_log_int(rng, 1, 190), R=rng.randint(1, 24), steps=rng.randint(12, 60),
                    n_T=_log_int(rng, 25, 200))
    while True:
        name, two_s, lo = rng.choice((("icosahedron", 1, 0), ("icosahedron", 2, 0), ("icosahedron", 3, 0),
                                      ("cuboctahedron", 1, 0), ("cuboctahedron", 2, 0), ("cuboctahedron", 3, 0),
                                      ("square:4x4", 1, 0), ("square:4x6:c2v", 1, 0), ("dodecahedron", 1, 0),
                                      ("dodecahedron", 2, 16), ("dodecahedron", 3, 28), ("icosidodecahedron", 1, 0)))
        n = cluster(name).n_sites
        two_M = 2 * rng.randint(lo // 2, max(lo // 2, n * two_s // 4))
        if n * two_s % 2:
            two_M += 1
        _, rhos = _symmetry(name)
        one = name not in SETS or rng.random() < 0.5
        irrep = rng.randrange(len(rhos)) if one else -1
        if _orbits(name, two_s, (n * two_s + two_M) // 2) < (60 if one else 12):
            continue  # smaller blocks may have no rows at all
        dtype = rng.choices(("f32", "f64", "f16"), (5, 3, 2))[0]
        table = rng.random() < 0.5
        c = dict(kind=kind, cluster=name, two_s=two_s, two_M=two_M, irrep=irrep, dtype=dtype)
        if kind == "hv":
            flip = two_M == 0 and one and rng.random() < 0.4
            api = "block" if one and dtype != "f16" and rng.random() < 0.4 else "packed"
            c.update(B=_log_int(rng, 1, 32), api=api, table=table, flip=flip)
            c["irrep"] = 2 * irrep + rng.randint(0, 1) if flip else irrep
        elif kind == "prepare":
            c.update(B=_log_int(rng, 1, 32), flip=False)
        else:
            # chains of blocks that hold many times their steps, as the campaigns' large sectors do
            c.update(sectors=1, R=rng.choice((1, 4, 24)), steps=rng.randint(8, 14),
                     rng=rng.choice(("gauss", "rademacher")), table=table)
            if not one and two_s * n >= 24:
                c["sectors"] = rng.randint(1, 4)
            if dtype == "f16" or _n_reps(c) < 1000:
                continue
        w = work(c)
        slow = 14 if dtype == "f64" else 1  # FP64 multiply-adds run at a fraction of the FP32 rate
        if kind == "lanczos":
            slow /= 4
        if w["bytes"] <= (1.5e10 if kind == "lanczos" else 4e9) and w["flops"] * slow <= 9e10 and _states(c) <= 2e9:
            return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# ---------------------------------------------------------------- group: closure, order, tabulated irreps


@functools.lru_cache(maxsize=None)
def _symmetry(name):
    """(permutations in canonical order, real-irreducible matrices in canonical irrep order) of a cluster's group."""
    gens = [tuple(int(v) for v in g) for g in cluster(name).gens]
    seen, todo = {tuple(range(len(gens[0])))}, [tuple(range(len(gens[0])))]
    while todo:
        p = todo.pop()
        for g in gens:
            q = tuple(g[k] for k in p)
            if q not in seen:
                seen.add(q)
                todo.append(q)
    perms = sorted(seen)
    index = {p: i for i, p in enumerate(perms)}
    G = len(perms)
    mult = np.array([[index[tuple(p[k] for k in q)] for q in perms] for p in perms])  # mult[g][h] = g h
    inv = np.argmax(mult == 0, axis=1)
    # a symmetric matrix commuting with the left regular representation: its eigenspaces are irreducible
    f = np.random.default_rng(7).standard_normal(G)
    f = f + f[inv]
    ev, Q = np.linalg.eigh(f[mult[inv]])
    found = {}
    for sel in np.split(np.arange(G), np.flatnonzero(np.diff(ev) > 1e-8) + 1):
        P = Q[:, sel] @ Q[:, sel].T
        basis = []
        for j in range(G):  # Gram-Schmidt over the projector's columns: independent of the solver's choice
            v = P[:, j].copy()
            for q in basis:
                v -= (q @ v) * q
            for q in basis:
                v -= (q @ v) * q
            if len(basis) < len(sel) and np.linalg.norm(v) > 1e-4:
                basis.append(v / np.linalg.norm(v))
        V = np.array(basis).T
        moved = np.empty((G,) + V.shape)
        for g in range(G):
            moved[g][mult[g]] = V  # (L(g) V)[g h] = V[h]
        rho = np.einsum("ha,ghb->gab", V, moved)
        chi = tuple(np.round(np.einsum("gaa->g", rho), 8) + 0.0)
        found.setdefault((rho.shape[1], tuple(-c for c in chi)), rho)
    return np.array(perms), [found[k] for k in sorted(found)]


def _group(name):
    c = cluster(name)
    g = F.ftlm_group_init(c.gens, c.bonds)
    F.ftlm_group_set_irreps(g, _symmetry(name)[1])
    return g


def _rhos(case):
    """Matrices [elements][d][d] of the case's blocks; with the spin flip the elements (g, 1) follow (g, 0)."""
    rhos = _symmetry(case["cluster"])[1]
    if case.get("flip"):
        rhos = [np.concatenate([r, s * r]) for r in rhos for s in (1.0, -1.0)]
    return rhos if case["irrep"] < 0 else [rhos[case["irrep"]]]


# ---------------------------------------------------------------- counts


def _bits(two_s):
    return max(1, math.ceil(math.log2(two_s + 1)))


@functools.lru_cache(maxsize=None)
def _ways(n, two_s):
    """Coefficients of (1 + x + ... + x^2s)^n as floats."""
    p = np.ones(1)
    for _ in range(n):
        p = np.convolve(p, np.ones(two_s + 1))
    return p


def _digit_sum(case, two_M=None):
    return (cluster(case["cluster"]).n_sites * case["two_s"] + (case["two_M"] if two_M is None else two_M)) // 2


def _states(case, two_M=None):
    return float(_ways(cluster(case["cluster"]).n_sites, case["two_s"])[_digit_sum(case, two_M)])


@functools.lru_cache(maxsize=None)
def _cycles(name):
    out = []
    for p in _symmetry(name)[0]:
        seen, lens = set(), []
        for k in range(len(p)):
            n = 0
            while k not in seen:
                seen.add(k)
                k = int(p[k])
                n += 1
            if n:
                lens.append(n)
        out.append(tuple(sorted(lens)))
    return out


@functools.lru_cache(maxsize=None)
def _orbits(name, two_s, total):
    """Orbits of the sector (Burnside)."""
    fixed = {}
    for lens in _cycles(name):
        if lens not in fixed:
            p = np.ones(1)
            for n in lens:
                q = np.zeros(n * two_s + 1)
                q[::n] = 1
                p = np.convolve(p, q)
            fixed[lens] = p[total]
    return sum(fixed[lens] for lens in _cycles(name)) / len(_cycles(name))


def _n_reps(case, two_M=None):
    n = _orbits(case["cluster"], case["two_s"], _digit_sum(case, two_M))
    return n / 2 if case.get("flip") else n


def _n_flips(case, two_M=None):
    """Ladder flips over the representatives: those of all states over the group order."""
    c = cluster(case["cluster"])
    a, s = _digit_sum(case, two_M), case["two_s"]
    rest = _ways(c.n_sites - 2, s)
    per_bond = sum(rest[a - i - j] for i in range(s) for j in range(1, s + 1) if 0 <= a - i - j < len(rest))
    G = len(_cycles(case["cluster"])) * (2 if case.get("flip") else 1)
    return 2.0 * c.n_bonds * per_bond / G


def _sectors(case):
    return [case["two_M"] + 2 * i for i in range(case.get("sectors", 1))]


def work(case):
    """Vectors, records (16 bytes) or entries (8 bytes a flip, 8 a representative) once; the contraction's flops."""
    if case["kind"] == "thermo":
        n = case["blocks"] * case["R"]
        return {"bytes": 16.0 * n * case["steps"] + 40.0 * case["n_T"],
                "flops": n * (30.0 * case["steps"] ** 2 + 12.0 * case["steps"] * case["n_T"])}
    dims = [r.shape[1] for r in _rhos(case)]
    W, dd, e = sum(dims), sum(d * d for d in dims), {"f64": 8, "f32": 4, "f16": 2}[case["dtype"]]
    by = fl = 0.0
    for two_M in _sectors(case):
        n, f = _n_reps(case, two_M), _n_flips(case, two_M)
        table = case["kind"] == "prepare" or case.get("table")
        tab = (8 * f + 24 * n) if table else 16 * n
        if case["kind"] == "lanczos":  # per step: u_j and u_{j-1} in, u_{j+1} out
            by += case["steps"] * (3 * n * W * case["R"] * e + tab)
            fl += case["steps"] * case["R"] * (2 * f * dd + 10 * n * W)
        else:
            B = case["B"]
            by += 2 * n * W * B * e + tab * (2 if case["kind"] == "prepare" else 1)
            fl += 2 * f * dd * B
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- preparation and the calls


def _sector(case, group, two_M=None):
    if case.get("flip"):
        return F.ftlm_build_sector_flip(group, case["two_s"])
    return F.ftlm_build_sector(group, case["two_s"], case["two_M"] if two_M is None else two_M)


def _set(case, sec):
    n = F.ftlm_sector_symmetry(sec)["n_irreps"]
    return F.ftlm_build_multiblock(sec, [case["irrep"]] if case["irrep"] >= 0 else list(range(n)))


def _normal(shape, dtype, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32).to(dtype)


def _stabilizers(masks):
    """(representatives with a nontrivial stabilizer, their 0/1 rows over the elements) from exported mask words."""
    order = np.bitwise_count(masks).sum(axis=1)
    rows = np.flatnonzero(order > 1)
    bits = (masks[rows][:, :, None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)
    return rows, bits.reshape(len(rows), 64 * masks.shape[1])


def _packed_input(case, n_reps, rows, stab, dtype, seed):
    """Random packed vectors [n_reps][W][B]: the segments of symmetric orbits lie in the projectors' range."""
    rhos = _rhos(case)
    x = _normal((n_reps, sum(r.shape[1] for r in rhos), case["B"]), torch.float32, seed)
    if len(rows):
        z = 0
        for P in _projectors(rhos, stab):
            d = P.shape[1]
            x[rows, z:z + d] = (P @ x[rows, z:z + d].double()).float()
            z += d
    return x.to(dtype)


def _projectors(rhos, stab):
    """P_k(r) = mean of rho_k over the stabilizer, per row of stab [n][elements]."""
    stab = stab.double()
    for r in rhos:
        t = torch.as_tensor(r, device=stab.device)
        P = (stab[:, :t.shape[0]] @ t.reshape(t.shape[0], -1)) / stab.sum(1, keepdim=True)
        yield P.reshape(-1, r.shape[1], r.shape[1])


def prepare(case, seed):
    if case["kind"] == "thermo":
        return {"case": case, "blocks": _thermo_blocks(case, seed), "T": _temperatures(case)}
    group = _group(case["cluster"])
    ft, tt = DTYPES[case["dtype"]]
    st = {"case": case, "group": group, "dtype": ft, "seed": seed}
    if case["kind"] == "lanczos":
        st["sectors"] = [_sector(case, group, m) for m in _sectors(case)]
        for s in st["sectors"]:
            if case["table"]:
                F.ftlm_sector_build_entries(s)
        if case["irrep"] >= 0:
            st["block"] = F.ftlm_build_block(st["sectors"][0], case["irrep"])
        else:
            st["sets"] = [_set(case, s) for s in st["sectors"]]
        return st
    sec = _sector(case, group)
    n = F.ftlm_sector_info(sec)["n_reps"]
    if case["kind"] == "hv" and case["api"] == "block":
        st["block"] = F.ftlm_build_block(sec, case["irrep"])
        st["x"] = _normal((F.ftlm_basis_info(st["block"])["dim"], case["B"]), tt, seed)
    else:
        rows, stab = _stabilizers(F.ftlm_sector_export(sec)[1])
        # element g of mask words 0-1 is (g, 0), of words 2-3 (g, 1): index g + z |G|
        stab = torch.as_tensor(stab.astype(np.float64), device=DEV)
        st["x"] = _packed_input(case, n, torch.as_tensor(rows, device=DEV), stab, tt, seed)
    st["y"] = torch.empty_like(st["x"])
    if case["kind"] == "hv":
        st["sector"] = sec
        if case["table"]:
            F.ftlm_sector_build_entries(sec)
        if case["api"] == "packed":
            st["set"] = _set(case, sec)
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "thermo":
        lnZ, E, C, chi, E0 = F.ftlm_thermo(st["blocks"], st["T"])
        return {"lnZ": lnZ, "E": E, "C": C, "chi": chi, "E0": E0}
    if case["kind"] == "hv":
        if case["api"] == "block":
            F.ftlm_hv(st["block"], st["dtype"], case["B"], st["x"], st["y"])
        else:
            F.ftlm_hv_packed(st["set"], st["dtype"], case["B"], st["x"], st["y"])
        return st["y"]
    if case["kind"] == "prepare":
        sec = _sector(case, st["group"])
        entries = F.ftlm_sector_build_entries(sec)
        mb = _set(case, sec)
        F.ftlm_hv_packed(mb, st["dtype"], case["B"], st["x"], st["y"])
        info = F.ftlm_sector_info(sec)
        return {"y": st["y"], "n_reps": info["n_reps"], "sector_dim": info["sector_dim"], "entries": entries}
    rng = F.GAUSS if case["rng"] == "gauss" else F.RADEMACHER
    if case["irrep"] >= 0:
        alpha, beta, steps = F.ftlm_lanczos(st["block"], st["dtype"], case["R"], case["steps"], st["seed"], 0, rng)
    else:
        n_sets, K = len(st["sets"]), len(_rhos(case))
        alpha, beta, steps = F.ftlm_lanczos_sets(st["sets"], st["dtype"], case["R"], case["steps"], st["seed"],
                                                 np.arange(n_sets * K).reshape(n_sets, K), rng)
    # the coefficients of chains on FP32 vectors are FP32 numbers handed over in float64 arrays
    t = np.float32 if case["dtype"] == "f32" else np.float64
    return {"alpha": alpha.astype(t), "beta": beta.astype(t), "steps": steps}


# ---------------------------------------------------------------- thermal sums


def _temperatures(case):
    return 0.02 * 5000.0 ** (np.arange(case["n_T"]) / max(1, case["n_T"] - 1))


def _thermo_blocks(case, seed):
    """Coefficients as chains of an s = 3/2 cluster give them: beta on a plateau that shrinks with M, little scatter."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["blocks"]):
        R, m = case["R"], case["steps"]
        short = min(m, 6 + 9 * i) if i < 4 else m  # the smallest blocks end early
        width = 13.0 * (1.0 - 0.03 * (i % 19))
        beta = width * (1.0 + 0.3 / (1.0 + np.arange(m))) + rng.normal(size=(R, m)) * 0.1
        alpha = 0.2 * (i % 10) + rng.normal(size=(R, m)) * 0.2
        alpha[:, short:] = 0
        beta[:, short:] = 0
        out.append(dict(two_M=2 * (i % 19), d_gamma=(1, 1, 3, 3, 3, 3, 4, 4, 5, 5)[i % 10], dim=100 + 37 * i,
                        alpha=alpha, beta=beta, steps=np.full(R, short, dtype=np.int32)))
    return out


def _exact_thermo(case, seed):
    T = _temperatures(case)[:, None]
    th, w, msq = [], [], []
    for b in _thermo_blocks(case, seed):
        m = int(b["steps"][0])
        A = np.zeros((case["R"], m, m))
        i = np.arange(m)
        A[:, i, i] = b["alpha"][:, :m]
        A[:, i[1:], i[:-1]] = b["beta"][:, :m - 1]
        ev, U = np.linalg.eigh(A)
        mult = 2.0 if b["two_M"] > 0 else 1.0
        th.append(ev.ravel())
        w.append((mult * b["d_gamma"] * b["dim"] / case["R"] * U[:, 0, :] ** 2).ravel())
        msq.append(np.full(ev.size, 0.25 * b["two_M"] ** 2))
    th, w, msq = np.concatenate(th), np.concatenate(w), np.concatenate(msq)
    E0 = th.min()
    z = w * np.exp(-(th - E0) / T)
    Z = z.sum(1)
    E = (z * th).sum(1) / Z
    C = (z * (th - E[:, None]) ** 2).sum(1) / Z / T[:, 0] ** 2
    return {"lnZ": np.log(Z) - E0 / T[:, 0], "E": E, "C": C, "chi": (z * msq).sum(1) / Z / T[:, 0], "E0": float(E0)}


# ---------------------------------------------------------------- exact: one sector from its definitions


class _Sector:
    """Representatives, stabilizers and flips of one S^z sector in plain 64-bit torch."""

    def __init__(self, case, two_M):
        c = cluster(case["cluster"])
        self.case, self.N, self.two_s, self.two_M = case, c.n_sites, case["two_s"], two_M
        self.bits, self.flip = _bits(case["two_s"]), bool(case.get("flip"))
        self.perms, self.bonds = _symmetry(case["cluster"])[0], c.bonds
        self.G = len(self.perms)
        self.flipc = sum(self.two_s << (self.bits * k) for k in range(self.N))
        self.rhos = [torch.as_tensor(r, device=DEV) for r in _rhos(case)]
        self._tables()
        self._representatives()

    def _tables(self):
        self.per = max(1, 12 // self.bits)  # sites per table
        self.starts = list(range(0, self.N, self.per))
        n = 1 << (self.bits * self.per)
        v = np.arange(n, dtype=np.int64)
        self.lut = np.zeros((self.G, len(self.starts), n), dtype=np.int64)
        for g in range(self.G):
            for t, k0 in enumerate(self.starts):
                for k in range(k0, min(k0 + self.per, self.N)):
                    d = (v >> (self.bits * (k - k0))) & ((1 << self.bits) - 1)
                    self.lut[g, t] |= d << (self.bits * int(self.perms[g][k]))
        self.lut = torch.as_tensor(self.lut, device=DEV)

    def images(self, n):
        """(element index, U(element) n) over all elements, the spin-flipped ones after G."""
        mask = (1 << (self.bits * self.per)) - 1
        parts = [(n >> (self.bits * k0)) & mask for k0 in self.starts]
        for z in range(2 if self.flip else 1):
            for g in range(self.G):
                v = self.lut[g, 0][parts[0]]
                for t in range(1, len(parts)):
                    v = v | self.lut[g, t][parts[t]]
                yield g + z * self.G, (self.flipc - v if z else v)

    def digit(self, n, k):
        return (n >> (self.bits * k)) & ((1 << self.bits) - 1)

    def _labels(self):
        """Labels of the sector in ascending order, in pieces: high half ascending, low halves of the missing sum."""
        total = (self.N * self.two_s + self.two_M) // 2
        n_lo = self.N // 2

        def halves(n):
            v = torch.zeros(1, dtype=torch.int64, device=DEV)
            s = v.clone()
            for k in range(n):
                d = torch.arange(self.two_s + 1, dtype=torch.int64, device=DEV)
                v = ((d[:, None] << (self.bits * k)) + v[None, :]).reshape(-1)
                s = (d[:, None] + s[None, :]).reshape(-1)
            return v, s

        lo, lo_sum = halves(n_lo)
        hi, hi_sum = halves(self.N - n_lo)
        order = torch.argsort(lo_sum, stable=True)  # ascending labels inside each sum
        lo = lo[order]
        count = torch.bincount(lo_sum, minlength=total + 1)
        first = torch.cumsum(count, 0) - count
        need = total - hi_sum
        ok = (need >= 0) & (need < count.numel())
        hi, need = hi[ok] << (self.bits * n_lo), need[ok]
        n = count[need]
        ends = torch.cumsum(n, 0)
        at = 0
        while at < hi.numel():
            base = int(ends[at - 1]) if at else 0
            to = max(at + 1, int(torch.searchsorted(ends, base + (1 << 25), right=True)))
            k = n[at:to]
            off = torch.arange(int(k.sum()), device=DEV) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
            yield torch.repeat_interleave(hi[at:to], k) + lo[torch.repeat_interleave(first[need[at:to]], k) + off]
            at = to

    def _representatives(self):
        kept = []
        for n in self._labels():
            mask = (1 << (self.bits * self.per)) - 1
            for z in range(2 if self.flip else 1):
                for g in range(self.G):
                    v = torch.zeros_like(n)
                    for t, k0 in enumerate(self.starts):
                        v |= self.lut[g, t][(n >> (self.bits * k0)) & mask]
                    if z:
                        v = self.flipc - v
                    n = n[v >= n]
            kept.append(n)
        self.reps = torch.cat(kept)
        self.n = self.reps.numel()
        size = torch.zeros(self.n, dtype=torch.int64, device=DEV)
        for lo in range(0, self.n, 1 << 22):
            r = self.reps[lo:lo + (1 << 22)]
            for _, v in self.images(r):
                size[lo:lo + r.numel()] += v == r
        self.rows = torch.nonzero(size > 1).reshape(-1)  # nontrivial stabilizers
        sub = self.reps[self.rows]
        self.stab = torch.stack([v == sub for _, v in self.images(sub)], 1).double() if sub.numel() else \
            torch.zeros((0, self.G), dtype=torch.float64, device=DEV)
        self.sqrtS = size.double().sqrt()
        self.P = list(_projectors([r.cpu().numpy() for r in self.rhos], self.stab))
        self.diag = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for i, j in self.bonds:
            self.diag += (self.digit(self.reps, int(i)) - 0.5 * self.two_s) * (self.digit(self.reps, int(j)) -
                                                                              0.5 * self.two_s)

    def flips(self):
        """(rows, target representatives, smallest minimising element, coefficient of Eq. 3), batch by batch."""
        s = 0.5 * self.two_s
        for lo in range(0, self.n, 1 << 20):
            n = self.reps[lo:lo + (1 << 20)]
            for i, j in self.bonds:
                for up, dn in ((int(i), int(j)), (int(j), int(i))):
                    mu, md = self.digit(n, up) - s, self.digit(n, dn) - s
                    ok = (mu < s) & (md > -s)
                    row = torch.nonzero(ok).reshape(-1)
                    if not row.numel():
                        continue
                    mu, md = mu[row], md[row]
                    a = n[row] + (1 << (self.bits * up)) - (1 << (self.bits * dn))
                    best = torch.full_like(a, torch.iinfo(torch.int64).max)
                    arg = torch.zeros_like(a)
                    for g, v in self.images(a):
                        less = v < best
                        best = torch.where(less, v, best)
                        arg = torch.where(less, torch.full_like(arg, g), arg)
                    c = 0.5 * torch.sqrt(s * (s + 1) - mu * (mu + 1)) * torch.sqrt(s * (s + 1) - md * (md - 1))
                    yield lo + row, torch.searchsorted(self.reps, best), arg, c

    def keep_flips(self):
        self._kept = list(self.flips())
        return self

    def apply(self, x):
        """H on lifted vectors [n][W][B] (Eqs. 15-16)."""
        y = torch.zeros_like(x)
        for row, tgt, g, c in getattr(self, "_kept", None) or self.flips():
            for lo in range(0, row.numel(), 1 << 18):
                t, gg = tgt[lo:lo + (1 << 18)], g[lo:lo + (1 << 18)]
                u = x[t] * (c[lo:lo + (1 << 18)] * self.sqrtS[t])[:, None, None]
                z, out = 0, []
                for r in self.rhos:
                    d = r.shape[1]
                    out.append((r[gg].unsqueeze(-1) * u[:, z:z + d].unsqueeze(2)).sum(1))  # rho(g*)^T u
                    z += d
                y.index_add_(0, row[lo:lo + (1 << 18)], torch.cat(out, 1))
        z = 0
        for P in self.P:
            d = P.shape[1]
            if self.rows.numel():
                y[self.rows, z:z + d] = (P @ y[self.rows, z:z + d]) / self.sqrtS[self.rows][:, None, None]
            z += d
        return y.addcmul_(self.diag[:, None, None], x)

    def columns(self, k):
        """(V [nontrivial][d][d], n_Gamma [n], row offsets [n]) of block k: Gram-Schmidt over the projector columns."""
        P = self.P[k]
        m, d = P.shape[0], self.rhos[k].shape[1]
        V = torch.zeros((m, d, d), dtype=torch.float64, device=DEV)
        count = torch.zeros(m, dtype=torch.int64, device=DEV)
        for j in range(d):
            v = P[:, :, j].clone()
            for q in range(d):
                v -= (V[:, :, q] * v).sum(1, keepdim=True) * V[:, :, q]
            nrm = v.norm(dim=1)
            ok = torch.nonzero(nrm > 1e-8).reshape(-1)
            V[ok, :, count[ok]] = v[ok] / nrm[ok, None]
            count[ok] += 1
        n_gamma = torch.full((self.n,), d, dtype=torch.int64, device=DEV)
        n_gamma[self.rows] = count
        return V, n_gamma, torch.cumsum(n_gamma, 0) - n_gamma

    def lift(self, k, value, B):
        """Lifted rows [n][d][B] of block k; value(rows) gives the block vector's entries [len(rows)][B]."""
        V, n_gamma, off = self.columns(k)
        d = self.rhos[k].shape[1]
        x = torch.empty((self.n, d, B), dtype=torch.float64, device=DEV)
        for q in range(d):
            x[:, q] = value(torch.clamp(off + q, max=max(0, int(n_gamma.sum()) - 1)))
            x[self.rows, q] *= (q < n_gamma[self.rows])[:, None]
        x[self.rows] = V @ x[self.rows]
        return x

    def lower(self, k, y):
        V, n_gamma, off = self.columns(k)
        out = torch.empty((int(n_gamma.sum()), y.shape[2]), dtype=torch.float64, device=DEV)
        y = y.clone()
        y[self.rows] = V.transpose(1, 2) @ y[self.rows]
        for q in range(y.shape[1]):
            ok = n_gamma > q
            out[off[ok] + q] = y[ok, q]
        return out


def _philox(row, chain, k0, k1, rng):
    """Start values of Section 2.2: Philox4x32-10 of (row, chain) under the key, Gaussian or +-1."""
    M = 0xFFFFFFFF
    shape = (row.shape[0], chain.shape[0])
    c = [(row & M)[:, None].expand(shape), (row >> 32)[:, None].expand(shape), chain[None, :].expand(shape),
         torch.zeros(shape, dtype=torch.int64, device=row.device)]

    def mulhilo(a, b):  # a: 32-bit constant
        p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
        lo = (p0 + ((p1 & 0xFFFF) << 16))
        return ((p1 >> 16) + (lo >> 32)) & M, lo & M

    for r in range(10):
        h0, l0 = mulhilo(0xD2511F53, c[0])
        h1, l1 = mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ ((k0 + r * 0x9E3779B9) & M), l1, h0 ^ c[3] ^ ((k1 + r * 0xBB67AE85) & M), l0]
    if rng == "rademacher":
        return 1.0 - 2.0 * (c[0] & 1).double()
    u1 = (((c[0] >> 5) << 26 | c[1] >> 6).double() + 0.5) * 2.0 ** -53
    u2 = ((c[2] >> 5) << 26 | c[3] >> 6).double() * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2)


def _exact_lanczos(case, seed):
    rhos = _rhos(case)
    R, m, K = case["R"], case["steps"], len(rhos)
    alpha = np.zeros((case["sectors"], K, R, m))
    beta = np.zeros_like(alpha)
    chain = torch.arange(R, device=DEV)
    for p, two_M in enumerate(_sectors(case)):
        sec = _Sector(case, two_M).keep_flips()
        v = torch.cat([sec.lift(k, lambda rows, k=k: _philox(rows, chain, seed & 0xFFFFFFFF, p * K + k, case["rng"]), R)
                       for k in range(K)], 1)
        cut = [0] + list(np.cumsum([r.shape[1] for r in rhos]))

        def dots(a, b):
            return torch.stack([(a[:, cut[k]:cut[k + 1]] * b[:, cut[k]:cut[k + 1]]).sum((0, 1)) for k in range(K)])

        def per_row(s):
            return torch.repeat_interleave(s, torch.as_tensor(np.diff(cut), device=DEV), 0)[None]

        v /= per_row(dots(v, v).sqrt())
        old, b = torch.zeros_like(v), torch.zeros((K, R), dtype=torch.float64, device=DEV)
        for j in range(m):
            w = sec.apply(v)
            a = dots(v, w)
            w -= per_row(a) * v + per_row(b) * old
            b = dots(w, w).sqrt()
            old, v = v, w / per_row(b)
            alpha[p, :, :, j], beta[p, :, :, j] = a.cpu().numpy(), b.cpu().numpy()
    if case["irrep"] >= 0:
        alpha, beta = alpha[0, 0], beta[0, 0]
    return {"alpha": alpha, "beta": beta, "steps": None}


def exact(case, seed):
    if case["kind"] == "thermo":
        return _exact_thermo(case, seed)
    if case["kind"] == "lanczos":
        return _exact_lanczos(case, seed)
    sec = _Sector(case, case["two_M"])
    tt = DTYPES[case["dtype"]][1]
    if case["kind"] == "hv" and case["api"] == "block":
        n_gamma = sec.columns(0)[1]
        x = _normal((int(n_gamma.sum()), case["B"]), tt, seed).double()
        return sec.lower(0, sec.apply(sec.lift(0, lambda rows: x[rows], case["B"])))
    x = _packed_input(case, sec.n, sec.rows, sec.stab, tt, seed).double()
    y = sec.apply(x)
    return y if case["kind"] == "hv" else {"y": y, "n_reps": None, "sector_dim": None, "entries": None}
