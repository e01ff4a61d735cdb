"""The work that a user of this library has it do, as cases to be measured.

A program that runs pole expansion and selected inversion keeps one plan per
sparsity pattern (the ordering and the device memory) and calls it with new
H and S: once per SCF cycle, k-point, chemical potential or MD step. So a
case's geometry fixes the pattern and the plan, which `prepare` keeps for
as long as cases of that geometry follow one another, and the seed gives the
values of H and S. The systems are the synthetic ones that the tests and the
benchmark use: chains, honeycomb sheets and water-like fluids of atoms with
4 to 13 orbitals, with exponentially decaying blocks inside a cutoff.

Keys of a case: `op` (the entry point), `kind`, `size` and `norb` (the
system), `table` (poles of the expansion), `first` and `poles` (the subrange
of it that the pass evaluates; a rank of a pole-parallel program takes such a
subrange), `split` (slices of the split-precision path, 0 = FP64), `batch`
(poles per device batch), `overlap` (False: S = I).
"""
import functools
import math

import numpy as np
import torch

from paper_1405_0194_gb300 import capi as px

BOHR = 1.0 / 0.529177210903
DELTA_E = 2.5  # half-width that covers the spectra of these systems, centred at MU
MU = 0.0
DEV = "cuda"


def listed():
    return [
        # one shift of a small molecule from host arrays (LDOS at one energy): the smallest call, latency
        dict(name="ldos_fluid24", op="selinv", kind="fluid", size=24, norb=0, table=2, first=0, poles=1, split=0, batch=1,
             overlap=True),
        # the whole 40-pole density matrix of the tiny chain: launches and short serial chains
        dict(name="dm_chain64", op="dm", kind="chain", size=64, norb=4, table=40, first=0, poles=40, split=0, batch=40,
             overlap=True),
        # a long thin system: many small fronts, many poles at once
        dict(name="dm_chain500", op="dm", kind="chain", size=500, norb=4, table=64, first=0, poles=64, split=0, batch=64,
             overlap=True),
        # an ordinary molecular system, part of its poles
        dict(name="dm_fluid96", op="dm", kind="fluid", size=96, norb=0, table=60, first=50, poles=8, split=0, batch=8,
             overlap=True),
        # a 2D sheet: wide separators, uneven tree
        dict(name="dm_sheet14", op="dm", kind="sheet", size=14, norb=13, table=60, first=40, poles=4, split=0, batch=4,
             overlap=True),
        # one pole of the benchmark's system: the largest FP64 work
        dict(name="dm_fluid512", op="dm", kind="fluid", size=512, norb=0, table=60, first=50, poles=1, split=0, batch=1,
             overlap=True),
        # the same system on the split-precision path, a batch of poles
        dict(name="dm_fluid512_split", op="dm", kind="fluid", size=512, norb=0, table=60, first=44, poles=8, split=6,
             batch=8, overlap=True),
        # inertia counts that bracket the chemical potential: real shifts, no selected inversion
        dict(name="inertia_fluid256", op="inertia", kind="fluid", size=256, norb=0, table=0, first=0, poles=16, split=0,
             batch=8, overlap=True),
        # the same on the split-precision path
        dict(name="inertia_sheet16_split", op="inertia", kind="sheet", size=16, norb=13, table=0, first=0, poles=8,
             split=6, batch=4, overlap=True),
        # a k-point or spin-orbit calculation: complex Hermitian H and S
        dict(name="herm_fluid64", op="herm", kind="fluid", size=64, norb=0, table=60, first=48, poles=6, split=0, batch=6,
             overlap=True),
        # the chain, the fluid and the sheet of that size side by side in one set of launches
        dict(name="group_small_split", op="group", kind="mixed", size=8, norb=0, table=64, first=40, poles=16, split=6,
             batch=16, overlap=True),
        # Tr[DM S], Tr[EDM S], Tr[FDM S] of stored matrices, inside another program's capture or loop
        dict(name="trace_fluid512", op="trace", kind="fluid", size=512, norb=0, table=0, first=0, poles=0, split=0, batch=1,
             overlap=True),
    ]


def draw(rng):
    """Another case of these ranges."""
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["selinv", "dm", "dm", "dm", "inertia", "herm", "group", "trace"])
    c = dict(op=op, kind=rng.choice(["chain", "fluid", "sheet"]), size=0, norb=0, table=0, first=0, poles=0, split=0, batch=1,
             overlap=op not in ("selinv", "inertia") or rng.random() < 0.7)
    # poles that cost no more than the largest listed case, by the size of the system's dense separators
    if c["kind"] == "chain":
        c["size"], c["norb"], most = between(20, 2000), rng.choice([3, 4, 5, 7]), 40
    elif c["kind"] == "fluid":
        c["size"] = between(12, 256)
        most = max(2, min(24, int(600 * (60.0 / c["size"]) ** 2.3)) // (2 if op == "herm" else 1))
        most = min(most, 3) if c["size"] > 150 else most
    else:
        c["size"], c["norb"] = between(4, 14), rng.choice([11, 13])
        most = max(2, min(24, int(24 * (8.0 / c["size"]) ** 3.5)))
    if op in ("dm", "inertia", "group"):
        c["split"] = rng.choice([0, 6])
    if op == "group":
        c.update(kind="mixed", size=rng.randint(4, 10), norb=0)
        most = 8
    if op == "selinv":
        c.update(table=2, poles=1)
    elif op == "inertia":
        c.update(poles=rng.randint(2, most + 2))
    elif op != "trace":
        c.update(table=2 * rng.randint(10, 32), poles=rng.randint(1, most))
        c["poles"] = min(c["poles"], c["table"])
        c["first"] = rng.randint(0, c["table"] - c["poles"])
    c["batch"] = max(1, c["poles"] if rng.random() < 0.7 else (c["poles"] + 1) // 2)
    return c


# ---------------------------------------------------------------- systems
def _positions(kind, size, norb):
    """Atom positions, orbitals per atom, cutoff, decay length, lattice (rows) or None, beta."""
    if kind == "chain":
        pos = np.zeros((size, 3))
        pos[:, 0] = 2.5 * np.arange(size)
        return pos, np.full(size, norb), 6.0, 2.0, None, 1000.0
    if kind == "sheet":
        a = 1.42 * math.sqrt(3.0) * BOHR
        a1, a2 = np.array([a, 0.0, 0.0]), np.array([0.5 * a, 0.5 * math.sqrt(3.0) * a, 0.0])
        i, j, b = np.meshgrid(np.arange(size), np.arange(size), np.arange(2), indexing="ij")
        pos = (i[..., None] * a1 + j[..., None] * a2 + b[..., None] * (a1 + a2) / 3.0).reshape(-1, 3)
        lattice = np.stack([size * a1, size * a2, np.array([0.0, 0.0, 1.0e6])])
        return pos, np.full(pos.shape[0], norb), 8.0 * BOHR, 3.0, lattice, 2000.0
    box, n = 46.9 * (size / 512.0) ** (1.0 / 3.0), 3 * size
    rng = np.random.default_rng(1000 + size)
    pos, k = np.zeros((n, 3)), 0
    while k < n:  # at least 2 bohr apart
        cand = rng.uniform(0.0, box, size=3)
        d = pos[:k] - cand
        d -= box * np.round(d / box)
        if k == 0 or np.min(np.einsum("ij,ij->i", d, d)) >= 4.0:
            pos[k] = cand
            k += 1
    return pos, np.array([13] * size + [5] * (2 * size)), 10.0, 3.0, np.diag([box, box, box]), 1000.0


@functools.lru_cache(maxsize=4)
def _pattern(kind, size, norb):
    """The CSC pattern and, per entry on the device, its distance factor, the entry that gives its value and its sign."""
    pos, no, cutoff, lam, lattice, beta = _positions(kind, size, norb)
    first = np.concatenate([[0], np.cumsum(no)])
    n, inv = int(first[-1]), None if lattice is None else np.linalg.inv(lattice)
    colptr, rows, decay = [np.zeros(1, np.int64)], [], []
    for J in range(pos.shape[0]):
        d = pos - pos[J]
        if lattice is not None:
            f = d @ inv
            d = (f - np.round(f)) @ lattice
        r = np.sqrt(np.einsum("ij,ij->i", d, d))
        near = np.nonzero(r <= cutoff)[0]
        rl = np.concatenate([np.arange(first[i], first[i + 1]) for i in near])
        dl = np.repeat(np.where(near == J, 0.0, np.exp(-r[near] / lam)), no[near])
        rows.append(np.tile(rl, no[J]))
        decay.append(np.tile(dl, no[J]))
        colptr.append(colptr[-1][-1:] + rl.size * np.arange(1, no[J] + 1))
    colptr, rows = np.concatenate(colptr).astype(np.int64), np.concatenate(rows).astype(np.int32)
    r = torch.from_numpy(rows).to(DEV).long()
    c = torch.from_numpy(np.repeat(np.arange(n), np.diff(colptr))).to(DEV)
    transposed = torch.argsort(r * n + c)  # the pattern is symmetric: entry of (c, r) for each (r, c)
    e = torch.arange(r.numel(), device=DEV)
    source = torch.where(r <= c, e, transposed)
    return dict(n=n, colptr=colptr, rowind=rows, beta=beta, r=r, c=c, source=source,
                lengths=torch.from_numpy(np.diff(colptr)).to(DEV),
                decay=torch.from_numpy(np.concatenate(decay)).to(DEV), sign=torch.sign(c - r).double())


def _values(pat, seed, hermitian):
    """H and S on the pattern: on-site blocks of H in [-1, 1] with 0.1 N(0, 1) couplings, pair blocks N(0, 1) exp(-d / lam);
    S diagonally dominant."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    r, c, src, decay = pat["r"], pat["c"], pat["source"], pat["decay"]
    nnz = r.numel()

    def normal():
        return torch.randn(nnz, generator=g, device=DEV, dtype=torch.float64)

    on_site, diag = decay == 0.0, r == c
    h = (normal() * torch.where(on_site, 0.1, decay))[src]
    h = torch.where(diag, 2.0 * torch.rand(nnz, generator=g, device=DEV, dtype=torch.float64) - 1.0, h)
    s = (0.05 * normal() * decay)[src]
    if hermitian:
        h = torch.complex(h, pat["sign"] * (0.2 * normal())[src] * h.abs())
        s = torch.complex(s, pat["sign"] * (0.1 * normal())[src] * s.abs())
    row_sum = torch.segment_reduce(s.abs() * ~diag, "sum", lengths=pat["lengths"])  # column by column, always in one order
    s = torch.where(diag, (1.1 + row_sum)[c].to(s.dtype), s)
    return h.contiguous(), s.contiguous()


def _systems(case):
    """(kind, size, norb) of each system of a case."""
    if case["op"] == "group":
        k = case["size"]
        return [("chain", 60 * k + 20, 4), ("fluid", k * k, 0), ("sheet", k, 13)]
    return [(case["kind"], case["size"], case["norb"])]


class _Plan:
    """A plan or a group, released with its last user."""

    def __init__(self, case):
        opts = px.pexsi_opts_default(max_batch=int(case["batch"]), split_slices=int(case["split"]))
        host = px.pexsi_opts_default(device=-1)
        pats = [_pattern(*s) for s in _systems(case)]
        self.group = case["op"] == "group"
        plans = [px.pexsi_setup(p["n"], p["colptr"], p["rowind"], opts=host if self.group else opts) for p in pats]
        self.handle = px.pexsi_group_create(plans, opts) if self.group else plans[0]
        if self.group:
            for p in plans:
                px.pexsi_plan_destroy(p)

    def __del__(self):
        (px.pexsi_group_destroy if self.group else px.pexsi_plan_destroy)(self.handle)


_kept = {}


def _plan(case):
    key = (case["op"] == "group", tuple(_systems(case)), case["batch"], case["split"])
    if key not in _kept:
        _kept.clear()  # one geometry at a time
        _kept[key] = _Plan(case)
    return _kept[key]


def prepare(case, seed):
    systems = []
    for k, key in enumerate(_systems(case)):
        pat = _pattern(*key)
        h, s = _values(pat, 1000003 * k + seed, case["op"] == "herm")
        systems.append(dict(pat=pat, H=h, S=s if case["overlap"] else None, out=[torch.zeros_like(h) for _ in range(3)]))
    st = dict(case=case, systems=systems)
    op, one = case["op"], systems[0]
    if op == "trace":
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 7)
        one["out"] = [torch.randn(one["H"].numel(), generator=g, device=DEV, dtype=torch.float64) for _ in range(3)]
        st["traces"] = torch.zeros(3, device=DEV, dtype=torch.float64)
        return st
    st["plan"] = _plan(case)
    rng = np.random.default_rng(seed)
    if op == "inertia":  # shifts over the middle of the spectrum
        st["shifts"] = np.sort(rng.uniform(-0.8, 0.8, case["poles"]))
    if op == "selinv":
        st["host"] = [None if x is None else x.cpu().numpy() for x in (one["H"], one["S"])]
        st["z"] = complex(rng.uniform(-0.5, 0.5), 0.01)
    torch.cuda.synchronize()
    return st


def run(st):
    case, systems = st["case"], st["systems"]
    op, one = case["op"], systems[0]
    stream = torch.cuda.current_stream().cuda_stream

    def addr(x):
        return 0 if x is None else x.data_ptr()

    if op == "trace":
        px.pexsi_trace_noalloc(*[addr(x) for x in one["out"]], addr(one["S"]), one["H"].numel(), addr(st["traces"]), stream)
        return st["traces"]
    h = st["plan"].handle
    if op == "selinv":
        return px.pexsi_selinv(h, *st["host"], st["z"])
    if op == "inertia":
        return px.pexsi_inertia_device(h, addr(one["H"]), addr(one["S"]), st["shifts"], stream)
    lo, hi = case["first"], case["first"] + case["poles"]
    if op == "group":
        k = len(systems)
        px.pexsi_group_dm_device(h, [addr(s["H"]) for s in systems], [addr(s["S"]) for s in systems], [MU] * k,
                                 [s["pat"]["beta"] for s in systems], case["table"], [DELTA_E] * k, lo, hi, 0,
                                 *[[addr(s["out"][q]) for s in systems] for q in range(3)], stream=stream)
        return [s["out"] for s in systems]
    call = px.pexsi_dm_hermitian_device if op == "herm" else px.pexsi_dm_device
    call(h, addr(one["H"]), addr(one["S"]), MU, one["pat"]["beta"], case["table"], DELTA_E, lo, hi, 0,
         *[addr(x) for x in one["out"]], stream=stream)
    return one["out"]


@functools.lru_cache(maxsize=64)
def _counts(kind, size, norb):
    """nnz and the flops of one pole's factorisation and selected inversion over the front structure (complex symmetric)."""
    pat = _pattern(kind, size, norb)
    plan = px.pexsi_setup(pat["n"], pat["colptr"], pat["rowind"], opts=px.pexsi_opts_default(device=-1))
    st = px.pexsi_plan_get_stats(plan)
    px.pexsi_plan_destroy(plan)
    return st["nnz"], st["factor_gemm_flops"], st["selinv_gemm_flops"]


def work(case):
    out = dict(bytes=0.0, flops=0.0)
    for key in _systems(case):
        nnz, factor, selinv = _counts(*key)
        values = 2 if case["overlap"] else 1
        if case["op"] == "trace":
            out["bytes"] += 32.0 * nnz
            out["flops"] += 6.0 * nnz
        elif case["op"] == "inertia":  # real arithmetic: 2 flops per multiply-add instead of 8
            out["bytes"] += 8.0 * nnz * values
            out["flops"] += case["poles"] * factor / 4.0
        elif case["op"] == "selinv":
            out["bytes"] += 8.0 * nnz * values + 16.0 * nnz
            out["flops"] += factor + selinv
        else:
            wide = 2 if case["op"] == "herm" else 1
            out["bytes"] += 8.0 * nnz * wide * (values + 3)
            out["flops"] += wide * case["poles"] * (factor + selinv)
    return out


# ---------------------------------------------------------------- 64-bit values
def _elliptic(u, k, k1):
    """sn, cn, dn of real u for modulus k (complementary modulus k1), by the arithmetic-geometric mean and descending Landen
    steps (Abramowitz and Stegun 16.4)."""
    a, c, b = [np.longdouble(1)], [np.longdouble(k)], np.longdouble(k1)
    while c[-1] > 1e-19 and len(a) < 40:
        a0 = a[-1]
        a.append((a0 + b) / 2)
        c.append((a0 - b) / 2)
        b = np.sqrt(a0 * b)
    phi = (2.0 ** (len(a) - 1)) * a[-1] * u
    for q in range(len(a) - 1, 0, -1):
        phi = (phi + np.arcsin(c[q] / a[q] * np.sin(phi))) / 2
    s, co = np.sin(phi), np.cos(phi)
    return s, co, np.sqrt(co * co + (np.longdouble(k1) * s) ** 2)


def _agm(b):
    a = np.longdouble(1)
    for _ in range(60):
        a, b = (a + b) / 2, np.sqrt(a * b)
    return a


def _poles(beta, n):
    """Shifts and the three weight sets of the n-pole expansion at (MU, beta, DELTA_E): the trapezoidal rule on the conformal
    map of Hale, Higham and Trefethen for xi = x^2 + (pi / beta)^2, in extended precision."""
    ld = np.longdouble
    pi = 4 * np.arctan(ld(1))
    beta = ld(beta)
    m = (pi / beta) ** 2
    M = ld(DELTA_E) ** 2 + m
    q = np.sqrt(M / m)
    k, k1 = (q - 1) / (q + 1), 2 * np.sqrt(q) / (q + 1)
    K, Kp = pi / (2 * _agm(k1)), pi / (2 * _agm(k))
    h = 4 * K / n
    x = -K + (np.arange(1, n + 1) - ld(0.5)) * h
    s, c, d = _elliptic(x, k, k1)
    s1, c1, d1 = _elliptic(np.full(n, Kp / 2), k1, k)
    den = c1 * c1 + k * k * s * s * s1 * s1
    i = np.clongdouble(1j)
    sn, cn, dn = (s * d1 + i * c * d * s1 * c1) / den, (c * c1 - i * s * d * s1 * d1) / den, (d * c1 * d1 - i * k * k * s * c * s1) / den
    root = np.sqrt(m * M)
    x = np.sqrt(root * (1 / k + sn) / (1 / k - sn) - m)
    w = -h * root * (2 / k) * cn * dn / (1 / k - sn) ** 2 / (4 * i * pi * x)

    def fermi(y):
        e = np.exp(-beta * np.where(y.real >= 0, y, -y))
        return np.where(y.real >= 0, 2 * e / (1 + e), 2 / (1 + e))

    def grand(y):
        right = y.real >= 0
        return -(2 / beta) * (np.log(1 + np.exp(-beta * np.where(right, y, -y))) - np.where(right, 0, beta * y))

    y = np.concatenate([x, -x])
    sgn = np.concatenate([-w, w])
    up = y.imag > 0
    y, sgn = y[up], 2 * i * sgn[up]
    f = fermi(y)
    return [v.astype(np.complex128) for v in (y + MU, sgn * f, sgn * (y + MU) * f, sgn * grand(y))]


def _inverse_on_pattern(s, z):
    pat = s["pat"]
    n, dt = pat["n"], torch.complex128
    A = torch.zeros(n, n, device=DEV, dtype=dt)
    over = (pat["r"] == pat["c"]).to(dt) if s["S"] is None else s["S"].to(dt)
    A[pat["r"], pat["c"]] = s["H"].to(dt) - complex(z) * over
    return torch.linalg.inv(A)


def exact(case, seed):
    op = case["op"]
    size = max(_pattern(*k)["n"] for k in _systems(case))
    if op == "inertia" or (op != "trace" and max(1, case["poles"]) * float(size) ** 3 > 6e11):
        return None  # whole numbers; or dense inverses that would take too long
    systems = []
    for k, key in enumerate(_systems(case)):
        pat = _pattern(*key)
        h, s = _values(pat, 1000003 * k + seed, op == "herm")
        systems.append(dict(pat=pat, H=h, S=s if case["overlap"] else None))
    one = systems[0]
    if op == "trace":
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 7)
        return torch.stack([torch.sum(torch.randn(one["H"].numel(), generator=g, device=DEV, dtype=torch.float64) * one["S"])
                            for _ in range(3)])
    if op == "selinv":
        G = _inverse_on_pattern(one, complex(np.random.default_rng(seed).uniform(-0.5, 0.5), 0.01))
        return G[one["pat"]["r"], one["pat"]["c"]].cpu().numpy()
    outs = []
    for s in systems:
        z, *weights = _poles(s["pat"]["beta"], case["table"])
        r, c = s["pat"]["r"], s["pat"]["c"]
        out = [torch.zeros_like(s["H"]) for _ in range(3)]
        for p in range(case["first"], case["first"] + case["poles"]):
            G = _inverse_on_pattern(s, z[p])
            up, down = G[r, c], G[c, r].conj()
            for o, w in zip(out, weights):
                wp = complex(w[p])
                if op == "herm":
                    o += (wp * up - wp.conjugate() * down) / 2j
                else:
                    o += (wp * up).imag
        outs.append(out)
    return outs if op == "group" else outs[0]
