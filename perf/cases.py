"""What a user of the library has it do, as measured cases.

Each case is one call (or, for `charge`, the short run of calls that belongs together) through the
public entry points of `paper_1003_4570_gb300.omen`, at the sizes of this repository's own
workloads: the 1,000,000-atom Si0.7Ge0.3 alloy, the delta-doped Si slabs, their Poisson grids.

    hx       y = (H - sigma) x, the product every Lanczos step repeats
    kbatch   the product of many Bloch wave vectors in one launch
    lowest   the lowest eigenpairs of an alloy block (thick-restart Lanczos)
    nearest  the states nearest an energy in the gap of a delta-doped slab (folded spectrum),
             the eigen-solve inside the Schroedinger-Poisson loop
    charge   electrons per atom from eigenvectors, their deposit on the Poisson grid, and the
             gather of a potential back to the atoms
    poisson  one solve of the finite-difference Poisson equation
    vff      a bounded valence-force-field relaxation and the bond strains it leaves
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1003_4570_gb300 import omen

A_NM = 0.5431                      # silicon lattice constant
GE_A_NM = 0.5658
GAP_VALENCE, GAP_CONDUCTION = -2.627017511981574, -1.6808215901542354   # of the gapped Si set
Q_E, EPS0 = 1.602176634e-19, 8.8541878128e-12
WALL, PERIODIC, BLOCH = 0, 1, 2
SITES = np.array([[0, 0, 0], [0, 2, 2], [2, 0, 2], [2, 2, 0], [1, 1, 1], [1, 3, 3], [3, 1, 3], [3, 3, 1]])
DIRS = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]])
PRECISION = {"f64": omen.OMEN_F64, "f32": omen.OMEN_F32, "refine": omen.OMEN_F32_REFINE64, "df": omen.OMEN_F64_DF}


def listed():
    return [
        # One product of the smallest slab of the self-consistent loop (1,280 complex rows): a call
        # whose time is its launch.
        hx("hx_slab_c128", (1, 1, 16), "slab", 10, "f64"),
        # The 1,000,000-atom alloy in FP64: the product of the paper's benchmark unit.
        hx("hx_alloy_f64", (50, 50, 50), "wall", 10, "f64"),
        # An alloy block of odd extents with FP32 vectors and stored blocks.
        hx("hx_alloy_f32", (37, 43, 41), "wall", 10, "f32"),
        # The 1,000,000-atom alloy without stored blocks, the option for the largest structures.
        hx("hx_alloy_matrix_free", (50, 50, 50), "wall", 10, "f32", matrix_free=True),
        # Spin-orbit rows (complex64 vectors, blocks of two for Kramers pairs) of a refined solve.
        hx("hx_spin_orbit_c64", (29, 31, 27), "wall", 10, "refine", spin_orbit=True, nvec=2),
        # 32 wave vectors of the 4x4x80-cell slab in one launch (k batching).
        kbatch("hx_kbatch_c64", (4, 4, 80), 32, "f32"),
        # 16 lowest eigenpairs of a 64,000-atom alloy block to 1e-9 eV.
        lowest("eigs_lowest_alloy", (20, 20, 20), "f64", 16, 96),
        # 8 states nearest an energy in the gap of the 1x1x16-cell slab: one step of the loop.
        nearest("eigs_nearest_slab", (1, 1, 16), 8, 48),
        # Charge of 16 states of 1,000,000 atoms, deposited and gathered on the 0.1 nm grid.
        charge("charge_alloy", (50, 50, 50), 16, (256, 256, 257)),
        # The Poisson grid of the 4x4x80-cell slab at the loop's tolerance.
        poisson("poisson_slab_grid", (11, 11, 217), "f64", 1e-13),
        # A device-sized grid with FP32 iterations and FP64 residuals.
        poisson("poisson_large_mixed", (256, 256, 257), "refine", 1e-10),
        # 100 conjugate-gradient steps of strain relaxation of 1,000,000 atoms.
        vff("vff_alloy", (50, 50, 50), 100),
    ]


def hx(name, cells, bc, basis, precision, matrix_free=False, spin_orbit=False, nvec=1):
    return dict(name=name, kind="hx", nx=cells[0], ny=cells[1], nz=cells[2], bc=bc, basis=basis, precision=precision,
                matrix_free=matrix_free, spin_orbit=spin_orbit, nvec=nvec)


def kbatch(name, cells, nk, precision):
    return dict(name=name, kind="kbatch", nx=cells[0], ny=cells[1], nz=cells[2], bc="slab", basis=10,
                precision=precision, spin_orbit=False, matrix_free=False, nk=nk)


def lowest(name, cells, precision, nev, basis_size):
    return dict(name=name, kind="lowest", nx=cells[0], ny=cells[1], nz=cells[2], bc="wall", basis=10,
                precision=precision, spin_orbit=False, matrix_free=False, nev=nev, basis_size=basis_size)


def nearest(name, cells, nev, basis_size):
    return dict(name=name, kind="nearest", nx=cells[0], ny=cells[1], nz=cells[2], bc="slab", basis=10, precision="f64",
                spin_orbit=False, matrix_free=False, nev=nev, basis_size=basis_size)


def charge(name, cells, nstates, grid):
    return dict(name=name, kind="charge", nx=cells[0], ny=cells[1], nz=cells[2], bc="wall", basis=10, precision="f64",
                spin_orbit=False, matrix_free=True, nstates=nstates, gx=grid[0], gy=grid[1], gz=grid[2])


def poisson(name, grid, precision, rtol):
    return dict(name=name, kind="poisson", gx=grid[0], gy=grid[1], gz=grid[2], precision=precision, rtol=rtol)


def vff(name, cells, steps):
    return dict(name=name, kind="vff", nx=cells[0], ny=cells[1], nz=cells[2], bc="wall", steps=steps)


def draw(rng):
    """A case of the same ranges: sizes over their logarithm, odd extents as likely as even ones."""
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def block(lo, hi):
        n = span(lo ** 3, hi ** 3) ** (1 / 3)
        c = [max(1, int(round(n * rng.uniform(0.8, 1.25)))) for _ in range(3)]
        while c[0] * c[1] * c[2] > hi ** 3:
            c[c.index(max(c))] -= 1
        return tuple(c)

    kind = rng.choice(["hx", "hx", "hx", "kbatch", "lowest", "nearest", "charge", "poisson", "poisson", "vff"])
    if kind == "hx":
        basis = rng.choice([5, 10, 10])
        if rng.random() < 0.3:
            c = hx("", (span(1, 4), span(1, 4), span(12, 80)), "slab", basis, rng.choice(["f64", "f32"]), nvec=rng.choice([1, 1, 3]))
        elif rng.random() < 0.3:
            c = hx("", block(4, 31), rng.choice(["wall", "periodic"]), basis, rng.choice(["refine", "f64"]), spin_orbit=True,
                   nvec=rng.choice([1, 2]))
        else:
            c = hx("", block(4, 50), rng.choice(["wall", "wall", "periodic"]), basis, rng.choice(["f64", "f32", "refine"]),
                   matrix_free=rng.random() < 0.3, nvec=rng.choice([1, 1, 2]))
            if c["nvec"] * c["nx"] * c["ny"] * c["nz"] > 125000:
                c["nvec"] = 1
    elif kind == "kbatch":
        c = kbatch("", (span(1, 4), span(1, 4), span(20, 80)), span(2, 32), rng.choice(["f32", "f64"]))
    elif kind == "lowest":
        c = lowest("", block(7, 20), rng.choice(["f64", "f64", "df"]), span(4, 16), 96)
    elif kind == "nearest":
        c = nearest("", (1, 1, span(8, 16)), span(4, 8), 48)
    elif kind == "charge":
        cells = block(8, 50)
        h = rng.uniform(0.1, 0.25)
        c = charge("", cells, span(4, 16), tuple(max(2, int(n * A_NM / h)) + d for n, d in zip(cells, (0, 0, 1))))
        while c["gx"] * c["gy"] * c["gz"] > 256 ** 3:
            c["gx"], c["gy"], c["gz"] = (int(c[k] * 0.95) for k in ("gx", "gy", "gz"))
    elif kind == "poisson":
        if rng.random() < 0.5:
            c = poisson("", (span(1, 16), span(1, 16), span(20, 240)), "f64", 1e-13)
        else:
            g = [span(24, 256) for _ in range(3)]
            c = poisson("", (g[0], g[1], g[2] + 1), "refine" if g[0] * g[1] * g[2] > 500_000 else rng.choice(["f64", "refine"]), 1e-10)
    else:
        c = vff("", block(6, 50), span(25, 100))
    del c["name"]
    return c


# ---- inputs -----------------------------------------------------------------------------

_CTX = []


def context():
    if not _CTX:
        _CTX.append(omen.omen_create(0, torch.cuda.current_stream().cuda_stream))
    return _CTX[0]


def generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def cells_of(case):
    return case["nx"] * case["ny"] * case["nz"]


def structure(case, seed):
    """Species, bond strains and boundaries: a strained Si0.7Ge0.3 alloy block, or an unstrained Si slab."""
    rng = np.random.default_rng([seed, 1])
    n = cells_of(case)
    slab = case["bc"] == "slab"
    species = np.zeros(8 * n, np.uint8) if slab else (rng.random(8 * n, dtype=np.float32) < 0.3).astype(np.uint8)
    strain = None if slab or case["kind"] in ("charge", "vff") else rng.uniform(-0.02, 0.02, 16 * n)
    per = {"wall": (WALL,) * 3, "periodic": (PERIODIC,) * 3, "slab": (BLOCH, BLOCH, WALL)}[case["bc"]]
    return SimpleNamespace(nx=case["nx"], ny=case["ny"], nz=case["nz"], periodic=per, a_nm=A_NM, species=species, strain=strain)


def parameters(case, seed):
    """Tight-binding parameters in the ranges of the repository's draws; slabs take its gapped Si set."""
    slab = case["bc"] == "slab"
    ns = 1 if slab else 2
    basis = case["basis"]
    g = np.random.default_rng(np.random.SeedSequence([163, 0])) if slab else np.random.default_rng([seed, 2])
    onsite, own, lam = np.zeros((ns, 4)), np.zeros((ns, 14)), np.zeros(ns)
    for s in range(ns):
        onsite[s] = [g.uniform(-6, -3), g.uniform(0, 3), g.uniform(3, 6), g.uniform(5, 8)]
        own[s] = g.uniform(-3, 3, size=14)
        lam[s] = g.uniform(0.01, 0.3)
    if basis == 5:
        onsite[:, 2] = 0.0
        own[:, [5, 6, 9, 10, 11, 12, 13]] = 0.0
    V = 0.5 * (own[:, None] + own[None, :])
    return SimpleNamespace(basis=basis, onsite=onsite, V=V, lambda_so=lam, eta=2.0)


def wave_vectors(case, seed, n):
    """Wave vectors of the slab's lateral zone (1/nm)."""
    rng = np.random.default_rng([seed, 3])
    k = np.zeros((n, 3))
    k[:, 0] = rng.uniform(0.05, 0.95, n) * math.pi / (case["nx"] * A_NM)
    k[:, 1] = rng.uniform(0.05, 0.95, n) * math.pi / (case["ny"] * A_NM)
    return k


def potential(case, seed):
    """Onsite potential energy per atom (eV): a screened sheet's well at mid-height and a few meV of disorder."""
    rng = np.random.default_rng([seed, 4])
    n = cells_of(case)
    cell = np.arange(n)
    z = (4.0 * (cell // (case["nx"] * case["ny"]))[None, :] + SITES[:, 2:3]) * (A_NM / 4)
    depth, length = rng.uniform(0.05, 0.3), rng.uniform(1.0, 5.0)
    u = -depth * np.exp(-np.abs(z - 0.5 * case["nz"] * A_NM) / length) + rng.uniform(-0.002, 0.002, z.shape)
    return torch.from_numpy(u.ravel()).cuda()


def is_complex(case):
    return case["spin_orbit"] or case["bc"] == "slab"


def vector_type(case):
    single = case["precision"] in ("f32", "refine")
    if is_complex(case):
        return torch.complex64 if single else torch.complex128
    return torch.float32 if single else torch.float64


def vectors(case, seed, n):
    """n vectors of components in [-1, 1]."""
    rows = 8 * cells_of(case) * case["basis"] * (2 if case["spin_orbit"] else 1)
    t = vector_type(case)
    part = torch.float32 if t in (torch.float32, torch.complex64) else torch.float64
    width = 2 if t.is_complex else 1
    x = torch.rand((n, rows * width), generator=generator(seed), device="cuda", dtype=part).mul_(2).sub_(1)
    return torch.view_as_complex(x.view(n, rows, 2)) if t.is_complex else x


def charge_density(case, seed):
    """A doping sheet at mid-height, its opposite charge spread wider, and the grain of single atoms (C/m^3)."""
    g = generator(seed)
    nz = case["gz"]
    z = torch.arange(1, nz, device="cuda", dtype=torch.float64) / nz - 0.5
    a, b, c = torch.rand(3, generator=g, device="cuda", dtype=torch.float64).tolist()
    sheet = 1e6 * (1 + a) * (torch.exp(-(z / (0.02 + 0.03 * b)) ** 2) - 0.3 * torch.exp(-(z / (0.08 + 0.05 * c)) ** 2))
    grain = torch.rand((nz - 1, case["gy"], case["gx"]), generator=g, device="cuda", dtype=torch.float64)
    return (sheet[:, None, None] + 1e6 * (grain - 0.5)).contiguous()


def grid_of(case, lengths=None):
    l = lengths or (case["gx"] * 0.2, case["gy"] * 0.2, case["gz"] * 0.2)
    return SimpleNamespace(nx=case["gx"], ny=case["gy"], nz=case["gz"], Lx_nm=l[0], Ly_nm=l[1], Lz_nm=l[2], eps_r=11.7)


def block_grid(case):
    return grid_of(case, (case["nx"] * A_NM, case["ny"] * A_NM, case["nz"] * A_NM))


def vff_constants():
    per = 1.0 / 1.602176634e-19 * 1e-18     # 1 N/m in eV/nm^2
    return SimpleNamespace(a_nm=np.array([A_NM, GE_A_NM]), alpha=np.array([48.5, 38.7]) * per, beta=np.array([13.8, 11.4]) * per)


def prepare(case, seed):
    ctx, kind = context(), case["kind"]
    s = SimpleNamespace(case=case, ctx=ctx)
    if kind == "poisson":
        s.grid = grid_of(case)
        s.rho = charge_density(case, seed)
        s.phi = torch.empty_like(s.rho)
        return s
    s.lat = omen.omen_build_lattice(ctx, structure(case, seed))
    if kind == "vff":
        s.constants = vff_constants()
        s.u = torch.empty((3, 8 * cells_of(case)), dtype=torch.float64, device="cuda")
        s.strain = torch.empty(16 * cells_of(case), dtype=torch.float64, device="cuda")
        s.start = torch.rand(s.u.shape, generator=generator(seed), device="cuda", dtype=torch.float64).sub_(0.5).mul_(2e-3)
        return s
    p = parameters(case, seed)
    k = wave_vectors(case, seed, 1)[0] if case["bc"] == "slab" else None
    s.u = potential(case, seed)
    s.ham = omen.omen_assemble_H(ctx, s.lat, p, spin_orbit=case["spin_orbit"], precision=PRECISION[case["precision"]],
                                 matrix_free=case["matrix_free"], k=k, U_atom_dev=s.u)
    if kind == "hx":
        s.x = vectors(case, seed, case["nvec"])
        s.y = torch.empty_like(s.x)
    elif kind == "kbatch":
        s.k = wave_vectors(case, seed, case["nk"])
        s.x = vectors(case, seed, case["nk"])
        s.y = torch.empty_like(s.x)
    elif kind == "charge":
        n = 8 * cells_of(case)
        s.grid = block_grid(case)
        s.psi = torch.rand((case["nstates"], 10 * n), generator=generator(seed), device="cuda", dtype=torch.float64)
        s.psi.sub_(0.5).mul_(math.sqrt(12.0 / (10 * n)))
        s.occ = np.linspace(1.0, 0.05, case["nstates"])
        s.density = torch.empty(n, dtype=torch.float64, device="cuda")
        s.rho = torch.empty((case["gz"] - 1, case["gy"], case["gx"]), dtype=torch.float64, device="cuda")
        s.phi = charge_density(case, seed + 1).mul_(1e-7)
        s.phi_atom = torch.empty(n, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case, ctx = s.case, s.ctx
    kind = case["kind"]
    if kind == "hx":
        omen.omen_hx(ctx, s.ham, s.x, s.y, nvec=case["nvec"], sigma=0.125)
        return s.y
    if kind == "kbatch":
        omen.omen_hx_kbatch(ctx, s.ham, s.k, s.x, s.y, sigma=0.125)
        return s.y
    if kind == "lowest":
        return omen.omen_eigs(ctx, s.ham, case["nev"], omen.OMEN_LOWEST, tol=1e-9, block=1, basis=case["basis_size"],
                              max_iter=20000)[0]
    if kind == "nearest":
        return omen.omen_eigs(ctx, s.ham, case["nev"], omen.OMEN_NEAREST, sigma=gap_energy(), tol=1e-9, block=1,
                              basis=case["basis_size"], max_iter=200000)[0]
    if kind == "charge":
        s.density.zero_()
        omen.omen_density_accum(ctx, s.ham, s.psi, case["nstates"], s.occ, 2.0, s.density)
        omen.omen_deposit(ctx, s.lat, s.grid, s.density * -Q_E, s.rho)
        omen.omen_gather(ctx, s.lat, s.grid, s.phi, s.phi_atom)
        return {"density": s.density, "rho": s.rho, "phi_atom": s.phi_atom}
    if kind == "poisson":
        s.phi.zero_()
        omen.omen_poisson(ctx, s.grid, s.rho, s.phi, rtol=case["rtol"], precision=PRECISION[case["precision"]])
        return s.phi
    s.u.copy_(s.start)
    info, _ = omen.omen_relax_vff(ctx, s.lat, s.constants, s.u, max_iter=case["steps"], strain_dev=s.strain, raise_on_noconv=False)
    return {"u": s.u, "strain": s.strain, "energy": info["energy"]}


def gap_energy():
    return GAP_CONDUCTION - 0.4 * (GAP_CONDUCTION - GAP_VALENCE)


# ---- least work ---------------------------------------------------------------------------

def work(case):
    """Inputs read once and outputs written once; operations of the plain definition."""
    kind = case["kind"]
    if kind == "poisson":
        n = case["gx"] * case["gy"] * (case["gz"] - 1)
        return {"bytes": 16.0 * n, "flops": 10.0 * n}
    cells = cells_of(case)
    atoms, bonds = 8 * cells, 16 * cells
    if kind == "vff":
        return {"bytes": float(case["steps"]) * atoms * 8 * 18, "flops": float(case["steps"]) * atoms * 700}
    rows = atoms * case["basis"] * (2 if case["spin_orbit"] else 1)
    if kind == "charge":
        nodes = case["gx"] * case["gy"] * (case["gz"] - 1)
        return {"bytes": 8.0 * (rows * case["nstates"] + 2 * atoms + 2 * nodes), "flops": 2.0 * rows * case["nstates"] + 80.0 * atoms}
    single = case["precision"] in ("f32", "refine")
    word = 4 if single else 8
    wide = 2 if is_complex(case) else 1
    per = rows * wide * word * 2.0
    fixed = bonds * word + atoms * 9.0
    flops = 2.0 * wide * rows * (4 * case["basis"] + 1)
    if kind == "hx":
        return {"bytes": fixed + per * case["nvec"], "flops": flops * case["nvec"]}
    if kind == "kbatch":
        return {"bytes": fixed + per * case["nk"], "flops": flops * case["nk"]}
    # a solve: some 500 products for the lowest levels, some 2,500 for a folded solve, and one pass
    # over half the basis for each
    steps = 500 if kind == "lowest" else 2500
    return {"bytes": steps * (fixed + per + 0.5 * case["basis_size"] * per), "flops": steps * (flops + 2.0 * case["basis_size"] * rows * wide)}


# ---- the same in 64 bits, in plain torch --------------------------------------------------

def sk_block(u, v12, v21, basis):
    """<atom 1 a|H|atom 2 b> for the bond direction u: the block of a bond along z, its orbitals rotated.
    V12 (V21): two-centre integrals with the first-named orbital on atom 1 (atom 2)."""
    def orbitals(r):
        x, y, z = r.T
        q = math.sqrt(3.0)
        d = [q * y * z, q * z * x, q * x * y, 0.5 * q * (x * x - y * y), z * z - 0.5 * (x * x + y * y)]
        return np.stack([np.ones_like(x), x, y, z] + (d if basis == 10 else []), axis=1)

    u = np.asarray(u, float) / np.linalg.norm(u)
    t = np.array([1.0, 0.0, 0.0]) if abs(u[0]) < 0.5 else np.array([0.0, 1.0, 0.0])
    e1 = np.cross(t, u)
    e1 /= np.linalg.norm(e1)
    frame = np.stack([e1, np.cross(u, e1), u])                # rows: the bond frame's axes
    r = np.random.default_rng(0).normal(size=(60, 3))
    r /= np.linalg.norm(r, axis=1, keepdims=True)
    rot = np.linalg.lstsq(orbitals(r), orbitals(r @ frame.T), rcond=None)[0]
    full = np.zeros((basis, basis))
    full[:basis - 1, :basis - 1] = rot                        # s, p, [d]
    full[-1, -1] = 1.0                                        # s*
    b = np.zeros((basis, basis))
    s, px, py, pz, e = 0, 1, 2, 3, basis - 1
    b[s, s], b[e, e], b[s, e], b[e, s] = v12[0], v12[1], v12[2], v21[2]
    b[s, pz], b[e, pz], b[pz, s], b[pz, e] = v12[3], v12[4], -v21[3], -v21[4]
    b[pz, pz], b[px, px], b[py, py] = v12[7], v12[8], v12[8]
    if basis == 10:
        yz, zx, xy, xx, zz = 4, 5, 6, 7, 8
        b[s, zz], b[e, zz], b[zz, s], b[zz, e] = v12[5], v12[6], v21[5], v21[6]
        b[pz, zz], b[zz, pz] = v12[9], -v21[9]
        b[px, zx] = b[py, yz] = v12[10]
        b[zx, px] = b[yz, py] = -v21[10]
        b[zz, zz], b[zx, zx], b[yz, yz], b[xy, xy], b[xx, xx] = v12[11], v12[12], v12[12], v12[13], v12[13]
    return full @ b @ full.T


def exact_product(case, seed, x, k, sigma):
    """(H - sigma) x for x [n, rows] in float64 or complex128; k: [3], or [n, 3] for one wave vector a row."""
    st, p = structure(case, seed), parameters(case, seed)
    basis, n = case["basis"], cells_of(case)
    spins = 2 if case["spin_orbit"] else 1
    nv = x.shape[0]
    x = x.view(nv, spins, basis, 8, n)
    species = torch.from_numpy(st.species.astype(np.int64)).cuda().view(8, n)
    strain = torch.zeros(16 * n, dtype=torch.float64, device="cuda") if st.strain is None else torch.from_numpy(st.strain).cuda()
    scale = (1.0 + strain).pow(-p.eta).view(4, 4, n)
    per_orbital = [0, 1, 1, 1] + ([2] * 5 if basis == 10 else []) + [3]
    onsite = torch.from_numpy(p.onsite[:, per_orbital]).cuda()
    diag = onsite[species].permute(2, 0, 1) + potential(case, seed).view(8, n)[None] - sigma
    y = x * diag[None, None]
    if case["spin_orbit"]:
        lam = torch.from_numpy(p.lambda_so).cuda()[species]
        pauli = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
        eps = np.zeros((3, 3, 3))
        for a, b, c in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
            eps[a, b, c], eps[a, c, b] = 1, -1
        for s1 in range(2):
            for s2 in range(2):
                m = torch.from_numpy(np.einsum("k,kab->ab", pauli[:, s1, s2], -1j * eps)).cuda()
                y[:, s1, 1:4] += torch.einsum("ab,vbsc->vasc", m, x[:, s2, 1:4]) * lam
    ns = p.onsite.shape[0]
    blocks = torch.from_numpy(np.array([[[sk_block(DIRS[d], p.V[i, j], p.V[j, i], basis) for d in range(4)] for j in range(ns)]
                                        for i in range(ns)])).cuda()
    cell = torch.arange(n, device="cuda")
    at = [cell % case["nx"], (cell // case["nx"]) % case["ny"], cell // (case["nx"] * case["ny"])]
    ext = (case["nx"], case["ny"], case["nz"])
    kk = None if k is None else torch.from_numpy(np.asarray(k, float).reshape(-1, 3)).cuda()
    for s in range(4):
        for d in range(4):
            target = SITES[s] + DIRS[d]
            off = np.floor_divide(target, 4)
            site = int(np.nonzero((SITES == target - 4 * off).all(axis=1))[0][0])
            ok = torch.ones(n, dtype=torch.bool, device="cuda")
            to, turn = [], torch.zeros((n, 3), dtype=torch.float64, device="cuda")
            for a in range(3):
                t = at[a] + int(off[a])
                out = (t < 0) | (t >= ext[a])
                if st.periodic[a] == WALL:
                    ok &= ~out
                elif st.periodic[a] == BLOCH:
                    turn[:, a] = torch.where(t < 0, -1.0, 0.0) + torch.where(t >= ext[a], 1.0, 0.0)
                to.append(t % ext[a])
            src = cell[ok]
            dst = ((to[2] * ext[1] + to[1]) * ext[0] + to[0])[ok]
            f = scale[d, s][ok]
            phase = None
            if kk is not None:
                length = torch.tensor([e * A_NM for e in ext], dtype=torch.float64, device="cuda")
                angle = kk @ (turn[ok] * length).T
                phase = torch.polar(torch.ones_like(angle), angle)[:, None, None, :]
            xa, xb = x[:, :, :, s][..., src], x[:, :, :, site][..., dst]
            if phase is not None:
                xb, xa = xb * phase, xa * phase.conj()
            sa, sb = species[s][src], species[site][dst]
            ya, yb = torch.zeros_like(xb), torch.zeros_like(xa)
            for i in range(ns):
                for j in range(ns):
                    g = torch.where((sa == i) & (sb == j), f, 0.0)
                    m = blocks[i, j, d].to(x.dtype)
                    ya += torch.einsum("ab,vqbc->vqac", m, xb * g)
                    yb += torch.einsum("ba,vqbc->vqac", m, xa * g)
            y[:, :, :, s].index_add_(3, src, ya)
            y[:, :, :, site].index_add_(3, dst, yb)
    return y.reshape(nv, -1)


def exact_levels(case, seed):
    rows = 8 * cells_of(case) * case["basis"]
    if rows > 5200:
        return None
    k = wave_vectors(case, seed, 1)[0] if case["bc"] == "slab" else None
    t = torch.complex128 if is_complex(case) else torch.float64
    e = torch.linalg.eigvalsh(exact_product(case, seed, torch.eye(rows, dtype=t, device="cuda"), k, 0.0).T)
    if case["kind"] == "lowest":
        return e[:case["nev"]].cpu().numpy()
    near = (e - gap_energy()).abs().argsort()[:case["nev"]]
    return e[near].sort().values.cpu().numpy()


def exact_poisson(case, seed):
    g = grid_of(case)
    b = charge_density(case, seed) / (EPS0 * g.eps_r)
    lam = []
    for n, length in ((g.nx, g.Lx_nm), (g.ny, g.Ly_nm)):
        j = torch.arange(n, device="cuda", dtype=torch.float64)
        lam.append(4 * torch.sin(math.pi * j / n) ** 2 / (length / n * 1e-9) ** 2)
    m = torch.arange(1, g.nz, device="cuda", dtype=torch.float64)
    sine = torch.sin(torch.outer(m, m) % (2 * g.nz) * (math.pi / g.nz))
    lz = 4 * torch.sin(math.pi * m / (2 * g.nz)) ** 2 / (g.Lz_nm / g.nz * 1e-9) ** 2
    f = torch.fft.fft2((sine @ b.view(g.nz - 1, -1)).view(b.shape))
    f /= lz[:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    return (sine @ torch.fft.ifft2(f).real.reshape(g.nz - 1, -1)).view(b.shape) * (2.0 / g.nz)


def exact_charge(case, seed):
    n, cells = 8 * cells_of(case), cells_of(case)
    g = block_grid(case)
    psi = torch.rand((case["nstates"], 10 * n), generator=generator(seed), device="cuda", dtype=torch.float64)
    psi.sub_(0.5).mul_(math.sqrt(12.0 / (10 * n)))
    density = torch.zeros(n, dtype=torch.float64, device="cuda")
    for f, v in zip(np.linspace(1.0, 0.05, case["nstates"]), psi):
        density += 2.0 * f * v.view(10, n).square().sum(0)
    cell = torch.arange(cells, device="cuda")
    ix = torch.stack([cell % case["nx"], (cell // case["nx"]) % case["ny"], cell // (case["nx"] * case["ny"])])
    pos = (4 * ix[:, None, :] + torch.from_numpy(SITES.T.copy()).cuda()[:, :, None]).reshape(3, n).double() * (A_NM / 4)
    h = torch.tensor([g.Lx_nm / g.nx, g.Ly_nm / g.ny, g.Lz_nm / g.nz], dtype=torch.float64, device="cuda")
    t = pos / h[:, None]
    lo = t.floor()
    frac, lo = t - lo, lo.long()
    nodes = torch.zeros((g.nz + 1) * g.ny * g.nx, dtype=torch.float64, device="cuda")
    padded = torch.zeros((g.nz + 1, g.ny, g.nx), dtype=torch.float64, device="cuda")
    padded[1:-1] = charge_density(case, seed + 1).mul_(1e-7)
    phi_atom = torch.zeros(n, dtype=torch.float64, device="cuda")
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                at = ((lo[2] + dz).clamp(0, g.nz) * g.ny + (lo[1] + dy) % g.ny) * g.nx + (lo[0] + dx) % g.nx
                w = 1.0
                for a, up in ((0, dx), (1, dy), (2, dz)):
                    w = w * (frac[a] if up else 1 - frac[a])
                nodes.index_add_(0, at, w * density * -Q_E)
                phi_atom += w * padded.view(-1)[at]
    rho = nodes.view(g.nz + 1, g.ny, g.nx)[1:-1] / float(h.prod() * 1e-27)
    return {"density": density, "rho": rho, "phi_atom": phi_atom}


def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        return exact_poisson(case, seed)
    if kind == "charge":
        return exact_charge(case, seed)
    if kind in ("lowest", "nearest"):
        return exact_levels(case, seed)
    if kind == "vff":
        return None                  # a path of many steps: no closed value
    if kind == "kbatch":
        x, k = vectors(case, seed, case["nk"]), wave_vectors(case, seed, case["nk"])
    else:
        x, k = vectors(case, seed, case["nvec"]), wave_vectors(case, seed, 1)[0] if case["bc"] == "slab" else None
    return exact_product(case, seed, x.to(torch.complex128 if x.is_complex() else torch.float64), k, 0.125)
