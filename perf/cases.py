"""Performance cases: the work that users of the library have it do, through its public entry points.

One real-time TDDFT step with numerical atomic orbitals builds the density matrix from the
coefficients, the density on the grid, the local Hamiltonian from the potential, propagates the
coefficients and, when the ions move, takes forces, the energy-density matrix, projector overlaps and
new neighbour lists; around it stand band structures (H(R), H(k)) and a serving loop that batches
systems of several sizes.  The listed cases take each of these calls at a size of the repository's own
workloads; draw() gives others of the same ranges.

    listed(), draw(rng), prepare(case, seed), run(state), work(case), exact(case, seed)

exact() evaluates the definitions (paper Eqs. 1-2 and Sec. 3.3.1-3.3.2) in float64 with plain torch
and numpy; it takes geometry and radial tables as data and none of the library's arithmetic.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2603_21835_gb300 import autograd as A
from paper_2603_21835_gb300 import gint as G
from paper_2603_21835_gb300 import inputs

DEV = "cuda"
F64 = torch.float64
DT = 0.05                      # propagation step (atomic time units)
MD_SKIN = 0.5                  # pair-set margin (Bohr) of the handle whose atoms move


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest system (8-atom cubic cell, images folded): launches and latency count
        dict(name="si8_rho_h", kind="rho_h", cells="1x1x1", grid="48x48x48", sigma=0.05),
        # the large production step: density and local H of 512 atoms in one call
        dict(name="si512_rho_h", kind="rho_h", cells="4x4x4", grid="192x192x192", sigma=0.05),
        # the backward direction: Pulay forces (and the density of the same pass)
        dict(name="si64_force", kind="force", cells="2x2x2", grid="96x96x96", sigma=0.1),
        # a molecule in vacuum: two species, 8-column atoms, many empty bricks; density, energy and
        # local H by separate calls as a self-consistency loop makes them
        dict(name="water32_scf", kind="water_scf", nmol=32, box=30.0, grid="144x144x144"),
        # a serving batch: five systems of different sizes, density + local H + forces, one call
        dict(name="batch_mixed", kind="batch", si="1x1x1 1x1x3 1x2x2", water="8 16", box=30.0,
             water_grid="144x144x144"),
        # band structure: H(R), then H(k) on a 2x2x2 mesh; a grid that is no multiple of anything
        dict(name="si64_hk", kind="hk", cells="2x2x2", grid="90x95x97", sigma=0.05, nk=8),
        # velocity-gauge projector overlaps, needed anew for every vector potential (float64)
        dict(name="si64_psibeta", kind="psibeta", cells="2x2x2", sigma=0.05),
        # density matrix of the 512-atom basis on the tensor cores
        dict(name="dm_mixed_6656", kind="dm_f16x3", n=6656, nocc=1024),
        # one propagation step and the new float64 density matrix, 64-atom basis
        dict(name="rt_step_832", kind="rt_step", n=832, nocc=128),
        # energy-density matrix for the overlap force, an odd size
        dict(name="edm_1601", kind="edm", n=1601),
        # float64 (the default precision): differentiable energy, forward and all three gradients
        dict(name="si8_fp64_grad", kind="fp64_grad", cells="1x1x1", grid="48x48x48", sigma=0.05),
        # ions move: new neighbour lists and the full pass set, two geometries in turn
        dict(name="si64_md", kind="md", cells="2x2x2", grid="96x96x96", sigma=0.05),
    ]


def _ints(text):
    return [int(x) for x in text.split("x")]


def _text(values):
    return "x".join(str(v) for v in values)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rho_h", "force", "water_scf", "batch", "hk", "psibeta", "dm_f16x3", "rt_step", "edm",
                       "fp64_grad", "md"])
    si_cells = ["1x1x1", "1x1x2", "1x1x3", "1x2x2", "1x2x3", "2x2x2", "1x3x3", "2x2x3", "2x3x3", "3x3x3"]

    def grid(cells, lo=47, hi=53):
        return _text(c * rng.randint(lo, hi) + rng.randint(0, 3) for c in _ints(cells))

    sigma = round(rng.uniform(0.01, 0.05), 3)
    if kind in ("rho_h", "force"):
        cells = rng.choice(si_cells)
        return dict(kind=kind, cells=cells, grid=grid(cells), sigma=sigma)
    if kind == "water_scf":
        return dict(kind=kind, nmol=rng.choice([4, 6, 8, 16, 32, 64]), box=30.0,
                    grid=_text(rng.randint(143, 153) for _ in range(3)))
    if kind == "batch":
        return dict(kind=kind, si=" ".join(rng.choice(si_cells[:5]) for _ in range(rng.randint(1, 4))),
                    water=" ".join(str(rng.choice([4, 6, 8, 16])) for _ in range(rng.randint(0, 2))), box=30.0,
                    water_grid=_text(rng.randint(132, 147) for _ in range(3)))
    if kind == "hk":
        cells = rng.choice(["1x1x1", "1x2x2", "2x2x2"])
        return dict(kind=kind, cells=cells, grid=grid(cells), sigma=sigma, nk=rng.randint(1, 8))
    if kind == "psibeta":
        return dict(kind=kind, cells=rng.choice(si_cells[:6]), sigma=sigma)
    if kind == "dm_f16x3":
        n = _log_int(rng, 100, 6656)
        return dict(kind=kind, n=n, nocc=max(1, int(n * rng.uniform(0.05, 0.16))))
    if kind == "rt_step":
        n = _log_int(rng, 104, 1500)
        return dict(kind=kind, n=n, nocc=max(1, int(n * rng.uniform(0.05, 0.2))))
    if kind == "edm":
        return dict(kind=kind, n=_log_int(rng, 104, 1601))
    if kind == "fp64_grad":
        cells = rng.choice(si_cells[:3])
        return dict(kind=kind, cells=cells, grid=grid(cells, 28, 48), sigma=sigma)
    cells = rng.choice(si_cells[:8])
    return dict(kind="md", cells=cells, grid=grid(cells), sigma=sigma)


# ------------------------------------------------------------------------------- systems and inputs
def _si_system(cells, grid, sigma, rng):
    sp = inputs.si_species()
    cell, pos = inputs.si_supercell(tuple(cells))
    pos = inputs.wrap_positions(cell, pos + rng.normal(0.0, sigma, pos.shape))
    return inputs.System(cell=cell, pos=pos, species=np.zeros(len(pos), np.int32), sp=[sp], grid=tuple(grid))


def _water_system(nmol, box, grid):
    # the serving pool's geometry of this size (V and D are drawn below)
    w = inputs.h2o_workload(nmol, 2000 + nmol, box, (8, 8, 8), dense_D=False)
    return dataclasses.replace(w.system, grid=tuple(grid))


def _systems(case):
    """The case's geometries (its own: block layouts follow from them; D, V and A come from the seed)."""
    rng = np.random.default_rng(11)
    if case["kind"] == "batch":  # one species list for all, as a batched launch wants it
        lib = inputs.serving_library()
        si = [_si_system(c, [48 * x for x in c], 0.05, rng) for c in map(_ints, case["si"].split())]
        wa = [_water_system(int(m), case["box"], _ints(case["water_grid"])) for m in case["water"].split()]
        return [inputs.on_species(s, lib) for s in si + wa]
    if case["kind"] == "water_scf":
        return [_water_system(case["nmol"], case["box"], _ints(case["grid"]))]
    return [_si_system(_ints(case["cells"]), _ints(case.get("grid", "8x8x8")), case["sigma"], rng)]


def _potential(sysm, rng):
    """20 periodic Gaussians (widths 1-3 Bohr) on the grid of an orthorhombic cell, float64, on the GPU."""
    L = np.diag(sysm.cell)
    cen, sig, amp = rng.random((20, 3)), rng.uniform(1.0, 3.0, 20), rng.normal(0.0, 0.5, 20)
    fac = []
    for d, n in enumerate(sysm.grid):
        x = np.arange(n)[None, :] / n * L[d] - cen[:, d:d + 1] * L[d]
        img = x[:, :, None] - np.arange(-2, 3) * L[d]
        fac.append(torch.from_numpy(np.exp(-img * img / (2 * sig[:, None, None] ** 2)).sum(-1)).to(DEV))
    a = torch.from_numpy(amp).to(DEV)
    return torch.einsum("g,gi,gj,gk->ijk", a, fac[0], fac[1], fac[2]).reshape(-1).contiguous()


def _dense_D(sysm, gen):
    """D = C C^T with one column per valence electron pair, on the GPU."""
    nocc = max(1, int(round(sum(inputs.OCCUPIED_PAIRS[sysm.sp[s].name] for s in sysm.species))))
    C = torch.randn(sysm.norb, nocc, dtype=F64, device=DEV, generator=gen) / 4
    D = C @ C.T
    return 0.5 * (D + D.T)


def _pairs(sysm, skin=0.0):
    """Atom pairs with an image closer than the sum of their supports (plus skin), sorted; their offsets."""
    rc = np.array([sysm.sp[s].rcut for s in sysm.species])
    no = np.array([sysm.sp[s].norb for s in sysm.species])
    lim = rc[:, None] + rc[None, :] + skin
    m = [int(math.ceil((2 * rc.max() + skin) / sysm.cell[d, d])) + 1 for d in range(3)]
    d0 = sysm.pos[None] - sysm.pos[:, None]
    best = np.full((len(rc), len(rc)), np.inf)
    for n in np.ndindex(*(2 * k + 1 for k in m)):
        x = d0 + (np.array(n) - m) @ sysm.cell
        best = np.minimum(best, np.einsum("ijc,ijc->ij", x, x))
    I, J = np.nonzero(np.sqrt(best) < lim)
    return I, J, np.concatenate([[0], np.cumsum(no[I] * no[J])])


def _block_index(sysm, I, J, off):
    """Flat index into the dense norb x norb matrix of every element of the pair blocks."""
    no = torch.tensor([sysm.sp[s].norb for s in sysm.species], device=DEV)
    ao = torch.cumsum(no, 0) - no
    I, J, off = (torch.as_tensor(x, device=DEV) for x in (I, J, off))
    p = torch.repeat_interleave(torch.arange(len(I), device=DEV), off[1:] - off[:-1])
    e = torch.arange(int(off[-1]), device=DEV) - off[p]
    nj = no[J[p]]
    return (ao[I[p]] + e // nj) * sysm.norb + ao[J[p]] + e % nj


def _grid_inputs(sysm, seed, k=0):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed * 1009 + k)
    return _dense_D(sysm, gen), _potential(sysm, np.random.default_rng([seed, k, 1]))


def _dense_inputs(case, seed):
    """Overlap and Hamiltonian of n localised functions at random centres (Gaussian decay, zero beyond
    14 Bohr, as between atoms whose supports do not touch), coefficients and occupations."""
    n, nocc = case["n"], case.get("nocc", max(1, case["n"] // 8))
    rng = np.random.default_rng(seed)
    L = (n / 13 * 135.0) ** (1 / 3)
    x = torch.from_numpy(rng.random((n, 3)) * L).to(DEV)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    out = {}
    if case["kind"] != "dm_f16x3":
        d2 = ((x[:, None] - x[None]) ** 2).sum(-1)
        K = torch.exp(-0.15 * d2) * (d2 < 196.0)
        R = torch.randn(n, n, dtype=F64, device=DEV, generator=gen)
        out["S"] = 0.8 * torch.eye(n, dtype=F64, device=DEV) + 0.2 * K
        H = 0.3 * K * (R + R.T)
        out["H"] = (H + torch.diag(torch.randn(n, dtype=F64, device=DEV, generator=gen))).contiguous()
    out["psi"] = torch.complex(*(torch.randn(nocc, n, dtype=F64, device=DEV, generator=gen) for _ in range(2))) / n**0.5
    out["f"] = 2.0 * torch.rand(nocc, dtype=F64, device=DEV, generator=gen)
    if case["kind"] == "edm":
        p = out.pop("psi")
        D = (p.conj() * out.pop("f")[:, None]).T @ p
        out["D"] = (0.5 * (D.real + D.real.T)).contiguous()
    return out


def _kpoints(nk):
    mesh = [(a, b, c) for a in (0.25, -0.25) for b in (0.25, -0.25) for c in (0.25, -0.25)]
    return np.array(mesh[:nk])


def _vector_potential(seed):
    return np.random.default_rng([seed, 3]).uniform(-0.15, 0.15, 3).tolist()


def _md_positions(sysm, seed):
    rng = np.random.default_rng([seed, 5])
    return [sysm.pos + rng.normal(0.0, 0.02, sysm.pos.shape) for _ in range(2)]


# ------------------------------------------------------------------------------------ prepare, run
def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind in ("dm_f16x3", "rt_step", "edm"):
        st.update(_dense_inputs(case, seed))
        st["cn"] = G.CrankNicolson(case["n"], case.get("nocc", 1))
        n = case["n"]
        st["out"] = torch.empty(n, n, dtype=F64, device=DEV)
        if kind == "rt_step":
            st["psi1"] = torch.empty_like(st["psi"])
        return st
    st["sys"] = systems = _systems(case)
    st["g"] = [G.Gint(s, skin=MD_SKIN if kind == "md" else 0.0) for s in systems]
    if kind == "psibeta":
        st["g"][0].set_projectors([inputs.si_projectors()])
        st["A"] = _vector_potential(seed)
        st["P"] = torch.empty(2 * st["g"][0].pb_nelems, dtype=F64, device=DEV)
        return st
    st["D"], st["V"], st["bufs"] = [], [], []
    for k, (s, g) in enumerate(zip(systems, st["g"])):
        D, V = _grid_inputs(s, seed, k)
        st["D"].append(D.reshape(-1)[_block_index(s, g.pair_IJ[:, 0], g.pair_IJ[:, 1], g.pair_off)].contiguous())
        st["V"].append(V)
        st["bufs"].append(tuple(torch.empty(m, dtype=F64, device=DEV) for m in (g.ngrid, g.nblock, (g.natoms, 3))))
    g = st["g"][0]
    if kind == "hk":
        g.layout_R()
        st["k"] = _kpoints(case["nk"])
        st["HR"] = torch.empty(g.nblock_R, dtype=F64, device=DEV)
        st["Hk"] = torch.empty(case["nk"] * 2 * g.nblock, dtype=F64, device=DEV)
    elif kind == "fp64_grad":
        st["pos"] = torch.from_numpy(systems[0].pos.copy()).to(DEV)
    elif kind == "md":
        st["pos"] = [torch.from_numpy(p).to(DEV) for p in _md_positions(systems[0], seed)]
        st["bufs"].append(tuple(torch.empty_like(b) for b in st["bufs"][0]))
    return st


def run(st):
    kind = st["kind"]
    if kind == "dm_f16x3":
        return st["cn"].density_matrix(st["psi"], st["f"], out=st["out"], precision="f16x3")
    if kind == "rt_step":
        psi1 = st["cn"].step(st["S"], st["H"], DT, st["psi"], out=st["psi1"])
        return [psi1, st["cn"].density_matrix(psi1, st["f"], out=st["out"])]
    if kind == "edm":
        return st["cn"].energy_density_matrix(st["S"], st["H"], st["D"], out=st["out"])
    g = st["g"][0]
    if kind == "psibeta":
        return g.psibeta(st["A"], out=st["P"])
    D, V = st["D"][0], st["V"][0]
    rho, H, F = st["bufs"][0]
    if kind == "rho_h":
        g.run(D, V, G.F16X3, rho=rho, H=H)
        return [rho, H]
    if kind == "force":
        return [g.force(D, V, G.F16X3, out=F, rho_out=rho), rho]
    if kind == "water_scf":
        g.rho(D, G.F16X3, out=rho)
        E = g.grid_dot(V, rho)
        g.vlocal(V, G.F16X3, out=H)
        return [rho, E, H]
    if kind == "batch":
        G.run_batch([G.Task(gg, D=d, V=v, rho=b[0], H=b[1], F=b[2])
                     for gg, d, v, b in zip(st["g"], st["D"], st["V"], st["bufs"])], G.F16X3)
        return [x for b in st["bufs"] for x in b]
    if kind == "hk":
        HR = g.vlocal_R(V, G.F16X3, out=st["HR"])
        return [HR, g.bloch(HR, st["k"], out=st["Hk"])]
    if kind == "fp64_grad":
        D, V, pos = (x.detach().requires_grad_() for x in (D, V, st["pos"]))
        E = A.grid_energy(g, D, V, pos)
        return [E.detach(), *torch.autograd.grad(E, (D, V, pos))]
    out = []
    for pos, (rho, H, F) in zip(st["pos"], st["bufs"]):  # md
        g.set_positions(pos)
        g.run(D, V, G.F16X3, rho=rho, H=H, F=F)
        out += [rho, H, F]
    return out


# -------------------------------------------------------------------------------------------- work
def _coverage(sysm):
    """W = sum over grid points of (orbitals covering the point)^2, from 1024 sampled points."""
    rng = np.random.default_rng(0)
    pts = rng.random((1024, 3)) @ sysm.cell
    n = np.zeros(1024)
    m = [int(math.ceil(max(s.rcut for s in sysm.sp) / sysm.cell[d, d])) for d in range(3)]
    for p, s in zip(sysm.pos, sysm.species):
        hit = np.zeros(1024, bool)
        for k in np.ndindex(*(2 * q + 1 for q in m)):
            hit |= ((pts - p - (np.array(k) - m) @ sysm.cell) ** 2).sum(-1) < sysm.sp[s].rcut ** 2
        n += hit * sysm.sp[s].norb
    return float(np.prod(sysm.grid)) * float((n * n).mean())


def work(case):
    kind = case["kind"]
    n, k = case.get("n", 0), case.get("nocc", 0)
    if kind == "dm_f16x3":  # D symmetric: n^2 / 2 products of length 2 nocc
        return dict(bytes=16 * n * k + 8 * k + 8 * n * n, flops=2.0 * n * n * k)
    if kind == "rt_step":
        return dict(bytes=8 * (3 * n * n) + 32 * n * k, flops=12.0 * n * n * k + 4 / 3 * n**3 + 2.0 * n * n * k)
    if kind == "edm":
        return dict(bytes=8 * 4 * n * n, flops=13 / 3 * n**3)
    nbytes = flops = 0.0
    for s in _systems(case):
        ng = float(np.prod(s.grid))
        if kind == "psibeta":
            # quadrature points times (13 orbitals from 5 radials, one phase, 2 radials x 13 complex sums)
            pairs, elems = _projector_pairs(s)
            nbytes += 16.0 * elems
            flops += pairs * 140 * 162 * 200.0
            continue
        nblk = float(_pairs(s, MD_SKIN if kind == "md" else 0.0)[2][-1])
        W = _coverage(s)  # one multiply-add per unordered pair and point for rho and for H, twice that for forces
        if kind in ("rho_h", "water_scf"):
            nbytes, flops = nbytes + 16 * (nblk + ng), flops + 2 * W
        elif kind == "force":
            nbytes, flops = nbytes + 8 * nblk + 16 * ng, flops + 2 * W
        elif kind == "batch":
            nbytes, flops = nbytes + 16 * (nblk + ng), flops + 3 * W
        elif kind == "md":
            nbytes, flops = nbytes + 2 * 16 * (nblk + ng), flops + 2 * 3 * W
        elif kind == "fp64_grad":
            nbytes, flops = nbytes + 16 * nblk + 16 * ng, flops + 4 * W
        else:
            nbytes, flops = nbytes + 8 * ng + 16 * nblk * case["nk"], flops + W + 4 * nblk * case["nk"]
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------- exact results (plain torch, float64)
def _radials(sp):
    """(l, rc, dr, f, f') of a species' radials with the tables on the GPU."""
    return [(r.l, r.rc, r.dr, torch.from_numpy(np.ascontiguousarray(r.f)).to(DEV),
             torch.from_numpy(np.ascontiguousarray(r.df)).to(DEV)) for r in sp.radials]


def _hermite(r, rc, dr, f, df):
    x = r / dr
    i = torch.clamp(x.floor().long(), max=len(f) - 2)
    t = x - i
    a, b, ga, gb = f[i], f[i + 1], df[i] * dr, df[i + 1] * dr
    val = a + (b - a) * t * t * (3 - 2 * t) + ga * t * (1 - t) ** 2 + gb * t * t * (t - 1)
    der = ((b - a) * 6 * t * (1 - t) + ga * (1 - t) * (1 - 3 * t) + gb * t * (3 * t - 2)) / dr
    inside = r < rc
    return torch.where(inside, val, 0.0), torch.where(inside, der, 0.0)


def _harmonics(l, u):
    """Real spherical harmonics (m = 0, +1, -1, +2, -2) as homogeneous polynomials of u, and gradients."""
    x, y, z = u.unbind(-1)
    o = torch.zeros_like(x)
    if l == 0:
        c = 0.5 / math.sqrt(math.pi)
        return [(o + c, (o, o, o))]
    if l == 1:
        c = o + math.sqrt(3 / (4 * math.pi))
        return [(c * z, (o, o, c)), (c * x, (c, o, o)), (c * y, (o, c, o))]
    c0, c1, c2 = (math.sqrt(v / math.pi) for v in (5 / 16, 15 / 4, 15 / 16))
    return [(c0 * (2 * z * z - x * x - y * y), (-2 * c0 * x, -2 * c0 * y, 4 * c0 * z)),
            (c1 * x * z, (c1 * z, o, c1 * x)), (c1 * y * z, (o, c1 * z, c1 * y)),
            (c2 * (x * x - y * y), (2 * c2 * x, -2 * c2 * y, o)), (c1 * x * y, (c1 * y, c1 * x, o))]


def _orbitals(rads, d, grad):
    """Orbitals at displacements d [..., 3]: [..., norb] (and gradients [..., norb, 3])."""
    r = d.norm(dim=-1)
    ir = torch.where(r > 1e-12, 1 / r, 0.0)
    u = d * ir[..., None]
    val, gra = [], []
    for l, rc, dr, f, df in rads:
        R, dR = _hermite(r, rc, dr, f, df)
        for Y, gY in _harmonics(l, u):
            val.append(R * Y)
            if grad:
                a = dR * Y - l * R * ir * Y
                gra.append(torch.stack([a * u[..., c] + R * ir * gY[c] for c in range(3)], -1))
    return torch.stack(val, -1), torch.stack(gra, -2) if grad else None


def _grid_exact(sysm, pos, D=None, V=None, want_rho=False, want_H=False, want_F=False, kfrac=None, nb=16):
    """rho, H (dense; [nk, norb, norb] complex when kfrac is given) and forces over blocks of nb^3 points:
    every (atom, image) whose support may reach the block has columns of its own."""
    cell = torch.from_numpy(sysm.cell).to(DEV)
    L = np.diag(sysm.cell)
    no = np.array([sysm.sp[s].norb for s in sysm.species])
    ao = np.cumsum(no) - no
    norb, w = int(no.sum()), abs(np.linalg.det(sysm.cell)) / float(np.prod(sysm.grid))
    rho = torch.zeros(sysm.grid, dtype=F64, device=DEV) if want_rho else None
    nk = 0 if kfrac is None else len(kfrac)
    H = None
    if want_H:
        H = torch.zeros(max(nk, 1) * norb * norb, dtype=torch.complex128 if nk else F64, device=DEV)
    F = torch.zeros(len(no), 3, dtype=F64, device=DEV) if want_F else None
    groups = []  # per species: radials, norb, image positions, atoms, lattice vectors
    for s, sp in enumerate(sysm.sp):
        at = np.nonzero(sysm.species == s)[0]
        if len(at) == 0:
            continue
        m = [int(math.ceil(sp.rcut / L[d])) + 1 for d in range(3)]
        n = np.array(list(np.ndindex(*(2 * q + 1 for q in m)))) - m
        T = (pos[at][:, None] + (n @ sysm.cell)[None]).reshape(-1, 3)
        keep = np.all((T > -sp.rcut) & (T < L + sp.rcut), axis=1)
        groups.append((_radials(sp), sp.norb, sp.rcut, T[keep], np.repeat(at, len(n))[keep],
                       np.tile(n, (len(at), 1))[keep]))
    Vg = V.reshape(sysm.grid) if V is not None else None
    axes = [np.arange(g) / g for g in sysm.grid]
    for i in range(0, sysm.grid[0], nb):
        for j in range(0, sysm.grid[1], nb):
            for k in range(0, sysm.grid[2], nb):
                box = [a[o:o + nb] for a, o in zip(axes, (i, j, k))]
                lo, hi = (np.array([b[e] for b in box]) * L for e in (0, -1))
                c, rad = 0.5 * (lo + hi), 0.5 * np.linalg.norm(hi - lo)
                fr = torch.from_numpy(np.stack(np.meshgrid(*box, indexing="ij"), -1).reshape(-1, 3)).to(DEV)
                pts = fr @ cell
                phi, gra, orb, img, atom = [], [], [], [], []
                for rads, nor, rc, T, at, n in groups:
                    q = np.nonzero(((T - c) ** 2).sum(1) < (rc + rad) ** 2)[0]
                    if len(q) == 0:
                        continue
                    v, gv = _orbitals(rads, pts[:, None] - torch.from_numpy(T[q]).to(DEV)[None], want_F)
                    phi.append(v.reshape(len(pts), -1))
                    if want_F:
                        gra.append(gv.reshape(len(pts), -1, 3))
                    orb.append((ao[at[q]][:, None] + np.arange(nor)).reshape(-1))
                    img.append(np.repeat(n[q], nor, axis=0))
                    atom.append(np.repeat(at[q], nor))
                if not phi:
                    continue
                sl = (slice(i, i + nb), slice(j, j + nb), slice(k, k + nb))
                phi = torch.cat(phi, 1)
                col = torch.from_numpy(np.concatenate(orb)).to(DEV)
                wv = (w * Vg[sl]).reshape(-1, 1) if V is not None else None
                if want_rho or want_F:
                    y = phi @ D[col][:, col]
                    if want_rho:
                        rho[sl] = (y * phi).sum(1).reshape(rho[sl].shape)
                    if want_F:
                        f = 2.0 * ((y * wv)[..., None] * torch.cat(gra, 1)).sum(0)
                        F.index_add_(0, torch.from_numpy(np.concatenate(atom)).to(DEV), f)
                if want_H:
                    t = (phi.T @ (phi * wv)).reshape(-1)
                    at2 = (col[:, None] * norb + col[None]).reshape(-1)
                    if not nk:
                        H.index_add_(0, at2, t)
                    else:
                        n = torch.from_numpy(np.concatenate(img).astype(np.float64)).to(DEV)
                        for q, kf in enumerate(kfrac):
                            ph = 2 * math.pi * (n @ torch.from_numpy(np.asarray(kf)).to(DEV))
                            z = torch.polar(torch.ones_like(ph), ph)
                            H.index_add_(0, at2 + q * norb * norb, t * (z.conj()[:, None] * z[None]).reshape(-1))
    return rho, H, F


def _projector_pairs(sysm):
    """(number of pairs, complex elements) of the projector overlaps of a Si system (4 x 13 blocks)."""
    n = len(_pairs_within(sysm, 2.5 + 7.0)[0])
    return n, 52 * n


def _pairs_within(sysm, reach):
    """Sorted (I, J) with an image of J closer than reach to I, and each pair's image positions."""
    L = np.diag(sysm.cell)
    m = [int(math.ceil(reach / L[d])) + 1 for d in range(3)]
    n = np.array(list(np.ndindex(*(2 * q + 1 for q in m)))) - m
    R = n @ sysm.cell
    I, J, img = [], [], []
    for a in range(len(sysm.pos)):
        for b in range(len(sysm.pos)):
            T = sysm.pos[b] + R
            T = T[((T - sysm.pos[a]) ** 2).sum(1) < reach * reach]
            if len(T):
                I.append(a)
                J.append(b)
                img.append(T)
    return I, J, img


def _psibeta_exact(sysm, avec):
    prj = inputs.si_projectors()
    rads, orb = _radials(prj), _radials(sysm.sp[0])
    x, wx = np.polynomial.legendre.leggauss(140)
    ct, wt = np.polynomial.legendre.leggauss(9)
    r, wr = 0.5 * (x + 1) * prj.rcut, 0.5 * wx * prj.rcut
    ph = 2 * np.pi * np.arange(18) / 18
    st = np.sqrt(1 - ct * ct)
    e = np.stack([st[:, None] * np.cos(ph), st[:, None] * np.sin(ph), np.repeat(ct[:, None], 18, 1)], -1).reshape(-1, 3)
    pts = torch.from_numpy((r[:, None, None] * e[None]).reshape(-1, 3)).to(DEV)
    wgt = torch.from_numpy(((wr * r * r)[:, None] * np.repeat(wt * 2 * np.pi / 18, 18)[None]).reshape(-1)).to(DEV)
    beta = (_orbitals(rads, pts, False)[0] * wgt[:, None]).T.contiguous()
    avec = torch.tensor(avec, dtype=F64, device=DEV)
    out = []
    for I, _, img in zip(*_pairs_within(sysm, prj.rcut + sysm.sp[0].rcut)):
        p = torch.from_numpy(sysm.pos[I]).to(DEV) + pts
        phi = sum(_orbitals(orb, p - torch.from_numpy(T).to(DEV), False)[0] for T in img)
        a = p @ avec
        out.append(torch.complex((beta * torch.cos(a)) @ phi, -(beta * torch.sin(a)) @ phi).reshape(-1))
    return torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dm_f16x3", "rt_step", "edm"):
        x = _dense_inputs(case, seed)
        if kind == "dm_f16x3":
            return _density(x["psi"], x["f"])
        if kind == "edm":
            X = torch.linalg.solve(x["S"], x["H"] @ x["D"])
            return 0.5 * (X + X.T)
        M = torch.complex(x["S"], 0.5 * DT * x["H"])
        psi1 = torch.linalg.solve(M, M.conj() @ x["psi"].T).T.contiguous()
        return [psi1, _density(psi1, x["f"])]
    systems = _systems(case)
    s = systems[0]
    if kind == "psibeta":
        return _psibeta_exact(s, _vector_potential(seed))
    out = []
    for k, s in enumerate(systems):
        D, V = _grid_inputs(s, seed, k)
        if kind == "hk":
            idx = _block_index(s, *_pairs(s))
            H = _grid_exact(s, s.pos, None, V, want_H=True, kfrac=_kpoints(case["nk"]))[1]
            return [None, H.reshape(case["nk"], -1)[:, idx]]  # H(R): keys depend on the grid blocks
        md = kind == "md"
        I, J, off = _pairs(s, MD_SKIN if md else 0.0)
        idx = _block_index(s, I, J, off)
        keep = torch.zeros(s.norb * s.norb, dtype=F64, device=DEV)
        keep[idx] = 1.0  # blocks of absent pairs are not stored
        Dk = (D.reshape(-1) * keep).reshape(s.norb, s.norb)
        for pos in (_md_positions(s, seed) if md else [s.pos]):
            rho, H, F = _grid_exact(s, pos, Dk, V, True, kind != "force",
                                    kind in ("force", "batch", "fp64_grad", "md"))
            H = H[idx] if H is not None else None
            rho = rho.reshape(-1)
            w = abs(np.linalg.det(s.cell)) / rho.numel()
            if kind == "rho_h":
                out += [rho, H]
            elif kind == "force":
                out += [F, rho]
            elif kind == "water_scf":
                out += [rho, (w * (rho * V).sum()).reshape(1), H]
            elif kind == "fp64_grad":
                out += [w * (rho * V).sum(), H, w * rho, -F]
            else:
                out += [rho, H, F]
    return out


def _density(psi, f):
    """Re(psi^T diag(f) conj(psi)), rows of psi the states."""
    a, b = psi.real, psi.imag
    return (a * f[:, None]).T @ a + (b * f[:, None]).T @ b
