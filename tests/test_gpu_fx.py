"""Float64 density, force and local-H passes on exact digit products, over the forms their kernels tell apart:
orbital counts of a brick that are no multiple of the 16-, 64- and 128-column tiles, atoms across a tile edge,
every compiled orbital shape and the general evaluator, radials that end early, atoms on grid points, ragged and
one-brick grids, empty bricks, bricks of more than 512 columns (the CUDA-core kernels), infinities and NaNs.
Tolerances of the float64 path: 1e-12 of the largest element for rho and H, 1e-11 for F, against the oracle."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2603_21835_gb300 import inputs
from tests.test_gpu_psibeta_shapes import ORB, _shorter, _sp

pytestmark = pytest.mark.gpu


def _system(names, nat, box, grid, on_grid=False):
    rng = np.random.default_rng(nat)
    sp = []
    for n in names:
        s = _sp(n, ORB[n.split()[0]])
        sp.append(_shorter(s, 1, 3.3337) if n.endswith("short") else s)
    cell = np.diag([box, box * 1.1, box * 0.95])
    frac = rng.random((nat, 3))
    if on_grid:
        frac = np.floor(frac * grid) / grid
    return inputs.System(cell=cell, pos=frac @ cell, species=(np.arange(nat) % len(names)).astype(np.int32), sp=sp, grid=grid)


@pytest.mark.parametrize("names,nat,box,grid,on_grid", [
    (("100",), 1, 11.0, (4, 4, 8), False), (("110",), 3, 15.0, (11, 9, 13), False), (("221", "110"), 9, 12.0, (8, 8, 8), False),
    (("221", "100"), 17, 12.0, (8, 5, 16), False), (("111", "210"), 6, 10.0, (12, 8, 8), True), (("unsorted",), 5, 13.0, (8, 8, 8), True),
    (("dd", "grids"), 7, 10.0, (8, 8, 8), False), (("221 short", "111 short"), 6, 9.0, (8, 8, 9), False),
    (("221",), 2, 40.0, (20, 20, 24), False), (("221",), 34, 10.0, (4, 8, 8), False), (("221",), 44, 10.0, (4, 8, 8), False)])
def test_passes_match_the_oracle(names, nat, box, grid, on_grid):
    import torch

    from paper_2603_21835_gb300 import gint as G

    s = _system(names, nat, box, grid, on_grid)
    rng = np.random.default_rng(nat + 1)
    o = Oracle(s)
    C = rng.normal(size=(o.norb, 5)) / 4
    D = C @ C.T
    V = rng.normal(size=int(np.prod(grid)))
    rho_o, H_o, F_o = o.rho(D).reshape(-1), o.vlocal(V), o.force(D, V)
    g = G.Gint(s)
    Db, Vd = torch.from_numpy(g.dense_to_blocks(D)).cuda(), torch.from_numpy(V).cuda()
    for _ in range(2):  # again: the scratch holds the last call's
        rho = g.rho(Db, G.FP64).cpu().numpy().reshape(-1)
        if nat < 44:
            H = g.blocks_to_dense(g.vlocal(Vd, G.FP64).cpu().numpy())
        else:  # more than 453 orbitals in a brick: refused in float64
            with pytest.raises(G.GintError):
                g.vlocal(Vd, G.FP64)
            H = H_o
        F = g.force(Db, Vd, G.FP64)
        F = (F[0] if isinstance(F, tuple) else F).cpu().numpy()
        g.sync()
        assert np.abs(rho - rho_o).max() <= 1e-12 * np.abs(rho_o).max()
        assert np.abs(H - H_o).max() <= 1e-12 * np.abs(H_o).max()
        assert np.abs(F - F_o).max() <= 1e-11 * np.abs(F_o).max()
    g.close()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_inputs_reach_the_same_results(bad):
    """One bad point of V, or one bad element of D: the same elements are non-finite as on the CUDA cores (FP32), the
    rest equals the clean run's."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    s = _system(("221", "110"), 6, 16.0, (16, 12, 16))
    rng = np.random.default_rng(3)
    g = G.Gint(s)
    C = rng.normal(size=(g.norb, 5)) / 4
    D = torch.from_numpy(g.dense_to_blocks(C @ C.T)).cuda()
    V = torch.from_numpy(rng.normal(size=g.ngrid)).cuda()
    H0, rho0 = g.vlocal(V, G.FP64).clone(), g.rho(D, G.FP64).clone()
    Vb = V.clone()
    Vb[g.ngrid // 2 + 37] = bad
    Hb, Hs = g.vlocal(Vb, G.FP64).clone(), g.vlocal(Vb, G.FP32).clone()
    ok = torch.isfinite(Hb)
    assert torch.equal(ok, torch.isfinite(Hs)) and not ok.all() and ok.any()
    assert float((Hb - H0)[ok].abs().max()) <= 1e-12 * float(H0.abs().max())
    M = C @ C.T
    M[3, 20] = M[20, 3] = bad
    Db = torch.from_numpy(g.dense_to_blocks(M)).cuda()
    rb, rs = g.rho(Db, G.FP64).clone().reshape(-1), g.rho(Db, G.FP32).clone().reshape(-1)
    ok = torch.isfinite(rb)
    assert torch.equal(ok, torch.isfinite(rs)) and not ok.all() and ok.any()
    assert float((rb - rho0.reshape(-1))[ok].abs().max()) <= 1e-12 * float(rho0.abs().max())
    g.sync()
    g.close()


def test_captured_passes_replay():
    """The float64 passes and the dense steps around them in one CUDA graph, replayed on new inputs: the direct calls'
    results (force and H sums in another order of atomics: 1e-13)."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    s = _system(("221", "110"), 6, 12.0, (16, 12, 16))
    rng = np.random.default_rng(5)
    g = G.Gint(s)
    n = g.norb
    C = rng.normal(size=(n, 5)) / 4
    D0, V0 = torch.from_numpy(g.dense_to_blocks(C @ C.T)).cuda(), torch.from_numpy(rng.normal(size=g.ngrid)).cuda()
    cn = G.CrankNicolson(n, 5)
    S = torch.eye(n, dtype=torch.float64, device="cuda")
    A = torch.from_numpy(rng.normal(size=(n, n))).cuda()
    A = 0.5 * (A + A.T)
    psi0 = torch.from_numpy(np.ascontiguousarray((rng.normal(size=(n, 5)) + 1j * rng.normal(size=(n, 5))).T)).cuda()
    f = torch.ones(5, dtype=torch.float64, device="cuda")
    D, V, psi = D0.clone(), V0.clone(), psi0.clone()
    out = [torch.empty(g.grid, dtype=torch.float64, device="cuda"), torch.empty_like(D), torch.empty((6, 3), dtype=torch.float64, device="cuda"),
           torch.empty_like(psi), torch.empty((n, n), dtype=torch.float64, device="cuda")]

    def calls():
        g.rho(D, G.FP64, out=out[0])
        g.vlocal(V, G.FP64, out=out[1])
        g.force(D, V, G.FP64, out=out[2])
        cn.step(S, A, 0.05, psi, out=out[3])
        cn.density_matrix(out[3], f, out=out[4])

    calls()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for scale in (1.0, -0.5):
        D.copy_(scale * D0)
        V.copy_(scale * V0)
        psi.copy_(scale * psi0)
        graph.replay()
        torch.cuda.synchronize()
        got = [x.clone() for x in out]
        calls()
        torch.cuda.synchronize()
        for a, b in zip(got, out):
            assert float((a - b).abs().max()) <= 1e-13 * float(b.abs().max())
    cn.close()
    g.close()


@pytest.mark.parametrize("rc,dr", [(5.0, 0.01), (5.0, 0.2), (10.0, 0.01), (10.0, 10.0 / 1023), (5.0, 5.0)])
def test_no_support_where_r_rounds_up_to_the_radius(rc, dr):
    """A grid point with r2 one ulp below rc^2, so that r rounds to rc, the last knot: outside, as for the oracle and
    the CUDA-core evaluator, whatever the parity of the knot count and the values at the table's end."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    sp = _sp("a", [(0, 0.3, rc)], dr)
    sp.radials[0].f[:] = 1.0
    sp.radials[0].df[:] = 0.0
    a, b = 3.0 * rc / 5.0, np.nextafter(4.0 * rc / 5.0, 0.0)
    r2 = b * b + a * a  # (the kernels' order: fma(dy, dy, dx dx), the product of b exact enough to agree)
    assert r2 == np.nextafter(rc * rc, 0.0) and np.sqrt(r2) == rc
    s = inputs.System(cell=np.diag([4.0 * rc] * 3), pos=np.array([[a, b, 0.0]]), species=np.zeros(1, np.int32), sp=[sp],
                      grid=(8, 8, 8))
    o = Oracle(s)
    D = np.array([[3.0]])
    V = np.ones(512)
    ref = o.rho(D).reshape(-1)
    assert ref[0] == 0.0 and ref.max() > 0.2
    g = G.Gint(s)
    Db, Vd = torch.from_numpy(g.dense_to_blocks(D)).cuda(), torch.from_numpy(V).cuda()
    rho = g.rho(Db, G.FP64).cpu().numpy().reshape(-1)
    rho_f = torch.empty(512, dtype=torch.float64, device="cuda")
    F = g.force(Db, Vd, G.FP64, rho_out=rho_f).cpu().numpy()
    H = g.vlocal(Vd, G.FP64).cpu().numpy()
    g.sync()
    assert rho[0] == 0.0 and rho_f[0].item() == 0.0
    assert np.abs(rho - ref).max() <= 1e-12 * ref.max() and np.abs(rho_f.cpu().numpy() - ref).max() <= 1e-12 * ref.max()
    assert np.abs(H - o.vlocal(V).reshape(-1)).max() <= 1e-12 * np.abs(o.vlocal(V)).max()
    assert np.abs(F - o.force(D, V)).max() <= 1e-11
    g.close()


def test_density_does_not_depend_on_the_scale_of_the_radials():
    """Radials times powers of two, D divided by them: the same density bit for bit, alone and in the force pass."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    power = [-20, 13, 5, -30, -9]
    names, nat, box, grid = ("221",), 9, 12.0, (8, 8, 16)
    s = _system(names, nat, box, grid)
    t = _system(names, nat, box, grid)
    for r, a in zip(t.sp[0].radials, power):
        r.f *= 2.0**a
        r.df *= 2.0**a
    c = np.tile(2.0 ** np.repeat(power, [2 * r.l + 1 for r in s.sp[0].radials]), nat)
    rng = np.random.default_rng(4)
    C = rng.normal(size=(len(c), 5)) / 4
    D, V = C @ C.T, rng.normal(size=int(np.prod(grid)))
    out = []
    for sys_, D_ in ((s, D), (t, D / c[:, None] / c)):
        g = G.Gint(sys_)
        Db, Vd = torch.from_numpy(g.dense_to_blocks(D_)).cuda(), torch.from_numpy(V).cuda()
        rho_f = torch.empty(V.size, dtype=torch.float64, device="cuda")
        g.force(Db, Vd, G.FP64, rho_out=rho_f)
        out.append((g.rho(Db, G.FP64).cpu().numpy().reshape(-1), rho_f.cpu().numpy()))
        g.sync()
        g.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_a_large_block_elsewhere_costs_a_brick_no_bits():
    """Atoms 0 and 1 share a block of D 2^40 above the rest: in bricks (4 x 4 x 8 points) that atom 1 does not reach, the
    density and the forces' density are those of a float64 chain, although the rows of atom 0 hold that block too."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    L, grid = 30.0, (16, 16, 16)
    sp = [_sp("a", ORB["221"])]
    s = inputs.System(cell=np.diag([L] * 3), pos=np.array([[10.1, 15.2, 14.9], [18.3, 15.1, 15.2], [11.9, 13.0, 15.0]]),
                      species=np.zeros(3, np.int32), sp=sp, grid=grid)
    o = Oracle(s)
    rng = np.random.default_rng(8)
    D = rng.normal(size=(o.norb, o.norb))
    D = D + D.T
    D[:13, 13:26] *= 2.0**40
    D[13:26, :13] *= 2.0**40
    x = [np.arange(n) / n * L for n in grid]
    pts = np.stack(np.meshgrid(*x, indexing="ij"), -1).reshape(-1, 3)
    near = (np.linalg.norm(pts - s.pos[1], axis=1) < 6.0).reshape(4, 4, 4, 4, 2, 8)
    far = np.broadcast_to(~near.any(axis=(1, 3, 5), keepdims=True), near.shape).reshape(-1)
    ref = o.rho(D).reshape(-1)
    g = G.Gint(s)
    Db, Vd = torch.from_numpy(g.dense_to_blocks(D)).cuda(), torch.ones(ref.size, dtype=torch.float64, device="cuda")
    rho_f = torch.empty_like(Vd)
    F = g.force(Db, Vd, G.FP64, rho_out=rho_f).cpu().numpy()
    rho = g.rho(Db, G.FP64).cpu().numpy().reshape(-1)
    g.sync()
    # the tolerance of the float64 path on either set of points
    for got in (rho, rho_f.cpu().numpy()):
        assert np.abs(got - ref)[far].max() <= 1e-12 * np.abs(ref[far]).max()
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    Fo = o.force(D, np.ones(ref.size))
    assert np.abs(F - Fo).max() <= 1e-11 * np.abs(Fo).max()
    g.close()
