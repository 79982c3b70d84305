"""Tensor-core density, forces and local H over the forms the brick kernel tells apart: the double-zeta-polarised
instance and the one of all shapes, slots of one image and of several (with atoms on grid points), the generic
evaluator; F16x3 against the float64 path with the tolerances of the parity tests (1e-6 of the largest element for
rho and H, 1e-5 Ha/Bohr for F), and a system alone against the same system in a batch, bit for bit."""
import numpy as np
import pytest

from tests.test_gpu_fx import _system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("names,nat,box,grid,on_grid", [
    (("221",), 4, 18.0, (28, 32, 24), False), (("221", "210"), 6, 9.0, (16, 16, 16), True), (("210",), 3, 16.0, (27, 29, 25), True),
    (("221", "110"), 5, 16.0, (24, 24, 24), True), (("111", "100"), 6, 8.0, (14, 16, 13), False),
    (("unsorted", "221"), 4, 15.0, (24, 24, 24), False), (("221 short",), 3, 9.0, (16, 16, 16), False)])
def test_force_passes_match_float64(names, nat, box, grid, on_grid):
    import torch

    from paper_2603_21835_gb300 import gint as G

    s = _system(names, nat, box, grid, on_grid)
    rng = np.random.default_rng(nat)
    g = G.Gint(s)
    C = rng.normal(size=(g.norb, 5)) / 8
    D = torch.from_numpy(g.dense_to_blocks(C @ C.T)).cuda()
    V = torch.from_numpy(rng.normal(size=g.ngrid) / 8).cuda()
    out = {}
    for prec in (G.FP64, G.F16X3):
        rho = torch.empty(g.grid, dtype=torch.float64, device="cuda")
        F = g.force(D, V, prec, rho_out=rho).clone()
        out[prec] = (F, rho, g.rho(D, prec).clone(), g.vlocal(V, prec).clone())
    g.sync()
    for k, (a, b) in enumerate(zip(out[G.F16X3], out[G.FP64])):
        tol = 1e-5 if k == 0 else 1e-6 * float(b.abs().max())
        assert float((a - b).abs().max()) <= tol, k
    g2 = G.Gint(s)
    one, *bufs = [[torch.empty_like(rho), torch.empty_like(out[G.FP64][3]), torch.empty_like(F)] for _ in range(3)]
    g.run(D, V, G.F16X3, rho=one[0], H=one[1], F=one[2])
    G.run_batch([G.Task(x, D=D, V=V, rho=b[0], H=b[1], F=b[2]) for x, b in zip((g, g2), bufs)], G.F16X3)
    g.sync()
    for b in bufs:
        assert torch.equal(b[0], one[0]) and torch.equal(b[1], one[1])
        assert float((b[2] - one[2]).abs().max()) <= 1e-12 * float(b[2].abs().max())
    g.close()
    g2.close()
