"""Cross-brick sums of the tensor-core local H where a pair's brick list is shorter than, as long as and a
little longer than the parts and batches it is cut into (16 parts for systems of few pairs, batches of 8), for
both reduction modes; against the float64 path (1e-6 of max |H|, the F16x3 tolerance) and each other (1e-10)."""
import numpy as np
import pytest

from paper_2603_21835_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nat,grid", [(1, (4, 4, 8)), (2, (8, 4, 8)), (2, (12, 12, 16)), (3, (20, 16, 24)), (2, (33, 29, 31)),
                                      (17, (24, 24, 24)), (18, (24, 20, 24))])
def test_short_and_ragged_lists(nat, grid):
    """17 atoms: 153 upper pairs where all overlap, the first system on the other side of the rule."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(nat)
    cell = np.diag([11.0, 11.0, 11.0])
    s = inputs.System(cell=cell, pos=rng.random((nat, 3)) @ cell, species=np.zeros(nat, np.int32), grid=grid,
                      sp=[inputs.species_dzp("X", 5.0, [(0, 1), (1, 1)])])
    g = G.Gint(s)
    V = torch.from_numpy(rng.normal(size=g.ngrid)).cuda()
    ref = g.vlocal(V, G.FP64)
    H = g.vlocal(V, G.F16X3)
    g.set_reduction("fp64")
    H64 = g.vlocal(V, G.F16X3)
    g.sync()
    m = float(ref.abs().max())
    assert float((H - ref).abs().max()) <= 1e-6 * m
    assert float((H - H64).abs().max()) <= 1e-10 * m
    g.close()


def test_many_pairs_and_moved_positions():
    """More upper pairs than the layout kernels keep cursors for in shared memory (24,576): the contribution lists
    then go through global memory.  Moved there and back, the blocks are those of the fresh handle bit for bit
    (the lists and their order depend on the positions only)."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(8)
    n = 13
    cell = np.diag([2.3 * n] * 3)
    pos = (np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * 2.3
    pos = pos + rng.normal(0.0, 0.1, pos.shape)
    s = inputs.System(cell=cell, pos=pos, species=np.zeros(len(pos), np.int32), grid=(90, 88, 92),
                      sp=[inputs.species_dzp("X", 2.6, [(0, 1), (1, 1)])])
    g = G.Gint(s, skin=0.3)
    I, J = g.pair_IJ.T
    assert (I <= J).sum() > 24576
    V = torch.from_numpy(rng.normal(size=g.ngrid)).cuda()
    ref = g.vlocal(V, G.FP64)
    H = g.vlocal(V, G.F16X3).clone()
    g.sync()
    assert float((H - ref).abs().max()) <= 1e-6 * float(ref.abs().max())
    p0 = torch.from_numpy(pos).cuda()
    g.set_positions(p0 + 0.05 * torch.randn(p0.shape, dtype=torch.float64, device="cuda"))
    ref1, H1 = g.vlocal(V, G.FP64), g.vlocal(V, G.F16X3)
    g.sync()
    assert float((H1 - ref1).abs().max()) <= 1e-6 * float(ref1.abs().max())
    g.set_positions(p0)
    assert torch.equal(g.vlocal(V, G.F16X3), H)
    g.sync()
    g.close()
