"""Tensor-core density matrix at the edges of its tiles and panels (one row, tiles of 128 short and over by one, panels
of 12 tiles short, full and over by one), fewer and more K chunks than stages and accumulators, and scales far outside
float32: the bound of the other sizes, 1e-6 of max_i sum_s |f_s| |psi_is|^2; symmetric bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nocc,e", [(1, 1, 0), (127, 32, 0), (129, 33, 300), (1536, 96, 0), (1537, 129, -300), (3200, 65, 0)])
def test_edges(n, nocc, e):
    import torch

    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(n)
    psi = (rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc))) / 32
    f = rng.uniform(-1, 2, size=nocc)
    cn = G.CrankNicolson(n, nocc)
    pd = torch.from_numpy(np.ascontiguousarray(psi.T) * 2.0 ** e).cuda()
    D = cn.density_matrix(pd, torch.from_numpy(f * 2.0 ** (-2 * e)).cuda(), precision="f16x3").cpu().numpy()
    assert cn.info() == 0
    cn.close()
    assert np.array_equal(D, D.T)
    ref = ((psi * f) @ psi.conj().T).real
    assert np.abs(D - ref).max() <= 1e-6 * (np.abs(psi) ** 2 @ np.abs(f)).max()


def test_an_infinity_or_nan_reaches_its_row_and_column():
    import torch

    from paper_2603_21835_gb300 import gint as G

    cn = G.CrankNicolson(300, 4)
    psi = torch.ones((4, 300), dtype=torch.complex128, device="cuda")
    psi[2, 130] = complex(0.0, float("nan"))
    D = cn.density_matrix(psi, torch.ones(4, dtype=torch.float64, device="cuda"), precision="f16x3")
    assert cn.info() == 0
    assert not torch.isfinite(D[130]).any() and not torch.isfinite(D[:, 130]).any()
    cn.close()
