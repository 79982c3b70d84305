"""Float64 products on the tensor cores (digit products, gint_sg.cu), reached through the dense steps.

The density matrix is one product D = (f psi) psi^T over K = 2 nocc real terms.  Its error has three
parts: the sum itself is rounded once per 1024 terms, the factors f psi are rounded once (2^-53 of each
product), and an operand is represented to 2^-62 of its row's largest magnitude (dropped digit products
included: below 2^-56 of the product of the two row maxima per term).  The bound below is their sum; the
reference is summed in extended precision."""
import numpy as np
import pytest

from oracle.dense import crank_nicolson, energy_density_matrix

pytestmark = pytest.mark.gpu


def _density(n, nocc, psi, f):
    import torch

    from paper_2603_21835_gb300 import gint as G

    cn = G.CrankNicolson(n, nocc)
    D = cn.density_matrix(torch.from_numpy(np.ascontiguousarray(psi.T)).cuda(), torch.from_numpy(f).cuda()).cpu().numpy()
    assert cn.info() == 0
    cn.close()
    return D


# tile edges (128 rows, 64 columns), digit chunks (16 terms), packing ranges (64), exact ranges (128) and
# contraction ranges (1024) met one short, exactly and one over
@pytest.mark.parametrize("n,nocc", [(1, 1), (63, 8), (64, 9), (65, 32), (127, 33), (128, 64), (129, 65), (33, 511), (40, 512),
                                    (20, 530)])
def test_density_matrix_error_bound(n, nocc):
    rng = np.random.default_rng(n + nocc)
    scale = 10.0 ** rng.uniform(-8, 8, size=(n, 1))  # rows of very different magnitude
    psi = scale * (rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc)))
    f = rng.uniform(-2, 2, size=nocc)
    D = _density(n, nocc, psi, f)
    a = np.stack([psi.real, psi.imag], -1).reshape(n, 2 * nocc).astype(np.longdouble)
    fa = a * np.repeat(f, 2)
    ref = fa @ a.T
    K = 2 * nocc
    ma, mb = np.abs(fa).max(1), np.abs(a).max(1)
    bound = 2.0**-53 * (np.abs(fa) @ np.abs(a.T) + (1 + K // 1024) * np.abs(ref)) + K * 2.0**-56 * np.outer(ma, mb)
    assert (np.abs(D - ref) <= bound).all()
    assert np.array_equal(D, D.T)


@pytest.mark.parametrize("nocc", [64, 100])
def test_aligned_digits_are_summed_exactly(nocc):
    """Every element 0x3f808080808080 2^-62: six of its digits are -128, so the level sums of a range of 128
    terms pass 2^23 and take the wide conversion; the result is one rounding of the exact sum."""
    q = 0x3F80808080808000
    x = float(q) * 2.0**-62
    assert int(x * 2.0**62) == q
    n = 70
    D = _density(n, nocc, np.full((n, nocc), x * (1 + 1j)), np.ones(nocc))
    exact = 2 * nocc * q * q  # times 2^-124
    assert (np.abs(D - float(exact) * 2.0**-124) <= np.spacing(D)).all()
    got = int(D[0, 0] * 2.0**100)
    assert abs(got - (exact >> 24)) <= (exact >> 24) * 2.0**-52


def test_extreme_exponents_and_zero_rows():
    rng = np.random.default_rng(5)
    n, nocc = 66, 20
    psi = rng.normal(size=(n, nocc)) + 0j
    psi[1] *= 1e-160
    psi[2] *= 1e150
    psi[3] = 0.0
    psi[4] *= 1e-300
    f = np.ones(nocc)
    D = _density(n, nocc, psi, f)
    ref = psi.real.astype(np.longdouble) @ psi.real.T.astype(np.longdouble)
    mx = np.abs(psi.real).max(1)
    tol = 2.0**-53 * 3 * (np.abs(psi.real) @ np.abs(psi.real.T)) + nocc * 2.0**-56 * np.outer(mx, mx) + 5e-324
    assert (np.abs(D - ref) <= tol).all()
    assert (D[3] == 0).all() and D[4, 4] == 0 and D[1, 1] != 0


def test_infinities_and_nans_stay_in_their_rows_and_columns():
    rng = np.random.default_rng(6)
    n, nocc = 130, 40
    psi = rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc))
    psi.real[7, 3], psi.imag[129, 0] = np.inf, np.nan
    f = rng.uniform(0.5, 2, size=nocc)
    D = _density(n, nocc, psi, f)
    a = np.stack([psi.real, psi.imag], -1).reshape(n, 2 * nocc)
    with np.errstate(invalid="ignore"):
        ref = (a * np.repeat(f, 2)) @ a.T
    ok = np.isfinite(ref)
    assert np.array_equal(np.isnan(D), np.isnan(ref)) and np.array_equal(np.isinf(D), np.isinf(ref))
    assert np.array_equal(D[np.isinf(ref)], ref[np.isinf(ref)])
    assert np.abs(D - ref)[ok].max() <= 1e-13 * np.abs(ref[ok]).max()


@pytest.mark.parametrize("n,k", [(1, 1), (2, 5), (31, 3), (32, 8), (33, 40), (63, 7), (64, 9), (65, 1), (97, 130)])
def test_step_at_block_edges(n, k):
    """Factorisation blocks of 32 (complex), more right-hand sides than rows included; 1e-12 of the
    largest entry as for the larger sizes."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(n)
    Q = rng.normal(size=(n, n))
    S, H = np.eye(n) + 0.5 * (Q @ Q.T) / n, 0.5 * (Q + Q.T)
    psi = rng.normal(size=(n, k)) + 1j * rng.normal(size=(n, k))
    cn = G.CrankNicolson(n, k)
    out = cn.step(*(torch.from_numpy(x).cuda() for x in (S, H)), 0.05,
                  torch.from_numpy(np.ascontiguousarray(psi.T)).cuda()).cpu().numpy().T
    assert cn.info() == 0
    cn.close()
    ref = crank_nicolson(S, H, 0.05, psi)
    assert np.abs(out - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 129, 200])
def test_energy_density_matrix_at_block_edges(n):
    import torch

    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(n)
    Q = rng.normal(size=(n, n))
    S, H, D = np.eye(n) + 0.5 * (Q @ Q.T) / n, 0.5 * (Q + Q.T), Q @ Q.T / n
    cn = G.CrankNicolson(n, 2)
    E = cn.energy_density_matrix(*(torch.from_numpy(x).cuda() for x in (S, H, D))).cpu().numpy()
    assert cn.info() == 0
    cn.close()
    ref = energy_density_matrix(S, H, D)
    assert np.abs(E - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.array_equal(E, E.T)
