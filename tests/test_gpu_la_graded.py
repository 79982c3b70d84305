"""Dense float64 steps on graded matrices, where a digit product keeps an operand to 2^-62 of its row's largest element:
basis functions of very different norms, and small pivots inside a matrix of unit diagonal.  Plain float64 elimination
is indifferent to the first and backward stable for the second."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrices(n, nocc, seed):
    rng = np.random.default_rng(seed)
    Q = rng.normal(size=(n, n))
    S, H, D = np.eye(n) + 0.5 * (Q @ Q.T) / n, 0.5 * (Q + Q.T), Q @ Q.T / n
    psi = rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc))
    return rng, S, H, D, psi


def _run(S, H, D, psi, dt=0.05):
    import torch

    from paper_2603_21835_gb300 import gint as G

    n, nocc = psi.shape
    cn = G.CrankNicolson(n, nocc)
    Sd, Hd, Dd = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (S, H, D))
    out = cn.step(Sd, Hd, dt, torch.from_numpy(np.ascontiguousarray(psi.T)).cuda()).cpu().numpy().T
    assert cn.info() == 0
    E = cn.energy_density_matrix(Sd, Hd, Dd).cpu().numpy()
    assert cn.info() == 0
    cn.close()
    return out, E


@pytest.mark.parametrize("n,nocc", [(33, 5), (130, 20), (1100, 24)])  # one and several blocks and contraction ranges
def test_results_do_not_depend_on_the_norms_of_the_basis(n, nocc):
    """Basis functions scaled by powers of two over a ratio of 2^28: the scaled results bit for bit."""
    rng, S, H, D, psi = _matrices(n, nocc, n)
    s = 2.0 ** rng.integers(-14, 15, size=n)
    out, E = _run(S, H, D, psi)
    out_s, E_s = _run(s[:, None] * S * s, s[:, None] * H * s, D / s[:, None] / s, psi / s[:, None])
    assert np.array_equal(out_s, out / s[:, None])
    assert np.array_equal(E_s, E / s[:, None] / s)


@pytest.mark.parametrize("small,cols", [(1e-8, 1), (1e-10, 4), (1e-12, 1), (1e-12, 4)])
def test_small_pivots_leave_the_solve_backward_stable(small, cols):
    """S of unit diagonal with pivots down to 1e-12 (columns of L up to 1e6): the residual of X = (psi_out + psi) / 2 in
    A X = S psi, A = S + i dt/2 H, against the bound of a float64 elimination, n 2^-53 of |X| (|L| |D| |L^T| is at most
    1 for a unit diagonal).  Digits relative to the rows of W = L D and of L left 4e-14 to 5e-12 of |X| here, a float64
    elimination on the host 5e-16 to 1e-15."""
    n, nocc, dt = 160, 8, 0.05
    rng = np.random.default_rng(cols)
    L, d = np.eye(n, dtype=np.longdouble), np.ones(n, dtype=np.longdouble)
    L += np.tril(rng.normal(size=(n, n)), -1) * 0.05
    for p in range(cols):
        k = 2 * p + 1
        d[k] = small
        L[k + 1:, k] = rng.normal(size=n - k - 1) * 0.3 / np.sqrt(small)
        L[k, k - 1] = 1.0
    S = (L * d) @ L.T
    s = 1 / np.sqrt(np.diag(S))
    S = (s[:, None] * S * s).astype(np.float64)
    S = 0.5 * (S + S.T)
    K = rng.normal(size=(n, n))
    H = S @ (K + K.T) @ S
    H = 0.5 * (H + H.T)
    psi = rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc))
    out, _ = _run(S, H, np.eye(n), psi, dt)
    X = (out.astype(np.clongdouble) + psi) / 2
    Sl, Hl = S.astype(np.longdouble), H.astype(np.longdouble)
    R = Sl @ X + 0.5j * dt * (Hl @ X) - Sl @ psi.astype(np.clongdouble)
    assert np.abs(R).max() <= n * 2.0**-53 * np.abs(X).max()


def test_density_matrix_of_functions_in_states_of_small_occupation():
    """Half of the functions have all their weight in states of occupation 1e-12: the error is relative to
    (D_ii D_jj)^(1/2), the operands' digits being those of f^(1/2) psi."""
    import torch

    from paper_2603_21835_gb300 import gint as G

    n, nocc = 70, 40
    rng = np.random.default_rng(3)
    psi = rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc))
    f = np.where(np.arange(nocc) < 10, 1.3, 1.7e-12)
    psi[: n // 2, :10] *= 1e-7
    cn = G.CrankNicolson(n, nocc)
    D = cn.density_matrix(torch.from_numpy(np.ascontiguousarray(psi.T)).cuda(), torch.from_numpy(f).cuda()).cpu().numpy()
    assert cn.info() == 0
    cn.close()
    a = np.stack([psi.real, psi.imag], -1).reshape(n, 2 * nocc).astype(np.longdouble)
    fa = a * np.repeat(f, 2)
    ref = fa @ a.T
    d = np.sqrt(np.diag(ref))
    # the factor f psi and the sum are rounded once each
    bound = 2.0**-53 * (np.abs(fa) @ np.abs(a.T) + np.abs(ref)) + 2 * nocc * 2.0**-57 * np.outer(d, d)
    assert (np.abs(D - ref) <= bound).all()
    assert np.array_equal(D, D.T)
