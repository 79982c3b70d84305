"""Propagation steps at the edges of the blocked solve, whose kernels cut the next product's operands themselves: sizes
one short of, at and over the 32- and 64-wide blocks, state counts around the eight vectors of a CTA; against the
oracle with the tolerance of the larger sizes, 1e-12 of the largest element."""
import numpy as np
import pytest

from oracle.dense import crank_nicolson, energy_density_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 97, 200])
@pytest.mark.parametrize("nocc", [1, 8, 9])
def test_step_and_energy_density_matrix(n, nocc):
    import torch

    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(100 * n + nocc)
    S = rng.normal(size=(n, n)) * 0.02
    S = np.eye(n) + 0.5 * (S + S.T)
    H = rng.normal(size=(n, n))
    H, R = 0.5 * (H + H.T), rng.normal(size=(n, n))
    R = 0.5 * (R + R.T)
    psi = rng.normal(size=(n, nocc)) + 1j * rng.normal(size=(n, nocc))
    cn = G.CrankNicolson(n, nocc)
    Sd, Hd, Rd = (torch.from_numpy(x).cuda() for x in (S, H, R))
    got = cn.step(Sd, Hd, 0.05, torch.from_numpy(np.ascontiguousarray(psi.T)).cuda()).cpu().numpy().T
    E = cn.energy_density_matrix(Sd, Hd, Rd).cpu().numpy()
    assert cn.info() == 0
    cn.close()
    ref, Eref = crank_nicolson(S, H, 0.05, psi), energy_density_matrix(S, H, R)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(E - Eref).max() <= 1e-12 * np.abs(Eref).max()
    assert np.array_equal(E, E.T)
