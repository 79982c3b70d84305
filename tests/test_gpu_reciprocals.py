"""The float64 reciprocals and reciprocal roots that the kernels form from float32 estimates and one third-order step,
against the exact functions over the exponents they meet, through entry points whose results are theirs.

1 / d: pivots of diagonal matrices.  The last operation is one fused multiply-add whose inputs are off by less than
2^-60, so a quotient is within one ulp (half, and a hair at ties).  1 / r and r: radials R(r) = r, whose interpolant is
exact, on one s and one p shell: the s orbital is Y_00 r, the p orbitals Y_1 d, whatever r.  Six roundings (the constant,
r / dr, the interpolant's two, u = d / r, the product) and the root's two: 8 x 2^-53."""
import numpy as np
import pytest

from paper_2603_21835_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_reciprocal_pivots():
    import torch

    from paper_2603_21835_gb300 import gint as G

    n = 256
    rng = np.random.default_rng(1)
    s = np.exp2(rng.uniform(-1000, 1000, n))
    s[:8] = [1.0, np.nextafter(1.0, 0.0), np.nextafter(1.0, 2.0), np.nextafter(2.0, 0.0), 2.0, 0.5, 2.0**-1000, 2.0**1000]
    cn = G.CrankNicolson(n, 1)
    one = torch.eye(n, dtype=torch.float64, device="cuda")
    E = cn.energy_density_matrix(torch.from_numpy(np.diag(s)).cuda(), one, one).cpu().numpy()
    assert cn.info() == 0
    q = 1.0 / s.astype(np.longdouble)
    assert np.all(np.abs(np.diag(E) - q) <= np.spacing(1.0 / s))
    assert np.count_nonzero(E - np.diag(np.diag(E))) == 0
    # complex: 1 / d = conj(d) / |d|^2, d = s (1 + i h dt / 2)
    s = np.exp2(rng.uniform(-400, 400, n))
    h, dt = rng.normal(size=n) * 10.0 ** rng.uniform(-3, 3, n), 0.05
    # (coefficients of a state: of the order of 1 / norm; far larger ones of small functions would share digits)
    psi = (rng.normal(size=(n, 1)) + 1j * rng.normal(size=(n, 1))) / np.sqrt(s)[:, None]
    out = cn.step(torch.from_numpy(np.diag(s)).cuda(), torch.from_numpy(np.diag(s * h)).cuda(), dt,
                  torch.from_numpy(np.ascontiguousarray(psi.T)).cuda()).cpu().numpy().T
    assert cn.info() == 0
    cn.close()
    z = 1j * (dt / 2) * (s * h).astype(np.longdouble)
    ref = (s - z) / (s + z) * psi[:, 0]
    # |d|^2 and the product with conj(d): two roundings each and the reciprocal's; 2 X - psi: |X| <= |psi|
    assert np.all(np.abs(out[:, 0] - ref) <= 16 * 2.0**-53 * np.abs(psi[:, 0]))


def test_radii_of_all_sizes():
    from paper_2603_21835_gb300 import gint as G

    rc, dr, L = 6.0, 2.0**-7, 40.0  # knots k dr and their differences are exact
    sp = inputs.Species(name="r", radials=[inputs.make_radial(l, 0.3, rc, dr) for l in (0, 1)])
    for r in sp.radials:
        r.f[:] = np.arange(r.npts) * dr
        r.df[:] = 1.0
    s = inputs.System(cell=np.diag([L] * 3), pos=np.zeros((1, 3)), species=np.zeros(1, np.int32), sp=[sp], grid=(8, 8, 8))
    rng = np.random.default_rng(2)
    u = rng.normal(size=(4000, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    d = u * np.exp(rng.uniform(np.log(1e-17), np.log(5.99), 4000))[:, None]
    g = G.Gint(s)
    phi, grad = g.orbitals(d, G.FP64)
    g.close()
    dl = d.astype(np.longdouble)
    r = np.sqrt((dl**2).sum(1))
    tol = 10 * 2.0**-53
    y0, y1 = np.longdouble("0.28209479177387814347"), np.longdouble("0.48860251190291992159")
    assert np.all(np.abs(phi[:, 0] - y0 * r) <= tol * y0 * r)
    for k, ax in enumerate((2, 0, 1)):  # m = 0, +1, -1: z, x, y
        assert np.all(np.abs(phi[:, 1 + k] - y1 * dl[:, ax]) <= tol * y1 * r)
        ref = np.zeros((len(d), 3))
        ref[:, ax] = 0.48860251190291992159
        far = r > 1e-11  # (nearer than 1e-12 the gradient takes its limit at the atom)
        assert np.abs(grad[far, 1 + k] - ref[far]).max() <= 64 * 2.0**-53
