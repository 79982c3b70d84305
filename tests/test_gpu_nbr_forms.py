"""Device neighbour lists over the forms their kernels tell apart: bricks with more entries than the counting
pass keeps (64: a tiny cell, many images), exactly one atom, more than 32 and 64 atoms near a brick, atoms
outside the cell, a strongly skewed cell, grids smaller than a brick, two species of very different support,
points and sphere centres on a common lattice (distances in the shell around rc).  Exact lists and
W = sum_g n_g^2 against a host brute force; entries within 1e-9 of the support boundary may go either way."""
import numpy as np
import pytest

from paper_2603_21835_gb300 import inputs
from tests.test_gpu_units import _brute_lists

pytestmark = pytest.mark.gpu


def _systems():
    rng = np.random.default_rng(3)
    s1 = inputs.species_dzp("A", 6.0, [(0, 1)])
    s2 = inputs.species_dzp("B", 1.3, [(0, 1), (1, 1)])
    box = np.diag([2.3, 2.4, 2.2])
    yield "many images", inputs.System(box, np.array([[0.4, 1.0, 2.0]]), np.zeros(1, np.int32), [s1], (8, 9, 12))
    box = np.diag([20.0, 18.0, 22.0])
    yield "one atom", inputs.System(box, np.array([[-30.0, 55.0, 7.3]]), np.zeros(1, np.int32), [s1], (20, 18, 23))
    box = np.diag([30.0, 12.0, 10.0])
    pos = rng.random((90, 3)) @ box
    yield "ninety atoms", inputs.System(box, pos, np.array([0] * 30 + [1] * 60, np.int32), [s2, s1][::-1], (31, 13, 11))
    skew = np.array([[9.0, 0.0, 0.0], [7.0, 6.0, 0.0], [-5.0, 4.0, 8.0]])
    yield "skewed", inputs.System(skew, rng.random((3, 3)) @ skew, np.array([0, 1, 0], np.int32), [s1, s2], (13, 9, 17))
    yield "tiny grid", inputs.System(np.diag([8.0, 8.0, 8.0]), rng.random((4, 3)) * 8, np.zeros(4, np.int32), [s1], (3, 2, 5))
    s3 = inputs.species_dzp("C", 3.0, [(0, 1)])
    yield "on the sphere", inputs.System(np.diag([12.0, 12.0, 12.0]), np.array([[6.0, 6.0, 6.0], [0.0, 0.0, 0.0]]),
                                         np.zeros(2, np.int32), [s3], (24, 24, 24))


@pytest.mark.parametrize("name,system", list(_systems()), ids=[n for n, _ in _systems()])
def test_lists_and_work(name, system):
    from paper_2603_21835_gb300 import gint as G

    g = G.Gint(system)
    b_off, slot_atom, slot_ent, epos = g.brick_lists()
    ref = _brute_lists(system)
    inv = np.linalg.inv(system.cell)
    biggest, boundary = 0, False
    for b, want in enumerate(ref):
        got = {}
        atoms = slot_atom[b_off[b]:b_off[b + 1]]
        assert (np.diff(atoms) > 0).all()
        for s in range(b_off[b], b_off[b + 1]):
            assert slot_ent[s + 1] > slot_ent[s]
            last = None
            for e in range(slot_ent[s], slot_ent[s + 1]):
                n = (epos[e] - system.pos[slot_atom[s]]) @ inv
                k = tuple(np.rint(n).astype(int))
                assert np.abs(n - k).max() < 1e-9 and (last is None or k > last)
                last = k
                got[(int(slot_atom[s]), *k)] = True
        must = {k for k, v in want.items() if v < -1e-9}
        assert must <= set(got) <= set(want), (name, b)
        boundary |= len(must) < len(want)
        biggest = max(biggest, len(got))
    if name == "many images":
        assert biggest > 64
    if not boundary:  # n_g is then unambiguous
        n = np.array(system.grid)
        pts = np.stack(np.meshgrid(*(np.arange(m) / m for m in n), indexing="ij"), -1).reshape(-1, 3) @ system.cell
        cov = np.zeros(len(pts))
        cov_at = {}
        for want in ref:
            for (a, *k) in want:
                cov_at.setdefault(a, set()).add(tuple(k))
        for a, ks in cov_at.items():
            hit = np.zeros(len(pts), bool)
            for k in ks:
                d = pts - system.pos[a] - np.array(k) @ system.cell
                hit |= (d * d).sum(1) < system.sp[system.species[a]].rcut ** 2
            cov += hit * system.sp[system.species[a]].norb
        assert g.stats()["W"] == float((cov * cov).sum())
    g.close()
