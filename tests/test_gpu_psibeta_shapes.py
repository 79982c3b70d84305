"""Projector overlaps over the forms the dispatch tells apart: every compiled orbital shape and the general
evaluator (unsorted radials, radials on different knot grids), radials that end at different radii, one to
three projector radials per species (odd counts, l = 0..2), species without projectors, and a cell small
enough for many images of a pair; float64 against the oracle to 1e-11 of max |P|, as for the larger cells."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2603_21835_gb300 import inputs
from tests.test_oracle_psibeta import angular_rule, radial_rule

pytestmark = pytest.mark.gpu


def _sp(name, spec, dr=0.01):
    """Species from (l, alpha, rc) radials."""
    return inputs.Species(name=name, radials=[inputs.make_radial(l, a, rc, dr) for l, a, rc in spec])


ORB = {
    "221": [(0, 0.3, 6.0), (0, 0.8, 6.0), (1, 0.3, 6.0), (1, 0.8, 6.0), (2, 0.3, 6.0)],
    "210": [(0, 0.3, 5.0), (0, 0.8, 5.0), (1, 0.5, 5.0)],
    "111": [(0, 0.3, 6.0), (1, 0.4, 6.0), (2, 0.5, 6.0)],
    "110": [(0, 0.3, 4.0), (1, 0.4, 4.0)],
    "100": [(0, 0.3, 6.0)],
    "unsorted": [(1, 0.3, 6.0), (0, 0.8, 6.0), (2, 0.5, 6.0)],
    "dd": [(2, 0.3, 6.0), (2, 0.6, 6.0)],
    "grids": [(0, 0.3, 6.0), (1, 0.4, 5.0)],
}
PRJ = [[(0, 6.0, 2.5), (1, 6.0, 2.5)], [(2, 4.0, 2.0)], [(0, 5.0, 2.2), (1, 6.0, 2.2), (2, 4.0, 2.2)], []]


def _shorter(sp, k, rc):
    """Radial k's table runs on, but its support ends at rc (between two knots)."""
    sp.radials[k].rc = rc
    return sp


@pytest.mark.parametrize("names,box", [(("221", "210"), 9.0), (("111", "110"), 14.0), (("100", "unsorted"), 10.0),
                                       (("dd", "grids"), 12.0), (("221 short", "111 short"), 11.0), (("221", "100"), 4.0)])
def test_shapes_match_the_oracle(names, box):
    from paper_2603_21835_gb300 import gint as G

    rng = np.random.default_rng(len(names[0]) + int(box))
    sp = []
    for n in names:
        s = _sp(n, ORB[n.split()[0]])
        sp.append(_shorter(s, 1, 4.3337) if n.endswith("short") else s)
    cell = np.diag([box, box * 1.1, box * 0.95])
    pos = rng.random((3, 3)) @ cell
    species = np.array([0, 1, 0], np.int32)
    grid = (12, 12, 16)
    s = inputs.System(cell=cell, pos=pos, species=species, sp=sp, grid=grid)
    g = G.Gint(s)
    A = np.array([0.12, -0.07, 0.05])
    for kp in range(len(PRJ)):
        prj = [_sp("a", PRJ[kp]), _sp("b", PRJ[(kp + 1) % len(PRJ)])]
        g.set_projectors(prj)
        P = g.psibeta(A).cpu().numpy()
        again = g.psibeta(A).cpu().numpy()
        assert np.array_equal(P, again)
        pmax = np.abs(P).max()
        o = Oracle(s)
        # the oracle takes projectors as the orbitals of a second system; a species without any is given a
        # radial that is not used
        op = Oracle(inputs.System(cell=cell, pos=pos, species=species, grid=grid,
                                  sp=[p if p.radials else _sp("x", [(0, 1.0, 1.0)]) for p in prj]))
        checked = 0
        for q, (I, J) in enumerate(g.pb_pairs):
            assert prj[species[I]].radials
            ref = o.psibeta(op, A, int(I), int(J), radial_rule(), angular_rule())
            got = P[g.pb_off[q]:g.pb_off[q + 1]].reshape(ref.shape)
            assert np.abs(got - ref).max() <= 1e-11 * pmax, (kp, I, J)
            checked += 1
        assert checked == len(g.pb_pairs) > 0
    g.close()
