"""The coefficient tables at small fields: the index keeps FP64's relative
precision down to zero, for the source in a cell and for the flux through a
face (inside a box and between boxes), so that a coefficient that starts from 0
is right to rounding.  Linear tables with a power of two as slope: every value
is the index itself times that power."""
from fractions import Fraction

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
E_MAX, N_TAB, DT = 35e6, 1000, 1e-13
# roundings on the way: the scale (2) and its product, the sum of two halves,
# the interpolation, then at most five products and sums, each 2^-53
TOL = 12 * 2.0 ** -53
INDICES = [1e-12, 2.5e-7, 3e-4, 0.37, 0.999, 1.0, 1.7, 2.3, 3.2, 3.99, 4.6, 57.3]


def _solver(dims):
    import paper_1708_08434_gb300 as p
    if dims == 3:
        g = p.Solver(synth.Domain(length=1e-3, nb=2, max_level=0, bc_type=(1,) * 6, bc_val=(0.0,) * 6), 9)
        g.build_octree()
        t = g.tables()
        return p, g, t["level"], t["ijk"]
    g = p.Quad(synth.Domain2(1e-3, 2, 0, synth.CARTESIAN, bc_type=(1,) * 4, bc_val=(0.0,) * 4), 5)
    t = g.tables()
    return p, g, t["level"], t["ij"]


def _table(slot, slope=2.0 ** -20):
    k = np.arange(N_TAB) * slope
    z = np.zeros(N_TAB)
    return {"e_max": E_MAX, "mu": np.full(N_TAB, 0.5) if slot == "alpha" else z,
            "diff": k if slot == "diff" else z, "alpha": k if slot == "alpha" else z}


@pytest.mark.parametrize("dims", [2, 3])
def test_source_in_a_cell(dims):
    p, g, level, _ = _solver(dims)
    g.set_table(_table("alpha"))
    cells = 8 ** dims
    n = len(level)
    x = np.array(INDICES)
    e = np.zeros((n, cells))
    e[level == 1, 5:5 + len(x)] = x * E_MAX / (N_TAB - 1)
    for var in (p.PHI, p.NI):
        g.upload(var, np.zeros((n, cells)))
    g.upload(p.EMAG, e)
    g.upload(p.NE, np.ones((n, cells)))
    g.fluid_stage(DT)
    got = g.download(p.NI)[level == 1]
    g.close()
    for i, ei in enumerate(e[level == 1][0, 5:5 + len(x)]):
        ei = Fraction(float(ei))
        want = Fraction(DT) * ei * (N_TAB - 1) / Fraction(E_MAX) / 2 ** 20 / 2 * ei
        for v in got[:, 5 + i]:
            assert abs(Fraction(float(v)) - want) <= Fraction(TOL) * want, (x[i], float(v), float(want))


@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("ratio", [1.0, 3.0, 0.0])  # of the second cell's |E| to the first's
def test_flux_through_a_face(dims, ratio):
    p, g, level, ij = _solver(dims)
    cells, n = 8 ** dims, len(level)
    g.set_table(_table("diff"))
    box = int(np.flatnonzero((level == 1) & (ij == 0).all(1))[0])
    right = int(np.flatnonzero((level == 1) & (ij[:, 0] == 1) & (ij[:, 1:] == 0).all(1))[0])
    row = 8 * 3 + (64 * 4 if dims == 3 else 0)
    h = Fraction(1e-3 / 16)
    for x in INDICES:
        for (b0, c0), (b1, c1) in (((box, row + 3), (box, row + 4)), ((box, row + 7), (right, row))):
            ne, e = np.zeros((n, cells)), np.full((n, cells), 1e7)
            ne[b0, c0] = 1.0
            e[b0, c0] = x * E_MAX / (N_TAB - 1)
            e[b1, c1] = ratio * e[b0, c0]
            for var, v in ((p.PHI, 0.0 * e), (p.NI, 0.0 * e), (p.EMAG, e), (p.NE, ne)):
                g.upload(var, v)
            g.fluid_stage(DT)
            got = Fraction(float(g.download(p.NE)[b1, c1]))
            ef = (Fraction(float(e[b0, c0])) + Fraction(float(e[b1, c1]))) / 2
            want = Fraction(DT) / h ** 2 * ef * (N_TAB - 1) / Fraction(E_MAX) / 2 ** 20
            assert abs(got - want) <= Fraction(TOL) * want, (x, b1 != b0, float(got), float(want))
    g.close()
