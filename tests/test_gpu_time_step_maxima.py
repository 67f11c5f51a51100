"""The time-step limits take their maxima over the cells whose terms are
numbers: a cell that holds a NaN leaves the limits of the others, and a
negative mobility counts by its size in the advective limit."""
import numpy as np
import pytest

import synth
from helpers import EPS0, Q, load_inputs, pair
from oracle import quad

pytestmark = pytest.mark.gpu


def _quad(mu=1.0):
    """A small mesh with its field, on both sides; mobilities times mu."""
    import paper_1708_08434_gb300 as p
    dom, st = synth.workload2("axi_small")
    o = quad.build_mesh(dom, st)
    t = o.tables()
    g = p.Quad(dom, len(t["level"]))
    synth.refine_all2(dom, st, g.level_ij, g.refine_level)
    ne, ni = synth.streamer_densities2(dom, st, t["level"], t["ij"])
    tab = synth.coefficient_table()
    tab["mu"] = mu * tab["mu"]
    for var, v in ((quad.NE, ne), (quad.NI, ni)):
        o.set(var, v)
    g.upload(p.NE, ne)
    g.upload(p.NI, ni)
    for s in (o, g):
        s.set_table(tab)
        s.charge_rhs(Q, EPS0)
        s.fmg(1e-10, 40)
        s.compute_field()
    return p, g, o, ne, np.flatnonzero(t["child"][:, 0] < 0)[3]


def _octree(mu=1.0):
    import paper_1708_08434_gb300 as p
    dom, st, o, g = pair("streamer_small")
    t = g.tables()
    load_inputs(dom, st, o, g)
    tab = synth.coefficient_table()
    tab["mu"] = mu * tab["mu"]
    for s in (o, g):
        s.set_table(tab)
        s.fmg(1e-10, 40)
        s.compute_field()
    return p, g, o, g.download(p.NE), np.flatnonzero(t["child"][:, 0] < 0)[3]


@pytest.mark.parametrize("make", [_quad, _octree])
@pytest.mark.parametrize("what", ["density", "potential"])
def test_nan_cell_leaves_the_other_limits(make, what):
    p, g, _, ne, b = make()
    phi = g.download(p.PHI)
    eps = EPS0 * (1e-6 if what == "density" else 1.0)  # the smaller one makes the relaxation time limit dt
    limit = g.dt_limit(Q, eps)
    assert 0.0 < limit < 1.0
    var, v = (p.NE, ne) if what == "density" else (p.PHI, phi)
    v = v.copy()
    v[b, 9] = np.nan
    g.upload(var, v)
    got = g.dt_limit(Q, eps)
    g.close()
    # the cell (and its neighbours, for the potential) is not the one that limits dt
    assert got == limit


@pytest.mark.parametrize("make", [_quad, _octree])
def test_negative_mobility_limits_by_its_size(make):
    p, g, o, _, _ = make(-1.0)
    a, b = g.dt_limit(Q, EPS0), o.dt_limit(Q, EPS0)
    g.close()
    assert abs(a - b) <= 1e-12 * b
