"""One-launch legs of quadtree levels (quadleg.cuh) where they can go wrong:
sweep counts, boundary mixes, a mesh with a level too large for them between
levels that have them, a base grid of one box.  Against the oracle after equal
cycles, 1e-12 of the potential (both sides FP64, rounding order differs)."""
import numpy as np
import pytest

import synth
from oracle import quad

pytestmark = pytest.mark.gpu


def _mesh(name, bct):
    if name == "through_large":  # base level of 128^2 boxes: more than are resident at once
        st = synth.Streamer2(refine_c=2.0, refine_tip=1.5e-3)
        dom = synth.Domain2(0.016, 128, 3, synth.AXISYMMETRIC, bc_val=(0.0, 0.0, 0.0, st.voltage))
    elif name == "single_base":
        st = synth.Streamer2(refine_c=2.0, refine_tip=8e-3, x_axis=0.008)
        dom = synth.Domain2(0.016, 1, 5, synth.CARTESIAN, bc_val=(0.0, 0.0, 0.0, st.voltage))
    else:
        dom, st = synth.workload2(name)
    if bct is not None:
        dom.bc_type = bct
    return dom, st


@pytest.mark.parametrize("name,nu1,nu2,bct", [
    ("axi_small", 2, 2, None), ("cart_small", 2, 2, (1, 0, 1, 1)), ("axi_small", 2, 2, (0, 1, 0, 1)),
    ("through_large", 2, 2, None), ("single_base", 2, 2, None),
    ("axi_small", 1, 1, None), ("cart_small", 1, 3, None), ("cart_small", 16, 16, None), ("single_base", 3, 1, None)])
def test_one_launch_legs(name, nu1, nu2, bct):
    import paper_1708_08434_gb300 as p
    dom, st = _mesh(name, bct)
    o = quad.build_mesh(dom, st)
    t = o.tables()
    g = p.Quad(dom, len(t["level"]), nu1, nu2)
    synth.refine_all2(dom, st, g.level_ij, g.refine_level)
    ne, ni = synth.streamer_densities2(dom, st, t["level"], t["ij"])
    for var, v in ((quad.NE, ne), (quad.NI, ni)):
        o.set(var, v)
    g.upload(p.NE, ne)
    g.upload(p.NI, ni)
    o.charge_rhs(synth.E_CHARGE, synth.EPS0)
    g.charge_rhs(synth.E_CHARGE, synth.EPS0)
    o.fmg(0.0, 4, nu1, nu2)
    g.fmg(0.0, 4)
    a, b = g.download(p.PHI), o.get(quad.PHI)
    g.close()
    assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


def test_advance_without_charge():
    """A Heun step with zero charge leaves a zero right-hand side behind, as
    the separate charge kernel did, not the one of the solve before."""
    import paper_1708_08434_gb300 as p
    dom, st = _mesh("axi_small", None)
    o = quad.build_mesh(dom, st)
    t = o.tables()
    g = p.Quad(dom, len(t["level"]))
    synth.refine_all2(dom, st, g.level_ij, g.refine_level)
    ne, ni = synth.streamer_densities2(dom, st, t["level"], t["ij"])
    g.upload(p.NE, ne)
    g.upload(p.NI, ni)
    g.set_table(synth.coefficient_table())
    g.charge_rhs(synth.E_CHARGE, synth.EPS0)
    g.fmg(1e-8, 40)
    g.compute_field()
    assert np.abs(g.download(p.RHS)).max() > 0.0
    g.advance(1e-13, 0.0, synth.EPS0, 1e-8, 40)
    rhs = g.download(p.RHS)[t["child"][:, 0] < 0]
    g.close()
    assert np.array_equal(rhs, np.zeros_like(rhs))
