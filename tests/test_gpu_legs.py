"""One-launch legs of small levels (mglevel.cuh) against the row kernels of
the same cycle: bit-identical potentials over sweep counts, boundary mixes
and meshes whose levels change between the two forms."""
import numpy as np
import pytest

import synth
from helpers import EPS0, Q, gpu_mesh

pytestmark = pytest.mark.gpu


def _mesh(name):
    """(domain, streamer or None): a refined mesh; one whose middle level (4096 boxes) is too large for a
    one-launch leg, between smaller levels; uniform levels only; refinement right above one box."""
    if name == "through_large":
        st = synth.Streamer(refine_c=2.0, refine_tip=3e-3)
        return synth.domain_streamer(16, 3, st), st
    if name == "single_base":
        st = synth.Streamer(refine_c=2.0, refine_tip=8e-3)
        return synth.domain_streamer(1, 4, st), st
    return synth.workload(name)


@pytest.mark.parametrize("name,nu1,nu2,bct", [
    ("streamer_small", 2, 2, None), ("streamer_small", 1, 1, None), ("streamer_small", 1, 3, None),
    ("streamer_small", 7, 7, None), ("streamer_small", 8, 2, None), ("streamer_small", 2, 2, (1, 0, 1, 1, 0, 1)),
    ("through_large", 2, 2, None), ("through_large", 1, 2, None), ("single_base", 2, 1, None),
    ("uniform32", 2, 2, (0, 1, 0, 0, 0, 0)), ("uniform64", 3, 1, (1, 1, 1, 1, 1, 1))])
def test_one_launch_legs_bit_identical(name, nu1, nu2, bct):
    import paper_1708_08434_gb300 as p
    dom, st = _mesh(name)
    if bct is not None:
        dom.bc_type = bct
    out = []
    for rows in (None, 0):
        g = gpu_mesh(dom, st, nu1=nu1, nu2=nu2)
        if rows is not None:
            g.set_row_kernels(rows)  # every level by rows: a launch per operation
        t = g.tables()
        if st is None:
            g.upload(p.RHO, synth.gaussian_charge(dom, t["level"], t["ijk"], np.arange(len(t["level"]))))
            g.charge_rhs(1.0, 1.0, True)
        else:
            ne, ni = synth.streamer_densities(dom, st, t["level"], t["ijk"])
            g.upload(p.NE, ne)
            g.upload(p.NI, ni)
            g.charge_rhs(Q, EPS0)
        r1 = g.fmg(1e-30, 3)
        a = g.download(p.PHI)
        r2 = g.solve(1e-30, 9)   # more V-cycles than the exchange tags count before they wrap
        g.vcycles(2)
        out.append((r1, r2, a, g.download(p.PHI)))
        g.close()
    (r1, r2, a, c), (s1, s2, b, d) = out
    assert r1 == s1 and r2 == s2
    assert np.array_equal(a, b) and np.array_equal(c, d)


def test_one_launch_legs_after_regrid_and_switch():
    """New meshes and a change of kernels between solves start the exchange anew."""
    import paper_1708_08434_gb300 as p
    dom, st = synth.workload("streamer_small")
    out = []
    for switch in (False, True):
        g = gpu_mesh(dom, st)
        t = g.tables()
        ne, ni = synth.streamer_densities(dom, st, t["level"], t["ijk"])
        g.upload(p.NE, ne)
        g.upload(p.NI, ni)
        got = []
        for step in range(3):
            g.charge_rhs(Q, EPS0)
            if switch:
                g.set_row_kernels(0)
            g.fmg(1e-9, 30)
            got.append(g.download(p.PHI))
            if switch:
                g.set_row_kernels(2048)
            g.solve(1e-30, 2)
            got.append(g.download(p.PHI))
            f = np.zeros(g.n_boxes, np.int8)
            lv = g.tables()
            leaf = np.flatnonzero((lv["child"][:, 0] < 0) & (lv["level"] == lv["level"].max() - 1))
            f[leaf[step::3]] = 1
            g.regrid(f)
        out.append(got)
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
