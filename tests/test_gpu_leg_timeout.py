"""A wait between the blocks of a one-launch leg that runs out: the call is
run again in a launch per operation from the potential it started with, so
its result is that of the row kernels bit for bit, and so are the following
ones; a new mesh has its legs back."""
import time

import numpy as np
import pytest

import synth
from helpers import EPS0, Q, gpu_mesh

pytestmark = pytest.mark.gpu


def _solver():
    import paper_1708_08434_gb300 as p
    dom, st = synth.workload("streamer_small")
    g = gpu_mesh(dom, st)
    t = g.tables()
    ne, ni = synth.streamer_densities(dom, st, t["level"], t["ijk"])
    g.upload(p.NE, ne)
    g.upload(p.NI, ni)
    g.set_table(synth.coefficient_table())
    g.charge_rhs(Q, EPS0)
    g.fmg(1e-4, 30)
    return p, g


CALLS = {
    "fmg": lambda g: g.fmg(1e-9, 30)[1:],
    "solve": lambda g: g.solve(1e-9, 30)[1:],
    "two_cycles": lambda g: g.solve(0.0, 2)[1:],
    "vcycles": lambda g: g.vcycles(2),
    "host_loop": lambda g: (g.set_graphs(False), g.solve(1e-9, 30)[1:], g.set_graphs(True))[1],
    "advance": lambda g: g.advance(1e-13, Q, EPS0, 1e-9, 30)[1:],
}


@pytest.mark.parametrize("call", sorted(CALLS))
def test_call_runs_again_without_legs(call):
    out = []
    for arm in (False, True):
        p, g = _solver()
        if call == "advance":
            g.compute_field()
        if arm:
            g.leg_wait_selftest()
            t0 = time.time()
        got = [CALLS[call](g), g.download(p.PHI), g.download(p.NE)]
        if arm:
            assert 0.02 < time.time() - t0 < 20.0
        n0 = g.launch_count()
        got += [g.solve(1e-30, 2)[1:], g.download(p.PHI)]
        launches = [g.launch_count() - n0]
        f = np.zeros(g.n_boxes, np.int8)
        t = g.tables()
        f[t["level"] == t["level"].max()] = -1
        assert g.regrid(f)[1] > 0
        n0 = g.launch_count()
        got += [g.solve(1e-30, 2)[1:], g.download(p.PHI)]
        launches.append(g.launch_count() - n0)
        out.append((got, launches))
        g.close()
    (a, la), (b, lb) = out
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert lb[0] > la[0] and lb[1] == la[1]
