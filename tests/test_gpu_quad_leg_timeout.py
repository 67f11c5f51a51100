"""A wait between the warps of a quadtree's one-launch leg that runs out: a
solve is run again in a launch per operation from the potential it started
with (1e-12 of the potential against the solve with legs: rounding order
differs); V-cycles, which are enqueued only, report it at the next call that
waits for the stream."""
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
Q, EPS0 = synth.E_CHARGE, synth.EPS0


def _quad():
    import paper_1708_08434_gb300 as p
    dom, st = synth.workload2("axi_small")
    g = p.Quad(dom, 1 << 12)
    synth.refine_all2(dom, st, g.level_ij, g.refine_level)
    t = g.tables()
    ne, ni = synth.streamer_densities2(dom, st, t["level"], t["ij"])
    g.upload(p.NE, ne)
    g.upload(p.NI, ni)
    g.set_table(synth.coefficient_table())
    g.charge_rhs(Q, EPS0)
    g.fmg(1e-4, 30)
    g.compute_field()
    return p, g


CALLS = {
    "fmg": lambda g: g.fmg(1e-9, 30)[2],
    "solve": lambda g: g.solve(1e-9, 30)[2],
    "two_cycles": lambda g: g.solve(0.0, 2)[2],
    "host_loop": lambda g: (g.set_graphs(False), g.solve(1e-9, 30)[2], g.set_graphs(True))[1],
    "advance": lambda g: g.advance(1e-13, Q, EPS0, 1e-9, 30)[2:],
}


@pytest.mark.parametrize("call", sorted(CALLS))
def test_solve_runs_again_without_legs(call):
    out = []
    for arm in (False, True):
        p, g = _quad()
        if arm:
            g.leg_wait_selftest()
            t0 = time.time()
        got = [CALLS[call](g), g.download(p.PHI), g.download(p.NE)]
        if arm:
            assert 0.02 < time.time() - t0 < 20.0
        n0 = g.launch_count()
        got += [g.solve(0.0, 2)[2], g.download(p.PHI)]
        launches = [g.launch_count() - n0]
        t = g.tables()
        assert g.regrid(np.where(t["level"] == t["level"].max(), -1, 0).astype(np.int8))[1] > 0
        n0 = g.launch_count()
        got += [g.solve(0.0, 2)[2], g.download(p.PHI)]
        launches.append(g.launch_count() - n0)
        out.append((got, launches))
        g.close()
    (a, la), (b, lb) = out
    for x, y in zip(a, b):
        if isinstance(x, np.ndarray):
            assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max()
        else:
            assert x == y
    assert lb[0] > la[0] and lb[1] == la[1]


REPORT = {
    "download": lambda p, g: g.download(p.PHI),
    "dt_limit": lambda p, g: g.dt_limit(Q, EPS0),
    "regrid": lambda p, g: g.regrid(np.where(g.tables()["level"] == g.n_levels - 1, -1, 0).astype(np.int8)),
}


@pytest.mark.parametrize("by", sorted(REPORT))
@pytest.mark.parametrize("graphs", [True, False])
def test_vcycles_report_at_the_next_wait(by, graphs):
    p, g = _quad()
    g.set_graphs(graphs)
    boxes = g.n_boxes
    g.leg_wait_selftest()
    g.vcycles(2)
    with pytest.raises(p.SmError) as e:
        REPORT[by](p, g)
    assert e.value.code == p.SM_ETIMEOUT and g.n_boxes == boxes
    REPORT[by](p, g)  # reported once
    g.close()


def test_solve_after_vcycles_that_ran_out():
    out = []
    for arm in (False, True):
        p, g = _quad()
        if arm:
            g.leg_wait_selftest()
        g.vcycles(1)
        rc, rel, _ = g.solve(1e-10, 40)
        assert rc == 0 and rel <= 1e-10
        out.append(g.download(p.PHI))
        g.close()
    # both are converged to 1e-10 of the right-hand side
    assert np.abs(out[0] - out[1]).max() <= 1e-7 * np.abs(out[0]).max()
