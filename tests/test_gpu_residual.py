"""The FP64 residual of leaf boxes formed in per-box fixed point (k_resnorm)
against the oracle's plain FP64 residual, on potentials whose boxes differ by
up to 24 orders of magnitude.  Bound: the map to fixed point errs by at most
6.5 2^-58 of the box's largest value and the oracle's sum by a few 2^-53 of
it, against a residual of the order of that value: 1e-13 with the divisions'
rounding, 1e-12 taken."""
import numpy as np
import pytest

import oracle
import synth
from helpers import gpu_mesh, load_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,decades,bct", [("streamer_small", 0, None), ("streamer_small", 12, None),
                                              ("streamer_small", 12, (1, 0, 1, 1, 0, 1)), ("uniform32", 12, None)])
def test_residual_over_magnitudes(name, decades, bct):
    import paper_1708_08434_gb300 as p
    dom, st = synth.workload(name)
    if bct is not None:
        dom.bc_type = bct
    o = oracle.build_mesh(dom, st)
    g = gpu_mesh(dom, st, precision=p.MIXED)
    t = o.tables()
    load_inputs(dom, st, o, g, t)
    r = np.random.default_rng(5)
    phi = o.get(oracle.PHI)
    phi = r.standard_normal(phi.shape) * 10.0 ** r.integers(-decades, decades + 1, (phi.shape[0], 1))
    g.upload(p.PHI, phi)
    rc, rel, cyc = g.solve(1e-30, 1)
    assert cyc == 1
    o.set(oracle.PHI, g.download(p.PHI))
    assert rel == pytest.approx(o.rel_residual(), rel=1e-12)

