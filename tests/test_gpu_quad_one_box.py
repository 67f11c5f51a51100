"""A quadtree of one box and no room for more: a regrid that changes nothing,
or that is refused for want of room, leaves the solver as it was."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flag", [0, 1])
def test_solve_after_regrid_on_one_box(flag):
    import paper_1708_08434_gb300 as p
    dom = synth.Domain2(0.016, 1, 1, synth.CARTESIAN, bc_val=(0.0, 0.0, 0.0, 1.0))
    g = p.Quad(dom, 1)
    rhs = np.random.default_rng(3).standard_normal((1, 64))
    out = []
    for again in range(2):
        g.upload(p.RHS, rhs)
        g.upload(p.PHI, np.zeros((1, 64)))
        g.solve(0.0, 1)
        out.append(g.download(p.PHI))
        if again:
            break
        if flag:
            with pytest.raises(p.SmError) as e:
                g.regrid(np.ones(1, np.int8))
            assert e.value.code == p.SM_ENOMEM
        else:
            assert g.regrid(np.zeros(1, np.int8)) == (0, 0, 0)
    g.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
