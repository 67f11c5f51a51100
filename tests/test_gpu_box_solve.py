"""sm_box_solve_noalloc at the problem counts where its split over blocks
changes, against the eigenvector solution in FP64 numpy."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _axis(lo, hi):
    """Eigenpairs of the 8-cell second difference with ghosts -phi (1) or phi (0)."""
    a = np.diag(np.full(8, -2.0)) + np.diag(np.ones(7), 1) + np.diag(np.ones(7), -1)
    a[0, 0] += -1.0 if lo else 1.0
    a[7, 7] += -1.0 if hi else 1.0
    return np.linalg.eigh(a)


@pytest.mark.parametrize("n", [1, 19, 20, 38, 39, 76, 77, 300])
def test_box_solve_split_edges(n):
    import torch
    import paper_1708_08434_gb300 as pkg
    rng = np.random.default_rng(n)
    length = 0.37
    h = length / 8
    f = rng.standard_normal((n, 512))
    bt = rng.integers(0, 2, (n, 6)).astype(np.int32)
    bt[np.arange(n), rng.integers(0, 6, n)] = 1
    bv = rng.standard_normal((n, 6))
    d = [torch.from_numpy(x).cuda() for x in (bt, bv, f)]
    phi = torch.full((n, 512), float("nan"), dtype=torch.float64, device="cuda")
    ptr = [C.c_void_p(x.data_ptr()) for x in d + [phi]]
    assert pkg.load().sm_box_solve_noalloc(length, n, *ptr, C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    got = phi.cpu().numpy()
    for p in range(n):
        u = f[p].reshape(8, 8, 8) * h * h  # [z][y][x]
        for face in range(6):
            if bt[p, face]:
                ix = [slice(None)] * 3
                ix[2 - face // 2] = -1 if face & 1 else 0
                u[tuple(ix)] -= 2.0 * bv[p, face]
        e = [_axis(*bt[p, 2 * a:2 * a + 2]) for a in (2, 1, 0)]
        c = np.einsum("zyx,za,yb,xc->abc", u, e[0][1], e[1][1], e[2][1])
        c /= e[0][0][:, None, None] + e[1][0][None, :, None] + e[2][0][None, None, :]
        want = np.einsum("abc,za,yb,xc->zyx", c, e[0][1], e[1][1], e[2][1]).reshape(512)
        assert np.abs(got[p] - want).max() <= 1e-12 * np.abs(want).max(), p
