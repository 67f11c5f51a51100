"""One call of sm_box_solve_noalloc outside a capture, of any problem count
(0 too), is enough for captures of every other count; without one a capture
is refused.  Each case runs in a process of its own, in which no kernel has
been loaded."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes as C, sys
import torch
import paper_1708_08434_gb300 as pkg
lib, first = pkg.load(), int(sys.argv[1])
torch.cuda.set_device(0)
g = torch.Generator(device="cuda").manual_seed(5)
boxes = {}
for n in (10, 30, 64, 100):  # one of each split of a box over blocks
    boxes[n] = [torch.ones(n, 6, dtype=torch.int32, device="cuda"),
                torch.randn(n, 6, generator=g, device="cuda", dtype=torch.float64),
                torch.randn(n, 512, generator=g, device="cuda", dtype=torch.float64)]
    boxes[n].append(torch.zeros_like(boxes[n][2]))
s = torch.cuda.Stream()
ptr = lambda t: C.c_void_p(t.data_ptr())
call = lambda n, d: lib.sm_box_solve_noalloc(0.7, n, *map(ptr, d), C.c_void_p(s.cuda_stream))
torch.cuda.synchronize()
if first >= 0:
    assert call(first, boxes[first or 10]) == 0
for n, d in boxes.items():
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        rc = call(n, d)
        d[3] += 0.0  # the capture holds something in either case
    if first < 0:
        assert rc == pkg.SM_ECUDA, (n, rc)
        continue
    assert rc == 0, (n, rc)
    graph.replay()
    torch.cuda.synchronize()
    captured = d[3].clone()
    assert call(n, d) == 0
    torch.cuda.synchronize()
    assert torch.isfinite(captured).all() and captured.abs().max() > 0 and torch.equal(captured, d[3]), n
"""


@pytest.mark.parametrize("first", [-1, 0, 64, 100])
def test_one_call_before_captures(first):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE, str(first)], cwd=root, timeout=300, capture_output=True, text=True,
                       env=dict(os.environ, CUDA_MODULE_LOADING="LAZY"))
    assert r.returncode == 0, r.stderr[-2000:]
