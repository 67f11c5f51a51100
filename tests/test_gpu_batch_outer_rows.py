"""The outer residual of the batched solve by 1, 2 and 4 rows a thread,
chosen by the number of columns: its sums are exact integers, so a solve's
potential is the same bit for bit whatever else is in the batch.  Odd sides,
sides that are no multiple of a column, walls of every kind."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SIDES = [7, 9, 15, 18, 20, 36, 48, 56]


def _solve(fill, bc_type, bc_val):
    import torch
    import paper_1708_08434_gb300 as p
    b = p.Batch(np.array(SIDES + [32] * fill, np.int32), 1.0, bc_type, bc_val)
    b.set_schedule(0, 8)  # one restriction kernel for every batch size
    for s, n in enumerate(SIDES):
        g = torch.Generator(device="cuda").manual_seed(100 + s)
        b.grid(b.rhs, s).copy_(torch.randn(n, n, n, generator=g, device="cuda", dtype=torch.float64))
    for s in range(len(SIDES), len(SIDES) + fill):
        b.grid(b.rhs, s).fill_(1.0)
    b.phi.zero_()
    rc, cyc, rel = b.solve(1e-9, 60)
    assert rc == 0
    out = [b.grid(b.phi, s).clone() for s in range(len(SIDES))], cyc[:len(SIDES)].tolist(), rel[:len(SIDES)].tolist()
    b.close()
    return out


@pytest.mark.parametrize("bc_type,bc_val", [((0, 0, 0, 0, 1, 1), (0.0,) * 5 + (1.0,)),
                                            ((0, 1, 0, 0, 0, 0), (0.0, 2.0, 0.0, 0.0, 0.0, 0.0)),
                                            ((1, 1, 1, 0, 1, 1), (0.3, -1.0, 0.7, 0.0, 1e-3, 5.0))])
def test_same_bits_for_every_number_of_columns(bc_type, bc_val):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cols = sum(-(-n // 32) * -(-n // 16) for n in SIDES)
    few, some, many = (_solve(max(0, -(-(c - cols) // 2)), bc_type, bc_val)
                       for c in (0, int(2.5 * sms), int(3.5 * sms)))  # a side of 32 has two columns
    for other in (some, many):
        assert few[1] == other[1] and few[2] == other[2]
        for x, y in zip(few[0], other[0]):
            assert torch.isfinite(x).all() and torch.equal(x, y)
