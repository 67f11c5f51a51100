"""The FP64 kernels' own square root, division, reciprocal and halving over
their ranges.  Each ends in a correction whose error before the last rounding
is far below an ulp (2^-65, 2^-92 relative), so it is at most one ulp from the
correctly rounded value; special values and halves are exact."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0x5EED, 77])
def test_against_the_library(seed):
    import paper_1708_08434_gb300 as pkg
    root, special, quotient, reciprocal, halves = pkg.check_arithmetic(1 << 26, seed)
    assert special == 0 and halves == 0
    assert root <= 1 and quotient <= 1 and reciprocal <= 1
