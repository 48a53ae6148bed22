"""The batch adds the FP32 sums of a level's 64 slots without their rounding, and so compares H with
the stop rule."""
import numpy as np
import pytest

from lbtest import lib

pytestmark = pytest.mark.gpu


# one row to a strip and a slot: 3 to 64 slots of 64, and rows that share slots' two halves
@pytest.mark.parametrize("rows", [3, 5, 11, 37, 61, 64])
@pytest.mark.parametrize("quad,N,nx", [("D2Q16-GH", 2, 32), ("D2Q36-GH", 3, 30), ("D2Q64-GH", 4, 20)])
@pytest.mark.parametrize("shape", [dict(), dict(warp_cells=1 << 20), dict(warp_cells=0)])
def test_sums_over_alike_rows_are_those_of_one_row(quad, N, nx, rows, shape):
    """A shear wave is the same in every row, so A and S, which are means over the rows, are bit for bit
    those of a grid of one row: the sum of up to 64 equal FP32 values takes 24 + 6 bits, which neither FP64
    nor a pair of FP32 rounds, and the one rounding of the normalised sum is the single row's (sums in
    FP32 round for 3, 5, ... rows).  The run ends at the same level (H is the row's times the rows)."""
    lib()
    from paper_0908_4520_gb300 import Batch

    b = Batch("f32", **shape)
    slots = [b.add(quad, N, nx, ny, 0.2, u0=1e-3, max_steps=400, stop_ratio=0.3) for ny in (1, rows)]
    b.run(0).sync()
    (a1, s1), (a, s) = (b.history(k) for k in slots)
    levels = [b.state(k)["level"] for k in slots]
    b.close()
    assert levels[0] == levels[1] and 20 < levels[0] < 400
    np.testing.assert_array_equal(a, a1)
    np.testing.assert_array_equal(s, s1)
