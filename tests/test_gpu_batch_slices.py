"""Four-warp groups that step on chip beside single warps of the groups that have run out of work:
each keeps to its own slice of the shared memory, at budgets that 16 warps do not share evenly."""
import numpy as np
import pytest

from lbtest import lib

pytestmark = pytest.mark.gpu

LARGEST = 227 * 1024 - 1156  # the largest on-chip budget that is accepted


# cells: the two buffers of a D2Q16-GH instance fill a four-warp group's slice to the last 16 to 112
# bytes (for the largest budget: of what the kernel's own shared memory leaves of it)
@pytest.mark.parametrize("precision,smem_bytes,cells", [("f32", 100000, 195), ("f16", 100000, 390),
                                                        ("f32", LARGEST, 437), ("f16", LARGEST, 875)])
def test_groups_keep_to_their_slices(precision, smem_bytes, cells):
    """2000 instances for the four-warp groups (of 7 to 30 strips, each far less than half of the launch's
    mean load) and 1000 for single warps: the histories are those of the run through global memory."""
    lib()
    from paper_0908_4520_gb300 import Batch

    mix = [("D2Q16-GH", 2, cells, 1, 0.1 + 0.0004 * i, 40 + i % 7) for i in range(2000)]
    mix += [("D2Q16-GH", 3, 20 + i % 13, 1, 0.3 + 0.001 * i, 40 + i % 50) for i in range(1000)]
    runs = []
    for budget in (0, smem_bytes):
        b = Batch(precision, smem_bytes=budget)
        slots = [b.add(*m[:5], u0=1e-3, max_steps=m[5], stop_ratio=0.0) for m in mix]
        b.run(0).sync()
        runs.append([b.history(s) for s in slots])
        b.close()
    for (a, s), (a0, s0) in zip(*runs):
        np.testing.assert_array_equal(a, a0)
        np.testing.assert_array_equal(s, s0)
