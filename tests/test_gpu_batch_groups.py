"""An instance's history does not depend on the group of warps that advances it: clusters, CTAs, four
warps or one, any launch shape, alone or among others, in chunks or in one launch."""
import numpy as np
import pytest

from lbtest import lib

pytestmark = pytest.mark.gpu

# rows below, at and above the 32 lanes of a ring strip, strips with tails of 1 to 30 cells, fewer and
# more strips than the 64 sums of a level
MIX = [("D2Q36-GH", 3, 2, 1, 0.3), ("D2Q16-GH", 2, 31, 3, 0.2), ("D2Q64-GH", 4, 32, 4, 0.7), ("D2Q36-GH", 4, 33, 1, 1.0),
       ("D2Q16-GH", 3, 61, 2, 0.1), ("D2Q36-GH", 2, 128, 4, 0.3), ("D2Q64-GH", 3, 256, 1, 2.0),
       ("D2Q16-GH", 4, 1024, 4, 0.01), ("D2Q64-GH", 2, 900, 5, 0.1)]


def _histories(mix, steps=90, chunk=0, precision="f32", **kw):
    from paper_0908_4520_gb300 import Batch

    b = Batch(precision, **kw)
    slots = [b.add(*m, u0=1e-3, max_steps=steps, stop_ratio=1e-3) for m in mix]
    for _ in range(1 if chunk == 0 else -(-(steps + 1) // chunk)):
        b.run(chunk)
    b.sync()
    out = [b.history(s) for s in slots]
    b.close()
    return out


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16"])
def test_history_is_the_same_in_every_group(precision):
    lib()
    ref = _histories(MIX, precision=precision)
    shapes = [dict(warp_cells=0), dict(warp_cells=1 << 20), dict(threads=64, warp_cells=0), dict(threads=96),
              dict(threads=128), dict(threads=256, smem_bytes=0), dict(smem_bytes=200 * 1024)]
    for kw in shapes:
        for (a, s), (a0, s0) in zip(_histories(MIX, precision=precision, **kw), ref):
            np.testing.assert_array_equal(a, a0)
            np.testing.assert_array_equal(s, s0)
    for (a, s), (a0, s0) in zip(_histories(MIX, chunk=7, precision=precision), ref):
        np.testing.assert_array_equal(a, a0)
        np.testing.assert_array_equal(s, s0)
    for m, (a0, s0) in zip(MIX, ref):  # alone: the whole card is its share
        (a, s), = _histories([m], precision=precision)
        np.testing.assert_array_equal(a, a0)
        np.testing.assert_array_equal(s, s0)


def test_largest_on_chip_budget_is_still_accepted():
    """The on-chip budget that the device's limit allows beside a kilobyte of the kernel's own."""
    Lattice, capi = lib()
    from paper_0908_4520_gb300 import Batch

    optin = 227 * 1024  # shared memory a block may opt in to
    (a, s), = _histories([MIX[1]], smem_bytes=optin - 1156)
    (a0, s0), = _histories([MIX[1]])
    np.testing.assert_array_equal(a, a0)
    with pytest.raises(capi.LBError):
        Batch("f32", smem_bytes=optin)
