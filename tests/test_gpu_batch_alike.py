"""Launches of alike instances: the group width chosen by waves gives the histories of whole CTAs."""
import numpy as np
import pytest

from lbtest import lib

pytestmark = pytest.mark.gpu


# counts below, at and above the waves of clusters (76), CTAs (152), four-warp groups (608) and warps (2432);
# one strip, strips for four warps, for a CTA and for clusters
@pytest.mark.parametrize("precision", ["f32", "f16"])
@pytest.mark.parametrize("quad,N,nx,ny,counts", [("D2Q16-GH", 2, 24, 1, (1, 2432, 2433)), ("D2Q36-GH", 3, 64, 1, (1, 608, 609, 1300)),
                                                 ("D2Q64-GH", 4, 250, 1, (76, 77, 153)), ("D2Q16-GH", 3, 130, 9, (1, 76, 152, 153))])
def test_histories_do_not_depend_on_the_count(quad, N, nx, ny, counts, precision):
    """The first and the last instance of each launch, with Kn of their own, against a launch that gives each
    instance a CTA; chunks keep the choice to itself in every launch, also when some have finished."""
    lib()
    from paper_0908_4520_gb300 import Batch

    def run(n, chunk, **kw):
        b = Batch(precision, max_slots=4096, **kw)
        slots = [b.add(quad, N, nx, ny, 0.2 + 1e-4 * i, u0=1e-3, max_steps=20 + i % 3, stop_ratio=0.0) for i in range(n)]
        for _ in range(1 if chunk == 0 else -(-23 // chunk)):
            b.run(chunk)
        b.sync()
        out = [b.history(slots[i]) for i in (0, n - 1)]
        b.close()
        return out

    ref = run(max(counts), 0, warp_cells=0)
    for n in counts:
        for chunk in (0, 8):
            got = run(n, chunk)
            np.testing.assert_array_equal(got[0], ref[0])
            if n == max(counts):
                np.testing.assert_array_equal(got[1], ref[1])
