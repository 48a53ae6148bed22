"""The batch's stop rule at a threshold that a level's H meets to FP32 rounding: every group of warps
stops at the same level, whether a plain sum decides or the exact one has to."""
import numpy as np
import pytest

from lbtest import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quad,N,nx,ny", [("D2Q16-GH", 2, 96, 3), ("D2Q36-GH", 3, 256, 1), ("D2Q64-GH", 4, 150, 9),
                                          ("D2Q16-GH", 3, 330, 7)])
def test_threshold_on_a_levels_h(quad, N, nx, ny):
    """stop_ratio = sqrt(H(n) / H(0)) of the single lattice's record, which the batch's H meets to some
    1e-7, nearer than the 2^-20 within which a plain FP32 sum does not decide.  H falls by far more than that
    a level, so the run ends at level n or n + 1, and at the same one with every shape."""
    Lattice, capi = lib()
    from paper_0908_4520_gb300 import Batch

    levels = (9, 10, 17, 30)
    with Lattice(quad, N, nx, ny, 0.2) as L:
        L.init_shear_wave(1e-3)
        L.step(40)
        h = L.diagnostics()["hnorm"]
    for n in levels:  # (from equilibrium H starts level)
        assert h[n] < (1 - 1e-4) * h[n - 1] and h[n + 1] < (1 - 1e-4) * h[n]
    ends = []
    for kw in (dict(), dict(warp_cells=1 << 20), dict(warp_cells=0), dict(threads=128), dict(threads=64, warp_cells=0)):
        b = Batch("f32", **kw)
        slots = [b.add(quad, N, nx, ny, 0.2, u0=1e-3, max_steps=60, stop_ratio=float(np.sqrt(h[n] / h[0]))) for n in levels]
        b.run(0).sync()
        ends.append([b.state(s)["level"] for s in slots])
        b.close()
    for n, end in zip(levels, ends[0]):
        assert end in (n + 1, n + 2), (n, end)  # levels run: 0 to n, or one more
    assert all(e == ends[0] for e in ends)
