"""Store-staged step kernel on grids with more tiles than blocks: every warp fills its
shared-memory slot again while its TMA store of the tile before may still be in flight."""
import numpy as np
import pytest

from lbtest import lib, random_fields

pytestmark = pytest.mark.gpu


# tiles of 9 rows (q = 64: 7) x 60 columns (16-bit: 56); the widths leave a last tile of a few cells
# in its first or its second half, the heights a partial last tile row
@pytest.mark.parametrize("quad,N,prec,nx,ny", [("D2Q36-GH", 3, "f32", 1028, 200), ("D2Q36-GH", 1, "f32", 996, 181),
                                               ("D2Q16-GH", 2, "f32", 1060, 190),
                                               ("D2Q36-GH", 3, "f16", 1016, 182), ("D2Q64-GH", 4, "bf16", 992, 148)])
def test_slots_filled_many_times_give_the_plain_kernels_bits(quad, N, prec, nx, ny):
    """Same per-cell arithmetic and rounding streams: equal populations, on fields that differ in every cell."""
    Lattice, capi = lib()
    fields = random_fields(nx, ny, nx + ny)
    runs = []
    for kernel in ("tma_store", "plain"):
        with Lattice(quad, N, nx, ny, 0.3, precision=prec, step_kernel=kernel) as L:
            assert L.info["tma_staged"] == (2 if kernel == "tma_store" else 0)
            L.init_fields(*fields)
            L.step(3).step(32)
            runs.append(L.populations())
    np.testing.assert_array_equal(*runs)
