"""The node-split FP64 step kernel where every warp takes several tiles, one after another, in the
same shared arrays: the automatic choice there, against the plain-load kernel."""
import numpy as np
import pytest

from lbtest import lib, random_fields

pytestmark = pytest.mark.gpu

CELLS = {"D2Q16-GH": 8, "D2Q36-GH": 5, "D2Q64-GH": 4}  # cells of a warp


@pytest.mark.parametrize("quad,N,nx,ny", [("D2Q64-GH", 4, 200, 100), ("D2Q64-GH", 3, 34, 600), ("D2Q36-GH", 3, 256, 64)])
@pytest.mark.parametrize("forced", [False, True])
def test_several_tiles_a_warp_give_the_plain_kernels_bits(quad, N, nx, ny, forced):
    """Equal populations after single levels and a chain.  The records' sums are FP64 sums in another
    order, each term in a chain of under a hundred additions (1e-14): within 1e-12 of the largest."""
    import torch

    Lattice, capi = lib()
    blocks = 4 * torch.cuda.get_device_properties(0).multi_processor_count  # at most, of four warps
    assert -(-nx // CELLS[quad]) * ny > 4 * blocks  # more tiles than warps
    kw = dict(precision="f64", force_amp=1e-3 if forced else 0.0, force_freq=1.0)
    fields = random_fields(nx, ny, nx + ny)
    runs = []
    for kernel in ("auto", "plain"):
        with Lattice(quad, N, nx, ny, 0.3, step_kernel=kernel, **kw) as L:
            assert L.info["node_split"] == (1 if kernel == "auto" else 0)
            L.init_fields(*fields)
            L.step(1).step(2).step(33)
            runs.append((L.populations(), L.diagnostics()))
    np.testing.assert_array_equal(runs[0][0], runs[1][0])
    for k in runs[0][1].dtype.names:
        a, b = runs[0][1][k], runs[1][1][k]
        scale = max(np.max(np.abs(b)), nx * ny if k == "mass" else 1e-2 * (nx * ny if k.startswith("mom") else 1.0))
        assert np.max(np.abs(a - b)) <= 1e-12 * scale, k


def test_the_small_grids_run_the_node_split_kernel():
    """Grids of part of a warp up to a few blocks' worth: the automatic choice for every product set, free
    and forced; upwind streaming, on-lattice sets and FP32 keep their kernels."""
    Lattice, capi = lib()
    for quad, N in (("D2Q16-GH", 2), ("D2Q36-GH", 3), ("D2Q64-GH", 4)):
        for nx, ny in ((2, 1), (6, 2), (34, 3), (40, 1), (130, 17)):
            for f in (0.0, 1e-3):
                with Lattice(quad, N, nx, ny, 0.3, precision="f64", force_amp=f) as L:
                    assert L.info["node_split"] == 1, (quad, nx, ny, f)
    for quad, kw in (("D2Q16-GH", dict(precision="f64", streaming="upwind2")), ("D2Q37", dict(precision="f64")),
                     ("D2Q16-GH", dict(precision="f32"))):
        with Lattice(quad, 2, 40, 1, 0.3, **kw) as L:
            assert L.info["node_split"] == 0
