"""The paths of small grids: the node-split FP64 step kernel against the plain-load one, and records
that a chained launch leaves to the launch behind it."""
import numpy as np
import pytest

from lbtest import lib, random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quad,N,forced", [("D2Q16-GH", 2, False), ("D2Q16-GH", 4, True), ("D2Q36-GH", 3, False),
                                           ("D2Q36-GH", 1, True), ("D2Q64-GH", 4, False), ("D2Q64-GH", 3, True)])
# cells of a warp: 8, 5 and 4; grids of one cell pair, of part of a warp, of whole and ragged warps,
# of more warps than SMs (blocks of several warps, several tiles a warp)
@pytest.mark.parametrize("nx,ny", [(2, 1), (6, 2), (34, 3), (40, 1), (130, 17)])
def test_node_split_and_plain_kernels_are_bitwise_equal(quad, N, forced, nx, ny):
    """Same per-cell arithmetic in the same order: equal populations.  The grid sums are FP64 sums in
    another order: within 1e-12 of the largest of their kind (1e4 terms of relative rounding 1e-16)."""
    Lattice, capi = lib()
    kw = dict(precision="f64", force_amp=1e-3 if forced else 0.0, force_freq=1.0, isothermal=N == 1)
    fields = random_fields(nx, ny, 11 + nx)
    runs = []
    for kernel in ("auto", "plain"):
        with Lattice(quad, N, nx, ny, 0.3, step_kernel=kernel, **kw) as L:
            L.init_fields(*fields)
            L.step(1).step(2).step(33)
            runs.append((L.populations(), L.diagnostics()))
    np.testing.assert_array_equal(runs[0][0], runs[1][0])
    for k in runs[0][1].dtype.names:
        a, b = runs[0][1][k], runs[1][1][k]
        scale = max(np.max(np.abs(b)), nx * ny if k == "mass" else 1e-2 * (nx * ny if k.startswith("mom") else 1.0))
        assert np.max(np.abs(a - b)) <= 1e-12 * scale, k


@pytest.mark.parametrize("quad,N,nx,ny,precision", [("D2Q16-GH", 2, 64, 1, "f64"), ("D2Q36-GH", 3, 70, 9, "f32"),
                                                    ("D2Q37", 3, 70, 9, "f32"), ("D2Q36-GH", 3, 70, 9, "f16")])
def test_records_of_chained_and_single_launches_are_equal(quad, N, nx, ny, precision):
    """A launch inside a chain leaves its record to the launch behind it; chains of 32, 2 and 1 levels
    and one level at a time give the same records and populations."""
    Lattice, capi = lib()
    fields = random_fields(nx, ny, 5)
    runs = []
    for steps in ((32, 2, 1, 67), (1,) * 102):
        with Lattice(quad, N, nx, ny, 0.2, precision=precision) as L:
            L.init_fields(*fields)
            for n in steps:
                L.step(n)
            runs.append((L.populations(), L.diagnostics()))
    np.testing.assert_array_equal(runs[0][0], runs[1][0])
    assert len(runs[0][1]) == len(runs[1][1]) == 103
    for k in runs[0][1].dtype.names:
        np.testing.assert_array_equal(runs[0][1][k], runs[1][1][k])


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_records_of_a_non_finite_state_are_flagged_in_a_chain(precision):
    """Every record of a state with a NaN in it carries the flag, also those that a chained launch
    leaves to the launch behind it, and the read-back reports the state."""
    import ctypes

    Lattice, capi = lib()
    rho, ux, uy, T = random_fields(32, 1, 3)
    uy = uy.copy()
    uy[0, 5] = np.nan
    with Lattice("D2Q16-GH", 2, 32, 1, 0.2, precision=precision) as L:
        L.init_fields(rho, ux, uy, T)
        L.step(40)
        out, n = (capi.lb_diag * 64)(), ctypes.c_int(0)
        assert capi.lib.lb_diagnostics(L.h, out, 64, ctypes.byref(n)) == capi.LB_ERR_UNSTABLE
        assert n.value == 41 and all(out[i].flags != 0.0 for i in range(41))
