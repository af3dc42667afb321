"""The FP32 2D kernel's two forms (warp tiles on grids up to 1.2M cells, block tiles above)."""
import time

import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TM = ["E0z", "B0x", "B0y"] + [k for k in W.FIELD_NAMES if k[1] == "1"]


def grid_of(nx, ny, bcx="periodic", bcy=None):
    b = W._bcs(bcx, bcy or bcx)
    return W.GridSpec(n=(nx, ny, 1), d=(0.05, 0.05, 0.05), dt=0.03, m=1.1, g=0.7, B_ext=(0.2, 0.9, 0.4), axion_bc=b, em_bc=b,
                      pml_cells=0 if (bcx, bcy or bcx) == ("periodic", "periodic") else 6, precision="fp32")


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


@pytest.mark.parametrize("bcx,bcy", [("periodic", "periodic"), ("pml", "pml"), ("periodic", "pml"), ("pml", "periodic")])
@pytest.mark.parametrize("nx,ny", [(58, 7), (60, 50), (116, 33), (250, 129), (252, 13), (502, 200)])
def test_warp_and_block_tiles_give_the_same_bits(nx, ny, bcx, bcy):
    """AUTO's warp tiles (58 columns) and the named kernel's block tiles (up to 250), both against
    the oracle (1e-4 normwise): widths around their strips, heights of less than a chunk."""
    from paper_2406_16796_gb300 import axp

    grid = grid_of(nx, ny, bcx, bcy)
    if min(ny, nx) < 2 * grid.pml_cells:
        grid = grid.replace(pml_cells=3)
    st = W.random_state(grid, seed=8, active=TM)
    out = []
    for kernel in (axp.AXP_KERNEL_AUTO, axp.AXP_KERNEL_TM2D):
        g = axp.Grid(grid)
        g.load(st)
        g.set_kernel(kernel)
        assert g.kernel_path() == axp.AXP_KERNEL_TM2D
        g.step(9)
        out.append(g.fields())
        g.close()
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    og.load(st)
    og.step(9)
    ref = og.fields()
    for k in list(W.FIELD_NAMES) + ["phi_cur", "phi_old"]:
        assert np.array_equal(out[0][k], out[1][k]), k
        assert rel(out[0][k], ref[k]) < 1e-4, (k, rel(out[0][k], ref[k]))


@pytest.mark.parametrize("nx,ny", [(1202, 1000), (60, 20010), (1000, 1200)])
@pytest.mark.parametrize("bcx,bcy", [("periodic", "periodic"), ("periodic", "pml"), ("pml", "periodic")])
def test_grids_around_the_line_between_the_forms(nx, ny, bcx, bcy):
    """1.2M cells and just above, where AUTO turns to block tiles."""
    from paper_2406_16796_gb300 import axp

    grid = grid_of(nx, ny, bcx, bcy)
    st = W.random_state(grid, seed=8, active=TM)
    g = axp.Grid(grid)
    g.load(st)
    g.step(2)
    got = g.fields()
    g.close()
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    og.load(st)
    og.step(2)
    ref = og.fields()
    for k in list(W.FIELD_NAMES) + ["phi_cur", "phi_old"]:
        assert rel(got[k], ref[k]) < 1e-4, (k, rel(got[k], ref[k]))


@pytest.mark.parametrize("bc", ["periodic", "pml"])
def test_single_steps_of_a_narrow_grid_are_not_bound_by_their_plan(bc):
    """The plan of the warp tiles is made once: searched on every call it took 0.36 ms of the
    host's time on this grid, seven steps' worth."""
    from paper_2406_16796_gb300 import axp

    g = axp.Grid(grid_of(16, 65536, bc))
    t = {}
    for n in (50, 1):
        g.step(n)
        best = 1e9
        for _ in range(5):
            g.synchronize()
            t0 = time.perf_counter()
            for _ in range(100 // n):
                g.step(n)
            g.synchronize()
            best = min(best, time.perf_counter() - t0)
        t[n] = best
    g.close()
    assert t[1] < 1.5 * t[50], t
