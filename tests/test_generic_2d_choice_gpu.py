"""FP32 2D grids of the generic kernel's path: AUTO keeps the generic kernel where the folded
passes, which go over the state four times, are slower; the fields are the oracle's either way."""
import time

import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ONE = [k for k in W.FIELD_NAMES if k[1] == "1"]
SETS = {"none": [], "tm": ["E0z", "B0x", "B0y"], "te": ["E0x", "E0y", "B0z"], "all": [k for k in W.FIELD_NAMES if k[1] == "0"]}


def grid_of(nx, ny, bcx, bcy):
    b = W._bcs(bcx, bcy)
    return W.GridSpec(n=(nx, ny, 1), d=(0.05, 0.05, 0.05), dt=0.02, m=1.1, g=0.7, B_ext=(0.2, 0.9, 0.3), axion_bc=b, em_bc=b,
                      pml_cells=8 if "pml" in (bcx, bcy) else 0, precision="fp32")


def us_per_step(g):
    best = 1e9
    g.step(10)
    for _ in range(5):
        g.synchronize()
        t0 = time.perf_counter()
        g.step(20)
        g.synchronize()
        best = min(best, (time.perf_counter() - t0) / 20)
    return best * 1e6


@pytest.mark.parametrize("nx,ny,bcx,bcy,comps", [(2048, 1024, "periodic", "periodic", "te"), (2048, 2048, "periodic", "periodic", "all"),
                                                 (2048, 2048, "reflect", "reflect", "none"), (1536, 1400, "periodic", "reflect", "tm"),
                                                 (4096, 2048, "periodic", "pml", "te"), (512, 512, "periodic", "periodic", "te"),
                                                 (1024, 1024, "pml", "pml", "te")])
def test_auto_is_not_slower_than_the_generic_kernel(nx, ny, bcx, bcy, comps):
    from paper_2406_16796_gb300 import axp

    t = []
    for kernel in (axp.AXP_KERNEL_AUTO, axp.AXP_KERNEL_FUSED):
        g = axp.Grid(grid_of(nx, ny, bcx, bcy))
        g.set_kernel(kernel)
        for k in SETS[comps] + ["phi_cur"]:
            g.write(k, np.full(g.shape, 1e-3))
        t.append(us_per_step(g))
        g.close()
    assert t[0] < 1.1 * t[1], t


@pytest.mark.parametrize("nx,ny,bcx,bcy,comps,per_step", [(1002, 800, "periodic", "periodic", "te", 1), (700, 700, "periodic", "periodic", "te", 4),
                                                          (1004, 1204, "reflect", "reflect", "none", 4), (1756, 900, "reflect", "reflect", "none", 1),
                                                          (1255, 1000, "periodic", "reflect", "all", 1)])
def test_either_choice_gives_the_oracles_fields(nx, ny, bcx, bcy, comps, per_step):
    from paper_2406_16796_gb300 import axp

    grid = grid_of(nx, ny, bcx, bcy)
    st = W.random_state(grid, seed=12, active=SETS[comps] + ONE)
    g, og = axp.Grid(grid), oracle.OracleGrid(grid.replace(precision="fp64"))
    g.load(st)
    og.load(st)
    assert g.kernel_path() == axp.AXP_KERNEL_FUSED
    g.step(1)
    n0 = g.launches()
    g.step(2)
    assert g.launches() - n0 == 2 * per_step
    og.step(3)
    got, ref = g.fields(), og.fields()
    for k in list(W.FIELD_NAMES) + ["phi_cur", "phi_old"]:
        nb = np.linalg.norm(ref[k])
        assert np.linalg.norm(got[k] - ref[k]) <= 1e-4 * (nb if nb > 0 else 1.0), k
    rec, want = g.diagnostics(), og.diagnostics()
    for key in ("H_phi", "H_g0", "H_g1"):
        assert rec[key] == pytest.approx(want[key], rel=1e-4), key
    g.close()
