"""The 2D kernel by name on small FP64 grids, which AUTO steps with the folded passes: the
soft source, the moving window, odd step counts and degenerate sizes keep their comparison
with the oracle, and the launches show which of the two ran (one a step against four)."""
import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

from test_soft_source_gpu import beam, grid2d, pair
from test_window_gpu import windowed_pair

pytestmark = pytest.mark.gpu

NAMES = list(W.FIELD_NAMES) + ["phi_cur", "phi_old"]
TM = ["E0z", "B0x", "B0y"] + [k for k in W.FIELD_NAMES if k[1] == "1"]


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


def same(g, og, tol):
    got, ref = g.fields(), og.fields()
    for k in NAMES:
        assert rel(got[k], ref[k]) <= tol, (k, rel(got[k], ref[k]))


def launches_of(g, steps):
    g.step(1)  # (the staggered state entered)
    n0 = g.launches()
    g.step(steps)
    return g.launches() - n0


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
@pytest.mark.parametrize("nx,ny,ybc", [(600, 150, "pml"), (300, 64, "periodic"), (301, 33, "pml")])
def test_soft_source(nx, ny, ybc, prec, tol):
    from paper_2406_16796_gb300 import axp

    src = beam(ny)
    g, og = pair(grid2d(nx, ny, prec, ybc=ybc), src, 120, axp.AXP_KERNEL_TM2D)
    same(g, og, tol)
    d, dr = g.diagnostics(), og.diagnostics()
    assert d["P_g2a"] == pytest.approx(dr["P_g2a"], rel=1e-10 if prec == "fp64" else 1e-3)
    assert launches_of(g, 5) == 5
    g.close()


def test_source_switched_mid_run():
    from paper_2406_16796_gb300 import axp

    grid, src = grid2d(300, 64, "fp64", ybc="periodic"), beam(64, plane=40)
    g, og = axp.Grid(grid), oracle.OracleGrid(grid)
    g.set_kernel(axp.AXP_KERNEL_TM2D)
    for s, n in ((None, 7), (src, 60), (None, 21)):
        for q in (g, og):
            q.set_soft_source(s)
            q.step(n)
    same(g, og, 1e-12)
    g.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
def test_windowed_run(prec, tol):
    from paper_2406_16796_gb300 import axp

    g, og, shifts, _ = windowed_pair(prec, axp.AXP_KERNEL_TM2D, 60)
    assert len(shifts) >= 5
    same(g, og, tol)
    assert g.diagnostics()["H_g0"] == pytest.approx(og.diagnostics()["H_g0"], rel=1e-10 if prec == "fp64" else 1e-4)
    g.close()


@pytest.mark.parametrize("kernel", ["TM2D", "TM2D_LIST"])
@pytest.mark.parametrize("axis,s", [(0, 4), (0, 16), (1, 7)])
def test_staggered_shift(axis, s, kernel):
    from paper_2406_16796_gb300 import axp

    w = W.pulse_2d(nx=300, ny=160, m=0.5 * W.K0, g=1e-2, precision="fp64")
    grid = w.grid.replace(pml_cells=10)
    L = W.LaserSpec(amplitude=0.01, k=(W.K0, 0.0, 0.0), pol=(0.0, 0.0, 1.0), centre=(4.0, 0.0, 0.0), waist=0.8, duration=1.0)
    a, b = axp.Grid(grid), axp.Grid(grid)
    for x in (a, b):
        x.set_kernel(getattr(axp, "AXP_KERNEL_" + kernel))
        x.inject_laser(L)
        x.step(25)
    a.shift_window(axis, s)  # staggered: the bands at the ends alone go through integer time
    axp.axp_set_background_field(b.h, grid.B_ext, grid.E_ext)  # the whole grid at integer time
    b.shift_window(axis, s)
    for steps in (0, 20):
        a.step(steps)
        b.step(steps)
        fa, fb = a.fields(), b.fields()
        for k in NAMES:
            assert rel(fa[k], fb[k]) <= 1e-12, (steps, k, rel(fa[k], fb[k]))
    a.close()
    b.close()


@pytest.mark.parametrize("steps", [1, 3, 7])
@pytest.mark.parametrize("n,bc", [((64, 90, 1), ("periodic", "pml")), ((5, 3, 1), ("periodic", "periodic")), ((8, 16, 1), ("pml", "pml"))])
def test_odd_step_counts_and_tiny_grids(n, bc, steps):
    from paper_2406_16796_gb300 import axp

    b = W._bcs(*bc)
    grid = W.GridSpec(n=n, d=(0.05, 0.07, 0.06), dt=0.02, m=2.0, g=1.3, B_ext=(0.1, -0.2, -1.0), axion_bc=b, em_bc=b,
                      pml_cells=2 if "pml" in bc else 0)
    st = W.random_state(grid, seed=77, active=TM)
    g, og = axp.Grid(grid), oracle.OracleGrid(grid)
    g.set_kernel(axp.AXP_KERNEL_TM2D)
    for q in (g, og):
        q.load(st)
        q.step(steps)
    same(g, og, 1e-12)
    assert not any(g.read(k).any() for k in ("E0x", "E0y", "B0z"))
    g.close()


LINES = [((836, 836, 1), ("pml", "pml"), 4), ((838, 836, 1), ("pml", "pml"), 1), ((70, 10001, 1), ("pml", "pml"), 1),
         ((70, 9999, 1), ("pml", "pml"), 4), ((512, 512, 1), ("periodic", "periodic"), 4), ((700, 700, 1), ("periodic", "periodic"), 1),
         ((2048, 340, 1), ("pml", "periodic"), 1), ((512, 1024, 1), ("pml", "periodic"), 4), ((836, 836, 1), ("periodic", "pml"), 1),
         ((300, 1000, 1), ("periodic", "pml"), 4)]


@pytest.mark.parametrize("n,bc,per_step", LINES)
def test_fp64_grids_around_the_line_between_passes_and_kernel(n, bc, per_step):
    """AUTO: the folded passes up to 700,000 cells with layers on every side, and up to where the
    2D kernel is the faster one with a periodic axis."""
    from paper_2406_16796_gb300 import axp

    b = W._bcs(*bc)
    grid = W.GridSpec(n=n, d=(0.05, 0.05, 0.05), dt=0.03, m=1.1, g=0.7, B_ext=(0.0, 0.2, 1.0), axion_bc=b, em_bc=b,
                      pml_cells=6 if "pml" in bc else 0)
    st = W.random_state(grid, seed=9, active=TM)
    g, og = axp.Grid(grid), oracle.OracleGrid(grid)
    g.load(st)
    og.load(st)
    assert launches_of(g, 2) == 2 * per_step
    og.step(3)
    same(g, og, 1e-12)
    g.close()


@pytest.mark.parametrize("nx,bc,one_launch", [(131072, "pml", True), (131073, "pml", False), (131072, "periodic", True),
                                              (131073, "periodic", False)])
def test_fp32_1d_grids_around_the_line_between_kernels(nx, bc, one_launch):
    """AUTO: the time-blocked 1D kernel up to 2^17 cells, a launch of the generic one per step above."""
    from paper_2406_16796_gb300 import axp

    b = W._bcs(bc)
    grid = W.GridSpec(n=(nx, 1, 1), d=(0.05, 0.05, 0.05), dt=0.035, m=1.1, g=0.7, B_ext=(0.3, 0.9, -0.2), axion_bc=b, em_bc=b,
                      pml_cells=20 if bc == "pml" else 0, precision="fp32")
    st = W.random_state(grid, seed=9, active=["E0y", "E0z", "B0y", "B0z"] + [k for k in W.FIELD_NAMES if k[1] == "1"])
    g, og = axp.Grid(grid), oracle.OracleGrid(grid.replace(precision="fp64"))
    g.load(st)
    og.load(st)
    assert launches_of(g, 9) == (1 if one_launch else 9)
    og.step(10)
    same(g, og, 1e-4)
    g.close()


@pytest.mark.parametrize("bc,prec,per_step", [("outflow", "fp64", 4), ("pml", "fp64", 4), ("pml", "fp32", 1)])
def test_boundary_benchmark_says_what_ran(bc, prec, per_step):
    from paper_2406_16796_gb300 import bccheck

    assert bccheck.reflectivity(bc, precision=prec, n=200, t_end=3.0)["launches_per_step"] == per_step


@pytest.mark.parametrize("n,bc", [((836, 836, 1), ("periodic", "periodic")), ((1300, 530, 1), ("periodic", "pml")),
                                  ((4096, 160, 1), ("pml", "periodic")), ((400, 400, 1), ("pml", "pml"))])
def test_auto_is_not_slower_than_the_named_kernel(n, bc):
    import time

    from paper_2406_16796_gb300 import axp

    b = W._bcs(*bc)
    t = []
    for kernel in (axp.AXP_KERNEL_AUTO, axp.AXP_KERNEL_TM2D):
        g = axp.Grid(W.GridSpec(n=n, d=(0.05, 0.05, 0.05), dt=0.03, m=1.1, g=0.7, B_ext=(0.0, 0.2, 1.0), axion_bc=b, em_bc=b,
                                pml_cells=6 if "pml" in bc else 0))
        g.set_kernel(kernel)
        g.write("E0z", np.full(g.shape, 1e-3))
        g.step(10)
        best = 1e9
        for _ in range(5):
            g.synchronize()
            t0 = time.perf_counter()
            g.step(20)
            g.synchronize()
            best = min(best, time.perf_counter() - t0)
        t.append(best)
        g.close()
    assert t[0] < 1.06 * t[1], t
