"""The time-blocked 1D kernel at the edges of what it takes: strong layers, the largest
windows, runs of one step."""
import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

from test_line1d_gpu import LASER, NAMES, line, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [3.9, 6.0, 50.0])
@pytest.mark.parametrize("nx,pml", [(300, 7), (2048, 20)])
@pytest.mark.parametrize("axion", [False, True])
def test_layers_of_any_strength_are_damped(axion, nx, pml, sigma):
    """sigma dt above 4 turns the sign of the layer's 1 - sigma h / 2: such cells are damped
    as the others are, with the generic kernel's bits (FP32, power-of-two cell size).  The
    axion's own layer is unstable from sigma dt = 2 on: with an axion only a few steps.
    Damped quotients below 1e-30 may differ in their last bit: 90 steps of at most 8 of them
    stay within 1e-30 x 2^-23 x 720 < 1e-34."""
    from paper_2406_16796_gb300 import axp

    grid = line(nx, "pml", "fp32", pml).replace(d=(1 / 16, 1 / 16, 1 / 16), dt=0.7 / 16, pml_sigma_max_dt=sigma)
    if not axion:
        grid = grid.replace(g=0.0)
    steps = 5 if axion else 90
    st = W.random_state(grid, seed=44, active=LASER)
    if not axion:
        for k in ("phi_cur", "phi_old"):
            st[k] = np.zeros_like(st[k])
    out = []
    for kernel in (axp.AXP_KERNEL_AUTO, axp.AXP_KERNEL_FUSED):
        g = axp.Grid(grid)
        g.load(st)
        g.set_kernel(kernel)
        g.step(steps)
        out.append(g.fields())
        g.close()
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    og.load(st)
    og.step(steps)
    ref = og.fields()
    for k in NAMES:
        assert np.all(np.abs(out[0][k] - out[1][k]) <= 1e-34), (k, rel(out[0][k], out[1][k]))
        assert rel(out[0][k], ref[k]) < 1e-4, (k, rel(out[0][k], ref[k]))


@pytest.mark.parametrize("nx", [118712, 118714, 131072, 146528])
def test_large_periodic_grids_keep_the_kernel(nx):
    """Up to 964 cells a block (152 SMs), chosen by AUTO and by name, with the generic
    kernel's fields."""
    from paper_2406_16796_gb300 import axp

    grid = line(nx, "periodic", "fp64")
    st = W.random_state(grid, seed=44, active=LASER)
    out = []
    for kernel in (axp.AXP_KERNEL_BLOCK1D, axp.AXP_KERNEL_FUSED):
        g = axp.Grid(grid)
        assert g.kernel_path() == axp.AXP_KERNEL_BLOCK1D
        g.load(st)
        g.set_kernel(kernel)
        g.step(40)
        out.append(g.fields())
        g.close()
    for k in NAMES:
        assert rel(out[0][k], out[1][k]) < 1e-12, (k, rel(out[0][k], out[1][k]))


def us_per_call(g, steps, calls=300):
    import time

    best = 1e9
    for _ in range(7):
        g.synchronize()
        t0 = time.perf_counter()
        for _ in range(calls):
            g.step(steps)
        g.synchronize()
        best = min(best, (time.perf_counter() - t0) / calls)
    return best * 1e6


@pytest.mark.parametrize("nx,bc", [(256, "periodic"), (4096, "periodic"), (65536, "periodic"), (2048, "pml")])
def test_single_steps_cost_no_more_than_a_launch_of_the_generic_kernel(nx, bc):
    """step(1) in FP32: a run of one window takes neither the counter's reset nor a
    cooperative launch (both together: 1.2 to 2.0 times the generic kernel's call)."""
    from paper_2406_16796_gb300 import axp

    t = []
    for kernel in (axp.AXP_KERNEL_AUTO, axp.AXP_KERNEL_FUSED):
        g = axp.Grid(line(nx, bc, "fp32"))
        g.load(W.random_state(g.spec, seed=44, active=LASER, scale0=1e-3))
        g.set_kernel(kernel)
        t.append(us_per_call(g, 1))
        g.close()
    assert t[0] < 1.15 * t[1], t


def test_runs_of_one_window_and_of_several_mix():
    """Any split of the steps, periodic FP64 too: the same bits, whichever launch a run takes."""
    from paper_2406_16796_gb300 import axp

    out = []
    for chunks in ([200], [1] * 20 + [14, 15, 16, 100, 35], [60, 1, 139]):
        g = axp.Grid(line(4999, "periodic", "fp64"))
        g.load(W.random_state(g.spec, seed=44, active=LASER))
        for c in chunks:
            g.step(c)
        out.append(g.fields())
        g.close()
    for k in NAMES:
        assert np.array_equal(out[0][k], out[1][k]) and np.array_equal(out[0][k], out[2][k]), k


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_record_beside_a_layer_that_stops_the_field(prec, tol):
    """One layer cell with sigma dt = 4 (1 - sigma h / 2 = 0): the record's divergence next to it
    takes E^n of that cell, which no half-step can be undone to."""
    grid = line(300, "pml", prec, 1).replace(d=(1 / 16, 1 / 16, 1 / 16), dt=1 / 32, pml_sigma_max_dt=4.0, g=0.0)
    st = W.random_state(grid, seed=44, active=LASER)
    for k in ("phi_cur", "phi_old"):
        st[k] = np.zeros_like(st[k])
    from paper_2406_16796_gb300 import axp

    g = axp.Grid(grid)
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    g.load(st)
    og.load(st)
    for n in (1, 30):
        g.step(n)
        og.step(n)
        rec, ref = g.diagnostics(), og.diagnostics()
        for key in ("H_g0", "H_g1", "gauss_l2", "sum_B1z2"):
            assert abs(rec[key] - ref[key]) <= tol * abs(ref[key]), (key, n, rec[key], ref[key])
    g.close()
