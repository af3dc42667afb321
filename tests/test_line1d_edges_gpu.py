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
