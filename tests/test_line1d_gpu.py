"""The time-blocked 1D kernel on the grids AUTO gives it beside periodic FP64 ones:
absorbing ends and FP32 split, against the oracle.

Tolerances: 1e-12 normwise in FP64, 1e-4 in FP32 split.  Sizes: blocks of 2 to 33 cells,
a last block that is not full, windows that hold both ends of a small grid, layers
wider than a block."""
import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NAMES = list(W.FIELD_NAMES) + ["phi_cur", "phi_old"]
LASER = ["E0y", "E0z", "B0y", "B0z"] + [k for k in W.FIELD_NAMES if k[1] == "1"]


def line(nx, bc, prec, pml=20):
    dx = 0.05
    b = W._bcs(bc)
    return W.GridSpec(n=(nx, 1, 1), d=(dx, dx, dx), dt=0.7 * dx, m=1.1, g=0.7, B_ext=(0.3, 0.9, -0.2), axion_bc=b, em_bc=b,
                      pml_cells=pml, precision=prec)


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


def pair(grid, every=0):
    from paper_2406_16796_gb300 import axp

    g = axp.Grid(grid, diag_every=every, diag_capacity=16 if every else 0)
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    st = W.random_state(grid, seed=44, active=LASER)
    g.load(st)
    og.load(st)
    return g, og


@pytest.mark.parametrize("bc,prec,tol", [("pml", "fp64", 1e-12), ("pml", "fp32", 1e-4), ("periodic", "fp32", 1e-4)])
@pytest.mark.parametrize("nx,pml", [(256, 20), (300, 7), (2048, 40), (4999, 20)])
def test_line_matches_the_oracle(nx, pml, bc, prec, tol):
    from paper_2406_16796_gb300 import axp

    grid = line(nx, bc, prec, pml)
    g, og = pair(grid)
    assert g.kernel_path() == axp.AXP_KERNEL_FUSED
    for n in (1, 70, 9):  # within a window, across windows
        og.step(n)
        g.step(n)
        n0 = g.launches()
        rec, ref = g.diagnostics(), og.diagnostics()
        assert g.launches() - n0 <= 3  # E^n was at hand
        for key in ("H_phi", "H_g0", "H_g1"):
            assert rec[key] == pytest.approx(ref[key], rel=1e-10 if prec == "fp64" else 1e-4), key
    n0 = g.launches()
    g.step(40)
    og.step(40)
    assert g.launches() - n0 == 1
    got, ref = g.fields(), og.fields()
    for k in NAMES:
        assert rel(got[k], ref[k]) < tol, (k, rel(got[k], ref[k]))
    g.close()


@pytest.mark.parametrize("bc,prec", [("pml", "fp64"), ("pml", "fp32"), ("periodic", "fp32")])
def test_any_split_of_the_steps_gives_the_same_bits(bc, prec):
    grid = line(777, bc, prec)
    runs = []
    for chunks in ([131], [1, 7, 56, 9, 3, 55]):
        g, _ = pair(grid, every=10)
        for c in chunks:
            g.step(c)
        runs.append((g.fields(), g.read_diagnostics()))
        g.close()
    for k in NAMES:
        assert np.array_equal(runs[0][0][k], runs[1][0][k]), k
    assert [r["step"] for r in runs[0][1]] == list(range(10, 131, 10))
    for a, b in zip(runs[0][1], runs[1][1]):
        assert a == b


@pytest.mark.parametrize("bc", ["pml", "periodic"])
@pytest.mark.parametrize("nx", [256, 1031])
def test_fp32_line_gives_the_generic_kernels_bits(nx, bc):
    """FP32 split: the time-blocked kernel takes the generic single-pass kernel's operations
    (a power-of-two cell size, as in the workloads; other sizes round 1/dx once more)."""
    from paper_2406_16796_gb300 import axp

    w = W.vacuum_1d(nx=nx, g=1e-2, m=0.5 * W.K0, precision="fp32")
    b = W._bcs(bc)
    grid = w.grid.replace(axion_bc=b, em_bc=b)
    out = []
    for kernel in (axp.AXP_KERNEL_AUTO, axp.AXP_KERNEL_FUSED):
        g = axp.Grid(grid)
        g.set_kernel(kernel)
        g.inject_laser(w.lasers[0])
        g.step(300)
        out.append(g.fields())
        g.close()
    for k in NAMES:
        assert np.array_equal(out[0][k], out[1][k]), k


def test_order0_x_components_keep_the_generic_kernel():
    """A layer damps E0x and B0x, which no curl drives: such a state stays with the
    kernel that treats them."""
    grid = line(512, "pml", "fp64")
    g, og = pair(grid)
    kick = W.random_state(grid, seed=45)["E0x"]
    g.write("E0x", kick)
    og.load({"E0x": kick})
    n0 = g.launches()
    g.step(12)
    og.step(12)
    assert g.launches() - n0 >= 12
    got, ref = g.fields(), og.fields()
    for k in NAMES:
        assert rel(got[k], ref[k]) < 1e-12, (k, rel(got[k], ref[k]))
    g.close()
