"""The folded multi-pass kernels that AUTO takes where no single-pass kernel fits
(outflow sides, a uniform E, FP64 3D, lasers outside the TM set), against the oracle.

Tolerances are the fused kernels': 1e-12 normwise in FP64 and 1e-4 in FP32 split,
after a few steps from a random state.  Sizes: ragged against the 256-thread blocks,
axes of 2 and 3 cells, an inactive middle axis, every boundary kind."""
import math

import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NAMES = list(W.FIELD_NAMES) + ["phi_cur", "phi_old"]
bcs = W._bcs
TE = ["E0x", "E0y", "B0z"] + [k for k in W.FIELD_NAMES if k[1] == "1"]
TM = ["E0z", "B0x", "B0y"] + [k for k in W.FIELD_NAMES if k[1] == "1"]
CASES = {
    # name: (grid, non-zero arrays or None, path)
    "1d_outflow": (dict(n=(263, 1, 1), B=(0.1, 0.9, 0.2), ax=bcs("outflow"), em=bcs("pml")), None, 1),
    "1d_outflow_tm": (dict(n=(70, 1, 1), B=(0.0, 0.9, 0.2), ax=bcs("outflow"), em=bcs("pml")), ["E0z", "B0y", "E1z"], 1),
    "2d_outflow_tm": (dict(n=(61, 37, 1), B=(0.0, 0.0, 1.0), ax=bcs("outflow", "outflow"), em=bcs("pml", "pml")), TM, 1),
    "2d_outflow_mixed": (dict(n=(36, 31, 1), B=(0.0, 0.4, 1.0), ax=bcs("outflow", ("reflect", "pml")),
                              em=bcs("pml", ("reflect", "pml")), E=(0.1, 0.0, -0.05)), None, 1),
    "2d_te_pml": (dict(n=(75, 44, 1), B=(0.2, 0.9, 0.0), ax=bcs("pml", "pml"), em=bcs("pml", "pml")), TE, 2),
    "2d_tm_pml": (dict(n=(61, 37, 1), B=(0.0, 0.0, 1.0), ax=bcs("pml", "pml"), em=bcs("pml", "pml")), TM, None),
    "2d_te_periodic": (dict(n=(50, 33, 1), B=(0.2, 0.9, 0.3)), TE, 2),
    "2d_all_reflect": (dict(n=(45, 29, 1), B=(0.2, 0.9, 0.3), ax=bcs("reflect", "pml"), em=bcs("reflect", "pml")), None, 2),
    "2d_no_laser_reflect": (dict(n=(45, 29, 1), B=(0.2, 0.9, 0.3), ax=bcs("reflect", "pml"), em=bcs("reflect", "pml")),
                            [k for k in W.FIELD_NAMES if k[1] == "1"], 2),
    "3d_pml_x": (dict(n=(19, 11, 7), B=(0.2, 0.9, 0.3), ax=bcs("pml"), em=bcs("pml")), None, 1),
    "3d_outflow": (dict(n=(9, 10, 11), B=(0.2, 0.9, 0.3), ax=bcs("outflow", "periodic", "outflow"),
                        em=bcs("pml", "periodic", "reflect"), E=(0.0, 0.2, 0.1)), None, 1),
    "3d_no_laser_pml": (dict(n=(9, 12, 8), B=(0.2, 0.9, 0.3), ax=bcs("pml", "pml", "pml"), em=bcs("pml", "pml", "pml")),
                        [k for k in W.FIELD_NAMES if k[1] == "1"], None),
    "xz_uniform_e": (dict(n=(21, 1, 13), B=(0.2, 0.9, 0.3), E=(0.3, 0.1, -0.2)), None, 1),
    "3d_tiny": (dict(n=(2, 3, 2), B=(0.2, 0.9, 0.3), E=(0.3, 0.1, -0.2)), None, 1),
}


def grid_of(n, B, ax=bcs(), em=bcs(), E=(0.0, 0.0, 0.0), prec="fp64", pml=3):
    d = (0.05, 0.07, 0.06)
    dt = 0.5 / math.sqrt(sum(1.0 / d[a] ** 2 for a in range(3) if n[a] > 1))
    return W.GridSpec(n=n, d=d, dt=dt, m=1.1, g=0.7, B_ext=B, E_ext=E, axion_bc=ax, em_bc=em, pml_cells=pml, precision=prec)


def ghosts_of(grid, seed):
    rng = np.random.default_rng(seed)
    return {(a, s): (rng.uniform(-1e-2, 1e-2, oracle.plane_shape(grid, a)), rng.uniform(-1e-2, 1e-2, oracle.plane_shape(grid, a)))
            for a in range(3) for s in range(2) if grid.axion_bc[a][s] == "outflow"}


def start(grid, active, kernel=None):
    from paper_2406_16796_gb300 import axp

    g = axp.Grid(grid)
    if kernel is not None:
        g.set_kernel(kernel)
    g.load(W.random_state(grid, seed=606, active=active))
    for (a, s), (cur, old) in ghosts_of(grid, 7).items():
        g.write_ghost(a, s, 0, cur)
        g.write_ghost(a, s, 1, old)
    return g


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
@pytest.mark.parametrize("case", sorted(CASES))
def test_staged_step_matches_the_oracle(case, prec, tol):
    kw, active, path = CASES[case]
    grid = grid_of(prec=prec, **kw)
    g = start(grid, active)
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    og.load(W.random_state(grid, seed=606, active=active))
    for (a, s), (cur, old) in ghosts_of(grid, 7).items():
        og.set_ghost(a, s, cur, old)
    if path is not None:
        assert g.kernel_path() == path
    for n in (1, 6):
        og.step(n)
        g.step(n)
        got, ref = g.fields(), og.fields()
        for k in NAMES:
            assert rel(got[k], ref[k]) < tol, (case, n, k, rel(got[k], ref[k]))
    for (a, s), _ in ghosts_of(grid, 7).items():
        assert rel(g.read_ghost(a, s, 0).reshape(og.ghost[a][s][0].shape), og.ghost[a][s][0]) < tol
    g.close()


@pytest.mark.parametrize("case", ["2d_outflow_mixed", "3d_pml_x", "1d_outflow"])
def test_any_split_of_the_steps_gives_the_same_bits(case):
    kw, active, _ = CASES[case]
    grid = grid_of(**kw)
    whole, parts, resumed = start(grid, active), start(grid, active), start(grid, active)
    whole.step(9)
    for n in (1, 3, 5):
        parts.step(n)
    resumed.step(4)
    image = resumed.save_state()
    again = start(grid, active)
    again.load_state(image)
    again.step(5)
    ref = whole.fields()
    for other in (parts, again):
        got = other.fields()
        for k in NAMES:
            assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
def test_staged_step_with_a_soft_source_matches_the_oracle(prec, tol):
    from paper_2406_16796_gb300 import axp

    grid = grid_of((60, 25, 1), (0.2, 0.9, 0.3), bcs("pml", "pml"), bcs("pml", "pml"), prec=prec)
    src = W.SourceSpec(amplitude=0.3, k=4.0, pol=(0.0, 0.8, 0.6), plane=12, centre=(0.5, 0.9, 0.0), waist=0.5, duration=0.8,
                       t_centre=0.4)
    g = axp.Grid(grid)
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    st = W.random_state(grid, seed=33)
    g.load(st)
    og.load(st)
    g.set_soft_source(src)
    og.set_soft_source(src)
    g.step(8)
    og.step(8)
    assert g.kernel_path() == axp.AXP_KERNEL_GENERAL
    got, ref = g.fields(), og.fields()
    for k in NAMES:
        assert rel(got[k], ref[k]) < tol, (k, rel(got[k], ref[k]))
