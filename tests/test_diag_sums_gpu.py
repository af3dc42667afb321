"""The diagnostics' sums against the oracle's on the state the grid holds (read back,
so FP32 rounding of the state itself does not enter), for every kernel form: active
axes, order-0 component sets, boundaries, and field magnitudes far apart.

FP64: 1e-11.  FP32 split: the level average phi^n and the 4-point B average are formed
in float, 2^-24 each, and enter differences of like size: 1e-5."""
import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

from test_staged_gpu import CASES, ghosts_of, grid_of

pytestmark = pytest.mark.gpu

KEYS = ("H_phi", "H_g0", "H_g1", "P_g2a", "P_a2g", "W", "sum_xB1z2", "sum_B1z2", "gauss_l2")


@pytest.mark.parametrize("scale1,scale_phi", [(1e-3, 1e-2), (1e-29, 1e-15), (1e15, 1e9)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 1e-5)])
@pytest.mark.parametrize("case", sorted(CASES))
def test_sums_match_the_oracle(case, prec, tol, scale1, scale_phi):
    from paper_2406_16796_gb300 import axp

    kw, active, _ = CASES[case]
    grid = grid_of(prec=prec, **kw)
    g = axp.Grid(grid)
    g.load(W.random_state(grid, seed=71, scale1=scale1, scale_phi=scale_phi, active=active))
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    og.load(g.fields())
    for (a, s), (cur, old) in ghosts_of(grid, 9).items():
        g.write_ghost(a, s, 0, cur * scale_phi)
        g.write_ghost(a, s, 1, old * scale_phi)
        og.set_ghost(a, s, g.read_ghost(a, s, 0).reshape(cur.shape), g.read_ghost(a, s, 1).reshape(cur.shape))
    ref = og.diagnostics()
    for _ in range(2):  # a second record finds the scratch as the first did
        rec = g.diagnostics()
        size = ref["H_phi"] + 2.0 * np.sqrt(ref["H_g0"] * ref["H_g1"])  # W's terms (Cauchy-Schwarz)
        size += 2.0 * np.sqrt(ref["H_g1"] * grid.cells * np.prod(grid.d))
        for key in KEYS:
            assert abs(rec[key] - ref[key]) <= tol * (size if key == "W" else abs(ref[key])) + 1e-300, (key, rec[key], ref[key])
    g.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_field_is_reported(bad):
    from paper_2406_16796_gb300 import axp

    grid = grid_of((40, 30, 1), (0.0, 0.0, 1.0), prec="fp32")
    st = W.random_state(grid, seed=5)
    st["B1x"][0, 11, 17] = bad
    g = axp.Grid(grid)
    g.load(st)
    with pytest.raises(axp.AxpError) as e:
        g.diagnostics()
    assert e.value.status == axp.AXP_E_NONFINITE
    g.close()
