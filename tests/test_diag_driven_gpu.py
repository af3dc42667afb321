"""Records of a grid whose laser drives a component it does not inject: a pulse
polarised in the plane (E along y) excites E0x, which the two E levels of the last
step must count as well."""
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_records_count_the_driven_components(prec, tol):
    from paper_2406_16796_gb300 import axp

    w = W.pulse_2d(nx=160, ny=128)
    grid = w.grid.replace(precision=prec, B_ext=(0.0, 1.0, 0.0))
    laser = W.LaserSpec(amplitude=0.01, k=(W.K0, 0.0, 0.0), pol=(0.0, 1.0, 0.0), centre=(2.5, 0.0, 0.0), waist=0.5,
                        duration=0.8)
    g = axp.Grid(grid, diag_every=2, diag_capacity=8)
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    g.inject_laser(laser)
    og.inject_laser(laser)
    g.step(8)
    for rec in g.read_diagnostics():
        og.step(2)
        ref = og.diagnostics()
        for key in ("H_phi", "H_g0", "H_g1", "P_g2a"):
            assert rec[key] == pytest.approx(ref[key], rel=tol), (rec["step"], key)
    g.close()
