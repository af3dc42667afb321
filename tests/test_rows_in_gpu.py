"""Rows of another grid into a grid that never saw an order-0 field: its records and its
steps take what the rows hold.

Tolerances: 1e-12 in FP64; FP32 split 1e-4 for stepped fields, 1e-5 for records of the same
state (the neighbours' averages are formed in float)."""
import math

import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import slab
from paper_2406_16796_gb300 import workloads as W

from test_staged_gpu import NAMES, TM, bcs, grid_of, rel

pytestmark = pytest.mark.gpu

KEYS = ("H_phi", "H_g0", "H_g1", "W", "sum_xB1z2", "sum_B1z2", "gauss_l2")
GRIDS = {
    "2d_uniform_e": dict(n=(40, 31, 1), B=(0.2, 0.9, 0.3), E=(0.3, 0.1, -0.2)),
    "2d_reflect": dict(n=(45, 29, 1), B=(0.2, 0.9, 0.3), ax=bcs("reflect", "pml"), em=bcs("reflect", "pml"), E=(0.1, 0.0, 0.0)),
    "3d_uniform_e": dict(n=(19, 11, 7), B=(0.2, 0.9, 0.3), E=(0.3, 0.1, -0.2)),
    "2d_generic": dict(n=(1255, 800, 1), B=(0.2, 0.9, 0.3), ax=bcs("periodic", "reflect"), em=bcs("periodic", "reflect")),
    "1d_generic": dict(n=(300, 1, 1), B=(0.2, 0.9, 0.3), ax=bcs("reflect"), em=bcs("reflect")),
    "1d_uniform_e": dict(n=(300, 1, 1), B=(0.2, 0.9, 0.3), E=(0.3, 0.1, -0.2)),
}


def rows_of(g):
    return max(a for a in range(3) if g.spec.n[a] > 1 or a == 0)


def hand_over(src, dst):
    import torch
    from paper_2406_16796_gb300 import axp

    n = src.spec.n[rows_of(src)]
    buf = torch.empty(axp.axp_rows_bytes(src.h, n), dtype=torch.uint8, device=src.device)
    axp.axp_pack_rows(src.h, 0, n, buf.data_ptr(), buf.numel())
    axp.axp_unpack_rows(dst.h, 0, n, buf.data_ptr(), buf.numel())
    torch.cuda.synchronize()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
@pytest.mark.parametrize("case", sorted(GRIDS))
def test_a_blank_grid_takes_every_row(case, prec, tol):
    from paper_2406_16796_gb300 import axp

    grid = grid_of(prec=prec, **GRIDS[case])
    st = W.random_state(grid, seed=31)
    src, dst = axp.Grid(grid), axp.Grid(grid)
    src.load(st)
    hand_over(src, dst)
    og = oracle.OracleGrid(grid.replace(precision="fp64"))
    og.load(src.fields())
    for step in (0, 4):
        dst.step(step)
        og.step(step)
        rec, ref = dst.diagnostics(), og.diagnostics()
        for key in KEYS:
            size = abs(ref[key]) if key != "W" else ref["H_phi"] + ref["H_g0"] + ref["H_g1"]
            assert abs(rec[key] - ref[key]) <= (1e-11 if prec == "fp64" else 1e-3 if step else 1e-5) * size, (key, step)
    got, want = dst.fields(), og.fields()
    for k in NAMES:
        assert rel(got[k], want[k]) < tol, (k, rel(got[k], want[k]))
    src.close()
    dst.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
@pytest.mark.parametrize("E", [(0.0, 0.0, 0.0), (0.2, 0.1, 0.0)])
def test_a_laser_crosses_the_cut(E, prec, tol):
    """Two slabs of a 2D grid, the laser's order-0 fields on the first one only (up to the row
    before the cut): the other slab's owned rows take it, in fields and records."""
    from paper_2406_16796_gb300 import axp

    n = (64, 96, 1)
    dt = 0.5 / math.sqrt(2.0) * 0.05
    glob = W.GridSpec(n=n, d=(0.05,) * 3, dt=dt, m=0.7, g=0.5, B_ext=(0.2, 0.1, 0.4), E_ext=E, precision=prec)
    st = W.random_state(glob, seed=17, active=TM)
    for k in ("E0z", "B0x", "B0y"):
        st[k][:, :30, :] = 0.0
        st[k][:, 47:, :] = 0.0
    k, rounds, world = 4, 4, 2
    runs = [slab.SlabRun(glob, r, world, k, slab.LocalComm()) for r in range(world)]
    for r in runs:
        r.load_global(st)
        for name in ("E0z", "B0x", "B0y"):  # the second slab's halo holds laser rows: it knows of none
            if r.plan.rank == 1:
                r.engine.grid.close()
                r.engine.grid = axp.Grid(r.plan.spec)
                blank = {q: np.zeros_like(v) if q in ("E0z", "B0x", "B0y") else v for q, v in st.items()}
                r.load_global(blank)
                break
    # the first exchange brings the halo rows of the laser
    for ph in range(2):
        bufs = {}
        for r in runs:
            send, _ = slab.schedule(r.plan)[ph]
            if send is not None:
                bufs[(r.plan.rank, send[0])] = r.engine.pack(*send[1])
        for r in runs:
            _, recv = slab.schedule(r.plan)[ph]
            if recv is not None:
                r.engine.unpack(recv[1][0], recv[1][1], bufs[(recv[0], r.plan.rank)])
    slab.run_local(runs, rounds)
    rec = slab.combine([r.engine.owned_record() for r in runs])
    got = {name: np.concatenate([r.owned(r.engine.fields())[name] for r in runs], axis=1) for name in NAMES}
    for r in runs:
        r.engine.close()
    og = oracle.OracleGrid(glob.replace(precision="fp64"))
    og.load(st)
    og.step(k * rounds)
    want, ref = og.fields(), og.diagnostics()
    for name in NAMES:
        assert rel(got[name], want[name]) < tol, (name, rel(got[name], want[name]))
    for key in KEYS:
        size = abs(ref[key]) if key != "W" else ref["H_phi"] + ref["H_g0"] + ref["H_g1"]
        assert abs(rec[key] - ref[key]) <= (1e-11 if prec == "fp64" else 1e-3) * size, (key, rec[key], ref[key])
