"""Groups with members of odd width: alone, together, and mixed with members of even width in
one launch a step.  A member's states are the same bits in any company, and the oracle's at
the FP32 split tolerance (1e-4)."""
import time

import numpy as np
import pytest

import oracle
from paper_2406_16796_gb300 import workloads as W

from test_group_gpu import NAMES, loaded, mods

pytestmark = pytest.mark.gpu

ODD = [dict(n=(301, 90), m=1.1, g=0.7, Bz=1.0, bc="periodic", steps=21), dict(n=(63, 47), m=0.0, g=0.3, Bz=0.5, bc="pml", steps=17),
       dict(n=(521, 131), m=0.4, g=0.9, Bz=2.0, bc="periodic_x_pml_y", steps=8)]
EVEN = [dict(n=(300, 90), m=1.1, g=0.7, Bz=1.0, bc="periodic", steps=13), dict(n=(64, 200), m=2.0, g=1.3, Bz=-1.0, bc="periodic_x_pml_y", steps=25),
        dict(n=(518, 33), m=0.4, g=0.9, Bz=2.0, bc="pml", steps=8)]


@pytest.mark.parametrize("graphs", [False, True])
def test_members_of_any_width_are_identical_alone_and_in_the_mix(graphs):
    import torch

    axp, group = mods()
    members = [m for pair in zip(ODD, EVEN) for m in pair]
    G = group.Group(8, 2000, stream=torch.cuda.Stream() if graphs else None, graphs=graphs)
    held = []
    for i, spec in enumerate(members):
        g, grid, st = loaded(axp, spec, 900 + i)
        held.append((g, G.add(g, spec["steps"]), grid, st))
    n0 = G.launches()
    for n in (1, 5, 24):
        G.run(n)
    assert G.launches() - n0 == 30  # one launch a step
    for (g, m, grid, st), spec, i in zip(held, members, range(len(members))):
        G.remove(m)
        assert g.step_count == spec["steps"]
        solo, _, _ = loaded(axp, spec, 900 + i)
        G1 = group.Group(1, 400)
        m1 = G1.add(solo, spec["steps"])
        G1.run(spec["steps"])
        G1.remove(m1)
        G1.close()
        og = oracle.OracleGrid(grid.replace(precision="fp64"))
        og.load(st)
        og.step(spec["steps"])
        a, b, ref = g.fields(), solo.fields(), og.fields()
        for k in NAMES:
            assert np.array_equal(a[k], b[k]), (spec, k)
            nb = np.linalg.norm(ref[k])
            assert np.linalg.norm(a[k] - ref[k]) <= 1e-4 * (nb if nb > 0 else 1.0), (spec, k)
        g.close()
        solo.close()
    G.close()


def test_a_mixed_group_is_not_two_groups_in_a_row():
    import torch

    axp, group = mods()

    def us(sizes):
        gs = [loaded(axp, dict(n=n, m=1.1, g=1e-3, Bz=1.0, bc="pml"), 3)[0] for n in sizes]
        G = group.Group(len(gs), 4096)
        ms = [G.add(g, 10 ** 9) for g in gs]
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            G.run(40)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        for m in ms:
            G.remove(m)
        G.close()
        for g in gs:
            g.close()
        return best / 40

    even, odd = us([(128, 64)] * 8), us([(127, 63)] * 8)
    both = us([(128, 64)] * 8 + [(127, 63)] * 8)
    assert both < 0.9 * (even + odd), (even, odd, both)
