"""Records of FP32 grids are sums in double or better of the floats the grid holds: against
exact sums (math.fsum over the products of two floats, which a double holds exactly).

Bound: a thread's sum is rounded once; the block's and the grid's trees add at most 5 + 3 + 3 + 5 +
3 roundings and the factors 4 more, all of positive terms: 24 x 2^-53 = 2.7e-15.  In a stripe
of cells that one thread sums, the other threads add zeros and only 8 x 2^-53 = 9e-16 is left."""
import math

import numpy as np
import pytest

from paper_2406_16796_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ORDER0 = [k for k in W.FIELD_NAMES if k[1] == "0"]
ORDER1 = [k for k in W.FIELD_NAMES if k[1] == "1"]
STRIDE = 456 * 256  # cells between two that one thread of a 2D record sums


def check(g, tol):
    rec, f = g.diagnostics(), g.fields()
    d = np.array(g.spec.d, dtype=np.float32).astype(np.float64)
    dV = d[0] * d[1] * d[2]
    total = lambda names: math.fsum(x for k in names for x in (f[k].ravel() ** 2).tolist())
    x = np.arange(1, g.spec.n[0] + 1, dtype=np.float64)[None, None, :]
    # (i + 1) B1z^2 needs more than a double's bits: the square split in two, each part exact
    b2 = f["B1z"] ** 2
    hi = b2.astype(np.float32).astype(np.float64)
    centroid = math.fsum((x * hi).ravel().tolist() + (x * (b2 - hi)).ravel().tolist())
    ref = {"H_g0": 0.5 * dV * total(ORDER0), "H_g1": 0.5 * dV * total(ORDER1), "sum_B1z2": dV * total(["B1z"]),
           "sum_xB1z2": d[0] * dV * centroid}
    for k, v in ref.items():
        assert abs(rec[k] - v) <= tol * v, (k, abs(rec[k] - v) / v)


def grid_of(n):
    return W.GridSpec(n=n, d=(0.05, 0.07, 0.06), dt=0.02, m=1.1, g=0.7, B_ext=(0.3, 0.9, 0.2), precision="fp32")


def random_fields(g, rng, keep=None):
    for k in W.FIELD_NAMES:
        a = rng.standard_normal(g.shape) * 10.0 ** rng.uniform(-3, 0, g.shape)
        if keep is not None:
            a = a * keep.reshape(g.shape)
        g.write(k, a)


@pytest.mark.parametrize("n", [(300, 1, 1), (64, 50, 1), (2048, 1024, 1), (96, 64, 40)])
def test_sums_of_many_cells(n):
    from paper_2406_16796_gb300 import axp

    g = axp.Grid(grid_of(n))
    random_fields(g, np.random.default_rng(5))
    check(g, 24 * 2.0 ** -53)
    g.close()


@pytest.mark.parametrize("seed", range(8))
def test_one_threads_sum_is_rounded_once(seed):
    from paper_2406_16796_gb300 import axp

    g = axp.Grid(grid_of((2048, 1024, 1)))
    keep = np.zeros(g.cells)
    keep[7 + seed::STRIDE] = 1.0
    random_fields(g, np.random.default_rng(seed), keep)
    check(g, 8 * 2.0 ** -53)
    g.close()


def test_positions_beyond_24_bits():
    """sum_xB1z2 of a 1D grid of more than 2^24 cells: the cell's number is not a float."""
    from paper_2406_16796_gb300 import axp

    n = (1 << 24) + 4099
    g = axp.Grid(W.GridSpec(n=(n, 1, 1), d=(0.5, 1.0, 1.0), dt=0.25, precision="fp32"))
    a = np.zeros(n)
    cells = [(1 << 24) + 2, (1 << 24) + 4098]
    for c in cells:
        a[c] = 1.5
    g.write("B1z", a)
    rec = g.diagnostics()
    assert rec["sum_xB1z2"] == 0.5 * 0.5 * 2.25 * sum(c + 1 for c in cells)
    g.close()
