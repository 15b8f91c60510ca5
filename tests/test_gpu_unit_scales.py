"""The FP32 gas kernels in units far from SI: densities and pressures that are
each well within FP32's range while their product is not, against the general
kernel on the same grid (relative L1 1e-5, the bar that these two have in SI
units).  Powers of two scale density and pressure; velocities scale with the
root of their ratio."""
import numpy as np
import pytest

import workloads as W
from gpu_util import rel_l1

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2111_11806_gb300.binding")


def waves(n, scale_rho, scale_p, walls=(0,) * 6):
    """A smooth state of 2 % waves without a body."""
    dim = len(n)
    wl = W.random_state(dim, n, 1, False, seed=801, body=False)
    X = W.cell_centres(wl.n, wl.lo, wl.hi)
    L = W.layout(dim, 1, False)
    s = sum(np.sin(2 * np.pi * (X[d] - 0.13 * d)) for d in range(dim)) / dim
    u = float(np.sqrt(scale_p / scale_rho))
    wl.prim[L["irho"]] = scale_rho * 1.2 * (1.0 + 0.02 * s)
    for d in range(dim):
        wl.prim[L["iu"] + d] = u * 60.0 * np.cos(2 * np.pi * X[d])
    wl.prim[L["ip"]] = scale_p * 1e5 * (1.0 + 0.02 * np.roll(s, 7))
    wl.prim[L["ir"]] = 0.0
    wl.walls = walls
    return wl


@pytest.mark.parametrize("scale_rho,scale_p", [(1.0, 1.0), (2.0 ** 61, 2.0 ** 51), (2.0 ** -72, 2.0 ** -72)],
                         ids=["si", "product_above", "product_below"])
@pytest.mark.parametrize("n", [(70, 44), (40, 26, 21)])
def test_gas_kernel_where_the_product_leaves_the_range(n, scale_rho, scale_p):
    wl = waves(n, scale_rho, scale_p, walls=(0, 1, 1, 0, 0, 0))
    got = []
    for general in (False, True):
        g = B.Grid.from_workload(wl, precision=B.DFV_FP32, general_stage=general)
        for _ in range(2):
            g.step(g.compute_dt(0.4))
        g.check()
        got.append(g.cons())
    assert np.all(np.isfinite(got[0]))
    err = rel_l1(got[0], got[1], wl)
    assert np.all(err <= 1e-5), err
