"""GPU parity of 3-D grids of two fluids (air and water, per-cell noise on every
primitive) against the oracle in both precisions: ragged tiles, a body at
rest, in prescribed motion and free, walls, and single cells in a direction.
The bars of the plain parity tests: relative L1 per plane FP64 <= 1e-12 after
one step and <= 1e-8 after several with the device's own dt, FP32 <= 1e-4."""
import numpy as np
import pytest

import workloads as W
from gpu_util import rel_l1, run_both

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2111_11806_gb300.binding")


def case(n, seed, **body):
    wl = W.random_state(3, n, 2, False, seed=seed)
    for k, v in body.items():
        setattr(wl, k, v)
    return wl


FREE = dict(body_dynamic=True, body_mass=30.0, body_x=(0.6, 0.45, 0.5), body_v=(5.0, -3.0, 2.0))
CASES = [
    ("rest_36x21x18", lambda: case((36, 21, 18), 701)),
    ("moving_33x17x19", lambda: case((33, 17, 19), 702, body_v=(25.0, -15.0, 20.0))),
    ("free_40x14x13", lambda: case((40, 14, 13), 703, **FREE)),
    ("walls_35x9x10", lambda: case((35, 9, 10), 704, walls=(0, 1, 1, 0, 1, 1))),
    ("exact_tiles_32x8x4", lambda: case((32, 8, 4), 705)),
    ("thin_31x1x2", lambda: case((31, 1, 2), 706)),
]


@pytest.mark.parametrize("precision,bar", [(B.DFV_FP64, 1e-12), (B.DFV_FP32, 1e-4)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_one_step(name, make, precision, bar):
    wl = make()
    o, g = run_both(wl, 1, precision)
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= bar), err


def test_several_steps_of_a_free_body_fp64():
    wl = CASES[2][1]()
    o, g = run_both(wl, 8, B.DFV_FP64, cfl=0.5, use_run=True)
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= 1e-8), err
    for got, want in zip(g.body(), o.body()):
        np.testing.assert_allclose(got, want, rtol=1e-8, atol=1e-8 * np.abs(want).max())
