"""Plastic-strain planes where a material's partial density fades out: cells
that a solid was absent from take masses that fall by orders of magnitude a
cell, down through the subnormal doubles, and the specific strain of such a
cell, the quotient of two of them, stays finite (FP64).  Against the oracle after
one step: masses, energy and strains, relative L1 1e-12.  (The stretch of the air
beside the fading solid hangs on the ratio of two vanishing shear impedances,
which a tie in the choice between face values can move by decades; it and later
steps are held to being finite.)"""
import numpy as np
import pytest

import workloads as W
from gpu_util import rel_l1, run_both

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2111_11806_gb300.binding")


def struck_plate():
    """Copper striking the wedge, its fraction exactly 0 in the air."""
    wl = W.with_history(W.impact_2d(96, solid_material=W.COPPER), seed=3, amp=0.01)
    L = W.layout(2, 2, True, True)
    block = wl.prim[L["iphi"]] > 0.5
    wl.prim[L["iphi"]] = np.where(block, 1.0, 0.0)
    wl.prim[L["iu"]] = np.where(block, 400.0, 0.0)
    wl.prim[L["iu"] + 1] = 0.0
    return wl, L


@pytest.mark.parametrize("solid", [W.COPPER, W.ALUMINIUM], ids=["johnson_cook", "perfectly_plastic"])
def test_masses_of_any_size_one_step(solid):
    """Fractions from 1e-290 to 1e-323 side by side: masses on both sides of
    the smallest normal double."""
    wl = W.with_history(W.impact_2d(40, solid_material=solid), seed=4, amp=0.01)
    L = W.layout(2, 2, True, True)
    air = wl.prim[L["iphi"]] < 0.5
    wl.prim[L["iphi"]] = np.where(air, 10.0 ** -np.linspace(290.0, 323.0, wl.ncell), wl.prim[L["iphi"]])
    mass = wl.prim[L["iphi"]][air] * solid["rho0"]
    assert np.any((mass > 0) & (mass < 2.2e-308))
    o, g = run_both(wl, 1, B.DFV_FP64)
    got = g.cons()
    assert np.all(np.isfinite(got))
    planes = [L["irho"], L["irho"] + 1, L["ip"], L["ih"], L["ih"] + 1]
    err = rel_l1(got, o.cons(), wl)[planes]
    assert np.all(err <= 1e-12), err


def test_fading_copper_stays_finite():
    wl, L = struck_plate()
    o, g = run_both(wl, 16, B.DFV_FP64, cfl=0.6)
    mass = o.cons()[L["irho"]]
    assert np.any((mass > 0) & (mass < 2.2e-308))
    assert np.all(np.isfinite(g.cons()))
