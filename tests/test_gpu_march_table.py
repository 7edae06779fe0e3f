"""The FP32 march's medium table: how many cubic pieces a profile takes, and rays
that leave the table (against the FP64 march, which checks every lookup)."""
import math

import numpy as np
import pytest

from oracle.swkb_oracle import rel_l2
from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def _bent(n_top, n_low=400, cols=1):
    """Nearly horizontal rays bent upwards by eps = 1 + 0.03 z: 3 units over a screen
    of 20 (from the highest ghost at 22 to about 26.3, less than the three ghost
    rays' 6 units, so that the screen stays covered), on a table ending n_top
    intervals of 1/8 above the grid's top at 16."""
    k, n_z, height = 2.0 * math.pi, 64, 16.0
    n_p = n_low + int(height * 8) + n_top
    xs = [0.0, 20.0, 40.0][:cols]
    prof = w._table(xs, -n_low / 8.0, 0.125, n_p, [w.f_linear(1.0, 0.03)] * cols)
    u0 = w.gaussian_beam(height / n_z * np.arange(n_z), k, 8.0, 2.0, 0.0)
    return w.Problem("bent", k, 0.0, height, n_z, w.BC_PERIODIC, 0.0, 20.0, 1, prof, u0, 0.5, 8, 8, 0.0, n_max=1)


@pytest.mark.parametrize("cols", [1, 3])
@pytest.mark.parametrize("precision", [swkb.SWKB_FP64, swkb.SWKB_MIXED])
def test_rays_leaving_the_table_are_an_error(precision, cols):
    # the plan's own reach check asks for 66 intervals, the rays for about 82
    statuses = []
    for n_top in range(60, 100):
        try:
            plan = swkb.Plan(_bent(n_top, cols=cols), precision)
        except swkb.SwkbError as e:
            assert e.status == swkb.SWKB_ERR_INVALID_ARG
            statuses.append("plan")
            continue
        try:
            plan.propagate()
            statuses.append("ok")
        except swkb.SwkbError as e:
            assert e.status == swkb.SWKB_ERR_RANGE
            statuses.append("range")
    # first refused at creation, then by the march, then carried
    assert statuses == sorted(statuses, key=["plan", "range", "ok"].index)
    assert "range" in statuses and "ok" in statuses
    # the two precisions agree on where the table is long enough
    if precision == swkb.SWKB_MIXED:
        n_ok = 60 + statuses.index("ok")
        with pytest.raises(swkb.SwkbError):
            swkb.Plan(_bent(n_ok - 1, cols=cols), swkb.SWKB_FP64).propagate()
        assert np.all(np.isfinite(swkb.Plan(_bent(n_ok, cols=cols), swkb.SWKB_FP64).propagate()))


@pytest.mark.parametrize("problem,pieces", [
    # curvature below the table's rounding, zero curvature, a lens the table resolves, a kinked duct
    (lambda: w.config_open_lens(n_z=8192, fc_patch=910, fc_overlap=248, n_screens=2), (1,)),
    (lambda: w.config_unit_periodic(n_screens=7), (1,)),
    (lambda: w.config_gaussian_lens_40km().with_(n_screens=2), (1,)),
    (lambda: w.config_surface_duct_small(n_screens=2), (2, 4, 8, 16)),
])
def test_pieces_and_mixed_parity(problem, pieces):
    pb = problem()
    plan = swkb.Plan(pb, swkb.SWKB_MIXED)
    assert plan.info.medium_pieces in pieces
    # the mixed path's bar against the FP64 path
    assert rel_l2(plan.propagate(), swkb.Plan(pb, swkb.SWKB_FP64).propagate()) < 1e-4


@pytest.mark.parametrize("dx", [50.0, 5.0, 1.0])
def test_pieces_follow_the_table_alone(dx):
    # the duct's 1 m blends ask for 16 pieces however short the screens are; a linear medium's curvature
    # is the table's rounding, for which one piece does
    duct = w.config_surface_duct_small().with_(dx=dx)
    assert swkb.Plan(duct, swkb.SWKB_MIXED).info.medium_pieces == 16
    assert swkb.Plan(w.config_unit_periodic().with_(dx=20.0 * dx / 50.0), swkb.SWKB_MIXED).info.medium_pieces == 1


def test_tables_with_ordinary_rounding_take_one_piece():
    # a broad lens given by its refractive index: eps = n^2 is rounded once more
    pb = w.config_gaussian_medium(a=2e-4, b=1e-6)
    pr = pb.profile
    pb = pb.with_(profile=w.Profile(pr.x_cols, pr.z0, pr.dz, np.sqrt(pr.eps) ** 2, pr.eps_z, pr.eps_zz))
    assert swkb.Plan(pb, swkb.SWKB_MIXED).info.medium_pieces == 1
