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


def _columns(pb, x_cols):
    """The problem with the medium of its first two columns on other range columns."""
    pr = pb.profile
    i = np.arange(len(x_cols)) % 2
    return pb.with_(profile=w.Profile(np.asarray(x_cols, float), pr.z0, pr.dz, pr.eps[i], pr.eps_z[i], pr.eps_zz[i]))


def _ducts():
    pb = w.config_surface_duct_small(n_screens=2)
    pr = pb.profile
    return pb.with_(profile=w._table([0.0, 50.0], pr.z0, pr.dz, pr.n_p,
                                     [w.f_trilinear_duct(12.0, -0.1), w.f_trilinear_duct(15.0, -0.1)]))


def test_mixed_tables_hold_each_column_once():
    pb = _ducts()
    infos = {n: swkb.Plan(_columns(pb, np.linspace(0.0, 200.0, n)), swkb.SWKB_MIXED).info for n in (3, 5, 9)}
    bytes_of = {n: i.device_bytes for n, i in infos.items()}
    column = (2 * (pb.profile.n_p - 1) + 1) * 16 * infos[3].medium_pieces   # mirrored and one more, 4 floats a piece
    assert bytes_of[5] - bytes_of[3] == 2 * column and bytes_of[9] - bytes_of[5] == 4 * column


@pytest.mark.parametrize("make", [_ducts, w.config_unit_periodic], ids=["grounded", "periodic"])
def test_small_and_large_tables_blend_alike(make):
    # FP64: small tables hold differences, larger ones (here by columns beyond the screens) do not; the blended
    # coefficients differ by a unit in the last place of e = eps - eps_ref, which is below 0.1 here: 2e-17 of k x / 2
    pb = make().with_(n_screens=2)
    xs = [0.0, 0.7 * pb.dx, 2.5 * pb.dx]
    small = swkb.Plan(_columns(pb, xs), swkb.SWKB_FP64)
    per = (pb.profile.n_p - 1) * 128
    far = 2.5 * pb.dx + np.arange(1, (8 << 20) // per + 3)
    large = swkb.Plan(_columns(pb, np.concatenate([xs, far])), swkb.SWKB_FP64)
    assert large.info.device_bytes - small.info.device_bytes < 0.6 * per * len(far) + (1 << 20)
    a, b = small.propagate(), large.propagate()
    assert rel_l2(a, b) < 1e-12


@pytest.mark.parametrize("precision", [swkb.SWKB_FP64, swkb.SWKB_MIXED])
def test_a_column_met_exactly_is_taken_exactly(precision):
    # screens between equal columns: whatever the blend's weight, the field of the column alone.  FP64 small tables
    # add zero differences, FP32 blends th c + (c - th c), a rounding per coefficient at most
    pb = _ducts()
    pr = pb.profile
    same = pb.with_(profile=w.Profile(np.array([0.0, 30.0, 110.0]), pr.z0, pr.dz, pr.eps[[0, 0, 0]], pr.eps_z[[0, 0, 0]],
                                      pr.eps_zz[[0, 0, 0]]))
    one = pb.with_(profile=w.Profile(np.array([0.0]), pr.z0, pr.dz, pr.eps[:1], pr.eps_z[:1], pr.eps_zz[:1]))
    a, b = (swkb.Plan(p, precision).propagate() for p in (same, one))
    if precision == swkb.SWKB_FP64:
        assert np.array_equal(a, b)
    else:
        assert rel_l2(a, b) < 1e-6
