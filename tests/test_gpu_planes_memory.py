"""Plans with inner planes when device memory is short: the arrays that let several planes be summed at once
are given up before the plan is."""
import ctypes

import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def _duct():
    return w.config_surface_duct_small(n_screens=2, rk4_steps=8)


def _bytes_one_by_one(pb, precision, planes):
    """Device bytes of a plan whose inner planes are summed one at a time (as they are with a single one)."""
    i = swkb.Plan(pb, precision, planes=2).info
    size = 8 if precision == swkb.SWKB_FP64 else 4
    return i.device_bytes + (planes - 2) * (3 * i.march_modes * i.n_rays_total + 2 * i.n_modes) * size


@pytest.mark.parametrize("precision", [swkb.SWKB_FP64, swkb.SWKB_MIXED])
def test_refused_plane_arrays_leave_one_plane_at_a_time(precision, monkeypatch):
    pb = _duct()
    plan = swkb.Plan(pb, precision, planes=8)
    want, full = plan.propagate_planes(8), plan.info.device_bytes
    least = _bytes_one_by_one(pb, precision, 8)
    assert full > least + (1 << 20)
    sizes = []
    for n in range(1, 64):
        monkeypatch.setenv("SWKB_FAIL_ALLOC_AT", str(n))
        try:
            plan = swkb.Plan(pb, precision, planes=8)
        except swkb.SwkbError as e:
            assert e.status == swkb.SWKB_ERR_OOM
            continue
        monkeypatch.delenv("SWKB_FAIL_ALLOC_AT")
        sizes.append(plan.info.device_bytes)
        assert np.array_equal(plan.propagate_planes(8), want)
        if sizes[-1] == full:      # n is past the last allocation
            break
    assert sizes[:-1] == [least] * 4 and sizes[-1] == full      # coefficients, partials and two bracket tables


def test_served_requests_take_no_plane_arrays():
    # a budget that holds the request's plan with one plane at a time holds the request
    pb = _duct()
    keep = swkb._Keep()
    prof, dom = swkb.make_profile(pb.profile, keep), swkb.swkb_domain(pb.z_a, pb.z_b, pb.x0, pb.bc)
    opt = swkb.options_for(pb, swkb.SWKB_MIXED, planes=8)
    u = np.ascontiguousarray(pb.u0, dtype=np.complex128)
    req = swkb.swkb_request(ctypes.pointer(prof), pb.k, ctypes.pointer(dom), pb.n_z, pb.dx, ctypes.pointer(opt),
                            u.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 0, pb.n_screens)
    srv = swkb.Server(_bytes_one_by_one(pb, swkb.SWKB_MIXED, 8) + 4096, max_slots=1)
    try:
        st, t = swkb.swkb_submit(srv.handle, req)
        assert st == swkb.SWKB_OK
        srv.n_z[t] = pb.n_z
        st, out = srv.poll(t)
        assert st == swkb.SWKB_OK
        assert np.array_equal(out, swkb.Plan(pb, swkb.SWKB_MIXED).propagate())
    finally:
        srv.close()


@pytest.mark.parametrize("precision", [swkb.SWKB_FP64, swkb.SWKB_MIXED])
def test_an_inner_plane_holds_its_rays_and_coefficients(precision):
    # three arrays of rays, the range-phase factors and the coefficients in polar form; nothing else
    pb = _duct()
    i, j = (swkb.Plan(pb, precision, planes=n).info for n in (0, 2))
    size = 8 if precision == swkb.SWKB_FP64 else 4
    assert j.device_bytes - i.device_bytes == (3 * i.march_modes * i.n_rays_total + 4 * i.n_modes) * size
