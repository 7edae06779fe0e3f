"""The overlapped sequence (march and brackets on streams of their own, two ray-buffer sets) against one
stream: the same kernels on the same arguments, so the fields are equal bit for bit."""
import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def _ducts(pb):
    pr = pb.profile
    return pb.with_(profile=w._table([0.0, 150.0], pr.z0, pr.dz, pr.n_p,
                                     [w.f_trilinear_duct(12.0, -0.1), w.f_trilinear_duct(15.0, -0.1)]))


CASES = {
    "duct": lambda: w.config_surface_duct_small(n_screens=5),
    "range": lambda: _ducts(w.config_surface_duct_small(n_screens=5)),
    "periodic": lambda: w.config_unit_periodic(n_screens=7),
    "open": lambda: w.config_open_lens(n_z=8000, fc_patch=800, fc_overlap=200, n_screens=5),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("precision", [swkb.SWKB_FP64, swkb.SWKB_MIXED])
def test_forced_overlap_gives_identical_fields(name, precision, monkeypatch):
    pb = CASES[name]()
    monkeypatch.setenv("SWKB_OVERLAP", "0")
    one = swkb.Plan(pb, precision)
    monkeypatch.setenv("SWKB_OVERLAP", "1")
    two = swkb.Plan(pb, precision)
    rays = one.info.march_modes * one.info.n_rays_total * (8 if precision == swkb.SWKB_FP64 else 4)
    assert two.info.device_bytes > one.info.device_bytes + 3 * rays       # a second set of ray buffers
    for every in (0, 1):
        assert np.array_equal(one.propagate(snapshot_every=every), two.propagate(snapshot_every=every))
    assert np.array_equal(one.propagate(q0=1, n_screens=4), two.propagate(q0=1, n_screens=4))


def test_long_fp64_marches_overlap_by_themselves(monkeypatch):
    # 489 modes x 2086 rays
    pb = w.config_surface_duct(rk4_steps=2).with_(n_screens=5)
    monkeypatch.delenv("SWKB_OVERLAP", raising=False)
    two = swkb.Plan(pb, swkb.SWKB_FP64)
    monkeypatch.setenv("SWKB_OVERLAP", "0")
    one = swkb.Plan(pb, swkb.SWKB_FP64)
    assert two.info.march_modes * two.info.n_rays_total >= 400000
    assert two.info.device_bytes > one.info.device_bytes + 3 * 400000 * 8
    assert np.array_equal(one.propagate(snapshot_every=1), two.propagate(snapshot_every=1))
