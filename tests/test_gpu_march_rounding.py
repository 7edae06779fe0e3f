"""Rounding of the ray march: its constants (in a homogeneous medium the landings are known exactly)
and the sums of its Runge-Kutta steps (the FP32 march against the FP64 one)."""
import math

import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,steps,dx,dz", [
    (swkb.SWKB_MIXED, 6, 13.0, 30.0 / 256), (swkb.SWKB_MIXED, 7, 19.0, 31.0 / 256),
    (swkb.SWKB_FP64, 7, 17.0, 36.0 / 256), (swkb.SWKB_FP64, 11, 13.0, 33.0 / 256),
])
def test_march_constants_are_rounded_once(precision, steps, dx, dz):
    # The mean relative error of the landings over the modes is that of the constants: one rounding,
    # u at most (u = 2^-24 or 2^-53), since the weights' own is carried by the last factor.  The
    # modes' own roundings (about u each, ~180 modes) leave 0.08 u; three times that is allowed for.
    pb = w.config_homogeneous(n_z=1024, height=1024 * dz, dx=dx, rk4_steps=steps, theta_deg=50.0, ray_stride=16)
    plan = swkb.Plan(pb, precision)
    got = plan.debug_screen(0, pb.u0)["delta"][:, plan.info.n_ghost]     # the ray launched at grid point 0
    n = np.arange(-plan.info.n_max, plan.info.n_max + 1).astype(np.longdouble)
    kappa = n / (np.longdouble(pb.z_b) - np.longdouble(pb.z_a))          # wavelength 1
    want = kappa / np.sqrt(1 - kappa * kappa) * np.longdouble(dx) / (np.longdouble(pb.z_b) / pb.n_z)
    err = (got[n != 0] - want[n != 0]) / want[n != 0]
    u = 2.0 ** (-24 if precision == swkb.SWKB_MIXED else -53)
    assert len(err) > 150
    assert abs(float(err.mean())) < 1.25 * u


def test_amplitudes_are_rounded_once_per_step():
    # Z_s stays near 1, so each of the 16 steps' sums rounds it by at most 2^-24 (rms 3.4e-8), and the
    # amplitude 1 / sqrt(Z_s) gains half of that: 6.9e-8 in all.  Its last factors (a root, an inverse
    # root, a quotient) add about 3.4e-8 rms each: 9.1e-8 together.
    pb = w.config_gaussian_lens_40km()
    a = [swkb.Plan(pb, p).debug_screen(0, pb.u0)["a"] for p in (swkb.SWKB_FP64, swkb.SWKB_MIXED)]
    err = a[1] / a[0] - 1.0
    assert math.sqrt(float((err * err).mean())) < 9.1e-8
