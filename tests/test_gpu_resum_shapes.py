"""Modal sums at the edges of their launch shapes: intervals shorter than a grid
step, windows of more than 32 rays, warps with more than 32 modes, runs of 16
points; the mixed sum against the FP64 one of the same plan."""
import math

import numpy as np
import pytest

from oracle.swkb_oracle import rel_l2
from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu

# FP32 terms: phases of up to four turns (2^-24 x 8 pi = 1.5e-6), the sine's
# 2^-21 and amplitudes and coefficients of a few 2^-24, over two screens; with a
# factor of two for the march's own rounding
TOL = 1e-5


def _lens(R):
    """A converging lens: landings up to 6 % closer than launches."""
    return w.config_gaussian_medium(a=0.02, b=0.01, ray_stride=R, n_screens=2)


def _open(R):
    return w.config_open_lens(n_z=8192, fc_patch=910, fc_overlap=248, n_screens=2, ray_stride=R)


@pytest.mark.parametrize("problem,tiling", [
    (lambda: _lens(1), None),                                        # intervals below one step
    (lambda: _lens(1), (64, 1, 4)),
    (lambda: _lens(2), (128, 2, 4)),                                 # 68 rays per window
    (lambda: w.config_surface_duct_small(n_screens=2), (512, 2, 16)),          # 36 rays, runs of 16
    (lambda: w.config_surface_duct_small(n_screens=2, bc=w.BC_DIRICHLET), (512, 20, 16)),
    (lambda: w.config_surface_duct_small(n_screens=2, ray_stride=64), None),   # 12 rays, runs of 16
    (lambda: w.config_gaussian_lens_40km().with_(n_screens=2), (64, 1, 8)),    # 134 modes per group
    (lambda: w.config_gaussian_lens_40km().with_(n_screens=2), (256, 1024, 8)),  # one mode per group
    (lambda: w.config_surface_duct_small(n_screens=2).with_(theta_max=math.radians(0.02)), None),
    # patch-wise: 36 rays per window, several hundred modes per group, R = 1
    (lambda: _open(8), (256, 1, 32)),
    (lambda: _open(8), (64, 1024, 32)),
    (lambda: _open(2), (128, 1, 32)),
    (lambda: _open(1), None),
])
def test_mixed_sum_matches_fp64(problem, tiling):
    pb = problem()
    got = swkb.Plan(pb, swkb.SWKB_MIXED, tiling=tiling).propagate()
    want = swkb.Plan(pb, swkb.SWKB_FP64).propagate()
    assert np.linalg.norm(want) > 0
    assert rel_l2(got, want) < TOL
