"""Patch DFTs that share twiddles between four patches (many patches, their number
not a multiple of four) against those of one patch per block: a field in a few
patches of a long homogeneous interval and of a short one."""
import numpy as np
import pytest

from oracle.swkb_oracle import rel_l2
from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu

PATCH, OVERLAP, STRIDE = 120, 48, 72
FEW, MANY = 8, 257        # 83 modes of 145-point periods: two blocks of bins per patch


def _pb(patches, u0=None):
    pb = w.config_open_lens(n_z=PATCH + (patches - 1) * STRIDE, fc_patch=PATCH, fc_overlap=OVERLAP, a=0.0,
                            n_screens=2, n_beams=1)
    return pb if u0 is None else pb.with_(u0=u0)


# the two sums differ in their order only: 2^-53 and 2^-24 times sqrt(145) and a
# dozen operations per value, over two screens; the march and the sum run on the
# same numbers shifted by whole ray strides
@pytest.mark.parametrize("precision,tol", [(swkb.SWKB_FP64, 1e-12), (swkb.SWKB_MIXED, 1e-5)])
@pytest.mark.parametrize("first", [0, 100, MANY - FEW])
def test_shared_twiddles_match_one_patch_per_block(precision, tol, first):
    few = _pb(FEW)
    z = np.arange(few.n_z) / 3.0
    u = w.gaussian_beam(z, few.k, few.n_z / 6.0, 6.0, 0.1) + 0.5 * w.gaussian_beam(z, few.k, few.n_z / 5.0, 9.0, -0.2)
    u[np.abs(z - few.n_z / 6.0) > few.n_z / 7.0] = 0.0
    want = swkb.Plan(_pb(FEW, u), precision).propagate()
    long = np.zeros(_pb(MANY).n_z, dtype=np.complex128)
    s = slice(first * STRIDE, first * STRIDE + few.n_z)
    long[s] = u
    got = swkb.Plan(_pb(MANY, long), precision).propagate()
    # away from the short interval's own ends, where its field is windowed out
    inner = slice(2 * OVERLAP, few.n_z - 2 * OVERLAP)
    assert np.linalg.norm(want) > 0
    assert rel_l2(got[s][inner], want[inner]) < tol
