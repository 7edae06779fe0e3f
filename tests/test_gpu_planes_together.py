"""Inner planes taken together: the same planes come out whatever number of them a
screen has (and so however they are grouped), on both output routes."""
import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def _rows(plan, pb, P, n, device):
    if not device:
        return plan.propagate_planes(P, n_screens=n)
    torch = pytest.importorskip("torch")
    u0 = torch.from_numpy(np.ascontiguousarray(pb.u0, dtype=np.complex128)).cuda()
    out = torch.full((n * P + 1, plan.n_z), 7.0, dtype=torch.complex128, device="cuda")
    plan.propagate_planes_device(P, u0.data_ptr(), out.data_ptr(), n_screens=n)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.all(got[-1] == 7.0)
    return got[:-1]


def _check(pb, prec, n, planes=(8, 4, 2)):
    want, top = None, planes[0]
    for P in planes:
        plan = swkb.Plan(pb, prec, planes=P)
        host, dev = (_rows(plan, pb, P, n, d) for d in (False, True))
        assert np.array_equal(host, dev)
        if want is None:
            want = host.reshape(n, top, -1)
        else:
            assert np.array_equal(host.reshape(n, P, -1), want[:, top // P - 1::top // P])


@pytest.mark.parametrize("prec", [swkb.SWKB_FP64, swkb.SWKB_MIXED])
@pytest.mark.parametrize("make", [
    lambda: w.config_unit_periodic(n_screens=2),
    lambda: w.config_homogeneous(eps0=1.04, bc=w.BC_DIRICHLET, ray_stride=2, rk4_steps=8, n_screens=2),
    lambda: w.config_surface_duct_small(n_screens=2, rk4_steps=8),
], ids=["periodic", "dirichlet", "neumann"])
def test_planes_do_not_depend_on_their_number(make, prec):
    _check(make(), prec, 2)


def test_planes_in_several_batches():
    # partials of a plane are some MB: 127 inner planes do not fit one batch of 256 MB
    pb = w.config_surface_duct_small(n_screens=1, rk4_steps=128)
    info = swkb.Plan(pb, swkb.SWKB_FP64, planes=128).info
    assert 127 * info.mode_groups * info.n_fft * 16 > 256 << 20
    _check(pb, swkb.SWKB_FP64, 1, (128, 64, 2))
