"""swkb_hill_propagate by the Chebyshev expansion (fields alone) against the
eigen-decomposition (fields with eigenvalues) over the forms both accept."""
import math

import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu

LAM = 0.05


def _inputs(bc, K, n_z, n_q, batch, height=50.0):
    rng = np.random.default_rng(7 + K)
    k = 2.0 * math.pi / LAM * np.linspace(0.8, 1.2, batch) if batch > 1 else np.array([2.0 * math.pi / LAM])
    eps, u0 = [], []
    for _ in range(batch):
        if bc == swkb.SWKB_BC_PERIODIC:
            z_a, z_b = -height, height
            eps.append(w.f_gaussian(2e-4, float(rng.uniform(1e-3, 5e-3)))(height * np.arange(n_q + 1) / n_q)[0])
        else:
            z_a, z_b = 0.0, height
            eps.append(w.f_trilinear_duct(float(rng.uniform(10, 20)), -0.15)(height * np.arange(n_q + 1) / n_q)[0])
        u = rng.standard_normal(n_z) + 1j * rng.standard_normal(n_z)
        u0.append(u)
    return k, np.array(eps), np.array(u0), swkb.hill_desc(bc, z_a, z_b, n_z, K, n_q, 0.0)


# both ways end in the same sums; A's rounding moves a mode's phase by about
# eps_mach k x / 2 (the eigen-solver's own by a multiple of that)
def _tol(k, x):
    return 1e-11 + 32 * np.finfo(float).eps * float(np.max(k)) * x


@pytest.mark.parametrize("bc", [swkb.SWKB_BC_PERIODIC, swkb.SWKB_BC_NEUMANN, swkb.SWKB_BC_DIRICHLET])
@pytest.mark.parametrize("K,n_z,n_q,batch,xs", [
    (1, 64, 2, 1, [30.0]),                          # a 2 x 2 matrix (with padding)
    (2, 64, 5, 1, [0.0, 10.0]),
    (33, 128, 66, 2, [20.0, 5.0]),                  # ranges out of order
    (64, 256, 129, 3, [100.0]),
    (40, 128, 100, 1, list(np.linspace(0.0, 60.0, 35))),   # more than 32 ranges
    (120, 512, 300, 1, [300.0, 150.0]),
    (120, 512, 300, 1, [30000.0]),                  # too many terms: both by eigenvectors
])
def test_expansion_matches_eigenvectors(bc, K, n_z, n_q, batch, xs):
    k, eps, u0, desc = _inputs(bc, K, n_z, n_q, batch)
    want, lam = swkb.swkb_hill_propagate(desc, k, eps, u0, xs, eigenvalues=True)
    got = swkb.swkb_hill_propagate(desc, k, eps, u0, xs)
    assert np.all(np.isfinite(lam))
    assert np.linalg.norm(want) > 0
    for r, x in enumerate(xs):
        assert np.linalg.norm(got[:, r] - want[:, r]) < _tol(k, x) * np.linalg.norm(want[:, r])


def test_evanescent_modes_take_the_eigenvectors():
    # kappa_K = 2 pi 300 / 10 > k: eigenvalues below zero
    k, eps, u0, desc = _inputs(swkb.SWKB_BC_NEUMANN, 300, 1024, 700, 1, height=5.0)
    want, lam = swkb.swkb_hill_propagate(desc, k, eps, u0, [3.0], eigenvalues=True)
    assert lam.min() < 0
    got = swkb.swkb_hill_propagate(desc, k, eps, u0, [3.0])
    assert np.linalg.norm(got - want) < _tol(k, 3.0) * np.linalg.norm(want)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_permittivity_is_refused(bad):
    k, eps, u0, desc = _inputs(swkb.SWKB_BC_NEUMANN, 20, 64, 40, 2)
    eps[1, 7] = bad
    with pytest.raises(swkb.SwkbError) as e:
        swkb.swkb_hill_propagate(desc, k, eps, u0, [5.0])
    assert e.value.status == swkb.SWKB_ERR_INVALID_ARG
