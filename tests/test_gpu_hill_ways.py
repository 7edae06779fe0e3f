"""Which way swkb_hill_propagate takes when no eigenvalues are asked for, and that the expansion agrees with the
eigenvectors wherever it is taken."""
import math

import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu

LAM = 0.05


def _inputs(bc, K, n_z, n_q, batch, height):
    rng = np.random.default_rng(11 + K)
    k = 2.0 * math.pi / LAM * np.linspace(0.9, 1.1, batch) if batch > 1 else np.array([2.0 * math.pi / LAM])
    s = height * np.arange(n_q + 1) / n_q
    if bc == swkb.SWKB_BC_PERIODIC:
        z_a, eps = -height, [w.f_gaussian(2e-4, float(rng.uniform(1e-3, 5e-3)))(s)[0] for _ in range(batch)]
    else:
        z_a, eps = 0.0, [w.f_trilinear_duct(float(rng.uniform(10, 20)), -0.15)(s)[0] for _ in range(batch)]
    u0 = rng.standard_normal((batch, n_z)) + 1j * rng.standard_normal((batch, n_z))
    return k, np.array(eps), u0, swkb.hill_desc(bc, z_a, height, n_z, K, n_q, 0.0)


def _both(inputs, xs):
    k, eps, u0, desc = inputs
    got = swkb.swkb_hill_propagate(desc, k, eps, u0, xs)
    products = swkb.swkb_hill_last_products()
    want, lam = swkb.swkb_hill_propagate(desc, k, eps, u0, xs, eigenvalues=True)
    assert swkb.swkb_hill_last_products() == 0 and np.all(np.isfinite(lam))
    for r, x in enumerate(xs):
        # A's rounding moves a mode's phase by about eps_mach k x / 2, the eigen-solver's own by a multiple
        tol = 1e-11 + 32 * np.finfo(float).eps * float(np.max(k)) * x
        assert np.linalg.norm(got[:, r] - want[:, r]) < tol * np.linalg.norm(want[:, r])
    return products


BCS = [swkb.SWKB_BC_PERIODIC, swkb.SWKB_BC_NEUMANN, swkb.SWKB_BC_DIRICHLET]


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("K,n_z,n_q,batch,xs", [
    (8, 64, 17, 1, [0.0]),                         # 9 cosine rows (padded to 10), nothing but the carrier
    (9, 64, 18, 1, [0.0, 3.0]),
    (16, 64, 33, 2, [5.0, 1.0]),                   # ranges out of order
    (40, 128, 100, 1, list(np.linspace(0.0, 60.0, 35))),
    (64, 256, 129, 3, [100.0]),
    (120, 512, 300, 1, [300.0, 150.0]),
])
def test_expansion_is_taken_and_agrees(bc, K, n_z, n_q, batch, xs):
    assert _both(_inputs(bc, K, n_z, n_q, batch, 50.0), xs) >= 24


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("K,n_z,n_q,height,xs", [
    (1, 64, 2, 50.0, [30.0]),                      # 2 rows: 24 terms are too many
    (120, 512, 300, 50.0, [30000.0]),              # thousands of terms on 122 rows
    (300, 1024, 700, 5.0, [3.0]),                  # evanescent modes
])
def test_eigenvectors_are_taken(bc, K, n_z, n_q, height, xs):
    assert _both(_inputs(bc, K, n_z, n_q, 1, height), xs) == 0


@pytest.mark.parametrize("K,n_z,height,xs", [
    (1501, 2048, 50.0, [185.0, 190.0, 195.0, 200.0, 204.0, 205.0]),      # 5750 terms: near 4 P
    (3001, 4096, 100.0, [195.0, 200.0, 205.0, 210.0]),                   # about 2 P
])
def test_large_expansions_are_not_given_up_for_rounding(K, n_z, height, xs):
    assert _both(_inputs(swkb.SWKB_BC_NEUMANN, K, n_z, 2 * K + 100, 1, height), xs) > 5000
