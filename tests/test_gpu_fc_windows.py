"""Patch-wise sums whose tiles hold few or many landings: ray strides beyond a tile, and rays compressed
more than four times on a tile but not on the tiles the limit is set for."""
import numpy as np
import pytest

import fc_pins as P
from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu
pytest.importorskip("mpmath")

from oracle.fc_oracle import FCOracle  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _err(got, want):
    return float(np.max(np.abs(got - want)) / np.max(np.abs(want)))


@pytest.mark.parametrize("precision,tol", [(swkb.SWKB_FP64, 1e-10), (swkb.SWKB_MIXED, 1e-4)])
@pytest.mark.parametrize("R", [256, 512, 1024, 2048])
def test_wide_ray_strides(R, precision, tol):
    # tiles of 128 points with a landing every R points: most hold none, the others one
    pb = P.open_problem(1024, 256, 5, 2048 * P.STEP, 3.0, 5.0, ray_stride=R)
    H = pb.z_b
    pb = pb.with_(profile=w._table([0.0], -5.0 * H, 0.25, int(11 * H / 0.25) + 1, [w.f_const(1.0)]))
    assert pb.n_z == 4096
    assert _err(swkb.Plan(pb, precision).propagate(), FCOracle(pb).propagate(pb.u0)) < tol


def _focusing(a, wid, dx, R, patches):
    """A strong lens over a long screen of nearly horizontal rays: five- to ninefold compression near its axis."""
    n_pat, n_ov = 768, 256
    H = ((patches - 1) * (n_pat - n_ov) + n_pat) * P.STEP
    return P.open_problem(n_pat, n_ov, patches, H / 2, 0.0, dx, medium=w.f_gaussian(a, 1 / wid ** 2, zc=H / 2 - wid * 0.07),
                          theta_deg=1.0, rk4_steps=64, ray_stride=R)


def _window(pb, tile):
    """Most rays (with the stencil's) on a tile."""
    o = FCOracle(pb)
    z = o.base.march(0, o.kappa[:, None], o.launch_points()[None, :])["z"]
    edges = pb.z_a + np.arange(0, pb.n_z + 1, tile) * o.h
    return max(int(np.diff(np.searchsorted(row, edges, side="right")).max()) + 4 for row in z)


# windows of 77 and 114 rays on 128 and 256 points (4 x 128 / 8 + 4 = 68 fit one tile, 132 the pair); 149 and 225 on
# 64 and 128 points at R = 2 (132 and 260).  Tiles of twice the size hold them at once: the same rays, and only the
# sums' rounding differs (FP64: phases of 64 turns, 5e-14 rad each; FP32: landings within a tile to 1.5e-5 points,
# 0.1 turns per point, 1e-5 rad each).
@pytest.mark.parametrize("precision,tol", [(swkb.SWKB_FP64, 1e-12), (swkb.SWKB_MIXED, 1e-4)])
@pytest.mark.parametrize("a,wid,dx,R,patches", [(0.085, 300.0, 1500.0, 8, 16), (0.085, 150.0, 750.0, 2, 8)])
def test_compression_on_one_tile(a, wid, dx, R, patches, precision, tol):
    pb = _focusing(a, wid, dx, R, patches)
    tile = 128 if R == 8 else 64
    assert _window(pb, tile) > 4 * tile // R + 4
    assert _window(pb, 2 * tile) <= 8 * tile // R + 4
    plan = swkb.Plan(pb, precision)
    assert plan.info.tile_points == tile
    want = swkb.Plan(pb, precision, tiling=(2 * tile, 8, 1)).propagate()
    assert np.max(np.abs(want)) > 0.1
    assert _err(plan.propagate(), want) < tol


def test_compression_on_a_pair_of_tiles_is_refused():
    pb = _focusing(0.105, 300.0, 1500.0, 8, 16)
    assert _window(pb, 256) > 132
    with pytest.raises(swkb.SwkbError) as e:
        swkb.Plan(pb, swkb.SWKB_FP64).propagate()
    assert e.value.status == 3
    # with the tile's size asked for, the limit is the tile's own
    pb = _focusing(0.085, 300.0, 1500.0, 8, 16)
    with pytest.raises(swkb.SwkbError) as e:
        swkb.Plan(pb, swkb.SWKB_FP64, tiling=(128, 8, 1)).propagate()
    assert e.value.status == 3
