"""The FP64 device functions of the march and the sums against long-double values: inverse root,
reciprocal, and the table sine with the plan's own table entries."""
import os
import subprocess

import numpy as np
import pytest

from paper_2301_03814_gb300 import build

pytestmark = pytest.mark.gpu

N = 1 << 18
ULP = 2.0 ** -53

SOURCE = r"""
#include <cstdio>
#include <cmath>
#include <vector>
#include "swkb_device.cuh"
using namespace swkb;

__global__ void k(const double* x, const double* a, const double* b, const double2* trig, int n,
                  double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = rsqrt64(x[i]);
  out[n + i] = rcp64(x[i]);
  sincos_table(trig, a[i], b[i], out + 2 * n + i, out + 3 * n + i);
}

int main(int argc, char** argv) {
  const int n = atoi(argv[1]);
  std::vector<double> in(3 * (size_t)n), out(4 * (size_t)n), trig = trig_table();
  FILE* f = fopen(argv[2], "rb");
  if (!f || fread(in.data(), sizeof(double), in.size(), f) != in.size()) return 2;
  fclose(f);
  double *d, *o, *t;
  if (cudaMalloc(&d, in.size() * 8) || cudaMalloc(&o, out.size() * 8) ||
      cudaMalloc(&t, trig.size() * 8))
    return 3;
  cudaMemcpy(d, in.data(), in.size() * 8, cudaMemcpyHostToDevice);
  cudaMemcpy(t, trig.data(), trig.size() * 8, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * (size_t)n, (const double2*)t, n, o);
  if (cudaMemcpy(out.data(), o, out.size() * 8, cudaMemcpyDeviceToHost)) return 4;
  f = fopen(argv[3], "wb");
  if (!f || fwrite(out.data(), sizeof(double), out.size(), f) != out.size()) return 5;
  fclose(f);
  return 0;
}
"""


@pytest.fixture(scope="module")
def values(tmp_path_factory):
    d = tmp_path_factory.mktemp("device_math")
    (d / "m.cu").write_text(SOURCE)
    exe = str(d / "m")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-ftz=true", "-prec-div=false",
                    "-prec-sqrt=false", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    str(d / "m.cu"), "-o", exe], check=True, capture_output=True)
    rng = np.random.default_rng(3)
    # P^2 and P_bar + P are near 1 and 2; intervals run from fractions of a grid step to long ones
    x = np.where(np.arange(N) % 2, rng.uniform(0.2, 4.0, N), np.exp(rng.uniform(np.log(1e-6), np.log(1e6), N)))
    # n m / N of the grid points of a run (multiples of 2^-20, a few turns of either sign), and the rays' phase
    a = np.round(rng.uniform(-2.5, 2.5, N) * 2 ** 20) / 2 ** 20
    b = np.where(np.arange(N) % 4 == 0, rng.uniform(-40.0, 40.0, N), rng.uniform(-1.0, 1.0, N))
    # small sines: the sum near a multiple of half a turn
    near = slice(0, N // 8)
    b[near] = -a[near] + np.round(2 * a[near]) / 2 + rng.uniform(-1e-4, 1e-4, N // 8)
    np.concatenate([x, a, b]).tofile(d / "in")
    subprocess.run([exe, str(N), str(d / "in"), str(d / "out")], check=True)
    return x, a, b, np.fromfile(d / "out").reshape(4, N)


def _worst(got, want):
    return float(np.max(np.abs((got - want) / want)))


def test_inverse_root(values):
    # the correction's rounding (x y enters it rounded: 1/2) and the last one: 1.5 halves of a unit,
    # and a remainder of third order below 2^-57
    x, _, _, out = values
    assert _worst(out[0].astype(np.longdouble), 1 / np.sqrt(x.astype(np.longdouble))) < 1.6 * ULP


def test_reciprocal(values):
    # one rounding (the division's own bound) and a remainder of third order below 2^-59
    x, _, _, out = values
    assert _worst(out[1].astype(np.longdouble), 1 / x.astype(np.longdouble)) < 1.02 * ULP


def test_table_sine(values):
    # the table entry and the last two operations are rounded to 2^-54 each: 1.5 x 2^-53 (and a little
    # from the small terms); nothing of the size of the phase
    _, a, b, out = values
    t = a.astype(np.longdouble) + b.astype(np.longdouble)
    t -= np.round(t)
    angle = 2 * np.arccos(np.longdouble(-1)) * t
    assert float(np.max(np.abs(out[2] - np.sin(angle)))) < 1.6 * ULP
    assert float(np.max(np.abs(out[3] - np.cos(angle)))) < 1.6 * ULP
    # near multiples of half a turn the sine keeps its relative accuracy: r, r^2, the polynomial and
    # two products, a rounding each
    s = slice(0, N // 8)
    small = np.abs(np.sin(angle[s])) > 0
    assert _worst(out[2][s][small], np.sin(angle[s][small])) < 6 * ULP
