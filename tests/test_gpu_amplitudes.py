"""Amplitude factors of the FP32 march: rounded once from what they are formed of."""
import os
import subprocess

import numpy as np
import pytest

from paper_2301_03814_gb300 import build, swkb
from paper_2301_03814_gb300 import workloads as w

pytestmark = pytest.mark.gpu

N = 1 << 16

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "swkb_device.cuh"

__global__ void k(const float* x, int n, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = swkb::amplitude(x[i], x[n + i], x[2 * n + i]);
}

int main(int argc, char** argv) {
  const int n = atoi(argv[1]);
  std::vector<float> in(3 * (size_t)n), out(n);
  FILE* f = fopen(argv[2], "rb");
  if (!f || fread(in.data(), 4, in.size(), f) != in.size()) return 2;
  fclose(f);
  float *d, *o;
  if (cudaMalloc(&d, in.size() * 4) || cudaMalloc(&o, out.size() * 4)) return 3;
  cudaMemcpy(d, in.data(), in.size() * 4, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, n, o);
  if (cudaMemcpy(out.data(), o, out.size() * 4, cudaMemcpyDeviceToHost)) return 4;
  f = fopen(argv[3], "wb");
  if (!f || fwrite(out.data(), 4, out.size(), f) != out.size()) return 5;
  fclose(f);
  return 0;
}
"""


def test_amplitudes_above_a_duct_have_no_bias():
    # In the linear gradient above the duct P0, P1 and Z stay near 1, and each factor is rounded to one
    # of a few neighbours of 1.  Rounded once, the mean over the rays is the few ties' (an eighth of
    # 2^-23 at most, where Z is rounded to steps of 2^-24); twice that is allowed.
    pb = w.config_surface_duct(height=100.0, n_z=4096, z_s=5.0, z_t_range=(10.0, 20.0), ray_stride=16)
    u = np.zeros(2 * pb.n_z, complex)
    u[pb.n_z:] = pb.u0
    a64, a = [swkb.Plan(pb, p).debug_screen(0, u)["a"] for p in (swkb.SWKB_FP64, swkb.SWKB_MIXED)]
    z = a.shape[1] // 2 + np.arange(a.shape[1] // 4, int(a.shape[1] * 0.45))   # launched at 50 .. 90 m
    err = a[:, z] / a64[:, z] - 1.0
    assert abs(float(err.mean())) < 0.5 * 2.0 ** -24


@pytest.mark.parametrize("p,z", [((0.9, 1.1), (0.9, 1.1)), ((0.01, 4.0), (1e-3, 1e3))])
def test_amplitude_is_rounded_once(tmp_path, p, z):
    # Half a unit in the last place, and the Newton step's own error: the first value's
    # (below 1e-6) squared, 1e-12 of the result or 2e-5 units.
    rng = np.random.default_rng(7)
    x = np.exp([rng.uniform(*np.log(b), N) for b in (p, p, z)]).astype(np.float32)
    x.tofile(tmp_path / "in")
    (tmp_path / "m.cu").write_text(SOURCE)
    exe = str(tmp_path / "m")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-ftz=true", "-prec-div=false",
                    "-prec-sqrt=false", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    "-o", exe, str(tmp_path / "m.cu")], check=True, capture_output=True)
    subprocess.run([exe, str(N), str(tmp_path / "in"), str(tmp_path / "out")], check=True, timeout=120)
    got = np.fromfile(tmp_path / "out", np.float32).astype(np.float64)
    P0sq, P1sq, Z = x.astype(np.float64)
    want = np.sqrt(np.sqrt(P0sq / P1sq) / Z)
    assert float(np.max(np.abs(got - want) / np.spacing(want.astype(np.float32)))) < 0.501
