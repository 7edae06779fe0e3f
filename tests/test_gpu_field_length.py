"""The FP32 sums' sine and coefficient: a term keeps its length on average, so that the field keeps
its own over many screens."""
import os
import subprocess

import numpy as np
import pytest

from paper_2301_03814_gb300 import build

pytestmark = pytest.mark.gpu

N = 1 << 18

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "swkb_device.cuh"

__global__ void k(const float* x, int n, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float2 pol = swkb::polar_turns<float>(make_float2(x[i], x[n + i]));
  float s, c;
  swkb::sincos_turns(x[2 * n + i], &s, &c);
  out[i] = pol.x;
  out[n + i] = s;
  out[2 * n + i] = c;
}

int main(int argc, char** argv) {
  const int n = atoi(argv[1]);
  std::vector<float> in(3 * (size_t)n), out(3 * (size_t)n);
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


@pytest.mark.parametrize("turns", [0.5, 1.5, 4.0])
def test_terms_keep_their_length(tmp_path, turns):
    # |c| (cos, sin) along the exact value, averaged over whole circles and over coefficients of
    # all mantissas.  What a term loses by rounding is random (2^-24 each, below 1e-9 on average over
    # 2^18 terms); the coefficient's factor is rounded to steps of 2^-23 of its square, which moves
    # its average over the mantissas by less than an eighth of 2^-24.  A quarter is allowed.
    rng = np.random.default_rng(3)
    mag, arg = np.exp(rng.uniform(-20.0, 3.0, N)), rng.uniform(0.0, 2.0 * np.pi, N)
    x = np.array([mag * np.cos(arg), mag * np.sin(arg), rng.uniform(-turns, turns, N)], np.float32)
    x.tofile(tmp_path / "in")
    (tmp_path / "m.cu").write_text(SOURCE)
    exe = str(tmp_path / "m")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-ftz=true", "-prec-div=false",
                    "-prec-sqrt=false", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    "-o", exe, str(tmp_path / "m.cu")], check=True, capture_output=True)
    subprocess.run([exe, str(N), str(tmp_path / "in"), str(tmp_path / "out")], check=True, timeout=120)
    pol, s, c = np.fromfile(tmp_path / "out", np.float32).astype(np.float64).reshape(3, N)
    x = x.astype(np.float64)
    t = 2.0 * np.pi * (x[2] - np.rint(x[2]))
    along = pol / np.hypot(x[0], x[1]) * (c * np.cos(t) + s * np.sin(t)) - 1.0
    assert abs(float(along.mean())) < 0.25 * 2.0 ** -24
