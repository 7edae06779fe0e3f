// swkb_modes_noalloc: step (a) of the screen step -- the pruned DFT of one
// screen field into its kept plane-wave coefficients -- for callers that must
// not allocate device memory.
//
// Who needs it: code that owns every byte of device memory itself (a host
// framework that pre-partitions HBM and forbids other allocators, or a
// latency-critical loop where cudaMalloc / cudaFree would synchronise the
// device and stall other streams).  Such callers still hand in their input
// and output buffers; the FFT's working storage lives here instead, in
// file-scope device arrays of a fixed size that every GPU loading this library
// holds until the process exits (3 MB per device).
//
// The arithmetic is an FP64 pruned two-pass DFT (k_fft1_pairs, then bins in pairs,
// k_fft2_pair).  The twiddles are those of the largest length, filled once:
// shorter ones are strided in it.  4096 points, 489 modes: 30.7 -> 12.3 us per call
// (before, each call filled a table and split the points into two rows only).

#include <mutex>
#include <string>

#include "swkb.h"
#include "swkb_internal.h"

namespace {

constexpr int kMaxN = 65536;   // largest FFT length accepted

// Scratch shared by every call on a device.  In host code these names are
// host-side stand-ins, not device addresses: the host must pass the address
// returned by cudaGetSymbolAddress to the kernels.
static __device__ __align__(256) double2 g_fft_mid[kMaxN];        // pass-1 output [N1][N2]
static __device__ __align__(256) double2 g_twiddle[kMaxN];        // exp(-2 pi i k / kMaxN)
// one entry per kept mode: 2 n_max + 1 <= n_fft - 1 < kMaxN
static __device__ __align__(256) double2 g_unit_phase[kMaxN];     // exp(i 0) per mode

struct DeviceScratch {
  bool ready = false;
  double2* mid = nullptr;
  double2* twiddle = nullptr;
  double2* unit_phase = nullptr;
};

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
DeviceScratch g_scratch[kMaxDevices];
swkb_status err(swkb_status s, const std::string& m) {
  swkb::set_last_error(m.c_str());
  return s;
}

__global__ void k_fill_twiddles(double2* tw, int N) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  double s, c;
  sincospi(2.0 * (double)k / (double)N, &s, &c);
  tw[k] = make_double2(c, -s);
}

__global__ void k_fill_unit(double2* v, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) v[k] = make_double2(1.0, 0.0);
}

// Once per device, with that device current: resolve the device addresses of
// the scratch arrays and set the kernels' shared-memory limits.
swkb_status setup(int dev, DeviceScratch** out) {
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  DeviceScratch& d = g_scratch[dev];
  if (!d.ready) {
    cudaError_t e = cudaGetSymbolAddress((void**)&d.mid, g_fft_mid);
    if (e == cudaSuccess) e = cudaGetSymbolAddress((void**)&d.twiddle, g_twiddle);
    if (e == cudaSuccess) e = cudaGetSymbolAddress((void**)&d.unit_phase, g_unit_phase);
    if (e == cudaSuccess) e = swkb::prepare_fft_kernels<double>();
    if (e == cudaSuccess) {
      k_fill_unit<<<(kMaxN + 255) / 256, 256>>>(d.unit_phase, kMaxN);
      k_fill_twiddles<<<(kMaxN + 255) / 256, 256>>>(d.twiddle, kMaxN);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess)
      return err(SWKB_ERR_CUDA, std::string("no-alloc set-up failed: ") + cudaGetErrorString(e));
    d.ready = true;
  }
  *out = &d;
  return SWKB_OK;
}

// N1 of n_fft = N1 N2: the smallest estimate of the FP64 instructions of the
// busiest of 152 SMs.  A pass-1 CTA of c columns forms c N1 sums of N1 / 4 terms of 8
// instructions, a pass-2 CTA a pair of sums of N2 terms of 4; the second
// kernel costs what an SM issues in 3 us.  Measured with about 11 us of launch and
// event overhead (pass 1 as N1 / 2 terms of 4 then, up to 1 us less), one kernel / the
// best split / this rule:
//   1024 points,   101 modes    14.8 / 14.8 / 14.9 us
//   4096 points,   489 modes    23.6 / 18.5 / 18.0
//   16384 points, 8001 modes     475 / 57.9 / 57.7
//   65536 points, 32001 modes   6905 /  246 / 247
int split(int n_fft, int n_max) {
  const long long sms = 152, launch = 12000;
  int best = 1;
  long long least = 0;
  for (int n1 = 1; n1 <= 64 && n1 <= n_fft / 32; n1 *= 2) {
    const long long n2 = n_fft / n1, cols = swkb::fft1_cols((int)n2);
    const long long cost =
        4 * n2 * ((swkb::fft2_pairs(n1, n_max) + sms - 1) / sms) +
        (n1 > 1 ? launch + 2 * n1 * n1 * cols * ((n2 / cols + sms - 1) / sms) : 0);
    if (n1 == 1 || cost < least) {
      best = n1;
      least = cost;
    }
  }
  return best;
}

bool is_device_pointer(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" swkb_status swkb_modes_noalloc(const double* u, int32_t n_fft, int32_t n_max,
                                          double* c, void* cuda_stream) {
  if (!u || !c) return err(SWKB_ERR_INVALID_ARG, "u and c must be device pointers");
  if (n_fft < 64 || n_fft > kMaxN || (n_fft & (n_fft - 1)))
    return err(SWKB_ERR_INVALID_ARG,
               "n_fft must be a power of two in [64, 65536] (the fixed scratch size)");
  if (n_max < 1 || n_max > n_fft / 2 - 1)
    return err(SWKB_ERR_INVALID_ARG, "n_max must be in [1, n_fft / 2 - 1]");
  if (!is_device_pointer(u) || !is_device_pointer(c))
    return err(SWKB_ERR_INVALID_ARG, "u and c must be device pointers");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return err(SWKB_ERR_CUDA, "no usable current device");
  DeviceScratch* d = nullptr;
  swkb_status st = setup(dev, &d);
  if (st != SWKB_OK) return st;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  swkb::FftArgs<double> f;
  f.u = reinterpret_cast<const double2*>(u);
  f.tw = d->twiddle;
  f.tw_shift = 0;
  while (n_fft << f.tw_shift < kMaxN) ++f.tw_shift;
  f.Y = d->mid;
  f.N = n_fft;
  f.N1 = split(n_fft, n_max);
  f.N2 = n_fft / f.N1;
  f.mirror = 0;
  f.part = nullptr;   // the caller's field is read directly
  f.n_part = 0;
  f.sym = 0;
  f.W = nullptr;
  f.log2N2 = 0;
  while ((1 << f.log2N2) < f.N2) ++f.log2N2;
  f.n_max = n_max;
  f.inv_N = 1.0 / n_fft;
  f.ephi = d->unit_phase;
  f.c = reinterpret_cast<double2*>(c);
  f.cpol = nullptr;
  e = swkb::launch_fft_pairs(f, s);
  if (e != cudaSuccess) return err(SWKB_ERR_CUDA, cudaGetErrorString(e));
  return SWKB_OK;
}
