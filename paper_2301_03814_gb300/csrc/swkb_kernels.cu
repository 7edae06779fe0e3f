// Device kernels of the screened-WKB screen step (sm_103a), templated on the
// arithmetic type T (double: the FP64 path; float: the mixed path, whose
// FP64 parts -- the range-phase carry exp(i Phi_n) and the launch tables --
// are prepared on the host).
//
// One screen Gamma_q -> Gamma_{q+1} (Algorithm 1) is, on the device:
//   k_reduce   sum the resummation partials, absorber window, reflection
//              projection u <- (u(z) +- u(2 z_a - z)) / 2   (Sec. 2.3)
//   k_fft1/2   pruned DFT of the screen field, c_n = w_n / N * exp(i Phi_n)
//              for |n| <= n_max                        (Eqs. fft_eq, ifft_eq)
//   k_march    RK4 across the slab for every (mode, ray): the x-form of the
//              characteristic system and its s-variation (Eqs. charsys,
//              charsys_s), amplitude sqrt(P0 / (P1 Z_s)) (corrected Eq.
//              delta_psi_eq_jac)
//   k_bracket  landing monotonicity / coverage checks, first bracket ray of
//              every resummation tile
//   k_resum    4-point Lagrange interpolation of phase and amplitude onto the
//              grid (Eq. ray_bundle_q_plus_1) fused with the modal sum
//
// The ray state is marched as deviations from the launch values:
//   dz = z - s,  dQ = Q - kappa_n,  rh = r - x P_bar_n,
// with P_bar_n = sqrt(eps_ref - kappa_n^2) and the table storing
// eps - eps_ref.  In exact arithmetic this is the same ODE as the plain form
// (RK4 is invariant under adding a constant to one right-hand side), but
// every stored quantity is small, so FP32 keeps ~1e-7 of the *deviation*.
// The dropped constant x P_bar_n is restored on the host, in FP64 and reduced
// mod 2 pi, as exp(i k dx P_bar_n) folded into c_n.

#include <utility>

#include <type_traits>

#include "swkb_device.cuh"

namespace swkb {

// ----------------------------------------------------------------------------
// launchers
// ----------------------------------------------------------------------------
namespace {
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     Args&&... args) {
  k<<<grid, block, smem, s>>>(std::forward<Args>(args)...);
  return cudaGetLastError();
}
}  // namespace

template <typename T>
cudaError_t launch_init(const double* u0, int n_z, int N, int mirror, typename C2<T>::type* u,
                        cudaStream_t s) {
  return launch_k(k_init<T>, dim3((N + 255) / 256), dim3(256), 0, s, u0, n_z, N, mirror, u);
}

template <typename T>
cudaError_t launch_reduce(const ReduceArgs<T>& a, cudaStream_t s) {
  const int n = (a.mirror || a.sym) ? a.N / 2 + 1 : a.N;
  return launch_k(k_reduce<T>, dim3((n + 255) / 256), dim3(256), 0, s, a);
}

template <typename T>
size_t fft1_smem_bytes(int N1, int cols) {
  const int E = N1 * cols;
  return (size_t)(E + N1 + (E < FFT1_THREADS ? PART_SUMS * E : 0)) * sizeof(typename C2<T>::type);
}

namespace {
// cos(2 pi k / 64) as the nearest double and what is missing from it.  A kernel argument:
// in constant memory it would be a bank more for every kernel of the library (0.3 us a
// launch: 40 screens on reused rays 488 -> 503 us).
struct Roots64 {
  double c[17][2];
};
constexpr Roots64 kRoots64 = {{
    {1.0, 0.0}, {0.9951847266721969, -4.248691367830441e-17},
    {0.9807852804032304, 1.8546939997825006e-17}, {0.9569403357322088, 4.05538698618757e-17},
    {0.9238795325112867, 1.7645047084336677e-17}, {0.881921264348355, -1.9843248405890562e-17},
    {0.8314696123025452, 1.4073856984728024e-18}, {0.773010453362737, -3.256590703364977e-17},
    {0.7071067811865476, -4.833646656726457e-17}, {0.6343932841636455, 1.0420901929280035e-17},
    {0.5555702330196022, 4.709410940561677e-17}, {0.47139673682599764, 6.516678136069013e-18},
    {0.3826834323650898, -1.0050772696461588e-17}, {0.2902846772544624, -1.892797870777425e-17},
    {0.19509032201612828, -7.991079068461731e-18}, {0.0980171403295606, -1.634582362244256e-18},
    {0.0, 0.0}}};

// exp(-2 pi i k / 64) and what is missing from it
__device__ __forceinline__ void root64(const Roots64& r, int k, double2& w, double2& lo) {
  const int q = k >> 4 & 3, m = k & 15;
  const double* c = r.c[q & 1 ? 16 - m : m];   // |cos|, |sin| of the angle
  const double* s = r.c[q & 1 ? m : 16 - m];
  const bool nc = q == 1 || q == 2, ns = q < 2;
  w = make_double2(nc ? -c[0] : c[0], ns ? -s[0] : s[0]);
  lo = make_double2(nc ? -c[1] : c[1], ns ? -s[1] : s[1]);
}

// Pass 1 in FP64 on a field read directly, rounding no more than rows of 2048 points
// summed directly would: the first radix-4 step of the columns (exact factors) as
// they are loaded, then sums of N1 / 4 terms in two chains, with what the roots of unity
// lack added back.  4096 to 65536 points, error 0.89 to 0.99 of the direct sums', against
// 1.05 to 1.09 with sums of N1 / 2 terms and rounded roots (k_fft1).  Latency bounds it,
// so every load is issued before the first wait and the roots are an argument (both
// passes back to back, 4096 points, 201 modes 12.4 -> 10.4 us, 489 modes 12.4; k_fft1 10.4
// and 11.4; 65536 points, 8001 modes 80.0 either way).  COLS columns per CTA, N1 >= 2.
template <int COLS>
__global__ void __launch_bounds__(FFT1_THREADS)
    k_fft1_pairs(const FftArgs<double> p, const __grid_constant__ Roots64 roots) {
  using V = double2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N1 = p.N1, E = N1 * COLS, tid = threadIdx.x, c0 = blockIdx.x * COLS;
  V* tile = reinterpret_cast<V*>(smem_raw);          // [N1][COLS]
  V* w1 = tile + E;                                  // [N1] roots, then what they lack
  const auto twiddle = [&](int e) {
    return p.tw[(long long)(c0 + e % COLS) * (e / COLS) << p.tw_shift];
  };
  // residue q of k1 modulo radix: tile rows q L .. q L + L - 1 hold its inputs n1 = 0 .. L - 1
  const int radix = N1 < 4 ? 2 : 4, L = N1 / radix, o = L * COLS;   // o <= 16 x 8
  V x[4], w2;   // every load before the first wait
  if (tid < o) {
    const V* u = p.u + (long long)(tid / COLS) * p.N2 + c0 + tid % COLS;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < radix) x[j] = u[(long long)j * L * p.N2];
  }
  if (tid < E) w2 = twiddle(tid);
  for (int k = tid; k < N1; k += FFT1_THREADS) root64(roots, k * (64 / N1), w1[k], w1[N1 + k]);
  if (tid < o) {
    V* t = tile + tid;
    if (radix == 2) {
      t[0] = make_double2(x[0].x + x[1].x, x[0].y + x[1].y);
      t[o] = make_double2(x[0].x - x[1].x, x[0].y - x[1].y);
    } else {
      const V s0 = make_double2(x[0].x + x[2].x, x[0].y + x[2].y);
      const V s1 = make_double2(x[1].x + x[3].x, x[1].y + x[3].y);
      const V d0 = make_double2(x[0].x - x[2].x, x[0].y - x[2].y);
      const V d1 = make_double2(x[1].x - x[3].x, x[1].y - x[3].y);
      t[0] = make_double2(s0.x + s1.x, s0.y + s1.y);
      t[o] = make_double2(d0.x + d1.y, d0.y - d1.x);       // d0 - i d1
      t[2 * o] = make_double2(s0.x - s1.x, s0.y - s1.y);
      t[3 * o] = make_double2(d0.x - d1.y, d0.y + d1.x);   // d0 + i d1
    }
  }
  __syncthreads();
  for (int e = tid; e < E; e += FFT1_THREADS) {
    const int c = e % COLS, k1 = e / COLS, n2 = c0 + c;
    if (e != tid) w2 = twiddle(e);
    const V* t = tile + (k1 & (radix - 1)) * L * COLS + c;
    const auto mac = [&](V& sum, int n1) {
      const int i = (n1 * k1) & (N1 - 1);
      cmac<double>(sum, t[n1 * COLS], w1[N1 + i]);
      cmac<double>(sum, t[n1 * COLS], w1[i]);
    };
    V s0 = t[0], s1 = make_double2(0.0, 0.0);
    if (L > 1) mac(s1, 1);
#pragma unroll 2
    for (int n1 = 2; n1 < L; n1 += 2) {
      mac(s0, n1);
      mac(s1, n1 + 1);
    }
    s0.x += s1.x; s0.y += s1.y;
    p.Y[(long long)k1 * p.N2 + n2] = cmul<double>(s0, w2);
  }
}

// Pass 2 in FP64 without a mirror: one CTA per pair of bins of a row, n = k1 + N1 k2
// and k1 - N1 k2, which share the products of the row's entries with the cosine
// and the sine (4 FMAs per entry for both bins; one by one 12 FP64 instructions).
// Pairs are counted by n (fft2_pairs); where only one bin is kept the other is not
// stored.
// Bound by FP64 issue at large sizes, by latency at small ones.
__global__ void __launch_bounds__(FFT2_THREADS) k_fft2_pair(const FftArgs<double> p) {
  using V = double2;
  __shared__ V sum[2][FFT2_THREADS / 32];
  const int tid = threadIdx.x;
  const int k1 = blockIdx.x & (p.N1 - 1), k2 = blockIdx.x / p.N1;
  const V* row = (p.N1 > 1 ? p.Y : p.u) + (long long)k1 * p.N2;
  double xc = 0.0, ys = 0.0, xs = 0.0, yc = 0.0;
#pragma unroll 8
  for (int n2 = tid; n2 < p.N2; n2 += FFT2_THREADS) {
    const unsigned e = (unsigned)(((long long)n2 * k2) & (p.N2 - 1));
    const V r = row[n2], w = twiddle2(p.tw, e, p.tw_shift, p.N1);
    xc += r.x * w.x;
    ys += r.y * w.y;
    xs += r.x * w.y;
    yc += r.y * w.x;
  }
  V s[2];
  s[0].x = xc - ys; s[0].y = yc + xs;   // n = k1 + N1 k2
  s[1].x = xc + ys; s[1].y = yc - xs;   // n = k1 - N1 k2
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s[h].x += __shfl_xor_sync(0xffffffffu, s[h].x, o);
      s[h].y += __shfl_xor_sync(0xffffffffu, s[h].y, o);
    }
    if ((tid & 31) == 0) sum[h][tid >> 5] = s[h];
  }
  __syncthreads();
  if (tid > 1 || (tid == 1 && k2 == 0)) return;
  const int n = tid == 0 ? k1 + p.N1 * k2 : k1 - p.N1 * k2;
  if (n > p.n_max || n < -p.n_max) return;
  V tot = sum[tid][0];
#pragma unroll
  for (int w = 1; w < FFT2_THREADS / 32; ++w) { tot.x += sum[tid][w].x; tot.y += sum[tid][w].y; }
  tot.x *= p.inv_N; tot.y *= p.inv_N;
  const int i = n + p.n_max;
  const V cv = cmul<double>(tot, p.ephi[i]);
  p.c[i] = cv;
  if (p.cpol) p.cpol[i] = polar_turns<double>(cv);
}

template <typename T>
cudaError_t launch_fft1(const FftArgs<T>& a, cudaStream_t s) {
  if (a.N1 == 1) return cudaSuccess;
  const int cols = fft1_cols(a.N2);
  return launch_k(cols == 4 ? k_fft1<T, 4> : k_fft1<T, 8>, dim3(a.N2 / cols), dim3(FFT1_THREADS),
                  fft1_smem_bytes<T>(a.N1, cols), s, a);
}
}  // namespace

template <typename T>
cudaError_t launch_fft(const FftArgs<T>& a, cudaStream_t s) {
  const cudaError_t e = launch_fft1<T>(a, s);
  if (e != cudaSuccess) return e;
  const int modes = a.mirror ? a.n_max + 1 : 2 * a.n_max + 1;
  return launch_k(k_fft2<T>, dim3(modes), dim3(FFT2_THREADS), 0, s, a);
}

cudaError_t launch_fft_pairs(const FftArgs<double>& a, cudaStream_t s) {
  if (a.N1 > 1) {
    const int cols = fft1_cols(a.N2);
    const cudaError_t e =
        launch_k(cols == 4 ? k_fft1_pairs<4> : k_fft1_pairs<8>, dim3(a.N2 / cols),
                 dim3(FFT1_THREADS), (size_t)(cols + 2) * a.N1 * sizeof(double2), s, a, kRoots64);
    if (e != cudaSuccess) return e;
  }
  return launch_k(k_fft2_pair, dim3(fft2_pairs(a.N1, a.n_max)), dim3(FFT2_THREADS), 0, s, a);
}

template <>
cudaError_t launch_march<double>(const MarchArgs<double>& a, bool multi_column, cudaStream_t s) {
  const long long threads = (long long)a.Mr * a.NRT;
  const dim3 block(MARCH64_THREADS),
      grid((unsigned)((threads + MARCH64_THREADS - 1) / MARCH64_THREADS));
  const auto launch = [&](auto planes) {
    constexpr bool P = decltype(planes)::value;
    return !multi_column ? launch_k(k_march<ONE_COLUMN, P>, grid, block, 0, s, a)
           : a.med.pairs ? launch_k(k_march<PAIRS, P>, grid, block, 0, s, a)
                         : launch_k(k_march<COLUMNS, P>, grid, block, 0, s, a);
  };
  return a.plane_steps > 0 ? launch(std::true_type{}) : launch(std::false_type{});
}

template <>
cudaError_t launch_march<float>(const MarchArgs<float>& a, bool multi_column, cudaStream_t s) {
  const long long threads = (long long)a.Mr * ((a.NRT + 1) / 2);
  const dim3 block(MARCH_THREADS),
      grid((unsigned)((threads + MARCH_THREADS - 1) / MARCH_THREADS));
  const bool pl = a.plane_steps > 0, cub = a.med.pieces > 0;
  if (cub) {
    if (pl)
      return multi_column ? launch_k(k_march_x2<true, true, true>, grid, block, 0, s, a)
                          : launch_k(k_march_x2<false, true, true>, grid, block, 0, s, a);
    return multi_column ? launch_k(k_march_x2<true, false, true>, grid, block, 0, s, a)
                        : launch_k(k_march_x2<false, false, true>, grid, block, 0, s, a);
  }
  if (pl)
    return multi_column ? launch_k(k_march_x2<true, true, false>, grid, block, 0, s, a)
                        : launch_k(k_march_x2<false, true, false>, grid, block, 0, s, a);
  return multi_column ? launch_k(k_march_x2<true, false, false>, grid, block, 0, s, a)
                      : launch_k(k_march_x2<false, false, false>, grid, block, 0, s, a);
}

// The inner planes of a screen: the screens' kernels over n planes at once.  A
// plane alone leaves the chip mostly idle (latency of its launches and of a small
// sum), and they are independent of one another.  8192 points, 3 screens of 4 planes:
// 596 -> 433 us per call (22 -> 11 launches per screen).
namespace {
template <typename T>
__global__ void __launch_bounds__(256) k_bracket_planes(BracketArgs<T> p, const PlaneStrides ps) {
  const long long z = blockIdx.z;
  p.d += z * ps.rays;
  p.jlo += z * ps.jlo;
  if (p.jlo_neg) p.jlo_neg += z * ps.jlo;
  const int rows = bracket_rows(p.NRT);
  for (int by = blockIdx.y; by < rows; by += gridDim.y)
    bracket_body<T, LD_PLAIN>(p, blockIdx.x, by, threadIdx.x);
}

template <typename T, int PW>
__global__ void __launch_bounds__(RESUM_WARPS * 32, sizeof(T) == 4 ? (PW < 16 ? 7 : 5) : 1)
    k_resum_planes(ResumArgs<T> p, const PlaneStrides ps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const long long y = blockIdx.y;
  p.d += y * ps.rays;
  p.ph += y * ps.rays;
  p.a += y * ps.rays;
  p.jlo += y * ps.jlo;
  if (p.jlo_neg) p.jlo_neg += y * ps.jlo;
  p.cpol += y * ps.modes;
  p.part += y * ps.part;
  resum_body<PW, LD_NC, 0>(p, blockIdx.x, threadIdx.x, smem_raw, 0);
}

// the field of the output points alone, as k_reduce and k_output form it
template <typename T>
__global__ void k_output_planes(const ReduceArgs<T> p, const PlaneStrides ps, int offset, int n_z,
                                double* __restrict__ out) {
  using V = typename C2<T>::type;
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n_z) return;
  const V* part = p.part + blockIdx.y * ps.part;
  const int i = offset + m;
  V a = parts_total<V, LD_PLAIN>(part + i, p.N, p.n_part);
  if (p.mirror && (!p.sym || i == p.N / 2)) {
    const int r = p.N - i;   // mirrored plans' outputs are points i >= N / 2
    const V b = r == i ? a : parts_total<V, LD_PLAIN>(part + r, p.N, p.n_part);
    const T sg = T(p.mirror);
    a.x = T(0.5) * (a.x + sg * b.x);
    a.y = T(0.5) * (a.y + sg * b.y);
  }
  double* o = out + 2 * ((long long)blockIdx.y * n_z + m);
  o[0] = double(a.x);
  o[1] = double(a.y);
}
}  // namespace

template <typename T>
cudaError_t launch_bracket(const BracketArgs<T>& a, cudaStream_t s) {
  const int rows = bracket_rows(a.NRT);
  dim3 grid((a.Mr + 255) / 256, rows < 65535 ? rows : 65535);
  return launch_k(k_bracket<T>, grid, dim3(256), 0, s, a);
}

template <typename T>
size_t resum_smem_bytes(int wcap, int tile_points) {
  const size_t per_warp = ((RESUM_CF + 3) * (size_t)wcap * sizeof(T) + 15) & ~(size_t)15;
  const size_t stage = (size_t)RESUM_WARPS * per_warp;
  // 32 runs of PW points, each padded to PW + 1 entries
  const size_t red = (size_t)RESUM_WARPS * (tile_points + 32) * sizeof(typename C2<T>::type);
  return stage > red ? stage : red;
}

template <typename T>
cudaError_t launch_resum(const ResumArgs<T>& a, cudaStream_t s) {
  const int grid = a.n_tiles_run * a.n_groups;
  const size_t smem = resum_smem_bytes<T>(a.wcap, a.TM);
  const int threads = RESUM_WARPS * 32;
  switch (a.PW) {
    case 2: return launch_k(k_resum<T, 2>, dim3(grid), dim3(threads), smem, s, a);
    case 4: return launch_k(k_resum<T, 4>, dim3(grid), dim3(threads), smem, s, a);
    case 8: return launch_k(k_resum<T, 8>, dim3(grid), dim3(threads), smem, s, a);
    case 16: return launch_k(k_resum<T, 16>, dim3(grid), dim3(threads), smem, s, a);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t prepare_kernels(int resum_smem) {
  // The limit is a per-device property of the kernel shared by every plan in
  // the process: raise it to the device's opt-in maximum (never lower it, or
  // a plan with smaller tiles would break another plan's launches).
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  if (resum_smem > optin) return cudaErrorInvalidValue;
  const void* fs[] = {(const void*)k_resum<T, 2>, (const void*)k_resum<T, 4>,
                      (const void*)k_resum<T, 8>, (const void*)k_resum<T, 16>,
                      (const void*)k_resum_planes<T, 2>, (const void*)k_resum_planes<T, 4>,
                      (const void*)k_resum_planes<T, 8>, (const void*)k_resum_planes<T, 16>};
  for (const void* f : fs) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t prepare_fft_kernels() {
  // k_fft1's dynamic shared memory is at most 5 E + N1 complex values at E = 128,
  // N1 = 32 and 9 N1 (k_fft1_pairs: 10 N1) at the largest N1 = 64, inside 48 KB; k_fft2
  // uses static shared memory only
  static_assert((5 * 128 + 32) * 16 <= 48 * 1024 && 10 * 64 * 16 <= 48 * 1024,
                "k_fft1 staging exceeds 48 KB");
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_cscale(const typename C2<T>::type* c, const typename C2<T>::type* f,
                          typename C2<T>::type* pol, int M, int n, cudaStream_t s) {
  return launch_k(k_cscale<T>, dim3((M + 255) / 256, n), dim3(256), 0, s, c, f, pol, M);
}

template <typename T>
cudaError_t launch_bracket_planes(const BracketArgs<T>& a, const PlaneStrides& ps, int n,
                                  cudaStream_t s) {
  const int rows = bracket_rows(a.NRT);
  const dim3 grid((a.Mr + 255) / 256, rows < 65535 ? rows : 65535, n);
  return launch_k(k_bracket_planes<T>, grid, dim3(256), 0, s, a, ps);
}

template <typename T>
cudaError_t launch_resum_planes(const ResumArgs<T>& a, const PlaneStrides& ps, int n,
                                cudaStream_t s) {
  const dim3 grid(a.n_tiles_run * a.n_groups, n), block(RESUM_WARPS * 32);
  const size_t smem = resum_smem_bytes<T>(a.wcap, a.TM);
  switch (a.PW) {
    case 2: return launch_k(k_resum_planes<T, 2>, grid, block, smem, s, a, ps);
    case 4: return launch_k(k_resum_planes<T, 4>, grid, block, smem, s, a, ps);
    case 8: return launch_k(k_resum_planes<T, 8>, grid, block, smem, s, a, ps);
    case 16: return launch_k(k_resum_planes<T, 16>, grid, block, smem, s, a, ps);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_output_planes(const ReduceArgs<T>& a, const PlaneStrides& ps, int offset,
                                 int n_z, int n, double* out, cudaStream_t s) {
  return launch_k(k_output_planes<T>, dim3((n_z + 255) / 256, n), dim3(256), 0, s, a, ps, offset,
                  n_z, out);
}

template <typename T>
cudaError_t launch_output(const typename C2<T>::type* u, int offset, int n, double* out,
                          cudaStream_t s) {
  return launch_k(k_output<T>, dim3((n + 255) / 256), dim3(256), 0, s, u, offset, n, out);
}

#define SWKB_INSTANTIATE(T)                                                                     \
  template cudaError_t launch_init<T>(const double*, int, int, int, C2<T>::type*, cudaStream_t); \
  template cudaError_t launch_reduce<T>(const ReduceArgs<T>&, cudaStream_t);                    \
  template cudaError_t launch_fft<T>(const FftArgs<T>&, cudaStream_t);                          \
  template cudaError_t launch_bracket<T>(const BracketArgs<T>&, cudaStream_t);                  \
  template cudaError_t launch_resum<T>(const ResumArgs<T>&, cudaStream_t);                      \
  template cudaError_t launch_output<T>(const C2<T>::type*, int, int, double*, cudaStream_t);   \
  template cudaError_t launch_cscale<T>(const C2<T>::type*, const C2<T>::type*, C2<T>::type*,   \
                                        int, int, cudaStream_t);                                \
  template cudaError_t launch_bracket_planes<T>(const BracketArgs<T>&, const PlaneStrides&, int, \
                                                cudaStream_t);                                  \
  template cudaError_t launch_resum_planes<T>(const ResumArgs<T>&, const PlaneStrides&, int,    \
                                              cudaStream_t);                                    \
  template cudaError_t launch_output_planes<T>(const ReduceArgs<T>&, const PlaneStrides&, int,  \
                                               int, int, double*, cudaStream_t);                \
  template size_t resum_smem_bytes<T>(int, int);                                                \
  template size_t fft1_smem_bytes<T>(int, int);                                                     \
  template cudaError_t prepare_kernels<T>(int);                                                 \
  template cudaError_t prepare_fft_kernels<T>();

SWKB_INSTANTIATE(float)
SWKB_INSTANTIATE(double)

}  // namespace swkb
