// Patch-wise Fourier-continuation screens (Sec. 2.2, Eq. ifft_eq_phi_patches):
// the two kernels that replace the periodic DFT and resummation on a
// non-periodic interval.  The ray march and the bracket search are the
// periodic ones: a ray depends only on its mode angle and launch point, so
// one family per mode serves every patch.
//
//   k_fc_modes  per patch: the patch's samples, its FC-Gram continuation to
//               N_p = n_pat + C points, and the kept modes of that sequence's DFT, w_n / N_p, rotated to the interval's
//               origin (exp(-2 pi i n s_p / N_p)) and carried over the screen
//               (exp(i k dx Pbar_n)): cf[p][n].  The continuation runs in
//               FP64 in every plan (the operator's entries reach 3e3, so its
//               cancellations need FP64); the DFT sums in the plan's type.
//   k_fc_resum  the interpolation fused with the modal sum, as the periodic
//               resummation, except that a ray's amplitude is complex: ray
//               (n, j) carries a_j (S^{p0}(z_j) cf[p0][n] + S^{p0+1}(z_j)
//               cf[p0+1][n]), p0 the first patch whose weight is non-zero at
//               z_j (at most two are), and the integer part of the phase is
//               2 pi (n m mod N_p) / N_p.
#include <cuda_runtime.h>

#include "swkb_device.cuh"
#include "swkb_fc_tables.h"

namespace swkb {

namespace {

constexpr int FC_MODES_PARTS = 8;        // parts of the sequence in a DFT block
constexpr int FC_MODES_BINS = 32;        // bins n >= 0 of one
constexpr int FC_MODES_THREADS = FC_MODES_PARTS * FC_MODES_BINS;
constexpr int FC_MODES_PATCHES = 4;      // patches sharing a block's twiddles
constexpr int FC_CHUNK = 16;             // samples summed before they join the total
constexpr int FC_WARPS = 4;
constexpr int FC_PF = 1;    // rounds of 32 rays prefetched one mode ahead
// Row of interval w: X_w, X_{w+1}, phase b0..b3, Re a r0..r3, Im a i0..i3.
// FP32: 20 floats (16 used) read as four 16-byte words; at an 80-byte stride
// the 8 lanes of a load phase touch 32 distinct banks.  FP64: 14 values read as
// 7 pairs.
template <typename T>
constexpr int FC_CF = sizeof(T) == 4 ? 20 : 14;

// x mod Np for x < 2^32 with magic = floor(2^32 / Np): the quotient
// estimate is floor(x / Np) or one less, so one correction finishes it.
__device__ __forceinline__ unsigned mod_np(unsigned x, unsigned Np, unsigned magic) {
  unsigned r = x - __umulhi(x, magic) * Np;
  return r >= Np ? r - Np : r;
}

template <typename T>
__host__ __device__ inline int fc_warp_bytes(int wcap) {
  return ((FC_CF<T> + 4) * wcap * (int)sizeof(T) + 15) & ~15;
}

// Twiddles of a DFT block, padded so that the samples behind them start on 16
// bytes.
__host__ __device__ inline int modes_pad(int Np) { return (Np + 1) & ~1; }

// CTA (PP patches from blockIdx.x PP, mode block blockIdx.y): the continuation
// in FP64, then the DFT in T (a mixed plan sums in FP32: exact twiddle indices,
// FP32 twiddles and samples).  A thread forms the bins n and -n of its PP
// patches over every eighth sample of the sequence (a warp each), from the sums of e cos and
// e sin they share, in chunks of 16 samples; the parts are added pairwise at the end.
// (Strided parts: neighbouring samples' terms are alike, so a part of consecutive
// ones sums to larger values; FP32 fields were 2 to 4 % further from FP64 with.)
//   What bounds it: per twiddle one gather from shared memory (several bank
// conflicts: lanes are consecutive n, so its stride is the sample's index) and
// its index, shared by PP patches and both bins.  188 patches of 945 points, 545
// modes: 35 us, against 95 with a warp per mode and patch (a gather and a sample
// per term); see launch_fc_modes for PP.
template <typename T, int PP>
__global__ void __launch_bounds__(FC_MODES_THREADS) k_fc_modes(const FcModesArgs<T> p) {
  using V = typename C2<T>::type;
  constexpr int PARTS = FC_MODES_PARTS, BINS = FC_MODES_BINS;
  static_assert(PARTS == 8, "the pairwise sum of the parts is written out");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* tw = reinterpret_cast<V*>(smem_raw);   // [N_p] exp(-2 pi i k / N_p)
  V* e = tw + modes_pad(p.Np);              // [N_p][PP] the continued sequences
  __shared__ double2 ends[PP][2 * FC_D];    // the d samples at each end, FP64
  const int pt0 = blockIdx.x * PP;
  const int np = min(PP, p.P - pt0);        // patches of this CTA
  for (int x = threadIdx.x; x < p.n_pat * PP; x += FC_MODES_THREADS) {
    const int k = x / PP, a = x % PP;
    V v;
    v.x = T(0); v.y = T(0);
    if (a < np) v = p.u[(long long)(pt0 + a) * p.stride + k];
    e[x] = v;
    if (k < FC_D) ends[a][FC_D + k] = make_double2((double)v.x, (double)v.y);
    if (k >= p.n_pat - FC_D)
      ends[a][k - (p.n_pat - FC_D)] = make_double2((double)v.x, (double)v.y);
  }
  for (int k = threadIdx.x; k < p.Np; k += FC_MODES_THREADS) {
    const double2 w = p.tw[k];
    V v;
    v.x = (T)w.x;
    v.y = (T)w.y;
    tw[k] = v;
  }
  __syncthreads();
  for (int x = threadIdx.x; x < FC_C * PP; x += FC_MODES_THREADS) {
    // value t past the right end: the right end's d samples (ends[0 .. d-1])
    // through row t; the same value counted backwards from the left end is
    // C - t steps before sample 0: the left end read backwards (sample
    // d - 1 - i = ends[2 d - 1 - i]) through row C - 1 - t
    const int t = x / PP, a = x % PP;
    double ar = 0.0, ai = 0.0;
    for (int i = 0; i < FC_D; ++i) {
      const double cr = p.cont[t * FC_D + i];
      const double cl = p.cont[(FC_C - 1 - t) * FC_D + i];
      const double2 fr = ends[a][i];
      const double2 fl = ends[a][2 * FC_D - 1 - i];
      ar += cr * fr.x + cl * fl.x;
      ai += cr * fr.y + cl * fl.y;
    }
    V v;
    v.x = (T)ar;
    v.y = (T)ai;
    e[(p.n_pat + t) * PP + a] = v;
  }
  __syncthreads();
  const unsigned Np = (unsigned)p.Np;
  const int lt = threadIdx.x % BINS, part = threadIdx.x / BINS;
  const int n = blockIdx.y * BINS + lt;      // bins n and -n, n <= n_max < Np / 2
  const unsigned nn = (unsigned)min(n, p.n_max);
  // sums of e cos and of e sin (the twiddle's parts) per patch
  T cr[PP], ci[PP], sr[PP], si[PP];
#pragma unroll
  for (int a = 0; a < PP; ++a) cr[a] = ci[a] = sr[a] = si[a] = T(0);
  int k = part;
  const unsigned step = mod_np(nn * (unsigned)PARTS, Np, p.np_magic);
  unsigned idx = mod_np(nn * (unsigned)part, Np, p.np_magic);
  while (k < p.Np) {
    const int stop = min(k + FC_CHUNK * PARTS, p.Np);
    T dr[PP], di[PP], fr[PP], fi[PP];
#pragma unroll
    for (int a = 0; a < PP; ++a) dr[a] = di[a] = fr[a] = fi[a] = T(0);
#pragma unroll 4
    for (; k < stop; k += PARTS) {
      const V w = tw[idx];
      idx += step;
      idx = min(idx, idx - Np);      // unsigned: the smaller is the one in [0, Np)
      V ev[PP];
      if constexpr (sizeof(T) == 4 && PP == 4) {
        const float4 x = *reinterpret_cast<const float4*>(e + k * PP);
        const float4 y = *reinterpret_cast<const float4*>(e + k * PP + 2);
        ev[0] = V{x.x, x.y}; ev[1] = V{x.z, x.w}; ev[2] = V{y.x, y.y}; ev[3] = V{y.z, y.w};
      } else {
#pragma unroll
        for (int a = 0; a < PP; ++a) ev[a] = e[k * PP + a];
      }
#pragma unroll
      for (int a = 0; a < PP; ++a) {
        const V v = ev[a];
        dr[a] += v.x * w.x;
        di[a] += v.y * w.x;
        fr[a] += v.x * w.y;
        fi[a] += v.y * w.y;
      }
    }
#pragma unroll
    for (int a = 0; a < PP; ++a) { cr[a] += dr[a]; ci[a] += di[a]; sr[a] += fr[a]; si[a] += fi[a]; }
  }
  // the other parts' sums through shared memory (over the samples)
  __syncthreads();
  T* red = reinterpret_cast<T*>(e);   // [PARTS - 1][4 PP][BINS]
  const T inv = (T)p.inv_Np;
  if (part > 0) {
    T* r = red + (part - 1) * 4 * PP * BINS + lt;
#pragma unroll
    for (int a = 0; a < PP; ++a) {
      r[(4 * a + 0) * BINS] = cr[a];
      r[(4 * a + 1) * BINS] = ci[a];
      r[(4 * a + 2) * BINS] = sr[a];
      r[(4 * a + 3) * BINS] = si[a];
    }
  }
  __syncthreads();
  if (part != 0 || n > p.n_max) return;
  const V ep = p.ephi[p.n_max + n], em = p.ephi[p.n_max - n];
#pragma unroll
  for (int a = 0; a < PP; ++a) {
    if (a >= np) break;
    const auto total = [&](T own, int v) {
      T q[PARTS];
      q[0] = own;
#pragma unroll
      for (int x = 1; x < PARTS; ++x) q[x] = red[((x - 1) * 4 * PP + 4 * a + v) * BINS + lt];
      return ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
    };
    const T ar = total(cr[a], 0), ai = total(ci[a], 1);
    const T br = total(sr[a], 2), bi = total(si[a], 3);
    // nn s0 < 2^11 2^20
    const V rot = tw[mod_np(nn * (unsigned)((long long)(pt0 + a) * p.stride), Np, p.np_magic)];
    // X_n = sum e w = (ar - bi) + i (ai + br), X_-n = sum e conj(w); each times
    // the patch's rotation (conjugated for -n), exp(i phi) and 1 / N_p
    const auto finish = [&](T xr, T xi, T ry, V ph) {
      const T zr = xr * rot.x - xi * ry, zi = xr * ry + xi * rot.x;
      V c;
      c.x = (zr * ph.x - zi * ph.y) * inv;
      c.y = (zr * ph.y + zi * ph.x) * inv;
      return c;
    };
    V* cf = p.cf + (long long)(pt0 + a) * p.M + p.n_max;
    cf[n] = finish(ar - bi, ai + br, rot.y, ep);
    if (n > 0) cf[-n] = finish(ar + bi, ai - br, -rot.y, em);
  }
}

template <typename T>
struct FcRow;

template <>
struct FcRow<float> {
  f2 c3, c2, c1, c0;   // (Re, Im) of the amplitude's cubic
  float X1, X2, b0, b1, b2, b3;
  __device__ __forceinline__ void load(const float* p) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(p);
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p + 4);
    const float4 x = *reinterpret_cast<const float4*>(p + 8);
    const float4 y = *reinterpret_cast<const float4*>(p + 12);
    c3.v = u.x; c2.v = u.y; c1.v = v.x; c0.v = v.y;
    X1 = x.x; X2 = x.y; b0 = x.z; b1 = x.w;
    b2 = y.x; b3 = y.y;
  }
};

template <>
struct FcRow<double> {
  double X1, X2, b0, b1, b2, b3, r0, r1, r2, r3, i0, i1, i2, i3;
  __device__ __forceinline__ void load(const double* p) {
    const double2* q = reinterpret_cast<const double2*>(p);
    const double2 a = q[0], b = q[1], c = q[2], d = q[3], e = q[4], f = q[5], g = q[6];
    X1 = a.x; X2 = a.y; b0 = b.x; b1 = b.y; b2 = c.x; b3 = c.y; r0 = d.x; r1 = d.y;
    r2 = e.x; r3 = e.y; i0 = f.x; i1 = f.y; i2 = g.x; i3 = g.y;
  }
};

// Rows of the intervals 1 .. W - 3 of a window (staged landings X, phases and
// complex amplitudes), a lane per interval; the last one's end is stored as
// infinity, so that no lane steps past it.  Returns whether every interval the
// lane built is at least a grid step long.
__device__ __forceinline__ bool build_rows(float* s_cf, const float* s_X, const float* s_ph,
                                           const float2* s_a, int W, int lane) {
  bool wide = true;
  for (int w = 1 + lane; w <= W - 3; w += 32) {
    const float X0 = s_X[w - 1], X1 = s_X[w], X2 = s_X[w + 1], X3 = s_X[w + 2];
    const float h21 = X2 - X1, h10 = X1 - X0;
    wide = wide && h21 >= 1.f;
    const float r21 = rcp_approx(h21), r10 = rcp_approx(h10), r32 = rcp_approx(X3 - X2);
    const float r20 = rcp_approx(X2 - X0), r31 = rcp_approx(X3 - X1), r30 = rcp_approx(X3 - X0);
    float b0, b1, b2, b3;
    cubic_through(s_ph[w - 1], s_ph[w], s_ph[w + 1], s_ph[w + 2], r21, r10, r32, r20, r31, r30,
                  h21, h10, b0, b1, b2, b3);
    const auto val = [&](int k) {
      f2 v;
      v.v = *reinterpret_cast<const unsigned long long*>(s_a + w + k);
      return v;
    };
    // the same Newton form for (Re, Im) together
    const f2 f0 = val(-1), f1 = val(0), fa = val(1), f3 = val(2);
    const f2 d12 = mul2(sub2(fa, f1), bc2(r21)), d01 = mul2(sub2(f1, f0), bc2(r10));
    const f2 d23 = mul2(sub2(f3, fa), bc2(r32));
    const f2 d012 = mul2(sub2(d12, d01), bc2(r20)), d123 = mul2(sub2(d23, d12), bc2(r31));
    const f2 c3 = mul2(sub2(d123, d012), bc2(r30));
    const f2 c1 = fma2(bc2(-h21), fma2(c3, bc2(h10), d012), d12);
    const f2 c2 = fma2(c3, bc2(h10 - h21), d012);
    float* row = s_cf + FC_CF<float> * w;
    *reinterpret_cast<ulonglong2*>(row) = make_ulonglong2(c3.v, c2.v);
    *reinterpret_cast<ulonglong2*>(row + 4) = make_ulonglong2(c1.v, f1.v);
    *reinterpret_cast<float4*>(row + 8) =
        make_float4(X1, w == W - 3 ? __int_as_float(0x7f800000) : X2,
                    minus_rint(b0), b1);           // whole turns do not matter
    *reinterpret_cast<float2*>(row + 12) = make_float2(b2, b3);
  }
  return wide;
}
__device__ __forceinline__ bool build_rows(double* s_cf, const double* s_X, const double* s_ph,
                                           const double2* s_a, int W, int lane) {
  bool wide = true;
  for (int w = 1 + lane; w <= W - 3; w += 32) {
    const double X0 = s_X[w - 1], X1 = s_X[w], X2 = s_X[w + 1], X3 = s_X[w + 2];
    const double h21 = X2 - X1, h10 = X1 - X0;
    wide = wide && h21 >= 1.0;
    const double r21 = rcp64(h21), r10 = rcp64(h10), r32 = rcp64(X3 - X2);
    const double r20 = rcp64(X2 - X0), r31 = rcp64(X3 - X1), r30 = rcp64(X3 - X0);
    const double2 f0 = s_a[w - 1], f1 = s_a[w], f2 = s_a[w + 1], f3 = s_a[w + 2];
    double b0, b1, b2, b3, c0, c1, c2, c3, d0, d1, d2, d3;
    cubic_through(s_ph[w - 1], s_ph[w], s_ph[w + 1], s_ph[w + 2], r21, r10, r32, r20, r31, r30,
                  h21, h10, b0, b1, b2, b3);
    cubic_through(f0.x, f1.x, f2.x, f3.x, r21, r10, r32, r20, r31, r30, h21, h10, c0, c1, c2, c3);
    cubic_through(f0.y, f1.y, f2.y, f3.y, r21, r10, r32, r20, r31, r30, h21, h10, d0, d1, d2, d3);
    double2* row = reinterpret_cast<double2*>(s_cf + FC_CF<double> * w);
    row[0] = make_double2(X1, w == W - 3 ? __longlong_as_double(0x7ff0000000000000ll) : X2);
    row[1] = make_double2(b0, b1);
    row[2] = make_double2(b2, b3);
    row[3] = make_double2(c0, c1);
    row[4] = make_double2(c2, c3);
    row[5] = make_double2(d0, d1);
    row[6] = make_double2(d2, d3);
  }
  return wide;
}

// The term of one point: tau from the row's X_w, t the phase in turns without
// the row's part.
__device__ __forceinline__ void add_term(const FcRow<float>& r, const double2*, float xv, float t,
                                         float& sr, float& si) {
  const float tau = xv - r.X1;
  const f2 tau2 = bc2(tau);
  float ar, ai, sn, cs;
  sp2(fma2(fma2(fma2(r.c3, tau2, r.c2), tau2, r.c1), tau2, r.c0), ar, ai);
  sincos_turns(t + (((r.b3 * tau + r.b2) * tau + r.b1) * tau + r.b0), &sn, &cs);
  sr += fmaf(ar, cs, -ai * sn);   // one rounding at the sum's size per term
  si += fmaf(ar, sn, ai * cs);
}
__device__ __forceinline__ void add_term(const FcRow<double>& r, const double2* trig, double xv,
                                         double t, double& sr, double& si) {
  const double tau = xv - r.X1;
  const double ar = ((r.r3 * tau + r.r2) * tau + r.r1) * tau + r.r0;
  const double ai = ((r.i3 * tau + r.i2) * tau + r.i1) * tau + r.i0;
  double sn, cs;
  sincos_table(trig, t, ((r.b3 * tau + r.b2) * tau + r.b1) * tau + r.b0, &sn, &cs);
  sr += fma(ar, cs, -ai * sn);
  si += fma(ar, sn, ai * cs);
}

template <typename T>
struct FcRay {
  T d, ph;
  typename C2<T>::type a;
};

// ray j of mode i: landing offset, phase and the complex amplitude
// a_j (S^{p0}(z_j) cf[p0][i] + S^{p0+1}(z_j) cf[p0+1][i])
template <typename T>
__device__ __forceinline__ FcRay<T> fc_ray(const FcResumArgs<T>& p, int i, int j, unsigned& st) {
  using V = typename C2<T>::type;
  // NRT M < 2^32 (at most 2^20 + 2 G rays of 2047 modes)
  const unsigned o = (unsigned)bchk((long long)((unsigned)j * (unsigned)p.M + (unsigned)i),
                                    (long long)p.NRT * p.M, st);
  FcRay<T> v;
  v.d = ld<LD_NC>(p.d + o);
  v.ph = ld<LD_NC>(p.ph + o);
  const T a = ld<LD_NC>(p.a + o);
  const int p0 = __ldg(p.win_p + j);
  const V sw = p.win_s[j];
  const V c0 = p.cf[bchk((long long)p0 * p.M + i, (long long)p.P * p.M, st)];
  T cr = sw.x * c0.x, ci = sw.x * c0.y;
  if (p0 + 1 < p.P) {
    const V c1 = p.cf[(long long)(p0 + 1) * p.M + i];
    cr += sw.y * c1.x;
    ci += sw.y * c1.y;
  }
  v.a.x = a * cr;
  v.a.y = a * ci;
  return v;
}

// Rays of the window between two brackets (0: skip).  A table left inconsistent by a
// failed screen (flagged by the bracket kernel) must not send the reads out of
// [0, NRT).
template <typename T>
__device__ __forceinline__ int fc_window(const FcResumArgs<T>& p, int jl, int jh) {
  return jl >= 1 && jh >= jl && jh <= p.NRT - 3 ? jh - jl + 4 : 0;
}

// The warps' sums in a fixed order, written as (ADD: added to) the group's partial.
template <typename T, int PW, bool ADD>
__device__ __forceinline__ void fc_block_sum(const FcResumArgs<T>& p, unsigned char* smem_raw,
                                             const T* accr, const T* acci, int tile, int group,
                                             unsigned st) {
  using V = typename C2<T>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, TM = p.TM, m0 = tile * TM;
  V* red = reinterpret_cast<V*>(smem_raw);
  const int TMP = 32 * (PW + 1);
#pragma unroll
  for (int q = 0; q < PW; ++q) {
    V v;
    v.x = accr[q];
    v.y = acci[q];
    red[warp * TMP + lane * (PW + 1) + q] = v;
  }
  __syncthreads();
  V* out = p.part + bchk((long long)group * p.N + m0, (long long)p.n_groups * p.N - (TM - 1), st);
  if (st) atomicOr(p.status, st);
  for (int x = threadIdx.x; x < TM; x += FC_WARPS * 32) {
    const int xs = (x / PW) * (PW + 1) + x % PW;
    V sum = red[xs];
#pragma unroll
    for (int k = 1; k < FC_WARPS; ++k) {
      const V v = red[k * TMP + xs];
      sum.x += v.x;
      sum.y += v.y;
    }
    if (ADD) { sum.x += out[x].x; sum.y += out[x].y; }
    out[x] = sum;
  }
}

// The modes of a tile whose rays are compressed beyond a window (wcap rays), up to wlim
// on the tile or its pair of tiles (lim_pair): wcap rays at a time.  A function of its
// own: within the main loop it takes that loop's registers (235 instead of 224 us on
// the 131072-point lens).
template <typename T, int PW>
__device__ __noinline__ void fc_resum_split(const FcResumArgs<T>& p, unsigned char* smem_raw,
                                            int tile, int group) {
  using V = typename C2<T>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wcap = p.wcap, m0 = tile * p.TM, x0 = lane * PW;
  T* s_cf = reinterpret_cast<T*>(smem_raw + (long long)warp * fc_warp_bytes<T>(wcap));
  V* s_a = reinterpret_cast<V*>(s_cf + FC_CF<T> * wcap);
  T* s_X = reinterpret_cast<T*>(s_a + wcap);
  T* s_ph = s_X + wcap;
  const int i1 = min(p.M, (group + 1) * p.modes_per_group);
  const unsigned Np = (unsigned)p.Np;
  const T invNp = T(1) / T(p.Np);
  unsigned st = 0;
  T accr[PW], acci[PW];
#pragma unroll
  for (int q = 0; q < PW; ++q) { accr[q] = T(0); acci[q] = T(0); }
  __syncthreads();   // the block's first sums are read
  for (int i = group * p.modes_per_group + warp; i < i1; i += FC_WARPS) {
    const auto bracket = [&](int t) {
      return p.jlo[bchk((long long)t * p.M + i, (long long)(p.n_tiles + 1) * p.M, st)];
    };
    const int jb = bracket(tile) - 1, W = fc_window(p, jb + 1, bracket(tile + 1));
    if (W <= wcap) continue;
    // (its own window too: beside an inconsistent bracket the pair's may be empty)
    if (W > p.wlim ||
        (p.lim_pair && fc_window(p, bracket(tile & ~1), bracket((tile | 1) + 1)) > p.wlim)) {
      st |= ST_CAUSTIC;
      continue;
    }
    const int base = (jb - p.G) * p.R - m0, n = i - p.n_max;
    const unsigned nn = (unsigned)(n < 0 ? n + p.Np : n);   // phases as in k_fc_resum
    T bc = T(mod_np(nn * (unsigned)(m0 + x0 + PW / 2), Np, p.np_magic)) * invNp;
    bc = bc >= T(0.5) ? bc - T(1) : bc;
    for (int w0 = 0; w0 < W - 3; w0 += wcap - 3) {
      const int Wp = min(wcap, W - w0);
      __syncwarp();
      for (int s = lane; s < Wp; s += 32) {
        const FcRay<T> v = fc_ray(p, i, jb + w0 + s, st);
        s_X[s] = T(base + (w0 + s) * p.R) + v.d;
        s_ph[s] = v.ph;
        s_a[s] = v.a;
      }
      __syncwarp();
      build_rows(s_cf, s_X, s_ph, s_a, Wp, lane);
      __syncwarp();
      int w = 1;
#pragma unroll
      for (int q = 0; q < PW; ++q) {   // the points of these rays' intervals
        const T xv = T(x0 + q);
        if ((w0 == 0 || s_X[1] <= xv) && (w0 + Wp == W || xv < s_X[Wp - 2])) {
          while (w < Wp - 3 && s_X[w + 1] <= xv) ++w;
          FcRow<T> r;
          r.load(s_cf + FC_CF<T> * w);
          add_term(r, p.trig, xv, fma(T(q - PW / 2), T(n) * invNp, bc), accr[q], acci[q]);
        }
      }
    }
  }
  __syncthreads();
  fc_block_sum<T, PW, true>(p, smem_raw, accr, acci, tile, group, st);
}

// One CTA: tile blk % n_tiles (TM = 32 PW points), mode group blk / n_tiles;
// its warps take the group's modes round-robin (the structure of the periodic
// sum: brackets of 32 modes looked up at once, the next mode's first rays loaded
// one mode ahead) and the CTA adds the warps' sums in a fixed order.
// Bound by instruction issue and by the warps its shared memory leaves (96 bytes
// per ray of a window): 131072-point lens, 545 modes, R = 8, 225 us per sum with
// 128-point tiles (256-point ones 306; 261 before, with per-mode bracket
// lookups, scalar amplitude cubics and library divisions).  FP64 8192-point lens
// 415 us (723).  FP32 7 CTAs per SM (72 registers); 6: 223 us, 8: 289.
template <typename T, int PW>
__global__ void __launch_bounds__(FC_WARPS * 32, sizeof(T) == 4 ? 7 : 1)
    k_fc_resum(const FcResumArgs<T> p) {
  using V = typename C2<T>::type;
  constexpr unsigned ALL = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = blockIdx.x % p.n_tiles, group = blockIdx.x / p.n_tiles;
  const int wcap = p.wcap, TM = p.TM, m0 = tile * TM;
  T* s_cf = reinterpret_cast<T*>(smem_raw + (long long)warp * fc_warp_bytes<T>(wcap));
  V* s_a = reinterpret_cast<V*>(s_cf + FC_CF<T> * wcap);
  T* s_X = reinterpret_cast<T*>(s_a + wcap);
  T* s_ph = s_X + wcap;
  const int i0 = group * p.modes_per_group, i1 = min(p.M, i0 + p.modes_per_group);
  const unsigned Np = (unsigned)p.Np;
  const T invNp = T(1) / T(p.Np);
  const long long nrays = (long long)p.NRT * p.M;
  const long long njlo = (long long)(p.n_tiles + 1) * p.M;
  const int x0 = lane * PW;
  const T xv0 = T(x0);
  unsigned st = 0;
  T accr[PW], acci[PW];
#pragma unroll
  for (int q = 0; q < PW; ++q) { accr[q] = T(0); acci[q] = T(0); }

  using RayVal = FcRay<T>;
  auto fetch = [&](int i, int j) { return fc_ray(p, i, j, st); };
  auto window = [&](int jl, int jh) { return fc_window(p, jl, jh); };
  constexpr unsigned OVER = 1u << 31;   // (in st) windows left to fc_resum_split
  RayVal pre[FC_PF];   // the next mode's first FC_PF rounds of 32 rays
  auto prefetch = [&](int i, int jb, int W) {
#pragma unroll
    for (int r = 0; r < FC_PF; ++r)
      if (lane + 32 * r < W) pre[r] = fetch(i, jb + lane + 32 * r);
  };

  for (int ib = i0 + warp; ib < i1; ib += 32 * FC_WARPS) {
    // lane k: window of mode ib + FC_WARPS k (first ray jb, W rays; 0: skip)
    int h_jb = 0, h_W = 0;
    {
      const int i = ib + FC_WARPS * lane;
      if (i < i1) {
        const int jl = p.jlo[bchk((long long)tile * p.M + i, njlo, st)];
        const int jh = p.jlo[bchk((long long)(tile + 1) * p.M + i, njlo, st)];
        h_W = window(jl, jh);
        if (h_W > wcap) { st |= OVER; h_W = 0; }
        h_jb = jl - 1;
      }
    }
    const int K = min(32, (i1 - ib + FC_WARPS - 1) / FC_WARPS);
    int jb = __shfl_sync(ALL, h_jb, 0), W = __shfl_sync(ALL, h_W, 0);
    prefetch(ib, jb, W);
    for (int k = 0; k < K; ++k) {
      const int i = ib + FC_WARPS * k;
      const int Wc = W, jc = jb, base = (jc - p.G) * p.R - m0;
      const auto put = [&](int w, const RayVal& v) {
        s_X[w] = T(base + w * p.R) + v.d;
        s_ph[w] = v.ph;
        s_a[w] = v.a;
      };
      __syncwarp();
#pragma unroll
      for (int r = 0; r < FC_PF; ++r)
        if (lane + 32 * r < Wc) put(lane + 32 * r, pre[r]);
      for (int w = lane + 32 * FC_PF; w < Wc; w += 32) put(w, fetch(i, jc + w));
      if (k + 1 < K) {
        jb = __shfl_sync(ALL, h_jb, k + 1);
        W = __shfl_sync(ALL, h_W, k + 1);
        prefetch(i + FC_WARPS, jb, W);
      }
      if (Wc == 0) continue;
      __syncwarp();
      bool wide = build_rows(s_cf, s_X, s_ph, s_a, Wc, lane);
      wide = __all_sync(ALL, wide);
      __syncwarp();
      // lane l sums the PW consecutive points l PW .. l PW + PW - 1 of the tile
      int w;
      {
        const float xf = (float)s_X[1];
        const float inv_sp = (float)(Wc - 3) * rcp_approx((float)s_X[Wc - 2] - xf);
        w = 1 + ifloor_small(((float)x0 - xf) * inv_sp);
        w = min(max(w, 1), Wc - 3);
        while (w > 1 && s_X[w] > xv0) --w;
        while (w < Wc - 3 && s_X[w + 1] <= xv0) ++w;
      }
      const T* row = s_cf + FC_CF<T> * w;
      FcRow<T> r;
      r.load(row);
      // the exact integer phase n m / Np mod 1 of the run's middle point,
      // moved into [-1/2, 1/2), and n / Np (|n / Np| < 1/2) per point from it:
      // the argument of the sine stays within about two turns
      const int n = i - p.n_max;   // |n| < Np / 2
      const unsigned nn = (unsigned)(n < 0 ? n + p.Np : n);
      // nn (m0 + x0 + PW / 2) < 2^11 2^20: no overflow
      T bc = T(mod_np(nn * (unsigned)(m0 + x0 + PW / 2), Np, p.np_magic)) * invNp;
      bc = bc >= T(0.5) ? bc - T(1) : bc;
      const T nNp = T(n) * invNp;
      T xv = xv0;   // exact
      if (wide) {   // at most one interval ends between two points
#pragma unroll
        for (int q = 0; q < PW; ++q) {
          if (q > 0) {
            xv += T(1);
            if (r.X2 <= xv) {
              row += FC_CF<T>;
              r.load(row);
            }
          }
          add_term(r, p.trig, xv, fma(T(q - PW / 2), nNp, bc), accr[q], acci[q]);
        }
      } else {
#pragma unroll
        for (int q = 0; q < PW; ++q) {
          if (q > 0) {
            xv += T(1);
            while (r.X2 <= xv) {
              row += FC_CF<T>;
              r.load(row);
            }
          }
          add_term(r, p.trig, xv, fma(T(q - PW / 2), nNp, bc), accr[q], acci[q]);
        }
      }
    }
  }
  const bool over = __syncthreads_or(st & OVER);
  fc_block_sum<T, PW, false>(p, smem_raw, accr, acci, tile, group, st & ~OVER);
  if (over) fc_resum_split<T, PW>(p, smem_raw, tile, group);
}

template <typename T, int PW>
cudaError_t resum_pw(const FcResumArgs<T>& a, cudaStream_t s) {
  const size_t smem = fc_resum_smem_bytes<T>(a.wcap, a.TM);
  k_fc_resum<T, PW><<<a.n_tiles * a.n_groups, FC_WARPS * 32, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

template <typename T>
size_t fc_resum_smem_bytes(int wcap, int tile_points) {
  const size_t rows = (size_t)FC_WARPS * fc_warp_bytes<T>(wcap);
  const int PW = tile_points / 32;
  const size_t red = (size_t)FC_WARPS * 32 * (PW + 1) * 2 * sizeof(T);
  return rows > red ? rows : red;
}

template <typename T>
size_t modes_smem(int Np, int patches) {
  const size_t tw = (size_t)modes_pad(Np) * sizeof(typename C2<T>::type);
  // the sums of the other parts overlie the samples
  const size_t stage = (size_t)patches * Np * sizeof(typename C2<T>::type);
  const size_t red = (size_t)(FC_MODES_PARTS - 1) * 4 * patches * FC_MODES_BINS * sizeof(T);
  return tw + (stage > red ? stage : red);
}

template <typename T>
size_t fc_modes_smem_bytes(int Np) {
  return modes_smem<T>(Np, FC_MODES_PATCHES);
}

template <typename T>
cudaError_t prepare_fc_kernels(int resum_smem, int modes_smem) {
  // The limit is a per-device property of the kernel shared by every plan in
  // the process: raise it to the device's opt-in maximum (never lower it, or a
  // plan with a shorter period or smaller tiles would break another plan's
  // launches).
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  if (resum_smem > optin ||
      modes_smem + (int)(FC_MODES_PATCHES * 2 * FC_D * sizeof(double2)) > optin)
    return cudaErrorInvalidValue;
  const void* fs[] = {(const void*)k_fc_modes<T, 1>, (const void*)k_fc_modes<T, FC_MODES_PATCHES>,
                      (const void*)k_fc_resum<T, 2>,
                      (const void*)k_fc_resum<T, 4>, (const void*)k_fc_resum<T, 8>};
  for (const void* f : fs) {
    // the dynamic limit plus the kernel's static shared memory must stay
    // within the opt-in maximum
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - (int)fa.sharedSizeBytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// out[p][n] = cf[p][n] f[n]: the patches' coefficients carried to a plane
// inside the screen (f: exp(i k (j / P - 1) dx Pbar_n)).
template <typename T>
__global__ void k_fc_cscale(const typename C2<T>::type* __restrict__ cf,
                            const typename C2<T>::type* __restrict__ f,
                            typename C2<T>::type* __restrict__ out, int PM, int M) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= PM) return;
  const typename C2<T>::type a = cf[k], b = f[k % M];
  typename C2<T>::type c;
  c.x = a.x * b.x - a.y * b.y;
  c.y = a.x * b.y + a.y * b.x;
  out[k] = c;
}

template <typename T>
cudaError_t launch_fc_cscale(const typename C2<T>::type* cf, const typename C2<T>::type* f,
                             typename C2<T>::type* out, int P, int M, cudaStream_t s) {
  const int PM = P * M;
  k_fc_cscale<T><<<(PM + 255) / 256, 256, 0, s>>>(cf, f, out, PM, M);
  return cudaGetLastError();
}

// Four patches per CTA share each twiddle where that still gives 128 CTAs: 188
// patches of 545 modes 35 us, against 49 with one patch per CTA; few patches
// take a CTA each (12 patches of 539 modes 13.5 us; FP64 41 us, against 125 with a
// warp per mode and patch).  Blocks of 128 bins and two parts: 32 and 22 us, and
// longer beside the march (730 instead of 708 us per screen on the 131072-point
// lens).
template <typename T>
cudaError_t launch_fc_modes(const FcModesArgs<T>& a, cudaStream_t s) {
  const int bx = (a.P + FC_MODES_PATCHES - 1) / FC_MODES_PATCHES;
  const int by = a.n_max / FC_MODES_BINS + 1;   // bins 0 .. n_max
  if (bx * by >= 128)
    k_fc_modes<T, FC_MODES_PATCHES><<<dim3(bx, by), FC_MODES_THREADS,
                                      modes_smem<T>(a.Np, FC_MODES_PATCHES), s>>>(a);
  else
    k_fc_modes<T, 1><<<dim3(a.P, by), FC_MODES_THREADS, modes_smem<T>(a.Np, 1), s>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fc_resum(const FcResumArgs<T>& a, cudaStream_t s) {
  switch (a.TM / 32) {
    case 2: return resum_pw<T, 2>(a, s);
    case 4: return resum_pw<T, 4>(a, s);
    case 8: return resum_pw<T, 8>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

const double* fc_continuation_host() { return &kFcContinuation[0][0]; }

template size_t fc_resum_smem_bytes<float>(int, int);
template size_t fc_resum_smem_bytes<double>(int, int);
template size_t fc_modes_smem_bytes<float>(int);
template size_t fc_modes_smem_bytes<double>(int);
template cudaError_t prepare_fc_kernels<float>(int, int);
template cudaError_t prepare_fc_kernels<double>(int, int);
template cudaError_t launch_fc_modes<float>(const FcModesArgs<float>&, cudaStream_t);
template cudaError_t launch_fc_modes<double>(const FcModesArgs<double>&, cudaStream_t);
template cudaError_t launch_fc_resum<float>(const FcResumArgs<float>&, cudaStream_t);
template cudaError_t launch_fc_cscale<float>(const float2*, const float2*, float2*, int, int,
                                             cudaStream_t);
template cudaError_t launch_fc_cscale<double>(const double2*, const double2*, double2*, int, int,
                                              cudaStream_t);
template cudaError_t launch_fc_resum<double>(const FcResumArgs<double>&, cudaStream_t);

}  // namespace swkb
