// Device bodies of the screened-WKB screen step (sm_103a), templated on the
// arithmetic type T.  Every step is a __device__ function of its (virtual)
// block index and thread index, called by the standalone kernels of
// swkb_kernels.cu (one launch per step) and by the persistent batch kernel of
// swkb_batch.cu (many instances' steps as work items of one launch), so both
// run the same arithmetic.  See swkb_kernels.cu for the step list.
#pragma once

#include <math.h>
#include <stdint.h>

#include <utility>

#include "swkb_internal.h"

namespace swkb {

// ----------------------------------------------------------------------------
// small helpers
// ----------------------------------------------------------------------------
// Bounds-checked builds (-DSWKB_BOUNDS_CHECK, libswkb_checked.so): an index
// outside [0, n) sets ST_BOUNDS in the kernel's status bits, which the host
// reports as an error, and is clamped into range so that the access stays
// inside its buffer.  Plain builds compile the check away.
__device__ __forceinline__ long long bchk(long long i, long long n, unsigned& st) {
#ifdef SWKB_BOUNDS_CHECK
  if (i < 0 || i >= n) {
    st |= ST_BOUNDS;
    return i < 0 ? 0 : n - 1;
  }
#else
  (void)n; (void)st;
#endif
  return i;
}

// Loads of data another kernel (or, in the persistent batch kernel, another
// work item of the same kernel) produced: LD_NC through the read-only
// (non-coherent) path, valid only when nothing writes the data during the
// kernel; LD_CG from L2, bypassing L1, for the persistent kernel, where the
// producer ran on another SM while this kernel was running.
enum { LD_PLAIN = 0, LD_NC = 1, LD_CG = 2 };
template <int LD, typename T>
__device__ __forceinline__ T ld(const T* p) {
  if constexpr (LD == LD_NC) return __ldg(p);
  else if constexpr (LD == LD_CG) return __ldcg(p);
  else return *p;
}

// Barrier over the threads running one virtual block: the whole CTA
// (BAR = 0, the standalone kernels), or one 128-thread half of it (BAR = 1:
// named barrier 1 + sub, the persistent kernel runs two such blocks per CTA).
template <int BAR>
__device__ __forceinline__ void vb_sync(int sub) {
  if constexpr (BAR == 0) {
    (void)sub;
    __syncthreads();
  } else {
    asm volatile("bar.sync %0, 128;" ::"r"(1 + sub) : "memory");
  }
}

// sin / cos of 2 pi t on the special-function unit: absolute error ~2^-21 for
// |t| <= 1/2.  The sums pass t within a turn and a half plus (q - PW / 2) n / N, so up to
// four turns more for the steepest modes of 16-point runs, whose argument's rounding (up to
// 1e-6) adds to it.  The pair is 7.35e-8 shorter than 1 on average over whole circles.
__device__ __forceinline__ void sincos_turns(float t, float* s, float* c) {
  __sincosf(6.28318530717958647692f * t, s, c);
}

// Exact integer/float steps of the resummation kept off the conversion units
// in FP32: floor of |y| < 2^22 by a round-down add of 1.5 * 2^23, the float
// of an integer k < 2^23 from its bits, and t - rint(t) for |t| < 2^22 by
// adding and subtracting 1.5 * 2^23 (round to nearest even, as rint).
__device__ __forceinline__ int ifloor_small(float y) {
  return (int)(__float_as_uint(__fadd_rd(y, 12582912.f)) - 0x4B400000u);
}
__device__ __forceinline__ float exact_u2f(unsigned k) {
  return __uint_as_float(0x4B000000u | k) - 8388608.f;
}
__device__ __forceinline__ float minus_rint(float t) {
  const float r = (t + 12582912.f) - 12582912.f;
  return t - r;
}

template <typename T>
__device__ __forceinline__ void load6(const T* p, T& a0, T& a1, T& a2, T& a3, T& a4, T& a5);

template <>
__device__ __forceinline__ void load6<float>(const float* p, float& a0, float& a1, float& a2,
                                             float& a3, float& a4, float& a5) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  const float2 w = __ldg(reinterpret_cast<const float2*>(p + 4));
  a0 = v.x; a1 = v.y; a2 = v.z; a3 = v.w; a4 = w.x; a5 = w.y;
}

template <>
__device__ __forceinline__ void load6<double>(const double* p, double& a0, double& a1, double& a2,
                                              double& a3, double& a4, double& a5) {
  const double2 u = __ldg(reinterpret_cast<const double2*>(p));
  const double2 v = __ldg(reinterpret_cast<const double2*>(p + 2));
  const double2 w = __ldg(reinterpret_cast<const double2*>(p + 4));
  a0 = u.x; a1 = u.y; a2 = v.x; a3 = v.y; a4 = w.x; a5 = w.y;
}

// ----------------------------------------------------------------------------
// (b) ray march
// ----------------------------------------------------------------------------
// Both precisions march the same system, scaled so that the right-hand side
// needs no constant factors (h the medium table's spacing, c = 1 / (2 h),
// e = eps - eps_ref, d1 and d2 the table's p' and p''/2 in units of h):
//   w  = (z - s) / h        w'  = 2c A          A = Q / P
//   dQ = Q - kappa          dQ' = c B           B = d1 / P
//   rh = r - x P_bar        rh' = D / (P_bar + P) + dQ A
//   N  = -Z_s               N'  = -c (S + A m) / P,   m = A S + B N
//   S  = Q_s / c            S'  = c (-4 d2 N + B m) / P
// This is the x-form of Eqs. charsys / charsys_s divided by x_t = 2P
//   z' = Q/P, Q' = eps_z/(2P), r' = (eps - kappa Q)/P,
//   P_s = (eps_z Z_s - 2 Q Q_s)/(2P), Z_s' = (Q_s - Q P_s/P)/P,
//   Q_s' = (eps_zz Z_s - eps_z P_s/P)/(2P)
// with D = e - dQ (2 kappa + dQ) = P^2 - P_bar^2, P - P_bar = D / (P_bar + P)
// and -P_s / P = c m / P.  The factors c, 2c, -c enter through the RK4 weights.

// 1/sqrt(x) and 1/x in FP64: the special-function unit's estimate (relative
// error ~2^-20) corrected by one step of third order (Householder's
// iterations: y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2, and y (1 + e + e^2)
// with e = 1 - x y), whose own error, ~2^-58, is below the rounding.  5 and 3
// FP64 operations, for normal positive x.
__device__ __forceinline__ double rsqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double rcp64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// FP64 medium lookup at table position u (intervals from the table origin;
// grounded domains: from the ground, the table even about it): p(t), p'(t) and
// p''(t)/2 of the interval's quintic.  The interval comes from the low bits of
// a round-down add of 1.5 * 2^52, so that only three additions of the lookup
// are FP64 work; positions outside the table (or its very top) take the slow
// branch.  The coefficients of two columns are blended with weight th: 12 FMAs, 6 where
// the table holds differences (PAIRS); a second polynomial and its blend would take 18.
enum { ONE_COLUMN = 0, COLUMNS = 1, PAIRS = 2 };
template <int MULTI>
__device__ __forceinline__ void med64(const MarchArgs<double>& p, int l, double u, double& e,
                                      double& d1, double& d2, unsigned& st) {
  constexpr int W = MULTI == PAIRS ? 16 : 8;
  const double magic = 6755399441055744.0;
  const double z = p.med.mirrored ? fabs(u) : u;
  const double v = __dadd_rd(z, magic);
  int i = __double2loint(v);
  double t = z - (v - magic);
  if (__double2hiint(v) != 0x43380000 || (unsigned)i >= (unsigned)p.med.n_int) {
    if (!(z >= 0.0 && z <= p.med.top)) st |= ST_RANGE;
    i = z > 0.0 ? p.med.n_int - 1 : 0;
    t = z > 0.0 ? 1.0 : 0.0;
  }
  const double* q = p.med.coef;
  long long o = (long long)i * W;
  double th = 0.0;
  if constexpr (MULTI != ONE_COLUMN) {
    o += (long long)__ldg(p.st.c + l) * p.med.col_stride;
    th = __ldg(p.st.th + l);
  }
  const long long next = MULTI == COLUMNS ? p.med.col_stride : MULTI == PAIRS ? 8 : 0;
  q += bchk(o, p.med.size - next - 7, st);
  double a[6];
  load6<double>(q, a[0], a[1], a[2], a[3], a[4], a[5]);
  if constexpr (MULTI != ONE_COLUMN) {
    double d[6];
    load6<double>(q + next, d[0], d[1], d[2], d[3], d[4], d[5]);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      a[k] = fma(th, d[k], MULTI == PAIRS ? a[k] : fma(-th, a[k], a[k]));
  }
  // Horner with derivatives (synthetic division)
  double b = a[5] * t + a[4];                             // coefficient 4
  d2 = a[5];                                              // coefficient 3
  d1 = a[5] * t + b;
  b = b * t + a[3];
  d2 = d2 * t + d1; d1 = d1 * t + b; b = b * t + a[2];    // coefficient 2
  d2 = d2 * t + d1; d1 = d1 * t + b; b = b * t + a[1];    // coefficient 1
  d2 = d2 * t + d1; d1 = d1 * t + b; b = b * t + a[0];    // coefficient 0
  e = b;
  // below the ground the slope changes sign (the sign bit of u)
  if (p.med.mirrored)
    d1 = __hiloint2double(__double2hiint(d1) ^ (__double2hiint(u) & (int)0x80000000),
                          __double2loint(d1));
}

struct Ray {
  double w, dQ, rh, N, S;
};

// Right-hand side without the factors 2c, c, 1, -c, c.  Turning points (P^2 <=
// 0) and caustics (N >= 0) are running extremes of the high words (as integers,
// off the FP64 pipe), tested once per ray.
template <int MULTI>
__device__ __forceinline__ Ray rhs64(const MarchArgs<double>& p, int l, double u, double kap,
                                     double pb, double pb2, const Ray& y, int& P2_lo, int& N_hi,
                                     unsigned& st) {
  double e, d1, d2;
  med64<MULTI>(p, l, u, e, d1, d2, st);
  const double Q = kap + y.dQ;
  const double D = fma(-y.dQ, Q + kap, e);                // e - dQ (2 kappa + dQ)
  const double P2 = pb2 + D;
  P2_lo = min(P2_lo, __double2hiint(P2));
  N_hi = max(N_hi, __double2hiint(y.N));
  const double iP = rsqrt64(P2);
  const double rden = rcp64(fma(P2, iP, pb));             // 1 / (P_bar + P)
  Ray d;
  d.w = Q * iP;
  d.dQ = d1 * iP;
  d.rh = fma(D, rden, y.dQ * d.w);
  const double m = fma(d.dQ, y.N, d.w * y.S);
  d.N = fma(d.w, m, y.S) * iP;
  d.S = fma(d.dQ, m, (-4.0 * d2) * y.N) * iP;
  return d;
}

// Thread t marches ray j of mode r, t = j Mr + r: a warp's lanes are
// consecutive modes at one launch height, so their table reads stay within a
// few intervals.  THREADS threads per block.
template <int MULTI, bool PLANES, int THREADS>
__device__ __forceinline__ void march64_body(const MarchArgs<double>& p, int blk, int tid) {
  const long long t = (long long)blk * THREADS + tid;
  if (t >= (long long)p.Mr * p.NRT) return;
  const int j = (int)(t / p.Mr);
  const int r = (int)(t - (long long)j * p.Mr);
  unsigned st = 0;
  const int i = r + p.mode_off;
  const double kap = p.kappa[i], pb = p.pbar[i], pb2 = p.pbar2[i];
  const double s = fma((double)((j - p.G) * p.R), p.u_dz, p.u_lo);   // launch height in intervals
  double e0, d0, d00;
  med64<MULTI>(p, 0, s, e0, d0, d00, st);
  double P0sq = pb2 + e0;
  if (!(P0sq > 0.0)) { st |= ST_TURNING; P0sq = pb2; }
  const double P0 = sqrt(P0sq);
  Ray y{0.0, 0.0, 0.0, -1.0, 0.0};
  const double H2 = p.s2, H = 2.0 * H2, W1 = 2.0 * H;
  const double H6 = p.s6, W6 = 2.0 * H6, h6 = p.h6;
  int P2_lo = 0x7fefffff, N_hi = (int)0x80000000;
  // landing quantities at RK4 stage l (the screen's end, or a plane inside it)
  auto land = [&](int l, double* od, double* oph, double* oa) {
    const long long o = bchk((long long)j * p.Mr + r, (long long)p.NRT * p.Mr, st);
    if (!(y.N < 0.0)) st |= ST_CAUSTIC;
    double e1, f1, g1;
    med64<MULTI>(p, l, s + y.w, e1, f1, g1, st);
    double P1sq = pb2 + e1 - y.dQ * (2.0 * kap + y.dQ);
    if (!(P1sq > 0.0)) { st |= ST_TURNING; P1sq = pb2; }
    const double Zs = y.N < 0.0 ? -y.N : 1.0;
    od[o] = y.w * p.w_out;
    oph[o] = y.rh * p.ph_out;
    oa[o] = sqrt(P0 * rsqrt(P1sq) / Zs);
  };
  // A step's slopes are summed (k1 + 2 k2 + 2 k3 + k4) before they join the state, so
  // that it is rounded once per step; a stage state needs no rh, and its w only as
  // the table position
  for (int n = 0; n < p.Nt; ++n) {
    const double u0 = s + y.w;
    Ray sum;
    auto add2x = [&](const Ray& k) {
      sum = Ray{fma(2.0, k.w, sum.w), fma(2.0, k.dQ, sum.dQ), fma(2.0, k.rh, sum.rh),
                fma(2.0, k.N, sum.N), fma(2.0, k.S, sum.S)};
    };
    auto stage = [&](const Ray& k, double gq) {
      return Ray{0.0, fma(gq, k.dQ, y.dQ), 0.0, fma(-gq, k.N, y.N), fma(gq, k.S, y.S)};
    };
    const Ray k1 = rhs64<MULTI>(p, 2 * n, u0, kap, pb, pb2, y, P2_lo, N_hi, st);
    sum = k1;
    const Ray k2 = rhs64<MULTI>(p, 2 * n + 1, fma(H, k1.w, u0), kap, pb, pb2, stage(k1, H2),
                                P2_lo, N_hi, st);
    add2x(k2);
    const Ray k3 = rhs64<MULTI>(p, 2 * n + 1, fma(H, k2.w, u0), kap, pb, pb2, stage(k2, H2),
                                P2_lo, N_hi, st);
    add2x(k3);
    const Ray k4 = rhs64<MULTI>(p, 2 * n + 2, fma(W1, k3.w, u0), kap, pb, pb2, stage(k3, H),
                                P2_lo, N_hi, st);
    y = Ray{fma(W6, sum.w + k4.w, y.w), fma(H6, sum.dQ + k4.dQ, y.dQ),
            fma(h6, sum.rh + k4.rh, y.rh), fma(-H6, sum.N + k4.N, y.N),
            fma(H6, sum.S + k4.S, y.S)};
    if (PLANES && (n + 1) % p.plane_steps == 0 && n + 1 < p.Nt) {
      const long long po = (long long)((n + 1) / p.plane_steps - 1) * p.NRT * p.Mr;
      land(2 * (n + 1), p.pl_d + po, p.pl_ph + po, p.pl_a + po);
    }
  }
  land(2 * p.Nt, p.out_d, p.out_ph, p.out_a);
  if (P2_lo <= 0) st |= ST_TURNING;
  if (N_hi >= 0) st |= ST_CAUSTIC;
  if (st) atomicOr(p.status, st);
}

// Bound by the FP64 pipe (2 operations per SM and clock, ~87 % busy): ~49 FP64
// operations per stage (12 of them the quintic, 8 the two special functions).
// On the 16384-point duct (489 modes x 2086 rays, 16 RK4 steps) 6.3 ms, against
// 9.1 ms with the unscaled system, library rsqrt and division, and FP64
// comparisons and conversions in the lookup (~66).  CTAs of 64 threads spread
// small plans evenly: 65 modes x 704 rays on 152 SMs take 0.18 ms, against
// 0.50 ms in CTAs of 256 (179 of them: two on some SMs, one on the others) that
// evaluated both columns of a lookup.
constexpr int MARCH64_THREADS = 64;

template <int MULTI, bool PLANES>
__global__ void __launch_bounds__(MARCH64_THREADS) k_march(const MarchArgs<double> p) {
  march64_body<MULTI, PLANES, MARCH64_THREADS>(p, blockIdx.x, threadIdx.x);
}

// ----------------------------------------------------------------------------
// (b) ray march, FP32 path with packed f32x2 arithmetic: each thread marches
// two rays of one mode (see march_x2_body for which).  The medium polynomials
// are evaluated per ray; the table positions, the right-hand side of the ray +
// variational system and the RK4 updates run on register pairs, halving their
// issue slots.
// ----------------------------------------------------------------------------
struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ f2 mk2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void sp2(f2 x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 bc2(float a) { return mk2(a, a); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {   // a b + c
  f2 r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// floor of both lanes' positions: a round-down add of 1.5 * 2^23 (exact for
// 0 <= u < 2^22), whose low bits are the integer
__device__ __forceinline__ f2 add2_rd(f2 a, f2 b) {
  f2 r;
  asm("add.rm.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Marched state of two rays (scaled as above).
struct Ray2 {
  f2 w, dQ, rh, N, S;
};

__device__ __forceinline__ void horner5(const float a[6], float t, float& e, float& d1,
                                        float& d2) {
  float b = a[5] * t + a[4];
  float c2 = a[5];
  float c1 = a[5] * t + b;
  b = b * t + a[3];
  c2 = c2 * t + c1; c1 = c1 * t + b; b = b * t + a[2];
  c2 = c2 * t + c1; c1 = c1 * t + b; b = b * t + a[1];
  c2 = c2 * t + c1; c1 = c1 * t + b; b = b * t + a[0];
  e = b; d1 = c1; d2 = c2;
}

// Cubic piece b0..b3 in tau: value, first derivative and half the second
// derivative by synthetic division (6 FMAs).
__device__ __forceinline__ void horner3(const float4 v, float t, float& e, float& d1, float& d2) {
  float b = v.w * t + v.z;
  float c1 = v.w * t + b;
  b = b * t + v.y;
  const float c2 = v.w * t + c1;
  c1 = c1 * t + b;
  b = b * t + v.x;
  e = b; d1 = c1; d2 = c2;
}

// Two coefficients of two columns blended with weight th (m = -th), exact at both ends.
__device__ __forceinline__ f2 blend2(f2 th, f2 m, f2 a, f2 b) {
  return fma2(th, b, fma2(m, a, a));
}

// One entry of the FP32 medium table at its local coordinate t: p(t), p'(t)
// and p''(t)/2.  MULTI: blended with the next column's entry (next values on)
// before the polynomial is evaluated (4 packed and 6 FMAs for a cubic piece;
// evaluating both columns and blending the results takes 18).
template <bool MULTI, bool CUBIC>
__device__ __forceinline__ void table_eval(const float* q, long long next, float t, float th,
                                           float& e, float& d1, float& d2) {
  const f2 th2 = bc2(th), m2 = bc2(-th);
  if constexpr (CUBIC) {
    float4 v = __ldg(reinterpret_cast<const float4*>(q));
    if constexpr (MULTI) {
      const float4 d = __ldg(reinterpret_cast<const float4*>(q + next));
      sp2(blend2(th2, m2, mk2(v.x, v.y), mk2(d.x, d.y)), v.x, v.y);
      sp2(blend2(th2, m2, mk2(v.z, v.w), mk2(d.z, d.w)), v.z, v.w);
    }
    horner3(v, t, e, d1, d2);
  } else {
    float a[6];
    load6<float>(q, a[0], a[1], a[2], a[3], a[4], a[5]);
    if constexpr (MULTI) {
      float d[6];
      load6<float>(q + next, d[0], d[1], d[2], d[3], d[4], d[5]);
#pragma unroll
      for (int k = 0; k < 6; k += 2)
        sp2(blend2(th2, m2, mk2(a[k], a[k + 1]), mk2(d[k], d[k + 1])), a[k], a[k + 1]);
    }
    horner5(a, t, e, d1, d2);
  }
}

// Running extremes of a ray pair, tested once per ray: table position, P^2
// (<= 0: turning point) and -Z_s (>= 0: caustic).  A ray that meets one goes on
// with values that are discarded; its table reads are clamped.  The
// comparisons drop NaNs: a ray that turns NaN stays NaN, and its landing is
// tested explicitly.
struct Extremes {
  float u_lo, u_hi, P2, N;
};

// FP32 medium lookup of both rays at table positions u2 (intervals or pieces
// from the table origin; the table stores the reflection, so there is no
// mirror step).
template <bool MULTI, bool CUBIC>
__device__ __forceinline__ void med32x2(const MarchArgs<float>& p, int l, f2 u2, f2& e, f2& d1,
                                        float& d2a, float& d2b, Extremes& x, unsigned& st) {
  constexpr int W = CUBIC ? 4 : 8;
  const f2 magic = bc2(12582912.f);
  const f2 v = add2_rd(u2, magic);
  const f2 t = sub2(u2, sub2(v, magic));
  float ua, ub, va, vb, ta, tb;
  sp2(u2, ua, ub);
  sp2(v, va, vb);
  sp2(t, ta, tb);
  x.u_lo = fminf(x.u_lo, fminf(ua, ub));
  x.u_hi = fmaxf(x.u_hi, fmaxf(ua, ub));
  // unsigned: positions below 0 and NaN wrap to large indices
  const unsigned n = (unsigned)p.med.n_int;
  const unsigned ia = min(__float_as_uint(va) - 0x4B400000u, n);
  const unsigned ib = min(__float_as_uint(vb) - 0x4B400000u, n);
  const float* base = p.med.coef;
  float th = 0.f;
  if constexpr (MULTI) {
    base += (long long)__ldg(p.st.c + l) * p.med.col_stride;
    th = __ldg(p.st.th + l);
  }
  const long long off = base - p.med.coef, next = MULTI ? p.med.col_stride : 0;
  const long long end = p.med.size - next - (W - 1);
  float ea, eb, d1a, d1b;
  table_eval<MULTI, CUBIC>(base + (bchk(off + (long long)ia * W, end, st) - off), next, ta, th,
                           ea, d1a, d2a);
  table_eval<MULTI, CUBIC>(base + (bchk(off + (long long)ib * W, end, st) - off), next, tb, th,
                           eb, d1b, d2b);
  e = mk2(ea, eb);
  d1 = mk2(d1a, d1b);
}

// Right-hand side of the scaled system above for two rays at table positions
// u2, without the factors 2c, c, 1, -c, c: d.w = A, d.dQ = B, ...
template <bool MULTI, bool CUBIC>
__device__ __forceinline__ Ray2 rhs2(const MarchArgs<float>& p, int l, f2 u2, f2 kap, f2 m2kap,
                                     f2 pb, f2 pb2v, const Ray2& y, Extremes& x, unsigned& st) {
  f2 e, d1;
  float d2a, d2b;
  med32x2<MULTI, CUBIC>(p, l, u2, e, d1, d2a, d2b, x, st);
  const f2 Q = add2(kap, y.dQ);
  const f2 D = fma2(y.dQ, sub2(m2kap, y.dQ), e);           // e - dQ (2 kappa + dQ)
  const f2 P2 = add2(pb2v, D);
  float P2a, P2b, Na, Nb;
  sp2(P2, P2a, P2b);
  sp2(y.N, Na, Nb);
  x.P2 = fminf(x.P2, fminf(P2a, P2b));
  x.N = fmaxf(x.N, fmaxf(Na, Nb));
  const f2 iP = mk2(rsqrtf(P2a), rsqrtf(P2b));
  float da, db;
  sp2(fma2(P2, iP, pb), da, db);                           // P_bar + P
  const f2 rden = mk2(rcp_approx(da), rcp_approx(db));
  Ray2 d;
  d.w = mul2(Q, iP);
  d.dQ = mul2(d1, iP);
  d.rh = fma2(D, rden, mul2(y.dQ, d.w));
  const f2 m = fma2(d.dQ, y.N, mul2(d.w, y.S));
  d.N = mul2(fma2(d.w, m, y.S), iP);
  d.S = mul2(fma2(d.dQ, m, mul2(mul2(mk2(d2a, d2b), bc2(-4.f)), y.N)), iP);
  return d;
}

// Amplitude factor sqrt(P0 / (P1 Z)) of P0^2, P1^2 and Z, rounded once: the approximate
// roots and the quotient lose 5e-8 on average where all three are near 1, the same
// way for every ray, and the field that much of its length at each screen.  One
// Newton step on a^4 P1^2 Z^2 = P0^2, whose left side is formed in two parts.
__device__ __forceinline__ float amplitude(float P0sq, float P1sq, float Z) {
  const float a = sqrtf(sqrtf(P0sq) * rsqrtf(P1sq) / Z);
  const float h = a * a, hl = fmaf(a, a, -h);
  const float u = h * Z, ul = fmaf(hl, Z, fmaf(h, Z, -u));
  const float w = u * u, wl = fmaf(2.f * u, ul, fmaf(u, u, -w));
  const float q = w * P1sq, ql = fmaf(wl, P1sq, fmaf(w, P1sq, -q));
  return fmaf(0.25f * a * rcp_approx(P0sq), (P0sq - q) - ql, a);
}

// Thread t marches rays q and q + NH of mode r, t = q Mr + r (NH = ceil(NRT / 2)):
// a warp's lanes are consecutive modes at one launch height (their table
// reads stay within a few intervals) and no lane idles at the end of a row.
// THREADS threads per block.
template <bool MULTI, bool PLANES, bool CUBIC, int THREADS>
__device__ __forceinline__ void march_x2_body(const MarchArgs<float>& p, int blk, int tid) {
  const int NH = (p.NRT + 1) >> 1;
  const int t = blk * THREADS + tid;
  if (t >= p.Mr * NH) return;
  const int ja = t / p.Mr;
  const int r = t - ja * p.Mr;
  const int jb = ja + NH;
  const bool has_b = jb < p.NRT;
  unsigned st = 0;
  const int i = r + p.mode_off;
  const float kap = p.kappa[i], pb = p.pbar[i], pb2 = p.pbar2[i];
  // launch heights in table intervals
  const float ua = fmaf(float((ja - p.G) * p.R), p.u_dz, p.u_lo);
  const float ub = has_b ? fmaf(float((jb - p.G) * p.R), p.u_dz, p.u_lo) : ua;
  const f2 s = mk2(ua, ub), kv = bc2(kap), m2kap = bc2(-2.f * kap);
  const f2 pbv = bc2(pb), pb2v = bc2(pb2);
  const f2 zero = bc2(0.f);
  Extremes x{ua, ua, 1.f, -1.f};   // P^2 and Z_s start at 1: none below
  f2 e0, d0;
  float t0, t1;
  med32x2<MULTI, CUBIC>(p, 0, s, e0, d0, t0, t1, x, st);
  float P0a, P0b;
  sp2(add2(pb2v, e0), P0a, P0b);
  if (!(P0a > 0.f)) { st |= ST_TURNING; P0a = pb2; }
  if (!(P0b > 0.f)) { st |= ST_TURNING; P0b = pb2; }
  Ray2 y{zero, zero, zero, bc2(-1.f), zero};
  // RK4 weights 1/2, 1, 1/6 times the factors of the scaled system
  const float s2 = p.s2, s6 = p.s6;
  const f2 two = bc2(2.f), H2 = bc2(s2), H1 = bc2(2.f * s2), W1 = bc2(4.f * s2);
  const f2 n2 = bc2(-s2), n1 = bc2(-2.f * s2);
  const f2 H6 = bc2(s6), n6 = bc2(-s6), W6 = bc2(2.f * s6), h6 = bc2(p.h6);
  const float w_out = p.w_out;
  // landing quantities at RK4 stage l (the screen's end, or a plane inside it)
  const auto land = [&](int l, float* od, float* oph, float* oam) {
    const long long nrm = (long long)p.NRT * p.Mr;
    const long long oa = bchk((long long)ja * p.Mr + r, nrm, st);
    const long long ob = has_b ? bchk((long long)jb * p.Mr + r, nrm, st) : oa;
    float wa, wb, dQa, dQb, rha, rhb, Na, Nb, u1a, u1b, e1a, e1b;
    sp2(y.w, wa, wb);
    sp2(y.dQ, dQa, dQb);
    sp2(y.rh, rha, rhb);
    sp2(y.N, Na, Nb);
    const f2 u1 = add2(s, y.w);
    sp2(u1, u1a, u1b);
    if (!(Na < 0.f) || !(Nb < 0.f)) st |= ST_CAUSTIC;
    if (!(u1a >= 0.f && u1a <= p.med.top) || !(u1b >= 0.f && u1b <= p.med.top)) st |= ST_RANGE;
    f2 e1, d1;
    float s0, s1;
    med32x2<MULTI, CUBIC>(p, l, u1, e1, d1, s0, s1, x, st);
    sp2(e1, e1a, e1b);
    float P1a = pb2 + e1a - dQa * (2.f * kap + dQa);
    float P1b = pb2 + e1b - dQb * (2.f * kap + dQb);
    if (!(P1a > 0.f)) { st |= ST_TURNING; P1a = pb2; }
    if (!(P1b > 0.f)) { st |= ST_TURNING; P1b = pb2; }
    const float Za = Na < 0.f ? -Na : 1.f, Zb = Nb < 0.f ? -Nb : 1.f;
    od[oa] = wa * w_out;
    oph[oa] = rha * p.ph_out;
    oam[oa] = amplitude(P0a, P1a, Za);
    if (has_b) {
      od[ob] = wb * w_out;
      oph[ob] = rhb * p.ph_out;
      oam[ob] = amplitude(P0b, P1b, Zb);
    }
  };
  // A step's slopes are summed (k1 + 2 k2 + 2 k3 + k4) before they join the state, so
  // that it is rounded once per step, not four times (amplitudes of a 1 km screen
  // 2.9 times closer, phases 1.6 times; as many operations).  A stage state needs
  // no rh, and its w only as the table position u.
  for (int n = 0; n < p.Nt; ++n) {
    const f2 u0 = add2(s, y.w);
    Ray2 sum;
    const auto add2x = [&](const Ray2& k) {
      sum = Ray2{fma2(two, k.w, sum.w), fma2(two, k.dQ, sum.dQ), fma2(two, k.rh, sum.rh),
                 fma2(two, k.N, sum.N), fma2(two, k.S, sum.S)};
    };
    const auto stage = [&](const Ray2& k, f2 gq, f2 gn) {
      return Ray2{zero, fma2(gq, k.dQ, y.dQ), zero, fma2(gn, k.N, y.N), fma2(gq, k.S, y.S)};
    };
    const Ray2 k1 = rhs2<MULTI, CUBIC>(p, 2 * n, u0, kv, m2kap, pbv, pb2v, y, x, st);
    sum = k1;
    const Ray2 k2 = rhs2<MULTI, CUBIC>(p, 2 * n + 1, fma2(H1, k1.w, u0), kv, m2kap, pbv, pb2v,
                                       stage(k1, H2, n2), x, st);
    add2x(k2);
    const Ray2 k3 = rhs2<MULTI, CUBIC>(p, 2 * n + 1, fma2(H1, k2.w, u0), kv, m2kap, pbv, pb2v,
                                       stage(k2, H2, n2), x, st);
    add2x(k3);
    const Ray2 k4 = rhs2<MULTI, CUBIC>(p, 2 * n + 2, fma2(W1, k3.w, u0), kv, m2kap, pbv, pb2v,
                                       stage(k3, H1, n1), x, st);
    y = Ray2{fma2(W6, add2(sum.w, k4.w), y.w), fma2(H6, add2(sum.dQ, k4.dQ), y.dQ),
             fma2(h6, add2(sum.rh, k4.rh), y.rh), fma2(n6, add2(sum.N, k4.N), y.N),
             fma2(H6, add2(sum.S, k4.S), y.S)};
    if (PLANES && (n + 1) % p.plane_steps == 0 && n + 1 < p.Nt) {
      const long long po = (long long)((n + 1) / p.plane_steps - 1) * p.NRT * p.Mr;
      land(2 * (n + 1), p.pl_d + po, p.pl_ph + po, p.pl_a + po);
    }
  }
  land(2 * p.Nt, p.out_d, p.out_ph, p.out_a);
  if (!(x.P2 > 0.f)) st |= ST_TURNING;
  if (!(x.N < 0.f)) st |= ST_CAUSTIC;
  if (!(x.u_lo >= 0.f && x.u_hi <= p.med.top)) st |= ST_RANGE;
  if (st) atomicOr(p.status, st);
}

// Bound by the FMA pipe: ~71 of its cycles per ray-pair stage (13 FFMA2, 8
// FMUL2, 7 FADD2 at two cycles each, 12 FFMA of the medium, 2 IMAD), busy 64 %
// of the time that CTAs are resident; 58 instructions in all.  On the
// 16384-point duct (489 modes x 2086 rays, 16 RK4 steps) 103 us, against 121
// with the unscaled system (35 packed operations, 80 instructions); 347
// against 485 us on a range-dependent table (698 modes x 4118 rays; 331 with the
// columns' differences stored, which doubles the table).
// 6 CTAs of 128 threads per SM (80 registers): 102 us; 3 of 256: 104; 4 of
// 256 (64 registers, spills): 112; 2 of 256: 107; all-scalar arithmetic: 110.  With
// inner planes 5 per SM (96 registers; 80 spill): 8192 points, 3 screens of 4 planes 447
// against 458 us per call.
constexpr int MARCH_THREADS = 128;

template <bool MULTI, bool PLANES, bool CUBIC>
__global__ void __launch_bounds__(MARCH_THREADS, PLANES ? 5 : 6)
    k_march_x2(const MarchArgs<float> p) {
  march_x2_body<MULTI, PLANES, CUBIC, MARCH_THREADS>(p, blockIdx.x, threadIdx.x);
}

// ----------------------------------------------------------------------------
// landing checks and tile brackets
// ----------------------------------------------------------------------------
// Landing of ray j in grid units: g_j = (j - G) R + d_j.  Tile t starts at
// grid point t TM; jlo[t][i] = the j with g_j <= t TM < g_{j+1}.

// Coverage of the screen by the landing pair (j, j + 1).
template <typename T>
__device__ __forceinline__ unsigned cover_pair(const BracketArgs<T>& p, int j, T d0, T d1) {
  const int b0 = (j - p.G) * p.R, b1 = b0 + p.R;
  unsigned st = 0;
  if (j == 1 && !(d0 <= T(-b0))) st |= ST_COVER;                  // g_1 <= 0
  if (j + 1 == p.NRT - 2 && !(d1 > T(p.N - b1))) st |= ST_COVER;  // g_{NRT-2} > N
  if (p.sym) {   // the mirror family g'_{j'} = N - g_{NRT-j'} must cover too
    if (j == 2 && !(d0 < T(-b0))) st |= ST_COVER;                 // g_2 < 0
    if (j + 1 == p.NRT - 1 && !(d1 >= T(p.N - b1))) st |= ST_COVER;  // g_{NRT-1} >= N
  }
  return st;
}

// A thread takes BRACKET_RUN consecutive landing pairs of one column, all its
// loads issued first; most runs bracket no tile start and leave after one test.
// Bound by the latency of those loads and, for large plans, by reading the
// landings: 489 x 2086 landings 8.1 us, 545 x 16398 20 us, FP64 489 x 2086 20 us
// (a thread per pair, each with its own estimates and loops for both families:
// 10.2, 39 and 38; runs of 2: 8.2, 30 and 18.5).
constexpr int BRACKET_RUN = 4;
// blocks along the rays
__host__ __device__ inline int bracket_rows(int NRT) {
  return (NRT - 1 + BRACKET_RUN - 1) / BRACKET_RUN;
}

template <typename T, int LD>
__device__ __forceinline__ void bracket_body(const BracketArgs<T>& p, int bx, int by, int tid) {
  const int i = bx * 256 + tid;
  if (i >= p.Mr) return;
  const int j0 = by * BRACKET_RUN;
  const int n = min(BRACKET_RUN, p.NRT - 1 - j0);   // pairs (j0 + k, j0 + k + 1), k < n
  unsigned st = 0;
  const long long nrm = (long long)p.NRT * p.Mr, o = (long long)j0 * p.Mr + i;
  T d[BRACKET_RUN + 1];
#pragma unroll
  for (int k = 0; k <= BRACKET_RUN; ++k)
    d[k] = ld<LD>(p.d + bchk(o + (long long)min(k, n) * p.Mr, nrm, st));
  bool rising = true;
#pragma unroll
  for (int k = 0; k < BRACKET_RUN; ++k)
    if (k < n) rising = rising && T(p.R) + d[k + 1] - d[k] > T(0);   // g_{j+1} > g_j
  if (!rising) st |= ST_CAUSTIC;
  if (j0 <= 2 || j0 + BRACKET_RUN >= p.NRT - 2) {
#pragma unroll
    for (int k = 0; k < BRACKET_RUN; ++k)
      if (k < n) st |= cover_pair(p, j0 + k, d[k], d[k + 1]);
  }
  // Multiples x = t TM within the run's landings, by a float estimate with a
  // margin of TM / 100, far above its rounding; exact tests decide.  Tile t of
  // the family starts at x, tile n_tiles - t of its mirror image (landings
  // N - g) at N - x.  (A run out of order, or NaN, is an error already: nothing
  // is written, and the sums check what they take from the table.)
  const float inv_tm = 1.0f / (float)p.TM;   // exact (TM is a power of two)
  const int b0 = (j0 - p.G) * p.R;           // |b0| <= N + G R < 2^31
  const float g0 = (float)b0 + (float)d[0];
  const float g1 = (float)(b0 + n * p.R) + (float)d[BRACKET_RUN];
  const int t0 = max((int)ceilf(g0 * inv_tm - 1e-2f), 0);
  const int t1 = rising ? min((int)floorf(g1 * inv_tm + 1e-2f), p.n_tiles) : -1;
  for (int t = t0; t <= t1; ++t) {
    const int x = t * p.TM;
    const long long nj = (long long)(p.n_tiles + 1) * p.Mr;
#pragma unroll
    for (int k = 0; k < BRACKET_RUN; ++k) {
      if (k >= n) break;
      const T lo = T(x - (b0 + k * p.R)), hi = T(x - (b0 + (k + 1) * p.R));
      if (d[k] <= lo && hi < d[k + 1])               // g_j <= x < g_{j+1}
        p.jlo[bchk((long long)t * p.Mr + i, nj, st)] = j0 + k;
      // bracket of the mirror family: g_j < x <= g_{j+1}
      if (p.sym && d[k] < lo && hi <= d[k + 1])
        p.jlo_neg[bchk((long long)(p.n_tiles - t) * p.Mr + i, nj, st)] = p.NRT - 1 - (j0 + k);
    }
  }
  if (st) atomicOr(p.status, st);
}

// Rows of landing pairs beyond the grid's y extent (65535) are taken in
// strides of gridDim.y.
template <typename T>
__global__ void __launch_bounds__(256) k_bracket(const BracketArgs<T> p) {
  const int rows = bracket_rows(p.NRT);
  for (int by = blockIdx.y; by < rows; by += gridDim.y)
    bracket_body<T, LD_PLAIN>(p, blockIdx.x, by, threadIdx.x);
}

// ----------------------------------------------------------------------------
// (c) + (d) interpolation fused with the modal sum
// ----------------------------------------------------------------------------
// A CTA owns one tile of TM = 32 PW consecutive grid points and one mode
// group; its RESUM_WARPS warps take the group's modes round-robin, each
// summing into registers (lane l holds points l PW .. l PW + PW - 1), and the CTA
// adds the warps' sums in a fixed order before writing one partial per
// (group, point).
//
// Per mode a warp
//  (1) stages the rays landing on the tile -- brackets jlo[t] .. jlo[t+1]
//      with stencil -1 / +2 -- in shared memory: landing X (grid units from
//      the tile start), phase, amplitude;
//  (2) one lane per interval [X_w, X_{w+1}): builds the 4-point Lagrange
//      polynomial through X_{w-1} .. X_{w+2} (Newton form, then monomial in
//      tau = x - X_w) for phase and amplitude into a shared-memory row;
//  (3) every lane evaluates its points: interval lookup (guessed from the
//      mean landing spacing, corrected by comparisons), two cubics, the
//      phase with its integer part exact (k kappa_n (z_m - z_lo) =
//      2 pi (n m mod N) / N), sincos, complex multiply-accumulate.
constexpr int RESUM_WARPS = 4;
constexpr int RESUM_CF = 12;      // values per interval row (X_w, X_{w+1}, two cubics, padding)

template <typename T>
__device__ __forceinline__ int resum_warp_bytes(int wcap) {
  return ((RESUM_CF + 3) * wcap * (int)sizeof(T) + 15) & ~15;
}

// Newton divided differences through (X1, X2, X0, X3), rewritten as a cubic
// in tau = x - X1:  b0 + b1 tau + b2 tau^2 + b3 tau^3.
template <typename T>
__device__ __forceinline__ void cubic_through(T f0, T f1, T f2, T f3, T r21, T r10, T r32, T r20,
                                              T r31, T r30, T h21, T h10, T& b0, T& b1, T& b2,
                                              T& b3) {
  const T d12 = (f2 - f1) * r21, d01 = (f1 - f0) * r10, d23 = (f3 - f2) * r32;
  const T d012 = (d12 - d01) * r20, d123 = (d23 - d12) * r31;
  const T d0123 = (d123 - d012) * r30;
  b0 = f1;
  b1 = d12 - h21 * (d012 + d0123 * h10);
  b2 = d012 + d0123 * (h10 - h21);
  b3 = d0123;
}

// Fixed-order sum of a block's four warps, written as its group's partial.
template <typename T, int PW, int BAR>
__device__ __forceinline__ void block_sum(const ResumArgs<T>& p, const T* accr, const T* acci,
                                          unsigned char* smem_raw, int group, int m0, int tid,
                                          int sub, unsigned st) {
  using V = typename C2<T>::type;
  const int lane = tid & 31, warp = tid >> 5, TM = p.TM;
  vb_sync<BAR>(sub);
  // per warp TM points as 32 runs of PW, each run padded to PW + 1 entries so
  // that the lanes' stores fall in different banks
  V* red = reinterpret_cast<V*>(smem_raw);
  const int TMP = 32 * (PW + 1);
#pragma unroll
  for (int q = 0; q < PW; ++q) {
    V v;
    v.x = accr[q];
    v.y = acci[q];
    red[warp * TMP + lane * (PW + 1) + q] = v;
  }
  vb_sync<BAR>(sub);
  V* out = p.part + bchk((long long)group * p.N + m0, (long long)p.n_groups * p.N - (TM - 1), st);
  if (st) atomicOr(p.status, st);
  for (int x = tid; x < TM; x += RESUM_WARPS * 32) {
    const int xs = (x / PW) * (PW + 1) + x % PW;
    V sum = red[xs];
#pragma unroll
    for (int w = 1; w < RESUM_WARPS; ++w) {
      const V v = red[w * TMP + xs];
      sum.x += v.x; sum.y += v.y;
    }
    out[x] = sum;
  }
}

// ---- FP32 ----
// Interval row: (X_w, X_w) | (b3, a3) | (b2, a2) | (b1, a1) | (b0, a0) | X_{w+1},
// the phase and amplitude cubics interleaved, so that three packed FMAs
// evaluate both and three 16-byte loads fetch a row.
struct Row32 {
  f2 X1, c3, c2, c1, c0;
  float X2;
};
__device__ __forceinline__ void load_row32(const float* p, Row32& r) {
  const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(p);
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p + 4);
  const float4 x = *reinterpret_cast<const float4*>(p + 8);
  r.X1.v = u.x; r.c3.v = u.y; r.c2.v = v.x; r.c1.v = v.y;
  r.c0 = mk2(x.x, x.y);
  r.X2 = x.z;
}

// One resummation block: blk its index in the launch, tid its thread index
// (0 .. 32 RESUM_WARPS - 1), smem_raw its shared memory (resum_smem_bytes),
// sub the virtual-block slot for the barrier (BAR).
template <int PW, int LD, int BAR>
__device__ __forceinline__ void resum_body(const ResumArgs<float>& p, int blk, int tid,
                                           unsigned char* smem_raw, int sub) {
  constexpr int LDC = LD == LD_NC ? LD_PLAIN : LD;   // mode coefficients
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int tt = blk % p.n_tiles_run;
  const int group = blk / p.n_tiles_run;
  const int half = p.n_tiles >> 1;
  const int tile = p.sym ? (tt < half ? half + tt : 0) : tt;
  const int wcap = p.wcap;
  const int TM = p.TM;
  unsigned char* wbase = smem_raw + (long long)warp * resum_warp_bytes<float>(wcap);
  float* s_cf = reinterpret_cast<float*>(wbase);               // [wcap][RESUM_CF], 16-byte aligned
  float2* s_pa = reinterpret_cast<float2*>(s_cf + RESUM_CF * wcap);   // phase, amplitude
  float* s_X = reinterpret_cast<float*>(s_pa + wcap);
  const int m0 = tile * TM;
  const int i0 = group * p.modes_per_group;
  const int i1 = min(p.M, i0 + p.modes_per_group);
  const float invN = scalbn(1.f, -(__ffs(p.N) - 1));           // exact
  const unsigned mask = (unsigned)p.N - 1u;
  const long long nrm = (long long)p.NRT * p.Mr;
  unsigned st = 0;

  float accr[PW], acci[PW];
#pragma unroll
  for (int q = 0; q < PW; ++q) { accr[q] = 0.f; acci[q] = 0.f; }

  // grounded: mode n < 0 is the mirror image of mode -n (column -n); its
  // ray j' is ray NRT - j' of mode -n, landing at N - g
  auto column = [&](int i, bool& mir) {
    const int n = i - p.n_max;
    mir = p.sym && n < 0;
    return p.sym ? (n < 0 ? -n : n) : i;
  };
  // One ray window per mode, its first 32 rays loaded one mode ahead.  r0: ray
  // of slot 0 (mirrored families run backwards), W: slots (0: skip the mode).
  float rd = 0.f, rph = 0.f, ra = 0.f;
  auto fetch = [&](int i, int r0, int w, float& d, float& ph, float& a) {
    bool mir;
    const int col = column(i, mir);
    const long long o = bchk((long long)(mir ? r0 - w : r0 + w) * p.Mr + col, nrm, st);
    d = ld<LD>(p.d + o);
    ph = ld<LD>(p.ph + o);
    a = ld<LD>(p.a + o);
  };

  // The warp's modes ib + RESUM_WARPS k, 32 at a time: lane k looks up the
  // brackets and the coefficient of mode k, which the loop takes by shuffles.
  for (int ib = i0 + warp; ib < i1; ib += 32 * RESUM_WARPS) {
    int h_r0 = 0, h_W = 0, h_base = 0;
    float h_mag = 0.f, h_arg = 0.f;
    {
      const int i = ib + RESUM_WARPS * lane;
      if (i < i1) {
        bool mir;
        const int col = column(i, mir);
        const int* jt = mir ? p.jlo_neg : p.jlo;
        const long long nj = (long long)(p.n_tiles + 1) * p.Mr;
        const int jl = ld<LD>(jt + bchk((long long)tile * p.Mr + col, nj, st));
        const int jh = ld<LD>(jt + bchk((long long)(tile + 1) * p.Mr + col, nj, st));
        // A bracket table left inconsistent by a failed screen (already flagged
        // by k_bracket) must not send the reads out of [0, NRT); a window wider
        // than the tile's capacity means rays compressed beyond it (flagged here).
        if (jl >= (mir ? 2 : 1) && jh >= jl && jh <= p.NRT - 3) {
          h_W = jh - jl + 4;
          if (h_W > wcap) { st |= ST_CAUSTIC; h_W = 0; }
        }
        const int jb = jl - 1;
        h_r0 = mir ? p.NRT - jb : jb;
        h_base = mir ? p.N - m0 - (p.NRT - jb - p.G) * p.R : (jb - p.G) * p.R - m0;
        // the mode coefficient in polar form (|c_n| scales the amplitudes,
        // arg c_n / 2 pi shifts the phases, in turns), formed by the DFT, so
        // that a term is two FMAs instead of a complex product
        const float2 cp = ld<LDC>(p.cpol + i);
        h_mag = cp.x;
        h_arg = cp.y;
      }
    }
    const int K = min(32, (i1 - ib + RESUM_WARPS - 1) / RESUM_WARPS);
    int r0 = __shfl_sync(ALL, h_r0, 0), W = __shfl_sync(ALL, h_W, 0);
    if (lane < W) fetch(ib, r0, lane, rd, rph, ra);
    for (int k = 0; k < K; ++k) {
      const int i = ib + RESUM_WARPS * k;
      const int Wc = W, rc = r0;
      const int base = __shfl_sync(ALL, h_base, k);
      const float cmag = __shfl_sync(ALL, h_mag, k);
      const float carg = __shfl_sync(ALL, h_arg, k);
      const float dsign = p.sym && i < p.n_max ? -1.f : 1.f;
      __syncwarp();
      if (lane < Wc) {
        s_X[lane] = fmaf(dsign, rd, (float)(base + lane * p.R));
        s_pa[lane] = make_float2(rph + carg, ra * cmag);
      }
      for (int w = lane + 32; w < Wc; w += 32) {   // beyond the prefetched rays
        float d, ph, a;
        fetch(i, rc, w, d, ph, a);
        s_X[w] = fmaf(dsign, d, (float)(base + w * p.R));
        s_pa[w] = make_float2(ph + carg, a * cmag);
      }
      // issue the next mode's window
      if (k + 1 < K) {
        r0 = __shfl_sync(ALL, h_r0, k + 1);
        W = __shfl_sync(ALL, h_W, k + 1);
        if (lane < W) fetch(i + RESUM_WARPS, r0, lane, rd, rph, ra);
      }
      if (Wc == 0) continue;
      __syncwarp();
      // Rows of the intervals 1 .. W - 3.  The last one's end is stored as
      // infinity: no lane steps past it.
      bool wide = true;
      for (int w = 1 + lane; w <= Wc - 3; w += 32) {
        const float X0 = s_X[w - 1], X1 = s_X[w], X2 = s_X[w + 1], X3 = s_X[w + 2];
        const float h21 = X2 - X1, h10 = X1 - X0;
        wide = wide && h21 >= 1.f;
        const f2 r21 = bc2(rcp_approx(h21)), r10 = bc2(rcp_approx(h10));
        const f2 r32 = bc2(rcp_approx(X3 - X2)), r20 = bc2(rcp_approx(X2 - X0));
        const f2 r31 = bc2(rcp_approx(X3 - X1)), r30 = bc2(rcp_approx(X3 - X0));
        const auto val = [&](int k) {
          f2 v;
          v.v = *reinterpret_cast<const unsigned long long*>(s_pa + w + k);
          return v;
        };
        // Newton divided differences through (X1, X2, X0, X3) of phase and
        // amplitude together, rewritten as cubics in tau = x - X1
        const f2 f0 = val(-1), f1 = val(0), fa = val(1), f3 = val(2);
        const f2 d12 = mul2(sub2(fa, f1), r21), d01 = mul2(sub2(f1, f0), r10);
        const f2 d23 = mul2(sub2(f3, fa), r32);
        const f2 d012 = mul2(sub2(d12, d01), r20), d123 = mul2(sub2(d23, d12), r31);
        const f2 c3 = mul2(sub2(d123, d012), r30);
        const f2 c1 = fma2(bc2(-h21), fma2(c3, bc2(h10), d012), d12);
        const f2 c2 = fma2(c3, bc2(h10 - h21), d012);
        float b0, a0;
        sp2(f1, b0, a0);
        b0 = minus_rint(b0);                       // whole turns do not matter
        float* row = s_cf + RESUM_CF * w;
        *reinterpret_cast<ulonglong2*>(row) = make_ulonglong2(bc2(X1).v, c3.v);
        *reinterpret_cast<ulonglong2*>(row + 4) = make_ulonglong2(c2.v, c1.v);
        *reinterpret_cast<float4*>(row + 8) =
            make_float4(b0, a0, w == Wc - 3 ? __int_as_float(0x7f800000) : X2, 0.f);
      }
      wide = __all_sync(ALL, wide);
      __syncwarp();
      // Lane l sums the PW consecutive points x = l PW + q.  The interval of its
      // first point (X_w <= x < X_{w+1}, w in [1, W-3]) is guessed from the mean
      // landing spacing and corrected by comparisons; later points only step
      // forward, loading the next row when they pass X_{w+1}: at most one row
      // per point where every interval is at least a grid step long.
      const int x0 = lane * PW;
      const float xv0 = (float)x0;
      int w;
      {
        const float xf = s_X[1];
        const float inv_sp = (float)(Wc - 3) * rcp_approx(s_X[Wc - 2] - xf);
        w = 1 + ifloor_small((xv0 - xf) * inv_sp);
        w = min(max(w, 1), Wc - 3);
        while (w > 1 && s_X[w] > xv0) --w;
        while (w < Wc - 3 && s_X[w + 1] <= xv0) ++w;
      }
      const float* row = s_cf + RESUM_CF * w;
      Row32 r;
      load_row32(row, r);
      // The exact integer phase n m / N mod 1 of the run's middle point,
      // moved into [-1/2, 1/2); the run's points differ from it by
      // (q - PW/2) n / N, exact in FP32 (multiples of 1/N below 2^(24 - log2 N)),
      // so each point's turn count costs one FMA.  The phase cubic is reduced
      // to (-1/2, 1/2] at its interval start, so the argument of the sine
      // stays within a few turns.
      const unsigned nn = (unsigned)(i - p.n_max);
      const unsigned nmc = (nn * (unsigned)(m0 + x0 + PW / 2)) & mask;
      float bc = exact_u2f(nmc) * invN;
      bc = bc >= 0.5f ? bc - 1.f : bc;
      const float nN = (float)(int)nn * invN;
      const f2 one = bc2(1.f);
      f2 xv = bc2(xv0);                     // the point, twice; exact
      const auto term = [&](int q) {
        const f2 tau = sub2(xv, r.X1);
        float phv, av;
        sp2(fma2(fma2(fma2(r.c3, tau, r.c2), tau, r.c1), tau, r.c0), phv, av);
        const float t = fmaf((float)(q - PW / 2), nN, bc) + phv;
        float sn, cs;
        sincos_turns(t, &sn, &cs);
        accr[q] = fmaf(av, cs, accr[q]);
        acci[q] = fmaf(av, sn, acci[q]);
      };
      const auto past = [&]() {
        float x, y;
        sp2(xv, x, y);
        return r.X2 <= x;
      };
      term(0);
      if (wide) {
#pragma unroll
        for (int q = 1; q < PW; ++q) {
          xv = add2(xv, one);
          if (past()) {
            row += RESUM_CF;
            load_row32(row, r);
          }
          term(q);
        }
      } else {
#pragma unroll
        for (int q = 1; q < PW; ++q) {
          xv = add2(xv, one);
          while (past()) {
            row += RESUM_CF;
            load_row32(row, r);
          }
          term(q);
        }
      }
    }
  }
  block_sum<float, PW, BAR>(p, accr, acci, smem_raw, group, m0, tid, sub, st);
}

// ---- FP64 ----
// sin / cos of 2 pi (a + b), a + b = k / TRIG_N + r with |r| <= 1 / (2 TRIG_N):
// the table's entry exp(2 pi i k / TRIG_N) rotated by the angle 2 pi r <= pi / 1024,
// whose sine and cosine - 1 need two and three Taylor terms (the next ones are
// below 2e-18).  a is a multiple of a small fraction of a turn (n m / N), so a - k /
// TRIG_N is exact and r takes no rounding of the size of a + b, only b's own.  14 FP64
// operations, absolute error about one unit in the last place of 1, small sines to
// a few units of their own; any |a + b| < 2^41.
__device__ __forceinline__ void sincos_table(const double2* trig, double a, double b, double* s,
                                             double* c) {
  const double magic = 6755399441055744.0;   // 1.5 * 2^52: rounds to an integer
  const double v = fma(a + b, (double)TRIG_N, magic);
  const double r = fma(v - magic, -1.0 / TRIG_N, a) + b;
  const double2 e = __ldg(trig + (__double2loint(v) & (TRIG_N - 1)));
  const double r2 = r * r;
  const double sr = r * fma(r2, fma(r2, 81.60524927607503, -41.34170224039975), 6.283185307179586);
  const double cr = r2 * fma(r2, 64.93939402266828, -19.73920880217872);   // cos - 1
  *c = fma(e.x, cr, fma(-e.y, sr, e.x));
  *s = fma(e.y, cr, fma(e.x, sr, e.y));
}

// Interval row: X_w, X_{w+1}, phase b0..b3, amplitude a0..a3.
struct Row64 {
  double X1, X2, b0, b1, b2, b3, a0, a1, a2, a3;
};
__device__ __forceinline__ Row64 load_row64(const double* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 u = q[0], v = q[1], w = q[2], x = q[3], y = q[4];
  return Row64{u.x, u.y, v.x, v.y, w.x, w.y, x.x, x.y, y.x, y.y};
}

// As the FP32 block; bound by the FP64 pipe, so reciprocals take 3 FP64
// operations (rcp64), a term 25, and a run's next interval is found by integer
// comparisons.
template <int PW, int LD, int BAR>
__device__ __forceinline__ void resum_body(const ResumArgs<double>& p, int blk, int tid,
                                           unsigned char* smem_raw, int sub) {
  constexpr int LDC = LD == LD_NC ? LD_PLAIN : LD;   // mode coefficients
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int tt = blk % p.n_tiles_run;
  const int group = blk / p.n_tiles_run;
  const int half = p.n_tiles >> 1;
  const int tile = p.sym ? (tt < half ? half + tt : 0) : tt;
  const int wcap = p.wcap;
  const int TM = p.TM;
  unsigned char* wbase = smem_raw + (long long)warp * resum_warp_bytes<double>(wcap);
  double* s_cf = reinterpret_cast<double*>(wbase);            // [wcap][RESUM_CF], 16-byte aligned
  double2* s_pa = reinterpret_cast<double2*>(s_cf + RESUM_CF * wcap);   // phase, amplitude
  double* s_X = reinterpret_cast<double*>(s_pa + wcap);
  const int m0 = tile * TM;
  const int i0 = group * p.modes_per_group;
  const int i1 = min(p.M, i0 + p.modes_per_group);
  const double invN = scalbn(1.0, -(__ffs(p.N) - 1));         // exact
  const unsigned mask = (unsigned)p.N - 1u;
  const long long nrm = (long long)p.NRT * p.Mr;
  const int x0 = lane * PW;
  const double xv0 = (double)x0;
  unsigned st = 0;

  double accr[PW], acci[PW];
#pragma unroll
  for (int q = 0; q < PW; ++q) { accr[q] = 0.0; acci[q] = 0.0; }

  auto column = [&](int i, bool& mir) {
    const int n = i - p.n_max;
    mir = p.sym && n < 0;
    return p.sym ? (n < 0 ? -n : n) : i;
  };
  double rd = 0.0, rph = 0.0, ra = 0.0;   // the next mode's first 32 rays
  auto fetch = [&](int i, int r0, int w, double& d, double& ph, double& a) {
    bool mir;
    const int col = column(i, mir);
    const long long o = bchk((long long)(mir ? r0 - w : r0 + w) * p.Mr + col, nrm, st);
    d = ld<LD>(p.d + o);
    ph = ld<LD>(p.ph + o);
    a = ld<LD>(p.a + o);
  };

  for (int ib = i0 + warp; ib < i1; ib += 32 * RESUM_WARPS) {
    // lane k: the brackets and coefficient of mode ib + RESUM_WARPS k
    int h_r0 = 0, h_W = 0, h_base = 0;
    double h_mag = 0.0, h_arg = 0.0;
    {
      const int i = ib + RESUM_WARPS * lane;
      if (i < i1) {
        bool mir;
        const int col = column(i, mir);
        const int* jt = mir ? p.jlo_neg : p.jlo;
        const long long nj = (long long)(p.n_tiles + 1) * p.Mr;
        const int jl = ld<LD>(jt + bchk((long long)tile * p.Mr + col, nj, st));
        const int jh = ld<LD>(jt + bchk((long long)(tile + 1) * p.Mr + col, nj, st));
        // (inconsistent or too wide windows: as in the FP32 block)
        if (jl >= (mir ? 2 : 1) && jh >= jl && jh <= p.NRT - 3) {
          h_W = jh - jl + 4;
          if (h_W > wcap) { st |= ST_CAUSTIC; h_W = 0; }
        }
        const int jb = jl - 1;
        h_r0 = mir ? p.NRT - jb : jb;
        h_base = mir ? p.N - m0 - (p.NRT - jb - p.G) * p.R : (jb - p.G) * p.R - m0;
        const double2 cp = ld<LDC>(p.cpol + i);
        h_mag = cp.x;
        h_arg = cp.y;
      }
    }
    const int K = min(32, (i1 - ib + RESUM_WARPS - 1) / RESUM_WARPS);
    int r0 = __shfl_sync(ALL, h_r0, 0), W = __shfl_sync(ALL, h_W, 0);
    if (lane < W) fetch(ib, r0, lane, rd, rph, ra);
    for (int k = 0; k < K; ++k) {
      const int i = ib + RESUM_WARPS * k;
      const int Wc = W, rc = r0;
      const int base = __shfl_sync(ALL, h_base, k);
      const double cmag = __shfl_sync(ALL, h_mag, k);
      const double carg = __shfl_sync(ALL, h_arg, k);
      const double dsign = p.sym && i < p.n_max ? -1.0 : 1.0;
      __syncwarp();
      if (lane < Wc) {
        s_X[lane] = fma(dsign, rd, (double)(base + lane * p.R));
        s_pa[lane] = make_double2(rph + carg, ra * cmag);
      }
      for (int w = lane + 32; w < Wc; w += 32) {   // beyond the prefetched rays
        double d, ph, a;
        fetch(i, rc, w, d, ph, a);
        s_X[w] = fma(dsign, d, (double)(base + w * p.R));
        s_pa[w] = make_double2(ph + carg, a * cmag);
      }
      if (k + 1 < K) {   // issue the next mode's window
        r0 = __shfl_sync(ALL, h_r0, k + 1);
        W = __shfl_sync(ALL, h_W, k + 1);
        if (lane < W) fetch(i + RESUM_WARPS, r0, lane, rd, rph, ra);
      }
      if (Wc == 0) continue;
      __syncwarp();
      bool wide = true;
      for (int w = 1 + lane; w <= Wc - 3; w += 32) {
        const double X0 = s_X[w - 1], X1 = s_X[w], X2 = s_X[w + 1], X3 = s_X[w + 2];
        const double2 f0 = s_pa[w - 1], f1 = s_pa[w], f2 = s_pa[w + 1], f3 = s_pa[w + 2];
        const double h21 = X2 - X1, h10 = X1 - X0;
        wide = wide && h21 >= 1.0;
        const double r21 = rcp64(h21), r10 = rcp64(h10), r32 = rcp64(X3 - X2);
        const double r20 = rcp64(X2 - X0), r31 = rcp64(X3 - X1), r30 = rcp64(X3 - X0);
        double b0, b1, b2, b3, a0, a1, a2, a3;
        cubic_through(f0.x, f1.x, f2.x, f3.x, r21, r10, r32, r20, r31, r30, h21, h10, b0, b1, b2,
                      b3);
        cubic_through(f0.y, f1.y, f2.y, f3.y, r21, r10, r32, r20, r31, r30, h21, h10, a0, a1, a2,
                      a3);
        double2* row = reinterpret_cast<double2*>(s_cf + RESUM_CF * w);
        // the last row's end is stored as infinity: no lane steps past it
        row[0] = make_double2(X1, w == Wc - 3 ? __longlong_as_double(0x7ff0000000000000ll) : X2);
        row[1] = make_double2(b0, b1);
        row[2] = make_double2(b2, b3);
        row[3] = make_double2(a0, a1);
        row[4] = make_double2(a2, a3);
      }
      wide = __all_sync(ALL, wide);
      __syncwarp();
      // interval of the lane's first point, as in the FP32 block
      int w;
      {
        const float xf = (float)s_X[1];
        const float inv_sp = (float)(Wc - 3) / ((float)s_X[Wc - 2] - xf);
        w = 1 + ifloor_small(((float)x0 - xf) * inv_sp);
        w = min(max(w, 1), Wc - 3);
        while (w > 1 && s_X[w] > xv0) --w;
        while (w < Wc - 3 && s_X[w + 1] <= xv0) ++w;
      }
      const double* row = s_cf + RESUM_CF * w;
      Row64 r;
      double t0;   // the run's first point in the row's tau
      int q_end;   // first point of the run past the row's interval
      const auto enter = [&]() {
        r = load_row64(row);
        t0 = xv0 - r.X1;
        const double d = r.X2 - xv0;          // exact where it decides
        q_end = d < (double)PW ? __double2int_ru(d) : PW;
      };
      enter();
      // exact integer phase of the run's middle point and n / N per point from
      // it, as in the FP32 block (exact: multiples of 1/N)
      const unsigned nn = (unsigned)(i - p.n_max);
      const double bc = (double)((nn * (unsigned)(m0 + x0 + PW / 2)) & mask) * invN;
      const double nN = (double)(int)nn * invN;
      const auto term = [&](int q) {
        const double tau = t0 + (double)q;
        const double phv = ((r.b3 * tau + r.b2) * tau + r.b1) * tau + r.b0;
        const double av = ((r.a3 * tau + r.a2) * tau + r.a1) * tau + r.a0;
        double sn, cs;
        sincos_table(p.trig, fma((double)(q - PW / 2), nN, bc), phv, &sn, &cs);
        accr[q] = fma(av, cs, accr[q]);
        acci[q] = fma(av, sn, acci[q]);
      };
      term(0);
      if (wide) {
#pragma unroll
        for (int q = 1; q < PW; ++q) {
          if (q >= q_end) {
            row += RESUM_CF;
            enter();
          }
          term(q);
        }
      } else {
#pragma unroll
        for (int q = 1; q < PW; ++q) {
          while (q >= q_end) {
            row += RESUM_CF;
            enter();
          }
          term(q);
        }
      }
    }
  }
  block_sum<double, PW, BAR>(p, accr, acci, smem_raw, group, m0, tid, sub, st);
}

// FP32, bound by instruction issue: 390 warp instructions per (mode, 256-point
// tile), 15 per point and lane and ~150 for the window, the rows and the search
// (477 with scalar cubics, per-mode bracket lookups and library divisions).
// 16384-point duct (977 modes x 16640 points) 34 us per sum against 41,
// 131072-point duct (1395 modes, R = 64) 221 against 372.  7 CTAs per SM (72
// registers: keeps the one-mode-ahead window), 5 for runs of 16 points (213 us,
// 230 at 72 registers, in an earlier build).  FP64, bound by its pipe: 1.04 ms on the 16384-point
// duct with 29 mode groups (1.78 with sincospi, library divisions and a complex
// coefficient per term; 25 FP64 operations per term instead of ~46).
template <typename T, int PW>
__global__ void __launch_bounds__(RESUM_WARPS * 32, sizeof(T) == 4 ? (PW < 16 ? 7 : 5) : 1)
    k_resum(const ResumArgs<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  resum_body<PW, LD_NC, 0>(p, blockIdx.x, threadIdx.x, smem_raw, 0);
}

// A point's partials are added in PART_SUMS interleaved sums (groups q, q +
// PART_SUMS, ... in order), then these in order, so that in pass 1 of the DFT several
// threads can share a point's loads.
constexpr int PART_SUMS = 4;

// interleaved sum q; loads issued 8 at a time
template <typename V, int LD>
__device__ __forceinline__ V parts_sum(const V* __restrict__ part, int N, int n_part, int q) {
  V s;
  s.x = s.y = 0;
  int g = q;
  for (; g + 7 * PART_SUMS < n_part; g += 8 * PART_SUMS) {
    V v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = ld<LD>(part + (long long)(g + k * PART_SUMS) * N);
#pragma unroll
    for (int k = 0; k < 8; ++k) { s.x += v[k].x; s.y += v[k].y; }
  }
#pragma unroll 4
  for (; g < n_part; g += PART_SUMS) {
    const V v = ld<LD>(part + (long long)g * N);
    s.x += v.x; s.y += v.y;
  }
  return s;
}

template <typename V>
__device__ __forceinline__ V parts_combine(V (&v)[PART_SUMS]) {
#pragma unroll
  for (int q = 1; q < PART_SUMS; ++q) { v[0].x += v[q].x; v[0].y += v[q].y; }
  return v[0];
}

// the four sums of one thread side by side
template <typename V, int LD>
__device__ __forceinline__ V parts_total(const V* __restrict__ part, int N, int n_part) {
  V a[PART_SUMS];
#pragma unroll
  for (int q = 0; q < PART_SUMS; ++q) a[q].x = a[q].y = 0;
  int g = 0;
  for (; g + 2 * PART_SUMS <= n_part; g += 2 * PART_SUMS) {
    V v[2 * PART_SUMS];
#pragma unroll
    for (int k = 0; k < 2 * PART_SUMS; ++k) v[k] = ld<LD>(part + (long long)(g + k) * N);
#pragma unroll
    for (int k = 0; k < 2 * PART_SUMS; ++k) {
      a[k % PART_SUMS].x += v[k].x;
      a[k % PART_SUMS].y += v[k].y;
    }
  }
#pragma unroll
  for (int k = 0; k < 2 * PART_SUMS; ++k) {
    if (g + k < n_part) {
      const V v = ld<LD>(part + (long long)(g + k) * N);
      a[k % PART_SUMS].x += v.x;
      a[k % PART_SUMS].y += v.y;
    }
  }
  return parts_combine(a);
}

// ----------------------------------------------------------------------------
// field bookkeeping: partial sums, absorber, reflection, I/O
// ----------------------------------------------------------------------------
template <typename T, int LD>
__device__ __forceinline__ void reduce_body(const ReduceArgs<T>& p, int k) {
  using V = typename C2<T>::type;
  auto sum_at = [&](int mm) {
    V s = parts_total<V, LD>(p.part + mm, p.N, p.n_part);
    if (p.W) { const T w = p.W[mm]; s.x *= w; s.y *= w; }
    return s;
  };
  const T sg = T(p.mirror);
  if (p.sym) {
    // partials hold the physical half m in [N/2, N) and m = 0; the other
    // half is its reflection
    if (k > p.N / 2) return;
    const int m = k < p.N / 2 ? p.N / 2 + k : 0;
    const V a = sum_at(m);
    if (m == 0 || m == p.N / 2) {
      V v;
      v.x = T(0.5) * (a.x + sg * a.x); v.y = T(0.5) * (a.y + sg * a.y);
      p.u[m] = v;
    } else {
      V b;
      b.x = sg * a.x; b.y = sg * a.y;
      p.u[m] = a;
      p.u[p.N - m] = b;
    }
    return;
  }
  const int m = k;
  if (!p.mirror) {
    if (m < p.N) p.u[m] = sum_at(m);
    return;
  }
  if (m > p.N / 2) return;
  const int mm = (p.N - m) & (p.N - 1);
  const V a = sum_at(m);
  const V b = (mm == m) ? a : sum_at(mm);
  V ua, ub;
  ua.x = T(0.5) * (a.x + sg * b.x); ua.y = T(0.5) * (a.y + sg * b.y);
  ub.x = T(0.5) * (b.x + sg * a.x); ub.y = T(0.5) * (b.y + sg * a.y);
  p.u[m] = ua;
  p.u[mm] = ub;
}

template <typename T>
__global__ void k_reduce(const ReduceArgs<T> p) {
  reduce_body<T, LD_PLAIN>(p, blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T>
__device__ __forceinline__ void init_body(const double* __restrict__ u0, int n_z, int N,
                                          int mirror, typename C2<T>::type* __restrict__ u,
                                          int m) {
  if (m >= N) return;
  typename C2<T>::type v;
  if (!mirror) {
    v.x = T(u0[2 * m]); v.y = T(u0[2 * m + 1]);
  } else if (m >= n_z) {
    v.x = T(u0[2 * (m - n_z)]); v.y = T(u0[2 * (m - n_z) + 1]);
  } else if (m > 0) {
    v.x = T(mirror) * T(u0[2 * (n_z - m)]); v.y = T(mirror) * T(u0[2 * (n_z - m) + 1]);
  } else {
    v.x = T(0); v.y = T(0);
  }
  u[m] = v;
}

template <typename T>
__global__ void k_init(const double* __restrict__ u0, int n_z, int N, int mirror,
                       typename C2<T>::type* __restrict__ u) {
  init_body<T>(u0, n_z, N, mirror, u, blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T, int LD>
__device__ __forceinline__ void output_body(const typename C2<T>::type* __restrict__ u,
                                            int offset, int n, double* __restrict__ out, int m) {
  if (m >= n) return;
  const typename C2<T>::type v = ld<LD>(u + offset + m);
  out[2 * m] = double(v.x);
  out[2 * m + 1] = double(v.y);
}

template <typename T>
__global__ void k_output(const typename C2<T>::type* __restrict__ u, int offset, int n,
                         double* __restrict__ out) {
  output_body<T, LD_PLAIN>(u, offset, n, out, blockIdx.x * blockDim.x + threadIdx.x);
}

// ----------------------------------------------------------------------------
// (a) pruned DFT: N = N1 N2, n = n1 N2 + n2, k = k1 + N1 k2
//   X[k1 + N1 k2] = sum_n2 w_{N2}^{n2 k2} w_N^{n2 k1} sum_n1 x[n1 N2 + n2] w_{N1}^{n1 k1}
// pass 1 (N1 > 1): direct length-N1 DFTs down the columns n2, then the twiddle
// w_N^{n2 k1};
// pass 2: one CTA per kept bin n (|n| <= n_max; n >= 0 for grounded fields),
// a direct length-N2 sum along its row k1, written as c_n.
// ----------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ typename C2<T>::type cmul(typename C2<T>::type a,
                                                     typename C2<T>::type b) {
  typename C2<T>::type r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}

// (|v|, arg(v) / 2 pi) of a complex value, the angle in turns in [-1/2, 1/2].
// FP32: |v| makes up for what sincos_turns falls short of (its square by 1.47e-7),
// which a field would lose at each screen whatever its shape; the root is the rounded
// one, since the approximate one loses 1.5e-8 more.
template <typename T>
__device__ __forceinline__ typename C2<T>::type polar_turns(typename C2<T>::type v) {
  typename C2<T>::type r;
  if constexpr (sizeof(T) == 8) r.x = hypot(v.x, v.y);
  else {
    const float q = fmaf(v.x, v.x, v.y * v.y);
    r.x = __fsqrt_rn(fmaf(q, 1.47e-7f, q));
  }
  r.y = atan2(v.y, v.x) * T(0.15915494309189533577);
  return r;
}

// Field value at grid point m formed from the resummation partials: the sum
// over mode groups times the absorber, with the reflection of grounded plans
// (same arithmetic as k_reduce).
template <typename T>
__device__ __forceinline__ int parts_source(const FftArgs<T>& p, int m) {
  return (p.sym && m > 0 && m < (p.N >> 1)) ? p.N - m : m;
}

template <typename T>
__device__ __forceinline__ typename C2<T>::type parts_finish(const FftArgs<T>& p, int m, int src,
                                                             typename C2<T>::type s) {
  const int half = p.N >> 1;
  if (p.W) { const T w = p.W[src]; s.x *= w; s.y *= w; }
  if (p.sym) {
    const T sg = T(p.mirror);
    if (m == 0 || m == half) {
      s.x = T(0.5) * (s.x + sg * s.x); s.y = T(0.5) * (s.y + sg * s.y);
    } else if (m < half) {
      s.x = sg * s.x; s.y = sg * s.y;
    }
  }
  return s;
}

// acc + a w: one rounding per product pair and sum in FP32 (as cmul and an
// addition), four FMAs in FP64, where issue bounds the sums
template <typename T>
__device__ __forceinline__ void cmac(typename C2<T>::type& s, typename C2<T>::type a,
                                     typename C2<T>::type w) {
  if constexpr (sizeof(T) == 8) {
    s.x = fma(a.x, w.x, fma(-a.y, w.y, s.x));
    s.y = fma(a.x, w.y, fma(a.y, w.x, s.y));
  } else {
    const typename C2<T>::type t = cmul<T>(a, w);
    s.x += t.x; s.y += t.y;
  }
}

// pass 1: a CTA takes COLS consecutive columns n2 (all N1 rows, one tile in shared
// memory) and forms Y[k1][n2] = w_N^{n2 k1} sum_n1 x[n1 N2 + n2] w_{N1}^{n1 k1} for
// all k1.  Two threads form rows k1 and k1 + N1 / 2 of a column, the sum and the
// difference of their sums over even and odd n1.  Latency bounds it on the plans'
// chain: few columns per CTA (fft1_cols), a point's partials summed by several threads.
// Both passes, 4096 points and 37 groups (lens): 12.1 -> 10.1 us; 8192 points (FP32
// duct) 12.0 -> 10.0; FP64, 32768 points: 33.3 -> 27.9 (with one thread per point's
// partials, 8 columns and every row formed alone; ~2 us are events).
// One block of 256 threads (blk its index, smem_raw its shared memory).
template <typename T, int LD, int COLS>
__device__ __forceinline__ void fft1_body(const FftArgs<T>& p, int blk, int tid,
                                          unsigned char* smem_raw) {
  using V = typename C2<T>::type;
  const int E = p.N1 * COLS;                         // a power of two
  V* tile = reinterpret_cast<V*>(smem_raw);          // [N1][COLS]
  V* w1 = tile + E;                                  // [N1] w_{N1}^k
  const int c0 = blk * COLS;
  for (int k = tid; k < p.N1; k += FFT1_THREADS) w1[k] = p.tw[(long long)k * p.N2 << p.tw_shift];
  if (p.part) {
    V* sums = w1 + p.N1;                             // [PART_SUMS][E], E < FFT1_THREADS
    const int m0 = c0 + (tid & (COLS - 1));
    if (E < FFT1_THREADS) {
      for (int i = tid; i < PART_SUMS * E; i += FFT1_THREADS) {
        const int src = parts_source(p, ((i & (E - 1)) / COLS) * p.N2 + m0);
        sums[i] = parts_sum<V, LD>(p.part + src, p.N, p.n_part, i / E);
      }
      __syncthreads();
    }
    for (int e = tid; e < E; e += FFT1_THREADS) {
      const int m = e / COLS * p.N2 + m0, src = parts_source(p, m);
      V s;
      if (E < FFT1_THREADS) {
        V v[PART_SUMS];
#pragma unroll
        for (int q = 0; q < PART_SUMS; ++q) v[q] = sums[q * E + e];
        s = parts_combine(v);
      } else {
        s = parts_total<V, LD>(p.part + src, p.N, p.n_part);
      }
      tile[e] = parts_finish(p, m, src, s);
    }
  } else {
    for (int e = tid; e < E; e += FFT1_THREADS) tile[e] = ld<LD>(p.u + e / COLS * p.N2 + c0 + e % COLS);
  }
  __syncthreads();
  for (int e0 = 0; e0 < E; e0 += FFT1_THREADS) {
    const int e = e0 + tid;                          // (k1, h, c); idle threads stay for the shuffle
    const int c = e % COLS, h = e / COLS & 1, k1 = e / (2 * COLS);
    const int row = k1 + h * (p.N1 / 2), n2 = c0 + c;
    V s;
    s.x = s.y = T(0);
    V w2 = s;
    if (e < E) {
      w2 = p.tw[(long long)n2 * row << p.tw_shift];
#pragma unroll 4
      for (int n1 = h; n1 < p.N1; n1 += 2)
        cmac<T>(s, tile[n1 * COLS + c], w1[(n1 * k1) & (p.N1 - 1)]);
    }
    V o;
    o.x = __shfl_xor_sync(0xffffffffu, s.x, COLS);
    o.y = __shfl_xor_sync(0xffffffffu, s.y, COLS);
    if (h) { s.x = o.x - s.x; s.y = o.y - s.y; }
    else { s.x += o.x; s.y += o.y; }
    if (e < E) p.Y[(long long)row * p.N2 + n2] = cmul<T>(s, w2);
  }
}

template <typename T, int COLS>
__global__ void __launch_bounds__(FFT1_THREADS) k_fft1(const FftArgs<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fft1_body<T, LD_PLAIN, COLS>(p, blockIdx.x, threadIdx.x, smem_raw);
}

// Polar form of c_i f_i (mode coefficients of the planes between screens, one per
// blockIdx.y).
template <typename T>
__global__ void k_cscale(const typename C2<T>::type* __restrict__ c,
                         const typename C2<T>::type* __restrict__ f,
                         typename C2<T>::type* __restrict__ pol, int M) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const long long o = (long long)blockIdx.y * M + i;
  pol[o] = polar_turns<T>(cmul<T>(c[i], f[o]));
}

// w_{N2}^{idx} from the table of w_N (w_{N2} = w_N^{N1}).
template <typename V>
__device__ __forceinline__ V twiddle2(const V* tw, unsigned idx, int shift, int N1) {
  return tw[(long long)idx * N1 << shift];
}

// pass 2: one CTA (4 warps) per kept mode n:
// X[k1 + N1 k2] = sum_n2 Y[k1][n2] w_{N2}^{n2 k2} (direct, pruned: only the
// 2 n_max + 1 kept bins are formed); c_n = X / N times the range-phase carry.
constexpr int FFT2_THREADS = 128;

// One pass-2 block of FFT2_THREADS threads: blk its index (one kept mode),
// wsum FFT2_THREADS / 32 values of shared memory, sub the barrier slot (BAR).
template <typename T, int LD, int BAR>
__device__ __forceinline__ void fft2_body(const FftArgs<T>& p, int blk, int tid,
                                          typename C2<T>::type* wsum, int sub) {
  using V = typename C2<T>::type;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  // grounded fields are even / odd, so c_{-n} = +-c_n: only n >= 0 is formed
  const int i = blk + (p.mirror ? p.n_max : 0);
  const int n = i - p.n_max;
  const int b = n >= 0 ? n : n + p.N;
  const int k1 = b & (p.N1 - 1);
  const int k2 = b / p.N1;
  const V* row = (p.N1 > 1 ? p.Y : p.u) + (long long)k1 * p.N2;
  const V ph = p.ephi[i];   // early: it is the last the chain needs
  V acc;
  acc.x = T(0); acc.y = T(0);
  // row entries and twiddles loaded 8 iterations at a time, summed in order
  constexpr int B = 8;
  int n2 = tid;
  for (; n2 + (B - 1) * FFT2_THREADS < p.N2; n2 += B * FFT2_THREADS) {
    V rv[B], tv[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const int m = n2 + k * FFT2_THREADS;
      const unsigned e = (unsigned)(((long long)m * k2) & (p.N2 - 1));
      rv[k] = ld<LD>(row + m);
      tv[k] = twiddle2(p.tw, e, p.tw_shift, p.N1);
    }
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const V t = cmul<T>(rv[k], tv[k]);
      acc.x += t.x; acc.y += t.y;
    }
  }
  for (; n2 < p.N2; n2 += FFT2_THREADS) {
    const unsigned e = (unsigned)(((long long)n2 * k2) & (p.N2 - 1));
    const V t = cmul<T>(ld<LD>(row + n2), twiddle2(p.tw, e, p.tw_shift, p.N1));
    acc.x += t.x; acc.y += t.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
  }
  if (lane == 0) wsum[warp] = acc;
  vb_sync<BAR>(sub);
  if (tid == 0) {
    V tot = wsum[0];
#pragma unroll
    for (int w = 1; w < FFT2_THREADS / 32; ++w) { tot.x += wsum[w].x; tot.y += wsum[w].y; }
    tot.x *= p.inv_N; tot.y *= p.inv_N;
    const V cv = cmul<T>(tot, ph);
    p.c[i] = cv;
    if (p.mirror && n > 0) {
      V cm;
      cm.x = T(p.mirror) * cv.x; cm.y = T(p.mirror) * cv.y;
      p.c[2 * p.n_max - i] = cm;
    }
    if (p.cpol) {   // |c_n| and arg(c_n) / 2 pi (turns, in (-1/2, 1/2])
      V pol = polar_turns<T>(cv);
      p.cpol[i] = pol;
      if (p.mirror && n > 0) {
        if (p.mirror < 0) pol.y = pol.y > T(0) ? pol.y - T(0.5) : pol.y + T(0.5);
        p.cpol[2 * p.n_max - i] = pol;
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(FFT2_THREADS) k_fft2(const FftArgs<T> p) {
  __shared__ typename C2<T>::type wsum[FFT2_THREADS / 32];
  fft2_body<T, LD_PLAIN, 0>(p, blockIdx.x, threadIdx.x, wsum, 0);
}

}  // namespace swkb
