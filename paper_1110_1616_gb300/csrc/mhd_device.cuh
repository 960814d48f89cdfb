// Device-side per-element formulas of the ideal-MHD advance, templated on the
// arithmetic type T (double for the FP64 path, float for the FP32 stencil of
// the mixed path). The evaluation order of every expression is the one the
// scheme fixes, so that the FP64 build without FMA contraction reproduces a
// plain FP64 implementation bit for bit.
//
// The paper names the hyperbolic advance of each grid (Abstract, Sec. 1) but not
// the scheme; the choices are:
//  * MUSCL-Hancock, unsplit, with the half-step predictor written in primitive
//    variables (the v div B term of the induction equation dropped).
//  * minmod(a, b): 0 unless a and b have the same strict sign, else the one of
//    smaller magnitude (a on a tie); a = backward, b = forward difference. The
//    slope of the normal B in its own direction is the face difference.
//  * HLLD (Miyoshi & Kusano 2005) with S_L = min(uL,uR) - max(cfL,cfR),
//    S_R = max(uL,uR) + max(cfL,cfR); degenerate star states when
//    |e| <= eps (|rho (S-u)(S-S_M)| + Bn^2); double-star states skipped when
//    Bn^2 <= eps p_T*; eps = 1e-12 in FP64 and 1e-6 in FP32; the normal field
//    is the mean of the two predicted face states' normal B.
//  * Edge EMFs: Gardiner & Stone upwinded average with the cell-centre
//    reference -(v x B) at the half step, upwinded by the face mass flux (the
//    mean of both sides when it is exactly 0).
#pragma once
#include <cuda_runtime.h>
#include "fp_bits.cuh"

namespace amrdev {

enum { RHO = 0, MX = 1, MY = 2, MZ = 3, EN = 4, BX = 5, BY = 6, BZ = 7 };

template <class T> struct Eps;
template <> struct Eps<double> { static __device__ __forceinline__ double v() { return 1e-12; } };
template <> struct Eps<float> { static __device__ __forceinline__ float v() { return 1e-6f; } };

__device__ __forceinline__ double dsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float dsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double dabs(double x) { return fabs(x); }
__device__ __forceinline__ float dabs(float x) { return fabsf(x); }

template <class T> __device__ __forceinline__ T mm(T a, T b) {
  if (a > T(0) && b > T(0)) return (a <= b) ? a : b;
  if (a < T(0) && b < T(0)) return (a >= b) ? a : b;
  return T(0);
}

// FP64: the same value from integer comparisons (fp_bits.cuh), which removes
// about 140 of the 350 FP64-pipe instructions of a 3D predictor cell (k_predict,
// 64^3 cells in 16^3 patches: 0.249 -> 0.193 ms)
template <> __device__ __forceinline__ double mm<double>(double a, double b) { return minmod_bits(a, b); }

// FP32: the median of a, b and 0, four minima and maxima instead of about seven
// comparisons and selections. The inner two pass a NaN on and the outer two drop
// it, so that a NaN gives 0 as the comparisons do: the same value for every pair.
__device__ __forceinline__ float min_nan(float a, float b) {
#ifdef __CUDA_ARCH__
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
#else
  return a != a || b != b ? NAN : fminf(a, b);
#endif
}
__device__ __forceinline__ float max_nan(float a, float b) {
#ifdef __CUDA_ARCH__
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
#else
  return a != a || b != b ? NAN : fmaxf(a, b);
#endif
}
template <> __device__ __forceinline__ float mm<float>(float a, float b) {
  return fmaxf(min_nan(a, b), fminf(max_nan(a, b), 0.0f));
}

template <class T> __device__ __forceinline__ T tmaxd(T a, T b) { return a > b ? a : b; }
template <class T> __device__ __forceinline__ T tmind(T a, T b) { return a < b ? a : b; }

// FP32 operations that round by themselves: the compiler contracts a product
// and a sum into an FMA or not by their surroundings, so the same formula could
// round one way in one kernel (or one unrolled copy of a loop) and another way
// in the next. Where results must not depend on that, the FMAs are written.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float xmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float xadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float xsub(float a, float b) { return __fsub_rn(a, b); }
#else
inline float xmul(float a, float b) { return a * b; }
inline float xadd(float a, float b) { return a + b; }
inline float xsub(float a, float b) { return a - b; }
#endif

// square of the fast magnetosonic speed along a direction with normal field bn
template <class T> __device__ __forceinline__ T cfast2(T rho, T p, T bn, T bt, T bu, T gamma) {
  T irho = T(1) / rho;
  T gp = gamma * p;
  T b2 = bn * bn + bt * bt + bu * bu;
  T a = (gp + b2) * irho;
  T disc = a * a - T(4) * (gp * irho) * (bn * bn * irho);
  if (disc < T(0)) disc = T(0);
  return T(0.5) * (a + dsqrt(disc));
}
// FP64: the same value (the factor 4 is exact), the clamp on the integer pipe
template <>
__device__ __forceinline__ double cfast2<double>(double rho, double p, double bn, double bt, double bu, double gamma) {
  const double irho = 1.0 / rho;
  const double gp = gamma * p;
  const double bn2 = bn * bn;
  const double b2 = bn2 + bt * bt + bu * bu;
  const double a = (gp + b2) * irho;
  const double y = (gp * irho) * (bn2 * irho);
  double disc = fma(-4.0, y, a * a);
  if (lt_zero(disc)) disc = 0.0;
  return 0.5 * (a + sqrt(disc));
}
// fast magnetosonic speed along a direction with normal field bn
template <class T> __device__ __forceinline__ T cfast(T rho, T p, T bn, T bt, T bu, T gamma) {
  return dsqrt(cfast2(rho, p, bn, bt, bu, gamma));
}

// conservative -> primitive, always in FP64: p = (g-1)(E - m.m/(2 rho) - B.B/2)
__device__ __forceinline__ void recover(const double* u, const double* bc, double gm1, double* w) {
  double r = u[0];
  double ir = 1.0 / r;
  double vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
  double ke = 0.5 * (u[1] * vx + u[2] * vy + u[3] * vz);
  double me = 0.5 * (bc[0] * bc[0] + bc[1] * bc[1] + bc[2] * bc[2]);
  w[0] = r; w[1] = vx; w[2] = vy; w[3] = vz;
  w[4] = gm1 * ((u[4] - ke) - me);
  w[5] = bc[0]; w[6] = bc[1]; w[7] = bc[2];
}

// Error-free FP32 transformations (Knuth two-sum, FMA two-product): a pair
// (hi, lo) represents hi + lo exactly or to ~2^-46 relative.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = a * b;
  e = fmaf(a, b, -p);
}
// (ah, al) + (bh, bl)
__device__ __forceinline__ void df_add(float ah, float al, float bh, float bl, float& h, float& l) {
  float s, e;
  two_sum(ah, bh, s, e);
  e += al + bl;
  h = s + e;
  l = e - (h - s);
}
// (ah, al)^2
__device__ __forceinline__ void df_sq(float ah, float al, float& h, float& l) {
  float p, e;
  two_prod(ah, ah, p, e);
  e = fmaf(2.0f * ah, al, e);
  h = p + e;
  l = e - (h - p);
}

// Recovery of one cell from stored values in the working type T. For T =
// double this is recover() exactly. For the mixed path (T = float) the pressure
// is the energy balance p = (g-1)(E - (ke + me)) in FP64, rounded to FP32
// (nearest even), with ke = |m|^2 / (2 rho) and me = |B_c|^2 / 2 formed from the
// FP32 inputs by error-free FP32 transformations (squares, sums, face means,
// the division by rho carried as hi + lo pairs, ~2^-46 relative); v = m / rho
// and B_c are FP32. The balance's FP64 instructions hold the FP64 pipe (2 lanes
// an SM) for longer than all of the recovery's FP32 work takes, so balance()
// carries it in pairs too and knows how far that can be from FP64: where every
// value in that interval rounds to the same FP32 number, that number is the
// FP64 balance's, bit for bit; else (about 1 cell in 2^16 at a pressure of a
// seventh of the energy) the FP64 instructions run. Four steps of the 128^3 blast,
// advance and CFL, take 1.655 ms with the balance in FP64 always and 1.602 ms
// with this; two of 256^3 5.71 and 5.48 ms.
template <class T> struct Gm1;  // gamma - 1 for recover_t
template <> struct Gm1<double> {
  double v;
  __host__ __device__ explicit Gm1(double gm1) : v(gm1) {}
};
template <> struct Gm1<float> {
  double v;
  float h, l;  // v as a pair
  __host__ __device__ explicit Gm1(double gm1) : v(gm1), h((float)gm1), l((float)(gm1 - (double)(float)gm1)) {}
  __host__ __device__ Gm1(double gm1, float hi, float lo) : v(gm1), h(hi), l(lo) {}
};
__device__ __forceinline__ void recover_t(const double* u, const double* bl, const double* br, Gm1<double> gm1,
                                          double* w) {
  double bc[3] = {0.5 * (bl[0] + br[0]), 0.5 * (bl[1] + br[1]), 0.5 * (bl[2] + br[2])};
  recover(u, bc, gm1.v, w);
}
// ke + me of a cell as a pair; irf = 1 / rho
__device__ __forceinline__ void ke_me(const float* u, const float* bl, const float* br, float irf, float& eh,
                                      float& el) {
  const float r = u[0];
  // |m|^2 as a pair
  float mh, ml, th, tl;
  two_prod(u[1], u[1], mh, ml);
  two_prod(u[2], u[2], th, tl);
  df_add(mh, ml, th, tl, mh, ml);
  two_prod(u[3], u[3], th, tl);
  df_add(mh, ml, th, tl, mh, ml);
  // ke = 0.5 |m|^2 / rho as a pair: q = mh/r, remainder (mh - q r + ml)/r
  const float q = mh * irf;
  const float q1 = (fmaf(-q, r, mh) + ml) * irf;
  const float q2 = (fmaf(-q1, r, fmaf(-q, r, mh) + ml)) * irf;
  float kh, kl;
  two_sum(q, q1 + q2, kh, kl);
  // |bl + br|^2 summed over components as a pair (me = that / 8)
  float bh = 0.0f, blo = 0.0f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float sh, se, qh, ql;
    two_sum(bl[c], br[c], sh, se);
    df_sq(sh, se, qh, ql);
    df_add(bh, blo, qh, ql, bh, blo);
  }
  // (ke + me) = 0.5 (kh, kl) + 0.125 (bh, blo): exact power-of-two scalings
  df_add(0.5f * kh, 0.5f * kl, 0.125f * bh, 0.125f * blo, eh, el);
}
// p = (g-1)(E - (eh + el)) rounded once; true if every value within
// tol (|E| + |eh|) (g-1) of it rounds to the same p. The pairs' own error: the
// difference's 2^-48 (|E| + 2 |eh|) and at most 2^-47 |eh| where it cancels, the
// product's under 2^-46 of |E| + |eh|; d > 2^-110 keeps every term clear of
// the range that FP32 flushes.
__device__ __forceinline__ bool balance(float E, float eh, float el, const Gm1<float>& gm1, float tol, float& p) {
  float s, t;
  two_sum(E, -eh, s, t);
  t = xsub(t, el);
  const float h = xadd(s, t), l = xsub(t, xsub(h, s));
  const float c = fmaf(h, gm1.l, xmul(l, gm1.h)), d = xmul(xadd(fabsf(E), fabsf(eh)), gm1.h * tol);
  p = fmaf(h, gm1.h, xadd(c, d));
  return p == fmaf(h, gm1.h, xsub(c, d)) && d > 0x1p-110f;
}
__device__ __forceinline__ void recover_t(const float* u, const float* bl, const float* br, Gm1<float> gm1, float* w) {
  const float irf = 1.0f / u[0];
  float eh, el, p;
  ke_me(u, bl, br, irf, eh, el);
  if (!balance(u[4], eh, el, gm1, 0x1p-43f, p))
    p = narrow_bits(gm1.v * (widen_bits(u[4]) - (widen_bits(eh) + widen_bits(el))));
  w[0] = u[0];
  w[1] = u[1] * irf;
  w[2] = u[2] * irf;
  w[3] = u[3] * irf;
  w[4] = p;
  w[5] = 0.5f * (bl[0] + br[0]);
  w[6] = 0.5f * (bl[1] + br[1]);
  w[7] = 0.5f * (bl[2] + br[2]);
}

// floors of the recovery (reading 12): the density before the recovery, the
// pressure after it; each raise counted
template <class T> __device__ __forceinline__ void floor_density(T* u, double rho_min, unsigned long long* events) {
  if (rho_min > 0.0 && u[0] < (T)rho_min) {
    u[0] = (T)rho_min;
    atomicAdd(events, 1ull);
  }
}
template <class T> __device__ __forceinline__ void floor_pressure(T* w, double p_min, unsigned long long* events) {
  if (p_min > 0.0 && w[4] < (T)p_min) {
    w[4] = (T)p_min;
    atomicAdd(events, 1ull);
  }
}

// A_d(W) s for the primitive predictor, direction d (n = d, t = d+1, u = d+2 mod 3)
template <class T, int D> __device__ __forceinline__ void prim_terms(const T* w, const T* s, T gamma, T ir, T* dw) {
  constexpr int n = D, t = (D + 1) % 3, u = (D + 2) % 3;
  const T rho = w[0], p = w[4];
  const T vn = w[1 + n];
  const T bn = w[5 + n], bt = w[5 + t], bu = w[5 + u];
  dw[0] = vn * s[0] + rho * s[1 + n];
  dw[1 + n] = vn * s[1 + n] + (s[4] + bt * s[5 + t] + bu * s[5 + u]) * ir;
  dw[1 + t] = vn * s[1 + t] - bn * s[5 + t] * ir;
  dw[1 + u] = vn * s[1 + u] - bn * s[5 + u] * ir;
  dw[4] = vn * s[4] + gamma * p * s[1 + n];
  dw[5 + n] = vn * s[5 + n];
  dw[5 + t] = vn * s[5 + t] - bn * s[1 + t] + bt * s[1 + n];
  dw[5 + u] = vn * s[5 + u] - bn * s[1 + u] + bu * s[1 + n];
}

// predicted states at a cell's high and low face: w +- s / 2 (in FP64 one
// instruction: 0.5 s is exact, so the fused sum rounds as the written one)
template <class T> __device__ __forceinline__ T plus_half(T w, T s) { return w + T(0.5) * s; }
template <class T> __device__ __forceinline__ T minus_half(T w, T s) { return w - T(0.5) * s; }
template <> __device__ __forceinline__ double plus_half<double>(double w, double s) { return fma(0.5, s, w); }
template <> __device__ __forceinline__ double minus_half<double>(double w, double s) { return fma(-0.5, s, w); }

// physical flux of a rotated state q = (rho, un, ut, uu, p, bt, bu); u = conserved
template <class T> __device__ __forceinline__ void phys_flux(const T* q, T bn, T igm1, T* f, T* u) {
  const T r = q[0], un = q[1], ut = q[2], uu = q[3], p = q[4], bt = q[5], bu = q[6];
  const T b2 = bn * bn + bt * bt + bu * bu;
  const T pt = p + T(0.5) * b2;
  const T e = p * igm1 + T(0.5) * r * (un * un + ut * ut + uu * uu) + T(0.5) * b2;
  const T vb = un * bn + ut * bt + uu * bu;
  f[0] = r * un;
  f[1] = r * un * un + pt - bn * bn;
  f[2] = r * un * ut - bn * bt;
  f[3] = r * un * uu - bn * bu;
  f[4] = (e + pt) * un - bn * vb;
  f[5] = bt * un - bn * ut;
  f[6] = bu * un - bn * uu;
  u[0] = r; u[1] = r * un; u[2] = r * ut; u[3] = r * uu; u[4] = e; u[5] = bt; u[6] = bu;
}

// 1 / (gamma - 1) of a face's flux: FP64 takes the host's quotient (the same
// value; an FP64 division costs about 10 instructions of the bound pipe), FP32
// forms it in place, where it holds no register between faces
template <class T> __device__ __forceinline__ T inv_gm1(T gamma, double igm1);
template <> __device__ __forceinline__ double inv_gm1<double>(double, double igm1) { return igm1; }
template <> __device__ __forceinline__ float inv_gm1<float>(float gamma, double) { return 1.0f / (gamma - 1.0f); }

// Quotients that share a divisor: FP64 divides each time (the written
// formula, bit for bit); FP32 multiplies by one reciprocal (the FP32 path
// compiles its divisions as a reciprocal and a product anyway).
template <class T> struct Quot {
  T d;
  __device__ __forceinline__ explicit Quot(T den) : d(den) {}
  __device__ __forceinline__ T operator()(T num) const { return num / d; }
};
template <> struct Quot<float> {
  float r;
  __device__ __forceinline__ explicit Quot(float den) : r(1.0f / den) {}
  __device__ __forceinline__ float operator()(float num) const { return num * r; }
};

// HLLD flux between rotated states ql, qr with common normal field bn;
// igm1 = 1 / (gamma - 1). The formula as written; hlld_flux is what the
// kernels call.
template <class T> __device__ void hlld_plain(const T* ql, const T* qr, T bn, T gamma, T igm1, T* f) {
  const T eps = Eps<T>::v();
  T fl[7], fr[7], ul[7], ur[7];
  phys_flux(ql, bn, igm1, fl, ul);
  phys_flux(qr, bn, igm1, fr, ur);
  // max(sqrt(a), sqrt(b)) = sqrt(max(a, b)): the square root is monotone and
  // correctly rounded, so one root serves both sides
  const T cl2 = cfast2(ql[0], ql[4], bn, ql[5], ql[6], gamma);
  const T cr2 = cfast2(qr[0], qr[4], bn, qr[5], qr[6], gamma);
  const T cmax = dsqrt(tmaxd(cl2, cr2));
  const T sl = tmind(ql[1], qr[1]) - cmax;
  const T sr = tmaxd(ql[1], qr[1]) + cmax;
  if (sl > T(0)) {
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = fl[k];
    return;
  }
  if (sr < T(0)) {
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = fr[k];
    return;
  }
  const T bn2 = bn * bn;
  const T rl = ql[0], rr = qr[0];
  const T uln = ql[1], urn = qr[1];
  const T ptl = ql[4] + T(0.5) * (bn2 + ql[5] * ql[5] + ql[6] * ql[6]);
  const T ptr = qr[4] + T(0.5) * (bn2 + qr[5] * qr[5] + qr[6] * qr[6]);
  const T dl = sl - uln, dr = sr - urn;
  const Quot<T> byden(dr * rr - dl * rl);
  const T sm = byden(dr * rr * urn - dl * rl * uln - ptr + ptl);
  const T pts = byden(dr * rr * ptl - dl * rl * ptr + rl * rr * dr * dl * (urn - uln));

  T rs[2], vs[2], ws[2], bts[2], bus[2], es[2], vbs[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const T* q = a == 0 ? ql : qr;
    const T sx = a == 0 ? sl : sr;
    const T da = sx - q[1];
    const T ssm = sx - sm;
    const Quot<T> byssm(ssm);
    rs[a] = byssm(q[0] * da);
    const T rds = q[0] * da * ssm;
    const T e = rds - bn2;
    if (dabs(e) <= eps * (dabs(rds) + bn2)) {
      vs[a] = q[2]; ws[a] = q[3]; bts[a] = q[5]; bus[a] = q[6];
    } else {
      const T ie = T(1) / e;
      const T tq = bn * (sm - q[1]) * ie;
      vs[a] = q[2] - q[5] * tq;
      ws[a] = q[3] - q[6] * tq;
      const T qq = (q[0] * da * da - bn2) * ie;
      bts[a] = q[5] * qq;
      bus[a] = q[6] * qq;
    }
    const T vb = q[1] * bn + q[2] * q[5] + q[3] * q[6];
    vbs[a] = sm * bn + vs[a] * bts[a] + ws[a] * bus[a];
    const T ea = a == 0 ? ul[4] : ur[4];
    es[a] = byssm(da * ea - (a == 0 ? ptl : ptr) * q[1] + pts * sm + bn * (vb - vbs[a]));
  }
  const T usl[7] = {rs[0], rs[0] * sm, rs[0] * vs[0], rs[0] * ws[0], es[0], bts[0], bus[0]};
  const T usr[7] = {rs[1], rs[1] * sm, rs[1] * vs[1], rs[1] * ws[1], es[1], bts[1], bus[1]};
  if (bn2 <= eps * pts) {
    if (sm >= T(0)) {
#pragma unroll
      for (int k = 0; k < 7; ++k) f[k] = fl[k] + sl * (usl[k] - ul[k]);
    } else {
#pragma unroll
      for (int k = 0; k < 7; ++k) f[k] = fr[k] + sr * (usr[k] - ur[k]);
    }
    return;
  }
  const T sql = dsqrt(rs[0]), sqr = dsqrt(rs[1]);
  const T abn = dabs(bn);
  const T sls = sm - abn / sql;
  const T srs = sm + abn / sqr;
  if (sls >= T(0)) {
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = fl[k] + sl * (usl[k] - ul[k]);
    return;
  }
  if (srs <= T(0)) {
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = fr[k] + sr * (usr[k] - ur[k]);
    return;
  }
  const T sgn = bn > T(0) ? T(1) : T(-1);
  const T idn = T(1) / (sql + sqr);
  const T vss = (sql * vs[0] + sqr * vs[1] + (bts[1] - bts[0]) * sgn) * idn;
  const T wss = (sql * ws[0] + sqr * ws[1] + (bus[1] - bus[0]) * sgn) * idn;
  const T btss = (sql * bts[1] + sqr * bts[0] + sql * sqr * (vs[1] - vs[0]) * sgn) * idn;
  const T buss = (sql * bus[1] + sqr * bus[0] + sql * sqr * (ws[1] - ws[0]) * sgn) * idn;
  const T vbss = sm * bn + vss * btss + wss * buss;
  if (sm >= T(0)) {
    const T ess = es[0] - sql * (vbs[0] - vbss) * sgn;
    const T uss[7] = {rs[0], rs[0] * sm, rs[0] * vss, rs[0] * wss, ess, btss, buss};
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = fl[k] + sls * uss[k] - (sls - sl) * usl[k] - sl * ul[k];
  } else {
    const T ess = es[1] + sqr * (vbs[1] - vbss) * sgn;
    const T uss[7] = {rs[1], rs[1] * sm, rs[1] * vss, rs[1] * wss, ess, btss, buss};
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = fr[k] + srs * uss[k] - (srs - sr) * usr[k] - sr * ur[k];
  }
}

// FP64: the value of hlld_plain bit for bit (no result of which depends on
// the sign of a zero), from fewer FP64-pipe instructions. The FP64 pipe (2
// lanes per SM) bounds every FP64 kernel of the advance; of the about 550
// FP64 instructions of hlld_plain per face, here:
//  * comparisons, minima and selections run on the integer pipe (fp_bits.cuh);
//  * the flux, energy and star energy are formed for the side the result is
//    taken from only, its operands selected first;
//  * a power-of-two factor is exact, so RN(c + RN(0.5 x)) = fma(0.5, x, c) and
//    RN(0.5 x y) = 0.5 RN(x y) (short of underflow).
// 64^3 cells in 16^3 patches, the fluxes of the three directions: 1.13 -> 0.81 ms
// (0.55 with k_flux's blocks of 64 and without ghost faces).
__device__ __forceinline__ void hlld_fp64(const double* ql, const double* qr, double bn, double gamma, double igm1,
                                          double* f) {
  constexpr double eps = 1e-12;
  const double bn2 = bn * bn;
  const double b2l = bn2 + ql[5] * ql[5] + ql[6] * ql[6], b2r = bn2 + qr[5] * qr[5] + qr[6] * qr[6];
  const double ptl = fma(0.5, b2l, ql[4]), ptr = fma(0.5, b2r, qr[4]);
  // twice cfast2 of both sides
  double c2[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const double* q = a == 0 ? ql : qr;
    const double irho = 1.0 / q[0];
    const double gp = gamma * q[4];
    const double x = (gp + (a == 0 ? b2l : b2r)) * irho;
    const double y = (gp * irho) * (bn2 * irho);
    double disc = fma(-4.0, y, x * x);
    if (lt_zero(disc)) disc = 0.0;
    c2[a] = x + sqrt(disc);
  }
  const double cmax = sqrt(0.5 * (gt_bits(c2[0], c2[1]) ? c2[0] : c2[1]));
  const bool uml = gt_bits(qr[1], ql[1]), uxl = gt_bits(ql[1], qr[1]);
  const double sl = (uml ? ql[1] : qr[1]) - cmax;
  const double sr = (uxl ? ql[1] : qr[1]) + cmax;
  const bool sup_l = gt_zero(sl), sup_r = lt_zero(sr);
  const double dl = sl - ql[1], dr = sr - qr[1];
  const double rdl = dl * ql[0], rdr = dr * qr[0];
  const double den = rdr - rdl;
  const double sm = (rdr * qr[1] - rdl * ql[1] - ptr + ptl) / den;
  const bool left = sup_l || (!sup_r && ge_zero(sm));
  // the side the flux is taken from
  double q[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) q[k] = left ? ql[k] : qr[k];
  const double b2 = left ? b2l : b2r, pt = left ? ptl : ptr;
  const double e = fma(0.5, b2, fma(0.5, q[0] * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]), q[4] * igm1));
  const double vb = q[1] * bn + q[2] * q[5] + q[3] * q[6];
  const double ru = q[0] * q[1];
  const double u[7] = {q[0], ru, q[0] * q[2], q[0] * q[3], e, q[5], q[6]};
  const double F[7] = {ru, ru * q[1] + pt - bn2, ru * q[2] - bn * q[5], ru * q[3] - bn * q[6],
                       (e + pt) * q[1] - bn * vb, q[5] * q[1] - bn * q[2], q[6] * q[1] - bn * q[3]};
  if (sup_l || sup_r) {
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = F[k];
    return;
  }
  const double pts = (rdr * ptl - rdl * ptr + ql[0] * qr[0] * dr * dl * (qr[1] - ql[1])) / den;
  double rs[2], vs[2], ws[2], bts[2], bus[2], ss[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const double* p = a == 0 ? ql : qr;
    const double da = a == 0 ? dl : dr, rd = a == 0 ? rdl : rdr;
    const double ssm = (a == 0 ? sl : sr) - sm;
    ss[a] = ssm;
    rs[a] = rd / ssm;
    const double rds = rd * ssm;
    const double ed = rds - bn2;
    if (abs_le(ed, eps * (fabs(rds) + bn2))) {
      vs[a] = p[2]; ws[a] = p[3]; bts[a] = p[5]; bus[a] = p[6];
    } else {
      const double ie = 1.0 / ed;
      const double tq = bn * (sm - p[1]) * ie;
      vs[a] = p[2] - p[5] * tq;
      ws[a] = p[3] - p[6] * tq;
      const double qq = (rd * da - bn2) * ie;
      bts[a] = p[5] * qq;
      bus[a] = p[6] * qq;
    }
  }
  const double S = left ? sl : sr, da = left ? dl : dr, ssm = left ? ss[0] : ss[1];
  const double r1 = left ? rs[0] : rs[1], v1 = left ? vs[0] : vs[1], w1 = left ? ws[0] : ws[1];
  const double bt1 = left ? bts[0] : bts[1], bu1 = left ? bus[0] : bus[1];
  const double vbs = sm * bn + v1 * bt1 + w1 * bu1;
  const double es = (da * e - pt * q[1] + pts * sm + bn * (vb - vbs)) / ssm;
  const double us[7] = {r1, r1 * sm, r1 * v1, r1 * w1, es, bt1, bu1};
  bool single = le_pos(bn2, eps * pts);
  double sql = 0.0, sqr = 0.0, Ss = 0.0;
  if (!single) {
    sql = sqrt(rs[0]);
    sqr = sqrt(rs[1]);
    const double abn = fabs(bn);
    // the star speed of the side: it is on the flux's side of the face exactly when the plain order of tests says so
    const double c = abn / (left ? sql : sqr);
    Ss = left ? sm - c : sm + c;
    single = left ? ge_zero(Ss) : le_zero(Ss);
  }
  if (single) {
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = F[k] + S * (us[k] - u[k]);
    return;
  }
  // times the sign of bn (-1 for a zero): a sign flip
  const uint64_t flip = gt_zero(bn) ? 0ull : F64_SIGN;
  auto sgn = [&](double x) { return f64_of(f64_bits(x) ^ flip); };
  const double idn = 1.0 / (sql + sqr), sqp = sql * sqr;
  const double vss = (sql * vs[0] + sqr * vs[1] + sgn(bts[1] - bts[0])) * idn;
  const double wss = (sql * ws[0] + sqr * ws[1] + sgn(bus[1] - bus[0])) * idn;
  const double btss = (sql * bts[1] + sqr * bts[0] + sgn(sqp * (vs[1] - vs[0]))) * idn;
  const double buss = (sql * bus[1] + sqr * bus[0] + sgn(sqp * (ws[1] - ws[0]))) * idn;
  const double vbss = sm * bn + vss * btss + wss * buss;
  const double t = sgn((left ? sql : sqr) * (vbs - vbss));
  const double ess = left ? es - t : es + t;
  const double uss[7] = {r1, us[1], r1 * vss, r1 * wss, ess, btss, buss};
  const double dS = Ss - S;
#pragma unroll
  for (int k = 0; k < 7; ++k) f[k] = F[k] + Ss * uss[k] - dS * us[k] - S * u[k];
}

// FP32: hlld_plain with every rounding written down (the FMAs, and xmul, xadd,
// xsub for the rest), so that a face has the same flux bit for bit in every
// kernel and launch shape, and only the side the result is taken from formed as
// in hlld_fp64; selections in place of the branches, which the faces of one
// warp take differently. SUM: the order of the roundings of the energy's sums,
// which is one for the fused 3D advance, one for the staged and the fused 2D
// kernels and one for the registers recomputed from a 3D level's state.
// The mass flux of gas nearly at rest is what this rounding leaves of it, and
// its sign decides what the edge EMFs upwind: another formula of the same
// accuracy moves single faces by 1e-3 of the field.
// About 250 instructions a face. With hlld_plain four steps of the 128^3 blast
// take 1.69 ms, two of 64^3 with a refined level 746 us; with this 1.60 ms, 698 us.
enum { HLLD_FUSED, HLLD_STAGED, HLLD_REGISTER };
template <int SUM>
__device__ __forceinline__ void hlld_fp32(const float* ql, const float* qr, float bn, float gamma, float igm1, float* f) {
  constexpr float eps = 1e-6f;
  const float bn2 = xmul(bn, bn);
  // twice the squares of the fast speeds
  float b2s[2], pts_[2], c2[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const float* q = a == 0 ? ql : qr;
    b2s[a] = fmaf(q[6], q[6], fmaf(q[5], q[5], bn2));
    pts_[a] = fmaf(0.5f, b2s[a], q[4]);
    const float irho = 1.0f / q[0];
    const float gp = xmul(gamma, q[4]);
    const float x = xmul(xadd(gp, b2s[a]), irho);
    float disc = fmaf(x, x, -4.0f * xmul(xmul(gp, irho), xmul(bn2, irho)));
    if (disc < 0.0f) disc = 0.0f;
    c2[a] = xadd(x, sqrtf(disc));
  }
  const float ptl = pts_[0], ptr = pts_[1];
  const float cmax = sqrtf(0.5f * tmaxd(c2[0], c2[1]));
  const float sl = xsub(tmind(ql[1], qr[1]), cmax), sr = xadd(tmaxd(ql[1], qr[1]), cmax);
  const bool sup_l = sl > 0.0f, sup_r = sr < 0.0f;
  const float dl = xsub(sl, ql[1]), dr = xsub(sr, qr[1]);
  const float rdl = xmul(dl, ql[0]), rdr = xmul(dr, qr[0]);
  const float iden = 1.0f / xsub(rdr, rdl);
  const float sm = xmul(xadd(xsub(fmaf(rdr, qr[1], -xmul(rdl, ql[1])), ptr), ptl), iden);
  const bool left = sup_l || (!sup_r && sm >= 0.0f);
  // the side the flux is taken from: its conserved state and flux
  float q[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) q[k] = left ? ql[k] : qr[k];
  const float pt = left ? ptl : ptr, b2 = left ? b2s[0] : b2s[1];
  const float hr = 0.5f * q[0], kk = fmaf(q[3], q[3], fmaf(q[1], q[1], xmul(q[2], q[2])));
  const float e = fmaf(0.5f, b2, SUM == HLLD_STAGED ? fmaf(hr, kk, xmul(q[4], igm1)) : fmaf(q[4], igm1, xmul(hr, kk)));
  const float vb = fmaf(q[3], q[6], fmaf(q[1], bn, xmul(q[2], q[5])));
  const float ru = xmul(q[0], q[1]);
  const float u[7] = {q[0], ru, xmul(q[0], q[2]), xmul(q[0], q[3]), e, q[5], q[6]};
  const float F[7] = {ru,
                      xsub(fmaf(ru, q[1], pt), bn2),
                      fmaf(ru, q[2], -xmul(bn, q[5])),
                      fmaf(ru, q[3], -xmul(bn, q[6])),
                      fmaf(xadd(e, pt), q[1], -xmul(bn, vb)),
                      fmaf(q[5], q[1], -xmul(bn, q[2])),
                      fmaf(q[6], q[1], -xmul(bn, q[3]))};
  const float pts = xmul(fmaf(xmul(xmul(xmul(ql[0], qr[0]), dr), dl), xsub(qr[1], ql[1]),
                              fmaf(rdr, ptl, -xmul(rdl, ptr))), iden);
  // star states of both sides
  float rs[2], vs[2], ws[2], bts[2], bus[2], iss[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const float* p = a == 0 ? ql : qr;
    const float da = a == 0 ? dl : dr, rd = a == 0 ? rdl : rdr;
    const float ssm = xsub(a == 0 ? sl : sr, sm);
    iss[a] = 1.0f / ssm;
    rs[a] = xmul(rd, iss[a]);
    const float rds = xmul(rd, ssm);
    const float ed = xsub(rds, bn2);
    const bool degen = fabsf(ed) <= xmul(eps, xadd(fabsf(rds), bn2));
    const float ie = 1.0f / ed;
    const float tq = degen ? 0.0f : xmul(xmul(bn, xsub(sm, p[1])), ie);
    const float qq = degen ? 1.0f : xmul(fmaf(rd, da, -bn2), ie);
    vs[a] = fmaf(-p[5], tq, p[2]);
    ws[a] = fmaf(-p[6], tq, p[3]);
    bts[a] = xmul(p[5], qq);
    bus[a] = xmul(p[6], qq);
  }
  const float S = left ? sl : sr, da = left ? dl : dr, is = left ? iss[0] : iss[1];
  const float r1 = left ? rs[0] : rs[1], v1 = left ? vs[0] : vs[1], w1 = left ? ws[0] : ws[1];
  const float bt1 = left ? bts[0] : bts[1], bu1 = left ? bus[0] : bus[1];
  const float vbs = fmaf(w1, bu1, SUM == HLLD_REGISTER ? fmaf(v1, bt1, xmul(sm, bn)) : fmaf(sm, bn, xmul(v1, bt1)));
  const float ea = fmaf(da, e, -xmul(pt, q[1]));
  const float eb = SUM == HLLD_FUSED ? fmaf(pts, sm, ea) : xadd(ea, xmul(pts, sm));
  const float es = xmul(fmaf(bn, xsub(vb, vbs), eb), is);
  const float us[7] = {r1, xmul(r1, sm), xmul(r1, v1), xmul(r1, w1), es, bt1, bu1};
  // the star speed of the side is on the flux's side of the face exactly when the plain order of tests says so
  const float sql = sqrtf(rs[0]), sqr = sqrtf(rs[1]);
  const float Ss = fmaf(left ? -fabsf(bn) : fabsf(bn), 1.0f / (left ? sql : sqr), sm);
  const bool single = bn2 <= xmul(eps, pts) || (left ? Ss >= 0.0f : Ss <= 0.0f);
  // double-star state
  const float sgn = bn > 0.0f ? 1.0f : -1.0f;
  const float idn = 1.0f / xadd(sql, sqr);
  const float sqp = xmul(sql, sqr);
  const float vss = xmul(fmaf(xsub(bts[1], bts[0]), sgn, fmaf(sql, vs[0], xmul(sqr, vs[1]))), idn);
  const float wss = xmul(fmaf(xsub(bus[1], bus[0]), sgn, fmaf(sql, ws[0], xmul(sqr, ws[1]))), idn);
  const float btss = xmul(fmaf(xmul(sqp, xsub(vs[1], vs[0])), sgn, fmaf(sql, bts[1], xmul(sqr, bts[0]))), idn);
  const float buss = xmul(fmaf(xmul(sqp, xsub(ws[1], ws[0])), sgn, fmaf(sql, bus[1], xmul(sqr, bus[0]))), idn);
  const float vbss =
      fmaf(wss, buss, SUM == HLLD_REGISTER ? fmaf(vss, btss, xmul(sm, bn)) : fmaf(sm, bn, xmul(vss, btss)));
  const float t = xmul(left ? sql : sqr, xsub(vbs, vbss));
  const float ess = fmaf(left ? -t : t, sgn, es);
  const float uss[7] = {r1, us[1], xmul(r1, vss), xmul(r1, wss), ess, btss, buss};
  const float dS = xsub(Ss, S);
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const float one = fmaf(S, xsub(us[k], u[k]), F[k]);
    const float two = fmaf(-S, u[k], fmaf(-dS, us[k], fmaf(Ss, uss[k], F[k])));
    f[k] = (sup_l || sup_r) ? F[k] : single ? one : two;
  }
}

template <class T, int SUM = HLLD_FUSED>
__device__ __forceinline__ void hlld_flux(const T* ql, const T* qr, T bn, T gamma, T igm1, T* f) {
  if constexpr (sizeof(T) == 8) hlld_fp64(ql, qr, bn, gamma, igm1, f);
  else hlld_fp32<SUM>(ql, qr, bn, gamma, igm1, f);
}

template <class T> __device__ __forceinline__ T upw(T fm, T lo, T hi) {
  if (fm > T(0)) return lo;
  if (fm < T(0)) return hi;
  return T(0.5) * (lo + hi);
}

// Gardiner-Stone edge EMF at (a-1/2, b-1/2); see the argument names of the
// cell references r[ab] (a-offset, b-offset) and face EMFs/mass fluxes.
template <class T>
__device__ __forceinline__ T gs_emf_plain(T ea_lo, T ea_hi, T eb_lo, T eb_hi, T r00, T r10, T r01, T r11, T fa_lo,
                                          T fa_hi, T fb_lo, T fb_hi) {
  const T db_hi = upw(fa_hi, r01 - eb_lo, r11 - eb_hi);
  const T db_lo = upw(fa_lo, eb_lo - r00, eb_hi - r10);
  const T da_hi = upw(fb_hi, r10 - ea_lo, r11 - ea_hi);
  const T da_lo = upw(fb_lo, ea_lo - r00, ea_hi - r01);
  return T(0.25) * (((ea_hi + ea_lo) + eb_hi) + eb_lo) + T(0.25) * (db_lo - db_hi) + T(0.25) * (da_lo - da_hi);
}
template <class T>
__device__ __forceinline__ T gs_emf(T ea_lo, T ea_hi, T eb_lo, T eb_hi, T r00, T r10, T r01, T r11, T fa_lo, T fa_hi,
                                    T fb_lo, T fb_hi) {
  return gs_emf_plain<T>(ea_lo, ea_hi, eb_lo, eb_hi, r00, r10, r01, r11, fa_lo, fa_hi, fb_lo, fb_hi);
}
// FP64: gs_emf_plain bit for bit (the factors 0.25 are exact): sign tests on
// the integer pipe and the operands selected before each one subtraction, 12
// instead of about 33 FP64 instructions; a mass flux of exactly 0 (or NaN)
// takes the formula as written
template <>
__device__ __forceinline__ double gs_emf<double>(double ea_lo, double ea_hi, double eb_lo, double eb_hi, double r00,
                                                 double r10, double r01, double r11, double fa_lo, double fa_hi,
                                                 double fb_lo, double fb_hi) {
  auto none = [](double f) { return !gt_zero(f) && !lt_zero(f); };
  if (none(fa_lo) || none(fa_hi) || none(fb_lo) || none(fb_hi))
    return gs_emf_plain<double>(ea_lo, ea_hi, eb_lo, eb_hi, r00, r10, r01, r11, fa_lo, fa_hi, fb_lo, fb_hi);
  auto neg = [](double f) { return (int64_t)f64_bits(f) < 0; };
  const bool ah = neg(fa_hi), al = neg(fa_lo), bh = neg(fb_hi), bl = neg(fb_lo);
  const double db_hi = (ah ? r11 : r01) - (ah ? eb_hi : eb_lo);
  const double db_lo = (al ? eb_hi : eb_lo) - (al ? r10 : r00);
  const double da_hi = (bh ? r11 : r10) - (bh ? ea_hi : ea_lo);
  const double da_lo = (bl ? ea_hi : ea_lo) - (bl ? r01 : r00);
  return 0.25 * ((((ea_hi + ea_lo) + eb_hi) + eb_lo) + (db_lo - db_hi) + (da_lo - da_hi));
}

__device__ __forceinline__ double tree2(double a, double b) { return a + b; }
__device__ __forceinline__ double tree4(double a, double b, double c, double d) { return (a + b) + (c + d); }
__device__ __forceinline__ double tree8(const double* v) {
  return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
}
// Mean of N = 2, 4 or 8 values, FP32: the sum in FP64, rounded once. Where the
// values lie within a factor of 2^16 of each other (or are all 0), that sum is
// exact, and so is the one by error-free FP32 transformations (they are
// multiples of one unit of which the errors' sum takes under 2^23 and the
// whole sum under 2^44), which spares the conversions and additions that hold
// the FP64 pipe; else, and where a value could be flushed, the FP64 sum runs.
// Two coarse steps of two 3D levels: 712 us with the FP64 sums always, 698 us
// with this; four of 512^2 with a refined level 723 and 695 us.
template <int N> __device__ __forceinline__ double mean(const double* v) {
  return N == 2 ? tree2(v[0], v[1]) * 0.5 : N == 4 ? tree4(v[0], v[1], v[2], v[3]) * 0.25 : tree8(v) * 0.125;
}
template <int N> __device__ __forceinline__ float mean(const float* v) {
  float hi = fabsf(v[0]), lo = hi;
#pragma unroll
  for (int i = 1; i < N; ++i) {
    hi = fmaxf(hi, fabsf(v[i]));
    lo = fminf(lo, fabsf(v[i]));
  }
  if (!(xmul(lo, 65536.0f) >= hi && hi < INFINITY && (lo > 0x1p-90f || hi == 0.0f))) {
    double d[N];
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = (double)v[i];
    return (float)mean<N>(d);
  }
  float s = v[0] * (1.0f / N), err = 0.0f;  // scaled first (exactly): no overflow where the mean has none
#pragma unroll
  for (int i = 1; i < N; ++i) {
    float e;
    two_sum(s, v[i] * (1.0f / N), s, e);
    err += e;
  }
  return s + err;
}

}  // namespace amrdev
