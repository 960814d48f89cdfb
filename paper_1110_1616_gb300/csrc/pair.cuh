// Pairs of FP32 values in one 64-bit register pair: sums, products and fused
// multiply-adds of both values are one instruction each (the packed f32x2
// forms of sm_100 and later), everything else works on the two values. The
// kernels that use them are bound by the issue of instructions, not by the
// FP32 pipe: a packed multiply-add takes one issue slot for two.
#pragma once
#include <cuda_runtime.h>

namespace amrdev {

struct Pair {
  float x, y;
};
struct Pred {  // a condition of each value
  bool x, y;
};
__device__ __forceinline__ Pair pair(float x, float y) { return {x, y}; }
__device__ __forceinline__ Pair pair(float v) { return {v, v}; }
__device__ __forceinline__ unsigned long long pack_bits(Pair a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ Pair unpack_bits(unsigned long long r) {
  Pair a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ Pair operator+(Pair a, Pair b) {
  unsigned long long r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack_bits(a)), "l"(pack_bits(b)));
  return unpack_bits(r);
}
__device__ __forceinline__ Pair operator*(Pair a, Pair b) {
  unsigned long long r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack_bits(a)), "l"(pack_bits(b)));
  return unpack_bits(r);
}
// a b + c
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
  unsigned long long r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack_bits(a)), "l"(pack_bits(b)), "l"(pack_bits(c)));
  return unpack_bits(r);
}
__device__ __forceinline__ Pair operator-(Pair a) { return {-a.x, -a.y}; }
// a - b as b (-1) + a: one instruction (the packed forms negate no operand)
__device__ __forceinline__ Pair operator-(Pair a, Pair b) { return fma2(b, pair(-1.0f), a); }
__device__ __forceinline__ Pair operator*(float a, Pair b) { return pair(a) * b; }
__device__ __forceinline__ Pair sel(Pred c, Pair a, Pair b) { return {c.x ? a.x : b.x, c.y ? a.y : b.y}; }
__device__ __forceinline__ Pair max2(Pair a, Pair b) { return {fmaxf(a.x, b.x), fmaxf(a.y, b.y)}; }
__device__ __forceinline__ Pair min2(Pair a, Pair b) { return {fminf(a.x, b.x), fminf(a.y, b.y)}; }
__device__ __forceinline__ Pair rcp2(Pair a) { return {1.0f / a.x, 1.0f / a.y}; }
__device__ __forceinline__ Pair sqrt2(Pair a) { return {sqrtf(a.x), sqrtf(a.y)}; }
__device__ __forceinline__ Pair rsqrt2(Pair a) { return {rsqrtf(a.x), rsqrtf(a.y)}; }
__device__ __forceinline__ Pair abs2(Pair a) { return {fabsf(a.x), fabsf(a.y)}; }
__device__ __forceinline__ Pred operator>(Pair a, float b) { return {a.x > b, a.y > b}; }
__device__ __forceinline__ Pred operator<(Pair a, float b) { return {a.x < b, a.y < b}; }
__device__ __forceinline__ Pred operator>=(Pair a, float b) { return {a.x >= b, a.y >= b}; }
__device__ __forceinline__ Pred operator<=(Pair a, float b) { return {a.x <= b, a.y <= b}; }
__device__ __forceinline__ Pred operator<=(Pair a, Pair b) { return {a.x <= b.x, a.y <= b.y}; }
__device__ __forceinline__ Pred operator||(Pred a, Pred b) { return {a.x || b.x, a.y || b.y}; }
__device__ __forceinline__ Pred operator&&(Pred a, Pred b) { return {a.x && b.x, a.y && b.y}; }
__device__ __forceinline__ Pred operator!(Pred a) { return {!a.x, !a.y}; }
__device__ __forceinline__ bool any(Pred a) { return a.x || a.y; }

// minmod: the median of a, b and 0
__device__ __forceinline__ Pair mm(Pair a, Pair b) {
  return max2(min2(a, b), min2(max2(a, b), pair(0.0f)));
}

// hlld_flux<float> (mhd_device.cuh) of two faces; ngm1 = -1 is folded into the
// products, bn the mean normal field
__device__ __forceinline__ void hlld_flux(const Pair* ql, const Pair* qr, Pair bn, float gamma, float igm1, Pair* f) {
  constexpr float eps = 1e-6f;
  const Pair bn2 = bn * bn, nbn = -bn;
  const Pair b2l = fma2(ql[6], ql[6], fma2(ql[5], ql[5], bn2)), b2r = fma2(qr[6], qr[6], fma2(qr[5], qr[5], bn2));
  const Pair ptl = fma2(pair(0.5f), b2l, ql[4]), ptr = fma2(pair(0.5f), b2r, qr[4]);
  const Pair irl = rcp2(ql[0]), irr = rcp2(qr[0]);
  const Pair g = pair(gamma);
  const Pair al = fma2(g, ql[4], b2l) * irl, ar = fma2(g, qr[4], b2r) * irr;
  const Pair yl = (g * ql[4]) * irl * (bn2 * irl), yr = (g * qr[4]) * irr * (bn2 * irr);
  const Pair cl = al + sqrt2(max2(fma2(pair(-4.0f), yl, al * al), pair(0.0f)));
  const Pair cr = ar + sqrt2(max2(fma2(pair(-4.0f), yr, ar * ar), pair(0.0f)));
  const Pair cmax = sqrt2(0.5f * Pair{cl.x > cr.x ? cl.x : cr.x, cl.y > cr.y ? cl.y : cr.y});
  const Pair sl = min2(ql[1], qr[1]) - cmax, sr = max2(ql[1], qr[1]) + cmax;
  const Pair rdl = (sl - ql[1]) * ql[0], rdr = (sr - qr[1]) * qr[0];
  const Pair iden = rcp2(rdr - rdl);
  const Pair du = qr[1] - ql[1], ndp = ptl - ptr;
  const Pair sml = fma2(rdr, du, ndp) * iden, smr = fma2(rdl, du, ndp) * iden;
  const Pair sm = ql[1] + sml;
  const Pred sup_l = sl > 0.0f, sup_r = sr < 0.0f, sup = sup_l || sup_r;
  const Pred left = sup_l || (!sup_r && sm >= 0.0f);
  Pair rs[2], vs[2], ws[2], bts[2], bus[2], iss[2];
  Pred degen[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const Pair* p = a == 0 ? ql : qr;
    const Pair d = a == 0 ? sml : smr, rd = a == 0 ? rdl : rdr;
    const Pair ssm = (a == 0 ? sl : sr) - sm;
    iss[a] = rcp2(ssm);
    rs[a] = fma2(p[0] * d, iss[a], p[0]);
    const Pair rds = rd * ssm;
    const Pair ed = rds - bn2;
    degen[a] = abs2(ed) <= eps * (abs2(rds) + bn2);
    const Pair die = sel(degen[a], pair(0.0f), d * rcp2(ed));
    const Pair ntq = nbn * die, kq = rd * die;
    vs[a] = fma2(p[5], ntq, p[2]);
    ws[a] = fma2(p[6], ntq, p[3]);
    bts[a] = fma2(p[5], kq, p[5]);
    bus[a] = fma2(p[6], kq, p[6]);
  }
  Pair r = sel(left, ql[0], qr[0]), un = sel(left, ql[1], qr[1]), ut = sel(left, ql[2], qr[2]),
       uu = sel(left, ql[3], qr[3]);
  Pair pt = sel(left, ptl, ptr), bt = sel(left, ql[5], qr[5]), bu = sel(left, ql[6], qr[6]);
  const Pair h = pair(0.5f);
  Pair e = fma2(h, sel(left, b2l, b2r), fma2(h * r, fma2(uu, uu, fma2(ut, ut, un * un)), sel(left, ql[4], qr[4]) * pair(igm1)));
  Pair vb = fma2(uu, bu, fma2(ut, bt, un * bn));
  // star state of the side
  const Pair d = sel(left, sml, smr), dpt = sel(left, rdl, rdr) * d;
  const Pair r1 = sel(left, rs[0], rs[1]);
  Pair v1 = sel(left, vs[0], vs[1]), w1 = sel(left, ws[0], ws[1]);
  Pair bt1 = sel(left, bts[0], bts[1]), bu1 = sel(left, bus[0], bus[1]);
  const Pair vb0 = fma2(w1, bu1, fma2(v1, bt1, sm * bn));
  Pair e1 = fma2(fma2(bn, vb - vb0, fma2(dpt, sm, d * (e + pt))), sel(left, iss[0], iss[1]), e);
  const Pair pt1 = pt + dpt;
  Pair vb1 = vb0;
  // double star
  const Pair il = rsqrt2(rs[0]), ir = rsqrt2(rs[1]);
  const Pair c = abs2(bn) * sel(left, il, ir);
  const Pair zl = sm - c, zr = sm + c;
  const Pred in = {left.x ? zl.x >= 0.0f : zr.x <= 0.0f, left.y ? zl.y >= 0.0f : zr.y <= 0.0f};
  const Pred dbl = !(bn2 <= eps * pt1 || in);
  const Pair sql = rs[0] * il, sqr = rs[1] * ir;
  const Pair sgn = {bn.x > 0.0f ? 1.0f : -1.0f, bn.y > 0.0f ? 1.0f : -1.0f};
  const Pair idn = rcp2(sql + sqr);
  const Pair other = sel(left, sqr, -sql), own = sel(left, sql, -sqr) * sgn;
  const Pair z0 = pair(0.0f);
  const Pair dv = sel(dbl, fma2(other, vs[1] - vs[0], sgn * (bts[1] - bts[0])) * idn, z0);
  const Pair dw = sel(dbl, fma2(other, ws[1] - ws[0], sgn * (bus[1] - bus[0])) * idn, z0);
  v1 = v1 + dv;
  w1 = w1 + dw;
  bt1 = fma2(own, dv, bt1);
  bu1 = fma2(own, dw, bu1);
  vb1 = fma2(w1, bu1, fma2(v1, bt1, sm * bn));
  e1 = fma2(own, vb1 - vb0, e1);
  // the state on the face
  r = sel(sup, r, r1);
  un = sel(sup, un, sm);
  ut = sel(sup, ut, v1);
  uu = sel(sup, uu, w1);
  pt = sel(sup, pt, pt1);
  bt = sel(sup, bt, bt1);
  bu = sel(sup, bu, bu1);
  e = sel(sup, e, e1);
  vb = sel(sup, vb, vb1);
  const Pair ru = r * un;
  f[0] = ru;
  f[1] = fma2(ru, un, pt) - bn2;
  f[2] = fma2(nbn, bt, ru * ut);
  f[3] = fma2(nbn, bu, ru * uu);
  f[4] = fma2(nbn, vb, (e + pt) * un);
  f[5] = fma2(nbn, ut, bt * un);
  f[6] = fma2(nbn, uu, bu * un);
}

}  // namespace amrdev
