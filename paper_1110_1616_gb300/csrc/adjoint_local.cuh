// Hand-written reverse mode of the costliest pointwise formulas of the
// advance: the HLLD flux (hlld_flux), the half-step primitive predictor
// (prim_terms summed over directions) and the recovery. Each function returns the exact
// transposed Jacobian-vector product of the formula in the compute type R
// (double: the FP64 forward; float: the FP32 stencil of the mixed-precision
// forward, with its own degenerate-state threshold), taking the branch the
// forward takes (wave-speed selection, supersonic, degenerate and
// double-star cases); it recomputes the forward's intermediates that decide a
// branch in the operation order of the formula as written. Included by
// adjoint.cu, which is compiled without FMA contraction, like the strict FP64
// forward: there every decision is the forward's. The FP32 forward contracts
// products into FMAs and divides approximately, so a float decision within a few
// roundings of its boundary, where the two regions' fluxes differ by as much,
// can be the other one. The adjoint's own sums contract by hand (Fm below).
#pragma once
#include <type_traits>

#include "mhd_device.cuh"

namespace amrdev {

// ------------------------------------------------------------------ contraction
// The adjoint's own sums contract into FMAs although the file is compiled
// without (the forward's values that decide its branches must round as the
// forward rounds them): a product with an adjoint value stays open (Pr) until
// it meets an addition. FP64 instructions bound these kernels.
template <class R> struct Pr { R a, b; };
template <class R> struct Fm {
  R v;
  __device__ __forceinline__ Fm() {}
  __device__ __forceinline__ Fm(R x) : v(x) {}
  __device__ __forceinline__ Fm(const Pr<R>& p) : v(p.a * p.b) {}
  friend __device__ __forceinline__ Pr<R> operator*(R a, const Fm& b) { return {a, b.v}; }
  friend __device__ __forceinline__ Pr<R> operator*(const Fm& a, R b) { return {a.v, b}; }
  friend __device__ __forceinline__ Pr<R> operator*(const Fm& a, const Fm& b) { return {a.v, b.v}; }
  friend __device__ __forceinline__ Fm operator+(const Fm& a, const Fm& b) { return a.v + b.v; }
  friend __device__ __forceinline__ Fm operator-(const Fm& a, const Fm& b) { return a.v - b.v; }
  friend __device__ __forceinline__ Fm operator-(const Fm& a) { return -a.v; }
  friend __device__ __forceinline__ Fm operator+(const Fm& a, const Pr<R>& p) { return fma(p.a, p.b, a.v); }
  friend __device__ __forceinline__ Fm operator+(const Pr<R>& p, const Fm& a) { return fma(p.a, p.b, a.v); }
  friend __device__ __forceinline__ Fm operator-(const Fm& a, const Pr<R>& p) { return fma(-p.a, p.b, a.v); }
  friend __device__ __forceinline__ Fm operator-(const Pr<R>& p, const Fm& a) { return fma(p.a, p.b, -a.v); }
  __device__ __forceinline__ Fm& operator+=(const Fm& b) { v = v + b.v; return *this; }
  __device__ __forceinline__ Fm& operator-=(const Fm& b) { v = v - b.v; return *this; }
  __device__ __forceinline__ Fm& operator+=(const Pr<R>& p) { v = fma(p.a, p.b, v); return *this; }
  __device__ __forceinline__ Fm& operator-=(const Pr<R>& p) { v = fma(-p.a, p.b, v); return *this; }
};
template <class R> __device__ __forceinline__ Fm<R> operator+(const Pr<R>& p, const Pr<R>& q) {
  return fma(p.a, p.b, q.a * q.b);
}
template <class R> __device__ __forceinline__ Fm<R> operator-(const Pr<R>& p, const Pr<R>& q) {
  return fma(p.a, p.b, -(q.a * q.b));
}
template <class R> __device__ __forceinline__ Fm<R> pick(bool c, const Fm<R>& a, const Fm<R>& b) {
  return Fm<R>(c ? a.v : b.v);
}
// sums start at -0, the identity of addition (x + 0 would cost an instruction)
template <class R> __device__ __forceinline__ Fm<R> none() { return Fm<R>(-R(0.0)); }

// fast speed cfast(rho, p, bn, bt, bu): value and transpose
template <class R> struct CFast {
  R irho, gp, b2, a, X, Y, sd, cf;
};
template <class R>
__device__ __forceinline__ CFast<R> cfast_fwd(R rho, R p, R bn, R bt, R bu, R gamma) {
  CFast<R> s;
  s.irho = R(1.0) / rho;
  s.gp = gamma * p;
  s.b2 = bn * bn + bt * bt + bu * bu;
  s.a = (s.gp + s.b2) * s.irho;
  s.X = s.gp * s.irho;
  s.Y = bn * bn * s.irho;
  R disc = s.a * s.a - R(4.0) * s.X * s.Y;
  if (disc < R(0.0)) disc = R(0.0);
  s.sd = sqrt(disc);
  s.cf = sqrt(R(0.5) * (s.a + s.sd));
  return s;
}
// d cf / d (rho, p, bn, bt, bu) * g in g5[0..4]; a discriminant at or clamped to
// zero passes nothing on
template <class R>
__device__ __forceinline__ void cfast_bwd(const CFast<R>& s, R bn, R bt, R bu, R gamma, Fm<R> g, Fm<R>* g5) {
  using F = Fm<R>;
  const F h = g * (R(0.25) / s.cf);  // of a and of sd
  const F gdisc = s.sd == R(0.0) ? F(R(0.0)) : F(h * (R(0.5) / s.sd));
  const F ga = h + (R(2.0) * s.a) * gdisc;
  const F gX = F(-R(4.0) * s.Y * gdisc), gY = F(-R(4.0) * s.X * gdisc);
  const F gi = s.gp * gX + bn * bn * gY + (s.gp + s.b2) * ga;  // of 1 / rho
  g5[0] = F(-(s.irho * s.irho) * gi);
  g5[1] = F(gamma * F(s.irho * (gX + ga)));
  g5[2] = F((R(2.0) * bn * s.irho) * (gY + ga));
  const F k = F(R(2.0) * F(s.irho * ga));
  g5[3] = F(bt * k);
  g5[4] = F(bu * k);
}

// the star state of one side: what its transpose reads
template <class R> struct Star {
  R ie, tq, qq, vs, ws, bts, bus;
  bool degen;
};
template <class R>
__device__ __forceinline__ Star<R> star_fwd(const R* q, R da, R ssm, R sm, R bn, R bn2, R eps) {
  using F = Fm<R>;
  Star<R> z;
  const R rds = q[0] * da * ssm;
  const R e = rds - bn2;
  z.degen = fabs(e) <= eps * (fabs(rds) + bn2);
  if (z.degen) {
    z.vs = q[2]; z.ws = q[3]; z.bts = q[5]; z.bus = q[6];
  } else {
    z.ie = R(1.0) / e;
    z.tq = bn * (sm - q[1]) * z.ie;
    z.qq = (q[0] * da * da - bn2) * z.ie;
    z.vs = (F(q[2]) - q[5] * F(z.tq)).v;
    z.ws = (F(q[3]) - q[6] * F(z.tq)).v;
    z.bts = q[5] * z.qq;
    z.bus = q[6] * z.qq;
  }
  return z;
}
// from the adjoints of (vs, ws, bts, bus, rs = r da / ssm): adds to the state's
// (gq), to those of da, ssm, sm and bn
template <class R>
__device__ __forceinline__ void star_bwd(const Star<R>& z, const R* q, R da, R ssm, R issm, R rs, R sm, R bn,
                                         Fm<R> gvs, Fm<R> gws, Fm<R> gbts, Fm<R> gbus, Fm<R> grs, Fm<R>* gq,
                                         Fm<R>& gda, Fm<R>& gssm, Fm<R>& gsm, Fm<R>& gbn) {
  using F = Fm<R>;
  gq[2] += gvs;
  gq[3] += gws;
  if (z.degen) {
    gq[5] += gbts;
    gq[6] += gbus;
  } else {
    // bts = bt qq, bus = bu qq, vs = ut - bt tq, ws = uu - bu tq
    const F gqq = q[5] * gbts + q[6] * gbus, gtq = -(q[5] * gvs + q[6] * gws);
    gq[5] += z.qq * gbts;
    gq[5] -= z.tq * gvs;
    gq[6] += z.qq * gbus;
    gq[6] -= z.tq * gws;
    // qq = (r da^2 - bn2) ie, tq = bn (sm - un) ie, ie = 1 / e, e = r da ssm - bn2
    const F h = F(z.ie * gqq), k = F(z.ie * gtq);
    const F ge = -(z.qq * h + z.tq * k);
    gq[0] += da * F(da * h + ssm * ge);
    gda += q[0] * F((R(2.0) * da) * h + ssm * ge);
    gssm += (q[0] * da) * ge;
    gbn -= (R(2.0) * bn) * (h + ge);
    gbn += (sm - q[1]) * k;
    gsm += bn * k;
    gq[1] -= bn * k;
  }
  const F m = F(issm * grs);
  gq[0] += da * m;
  gda += q[0] * m;
  gssm -= rs * m;
}

// gx[15] = J^T g of hlld_flux at x = (ql[7], qr[7], bn) (written).
// The flux is built on one side's state and star region (side s; the other is
// o), and the formulas are symmetric under exchanging the sides, so once the
// branch is known the sides are exchanged by selects and one code serves both:
// the energy, the physical flux and the conserved state of o pass nothing on,
// nor do its star fields outside the double-star region. About 560 FP64
// instructions a face where transposing both sides term by term took about 880
// (256^2 in 32^2 patches, and its refined level, a launch: 457 -> 231 us).
template <class R> __device__ void hlld_vjp(const R* x, const R* g, R gamma, R* gx) {
  using F = Fm<R>;
  const R* ql = x;
  const R* qr = x + 7;
  const R bn = x[14];
  const R eps = Eps<R>::v();
  const R igm1 = R(1.0) / (gamma - R(1.0));
  // the forward's wave speeds and branch, in its operation order
  CFast<R> cm;
  bool cmax_l;
  {
    const CFast<R> cL = cfast_fwd(ql[0], ql[4], bn, ql[5], ql[6], gamma);
    const CFast<R> cR = cfast_fwd(qr[0], qr[4], bn, qr[5], qr[6], gamma);
    cmax_l = cL.cf > cR.cf;  // tmaxd(cl, cr)
    cm.irho = cmax_l ? cL.irho : cR.irho;
    cm.gp = cmax_l ? cL.gp : cR.gp;
    cm.b2 = cmax_l ? cL.b2 : cR.b2;
    cm.a = cmax_l ? cL.a : cR.a;
    cm.X = cmax_l ? cL.X : cR.X;
    cm.Y = cmax_l ? cL.Y : cR.Y;
    cm.sd = cmax_l ? cL.sd : cR.sd;
    cm.cf = cmax_l ? cL.cf : cR.cf;
  }
  const bool smin_l = ql[1] < qr[1];  // tmind(uln, urn)
  const bool smax_l = ql[1] > qr[1];  // tmaxd(uln, urn)
  const R sl = (smin_l ? ql[1] : qr[1]) - cm.cf;
  const R sr = (smax_l ? ql[1] : qr[1]) + cm.cf;
  const R bn2 = bn * bn;
  const bool star = !(sl > R(0.0) || sr < R(0.0));
  bool left = sl > R(0.0), dbl = false;
  R sm = 0, pts = 0, den = 0, ptl = 0, ptr = 0, dl = 0, dr = 0, rsl = 0, rsr = 0, sql = 0, sqr = 0, sls = 0, srs = 0;
  if (star) {
    const R rl = ql[0], rr = qr[0], uln = ql[1], urn = qr[1];
    ptl = ql[4] + R(0.5) * (bn2 + ql[5] * ql[5] + ql[6] * ql[6]);
    ptr = qr[4] + R(0.5) * (bn2 + qr[5] * qr[5] + qr[6] * qr[6]);
    dl = sl - uln;
    dr = sr - urn;
    den = dr * rr - dl * rl;
    sm = (dr * rr * urn - dl * rl * uln - ptr + ptl) / den;
    pts = (dr * rr * ptl - dl * rl * ptr + rl * rr * dr * dl * (urn - uln)) / den;
    rsl = rl * dl / (sl - sm);
    rsr = rr * dr / (sr - sm);
    left = sm >= R(0.0);
    if (!(bn2 <= eps * pts)) {
      sql = sqrt(rsl);
      sqr = sqrt(rsr);
      const R abn = fabs(bn);
      sls = sm - abn / sql;
      srs = sm + abn / sqr;
      if (sls >= R(0.0)) left = true;
      else if (srs <= R(0.0)) left = false;
      else dbl = true;
    }
  }
  // side s first
  R q[7], o[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    q[k] = left ? ql[k] : qr[k];
    o[k] = left ? qr[k] : ql[k];
  }
  F gq[7], go[7], gbn, gSs = none<R>(), gSo = none<R>();
#pragma unroll
  for (int k = 0; k < 7; ++k) go[k] = none<R>();
  const F G[7] = {g[0], g[1], g[2], g[3], g[4], g[5], g[6]};
  const R B2 = bn * bn + q[5] * q[5] + q[6] * q[6];
  const R K = q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
  const R pt = q[4] + R(0.5) * B2;
  const R E = q[4] * igm1 + R(0.5) * q[0] * K + R(0.5) * B2;
  const R vb = q[1] * bn + q[2] * q[5] + q[3] * q[6];
  const R S = star ? (left ? sl : sr) : R(0.0);
  const R uS = q[1] - S;  // the flux less S times the conserved state, as the star fluxes hold it
  F gE = F(uS * G[4]), gpt = G[1] + q[1] * G[4], gv = -G[4];  // gv bn: of vb
  // the physical flux of s, and -S times its conserved state
  const F Q = G[0] + q[1] * G[1] + q[2] * G[2] + q[3] * G[3];
  gq[0] = F(uS * Q);
  F gm1 = Q + uS * G[1], gm2 = F(uS * G[2]), gm3 = F(uS * G[3]);  // velocity adjoints over rho
  gq[1] = (E + pt) * G[4] + q[5] * G[5] + q[6] * G[6];
  gq[2] = F(-bn * G[5]);
  gq[3] = F(-bn * G[6]);
  gq[5] = uS * G[5] - bn * G[2];
  gq[6] = uS * G[6] - bn * G[3];
  gbn = -((R(2.0) * bn) * G[1] + q[5] * G[2] + q[6] * G[3] + vb * G[4] + q[2] * G[5] + q[3] * G[6]);
  if (star) {
    const R So = left ? sr : sl;
    const R ds = left ? dl : dr, dn = left ? dr : dl;
    const R pto = left ? ptr : ptl;
    const R rs = left ? rsl : rsr, rso = left ? rsr : rsl;
    const R ssm = S - sm, issm = R(1.0) / ssm;
    const Star<R> z = star_fwd(q, ds, ssm, sm, bn, bn2, eps);
    const R vbs = (sm * F(bn) + z.vs * F(z.bts) + z.ws * F(z.bus)).v;
    const R es = (ds * F(E) - pt * F(q[1]) + pts * F(sm) + bn * F(vb - vbs)).v * issm;
    const R t = dbl ? (left ? sls : srs) : R(0.0);  // f = f_s + t uss + (S - t) us - S u
    const R c = S - t, crs = c * rs;
    gSs = F((rs - q[0]) * G[0]) + (rs * sm - q[0] * q[1]) * G[1] + (rs * z.vs - q[0] * q[2]) * G[2] +
          (rs * z.ws - q[0] * q[3]) * G[3] + (es - E) * G[4] + (z.bts - q[5]) * G[5] + (z.bus - q[6]) * G[6];
    F grs = S * F(G[0] + sm * G[1]) + c * F(z.vs * G[2] + z.ws * G[3]);
    F gsm = F((S * rs) * G[1]), ges = F(S * G[4]);
    F gvs = F(crs * G[2]), gws = F(crs * G[3]), gbts = F(c * G[5]), gbus = F(c * G[6]), gvbs = none<R>();
    if (dbl) {
      const R ls = left ? R(1.0) : -R(1.0);
      const R sp = bn > R(0.0) ? ls : -ls;
      const R sq = left ? sql : sqr, sqo = left ? sqr : sql;
      const R sso = So - sm;
      const Star<R> zo = star_fwd(o, dn, sso, sm, bn, bn2, eps);
      const R idn = R(1.0) / (sq + sqo), isq = R(1.0) / sq;
      const R dv = (zo.vs - z.vs) * sp, dw = (zo.ws - z.ws) * sp, ss2 = sq * sqo;
      const R vss = (sq * F(z.vs) + sqo * F(zo.vs) + sp * F(zo.bts - z.bts)).v * idn;
      const R wss = (sq * F(z.ws) + sqo * F(zo.ws) + sp * F(zo.bus - z.bus)).v * idn;
      const R bts2 = (sq * F(zo.bts) + sqo * F(z.bts) + ss2 * F(dv)).v * idn;
      const R bus2 = (sq * F(zo.bus) + sqo * F(z.bus) + ss2 * F(dw)).v * idn;
      const R vbss = (sm * F(bn) + vss * F(bts2) + wss * F(bus2)).v;
      const R D = (vbs - vbss) * sp;  // ess = es - sq D
      // of t, and of uss = (rs, rs sm, rs vss, rs wss, ess, btss, buss)
      const F gt = rs * F((vss - z.vs) * G[2] + (wss - z.ws) * G[3]) - (sq * D) * G[4] + (bts2 - z.bts) * G[5] +
                   (bus2 - z.bus) * G[6];
      const R trs = t * rs;
      grs += t * F(vss * G[2] + wss * G[3]);
      F gvss = F(trs * G[2]), gwss = F(trs * G[3]), gb2 = F(t * G[5]), gc2 = F(t * G[6]);
      const F gess = F(t * G[4]);
      const F gx2 = F((sq * sp) * gess);  // of vbss, and less of vbs
      gvbs = -gx2;
      gsm += bn * gx2;
      gbn += sm * gx2;
      gvss += bts2 * gx2;
      gb2 += vss * gx2;
      gwss += bus2 * gx2;
      gc2 += wss * gx2;
      const F gi = -F(idn * F(vss * gvss + wss * gwss + bts2 * gb2 + bus2 * gc2));  // of sq + sqo
      const F nv = F(idn * gvss), nw = F(idn * gwss), nb = F(idn * gb2), nc = F(idn * gc2);
      const F X = dv * nb + dw * nc;
      F gsq = gi + z.vs * nv + z.ws * nw + zo.bts * nb + zo.bus * nc + sqo * X - D * gess;
      const F gsqo = gi + zo.vs * nv + zo.ws * nw + z.bts * nb + z.bus * nc + sq * X;
      const R A = ss2 * sp;
      gvs += sq * nv;
      gvs -= A * nb;
      gws += sq * nw;
      gws -= A * nc;
      gbts += sqo * nb;
      gbts -= sp * nv;
      gbus += sqo * nc;
      gbus -= sp * nw;
      // t = sm -/+ |bn| / sq
      gsm += gt;
      const F gti = F(isq * gt);
      gsq += (ls * fabs(bn) * isq) * gti;
      gbn -= (bn == R(0.0) ? R(0.0) : sp) * gti;
      grs += (R(0.5) * isq) * gsq;
      F gda = none<R>(), gssm = none<R>();
      star_bwd(zo, o, dn, sso, R(1.0) / sso, rso, sm, bn, F(sqo * nv + A * nb), F(sqo * nw + A * nc),
               F(sq * nb + sp * nv), F(sq * nc + sp * nw), F((R(0.5) / sqo) * gsqo), go, gda, gssm, gsm, gbn);
      gSo = gssm + gda;
      gsm -= gssm;
      go[1] -= gda;
    }
    // es = (ds E - pt un + pts sm + bn (vb - vbs)) / ssm
    const F gn = F(issm * ges);
    F gssm = F(-es * gn), gda = F(E * gn);
    gE += ds * gn;
    gpt -= q[1] * gn;
    gq[1] -= pt * gn;
    F gpts = F(sm * gn);
    gsm += pts * gn;
    gbn += (vb - vbs) * gn;
    gv += gn;
    gvbs -= bn * gn;
    // vbs = sm bn + vs bts + ws bus
    gsm += bn * gvbs;
    gbn += sm * gvbs;
    gvs += z.bts * gvbs;
    gbts += z.vs * gvbs;
    gws += z.bus * gvbs;
    gbus += z.ws * gvbs;
    star_bwd(z, q, ds, ssm, issm, rs, sm, bn, gvs, gws, gbts, gbus, grs, gq, gda, gssm, gsm, gbn);
    gSs += gssm + gda;
    gsm -= gssm;
    gq[1] -= gda;
    // with the mass fluxes m = d rho: sm = (mo uo - ms us - pto + pt) / (mo - ms),
    // pts = (mo pt - ms pto + ms mo (uo - us)) / (mo - ms)
    const R iden = R(1.0) / (left ? den : -den);
    const R ms = ds * q[0], mo = dn * o[0], du = o[1] - q[1];
    const F a = F(iden * gsm), b = F(iden * gpts);
    const F gden = sm * a + pts * b;  // less
    const F gmo = o[1] * a + (pt + ms * du) * b - gden;
    const F gms = gden - q[1] * a + (mo * du - pto) * b;
    const F mmb = F((ms * mo) * b);
    go[1] += mo * a;
    go[1] += mmb;
    gq[1] -= ms * a;
    gq[1] -= mmb;
    gpt += a + mo * b;
    const F gpto = -(a + ms * b);
    go[4] += gpto;
    gbn += bn * gpto;
    go[5] += o[5] * gpto;
    go[6] += o[6] * gpto;
    const F gdo = F(o[0] * gmo), gds = F(q[0] * gms);
    go[0] += dn * gmo;
    gq[0] += ds * gms;
    gSo += gdo;
    go[1] -= gdo;
    gSs += gds;
    gq[1] -= gds;
  }
  // the energy, pt and vb of s
  const F w = gE + gpt, gvb = F(bn * gv);
  gm1 += q[1] * gE;
  gm2 += q[2] * gE;
  gm3 += q[3] * gE;
  gq[0] += (R(0.5) * K) * gE;
  gq[1] += q[0] * gm1;
  gq[1] += bn * gvb;
  gq[2] += q[0] * gm2;
  gq[2] += q[5] * gvb;
  gq[3] += q[0] * gm3;
  gq[3] += q[6] * gvb;
  gq[4] = gpt + igm1 * gE;
  gq[5] += q[2] * gvb;
  gq[5] += q[5] * w;
  gq[6] += q[3] * gvb;
  gq[6] += q[6] * w;
  gbn += q[1] * gvb;
  gbn += bn * w;
  F gl[7], gr[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    gl[k] = pick(left, gq[k], go[k]);
    gr[k] = pick(left, go[k], gq[k]);
  }
  if (star) {
    // sl = min(uln, urn) - cmax; sr = max(uln, urn) + cmax
    const F gsl = pick(left, gSs, gSo), gsr = pick(left, gSo, gSs);
    gl[1] += pick(smin_l, gsl, none<R>()) + pick(smax_l, gsr, none<R>());
    gr[1] += pick(smin_l, none<R>(), gsl) + pick(smax_l, none<R>(), gsr);
    F g5[5];
    cfast_bwd(cm, bn, cmax_l ? ql[5] : qr[5], cmax_l ? ql[6] : qr[6], gamma, gsr - gsl, g5);
    gbn += g5[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int f = k == 0 ? 0 : 3 + k, c = k < 2 ? k : k + 1;
      const F s = pick(cmax_l, gl[f], gr[f]) + g5[c];
      gl[f] = pick(cmax_l, s, gl[f]);
      gr[f] = pick(cmax_l, gr[f], s);
    }
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    gx[k] = gl[k].v;
    gx[7 + k] = gr[k].v;
  }
  gx[14] = gbn.v;
}

// transpose of dw = A_D(w) s (prim_terms) applied to G: accumulates into gw
// and the adjoint of ir = 1 / rho, writes gs
template <int D, class R>
__device__ __forceinline__ void prim_terms_vjp(const R* w, const R* s, R gamma, R ir, const Fm<R>* G, Fm<R>* gw,
                                               Fm<R>* gs, Fm<R>& gir) {
  using F = Fm<R>;
  constexpr int n = D, t = (D + 1) % 3, u = (D + 2) % 3;
  const R rho = w[0], p = w[4];
  const R vn = w[1 + n];
  const R bn = w[5 + n], bt = w[5 + t], bu = w[5 + u];
  // every component carries vn s_f: d/dvn = s . G, d/ds_f += vn G_f
  F sg = F(s[0] * G[0]);
#pragma unroll
  for (int f = 1; f < 8; ++f) sg += s[f] * G[f];
#pragma unroll
  for (int f = 0; f < 8; ++f) gs[f] = F(vn * G[f]);
  gw[1 + n] += sg;
  // dw0: rho s[1+n]
  gw[0] += s[1 + n] * G[0];
  gs[1 + n] += rho * G[0];
  // dw[1+n]: (s4 + bt s[5+t] + bu s[5+u]) ir
  const F iG = F(ir * G[1 + n]);
  gir += (F(s[4]) + bt * F(s[5 + t]) + bu * F(s[5 + u])).v * G[1 + n];
  gs[4] += iG;
  gs[5 + t] += bt * iG;
  gs[5 + u] += bu * iG;
  gw[5 + t] += s[5 + t] * iG;
  gw[5 + u] += s[5 + u] * iG;
  // dw[1+t], dw[1+u]: - bn s[5+t] ir, - bn s[5+u] ir
  const F sG = s[5 + t] * G[1 + t] + s[5 + u] * G[1 + u];
  const R bi = bn * ir;
  gw[5 + n] -= ir * sG;
  gs[5 + t] -= bi * G[1 + t];
  gs[5 + u] -= bi * G[1 + u];
  gir -= bn * sG;
  // dw4: gamma p s[1+n]
  const F gG = F(gamma * G[4]);
  gw[4] += s[1 + n] * gG;
  gs[1 + n] += p * gG;
  // dw[5+t], dw[5+u]: - bn s[1+t] + bt s[1+n], - bn s[1+u] + bu s[1+n]
  gw[5 + n] -= s[1 + t] * G[5 + t] + s[1 + u] * G[5 + u];
  gs[1 + t] -= bn * G[5 + t];
  gs[1 + u] -= bn * G[5 + u];
  gw[5 + t] += s[1 + n] * G[5 + t];
  gw[5 + u] += s[1 + n] * G[5 + u];
  gs[1 + n] += bt * G[5 + t] + bu * G[5 + u];
}

// gx = J^T g of the half-step predictor wh = w - sum_d h_d A_d(w) s_d at
// x = (w[8], s_0[8], .., s_{DIM-1}[8]); gx has 8 + 8 DIM entries (written)
template <int DIM, class R>
__device__ __forceinline__ void predict_vjp(const R* x, const R* g, R gamma, const R* h, R* gx) {
  using F = Fm<R>;
  const R* w = x;
  const R ir = R(1.0) / w[0];
  F gir = none<R>(), gw[8], gs[8], G[8];
#pragma unroll
  for (int f = 0; f < 8; ++f) gw[f] = F(g[f]);
  const auto dir = [&](auto D) {
    constexpr int d = decltype(D)::value;
#pragma unroll
    for (int f = 0; f < 8; ++f) G[f] = F(-h[d] * g[f]);
    prim_terms_vjp<d>(w, x + 8 + 8 * d, gamma, ir, G, gw, gs, gir);
#pragma unroll
    for (int f = 0; f < 8; ++f) gx[8 + 8 * d + f] = gs[f].v;
  };
  dir(std::integral_constant<int, 0>{});
  dir(std::integral_constant<int, 1>{});
  if constexpr (DIM == 3) dir(std::integral_constant<int, 2>{});
  gw[0] -= (ir * ir) * gir;
#pragma unroll
  for (int f = 0; f < 8; ++f) gx[f] = gw[f].v;
}

// gx[8] = J^T g of the FP64 recovery W(U, B_c) (recover() in mhd_device.cuh): x = (rho,
// m_x, m_y, m_z, E, B_cx, B_cy, B_cz), W = (rho, v, p, B_c), p = gm1 ((E - ke) - me)
__device__ __forceinline__ void recover_vjp(const double* x, const double* g, double gm1, double* gx) {
  const double r = x[0], ir = 1.0 / r;
  const double vx = x[1] * ir, vy = x[2] * ir, vz = x[3] * ir;
  const double gp = g[4];
  const double gke = -gm1 * gp, gme = -gm1 * gp;
  // ke = (m_x vx + m_y vy + m_z vz) / 2; v = m ir
  const double gvx = g[1] + 0.5 * x[1] * gke, gvy = g[2] + 0.5 * x[2] * gke, gvz = g[3] + 0.5 * x[3] * gke;
  const double gir = x[1] * gvx + x[2] * gvy + x[3] * gvz;
  gx[0] = g[0] - ir * ir * gir;
  gx[1] = 0.5 * vx * gke + ir * gvx;
  gx[2] = 0.5 * vy * gke + ir * gvy;
  gx[3] = 0.5 * vz * gke + ir * gvz;
  gx[4] = gm1 * gp;
  // me = |B_c|^2 / 2
  gx[5] = g[5] + x[5] * gme;
  gx[6] = g[6] + x[6] * gme;
  gx[7] = g[7] + x[7] * gme;
}

}  // namespace amrdev
