// mhd_riemann_vjp.cuh -- reverse-mode derivative of the face solve (riemann<RS> in mhd_device.cuh)
// for the adjoint of the step.
//
// For weights (lf, lap, lam, lus) the scalar g = sum_v lf[v] F[v] + lap alpha+ + lam alpha- +
// lus u* of one face is differentiated with respect to the 15 inputs (left and right face states
// and the normal field) in one reverse sweep. The forward values that decide a branch are recomputed
// with the same device functions (phys_speed, phys_flux, star_state) and the same roundings: the
// forward kernels are compiled without contraction, this file's with it, so a product that enters
// a sum on the way to a decision is a mul_rn here. Every branch -- the max/min of the wave speeds,
// the HLLD fan region, the side of the contact, the degenerate star state, the clamped discriminant
// -- is then the one the forward step took, also where two meet to rounding (a head-on collision of
// equal gases), and the derivative is the one of that branch (ties and zero square roots as in the
// forward-mode dual numbers). Each reverse statement is
// the transpose of one forward statement, in reverse order.
#pragma once
#include "mhd_device.cuh"

namespace mhd {

// adjoint of cf2 = A / (2 rho) of a state (phys_speed): accumulates into ds (rho and p) and dbn2, and
// returns the adjoint of its b2
__device__ __forceinline__ double speed_rev(const FaceState& s, double bn2, double b2, double A, double gam,
                                            double dcf2, FaceState& ds, double& dbn2) {
  const double P = gam * s.p;
  const double Sp = P + b2;
  const double disc0 = fma(Sp, Sp, -(times4(bn2) * P));
  const bool keep = gt0(disc0);  // (pmax(disc, 0); the square root's derivative at 0 is taken as 0)
  const double r = rcp(s.rho);
  double dSp = halve(dcf2) * r;  // A = Sp + sqrt(disc)
  ds.rho -= dSp * A * r;
  const double q = halve(rsqrt_(keep ? disc0 : 1.0)) * dSp;
  const double ddisc = keep ? q : 0.0;
  dSp = fma(2.0 * Sp, ddisc, dSp);
  const double d4 = -4.0 * ddisc;
  dbn2 = fma(P, d4, dbn2);
  ds.p = fma(gam, fma(bn2, d4, dSp), ds.p);
  return dSp;
}
// adjoint of b2 and pt of a state: accumulates into ds and dbn2
__device__ __forceinline__ void pt_rev(const FaceState& s, double db2, double dpt, FaceState& ds, double& dbn2) {
  const double t = fma(0.5, dpt, db2);
  ds.p += dpt;
  ds.by = fma(2.0 * s.by, t, ds.by);
  ds.bz = fma(2.0 * s.bz, t, ds.bz);
  dbn2 += t;
}

// adjoint of phys_flux (U, F, e of a state, given its b2 and pt): dU, dF, de in; accumulates
// into ds, dbn, db2, dpt
__device__ __forceinline__ void phys_flux_rev(const FaceState& s, double bn, double gm1inv, const PhysFlux& o,
                                              const double* dU, const double* dF, double de_extra, FaceState& ds,
                                              double& dbn, double& db2, double& dpt) {
  const double u2 = fma(s.u, s.u, fma(s.v, s.v, s.w * s.w));
  const double ub = fma(s.u, bn, fma(s.v, s.by, s.w * s.bz));
  const double mu = s.rho * s.u;
  const double e = o.e;
  double dmu = dU[1] + dF[0] + dF[1] * s.u + dF[2] * s.v + dF[3] * s.w;
  ds.rho += dU[0] + dU[2] * s.v + dU[3] * s.w;
  ds.v += dU[2] * s.rho + dF[2] * mu;
  ds.w += dU[3] * s.rho + dF[3] * mu;
  const double de = dU[4] + dF[4] * s.u + de_extra;
  ds.u += dF[1] * mu + dF[4] * (e + o.pt);
  dpt += dF[1] + dF[4] * s.u;
  double dbn2 = -dF[1];
  dbn += -dF[2] * s.by - dF[3] * s.bz - dF[4] * ub;
  ds.by -= dF[2] * bn;
  ds.bz -= dF[3] * bn;
  const double dub = -dF[4] * bn;
  ds.u += dub * bn;
  dbn += dub * s.u;
  ds.v += dub * s.by;
  ds.by += dub * s.v;
  ds.w += dub * s.bz;
  ds.bz += dub * s.w;
  ds.p += de * gm1inv;
  ds.rho += de * 0.5 * u2;
  const double du2 = de * 0.5 * s.rho;
  db2 += de * 0.5;
  ds.u += 2.0 * s.u * du2;
  ds.v += 2.0 * s.v * du2;
  ds.w += 2.0 * s.w * du2;
  ds.rho += dmu * s.u;
  ds.u += dmu * s.rho;
  dbn += 2.0 * bn * dbn2;
}

// adjoints of a star state's outputs
struct StarAdj {
  double rs, vs, ws, bys, bzs;
};

// adjoint of star_state(q, m, su, d, ssm, bn, bn2) with outputs o and ssminv (es: the energy
// formed with ssminv, des its adjoint; 0 where it is not formed): accumulates into dq (tangential
// components), dm, dsu, dd, dssm, dbn, dbn2
__device__ __forceinline__ void star_state_rev(const FaceState& q, double m, double su, double d, double ssm,
                                               double bn, double bn2, double ssminv, const StarT<double>& o,
                                               const StarAdj& g, double es, double des, FaceState& dq, double& dm,
                                               double& dsu, double& dd, double& dssm, double& dbn, double& dbn2) {
  // rs = m ssminv, es = X ssminv, ssminv = 1 / ssm
  dm += g.rs * ssminv;
  dssm -= fma(g.rs, o.rs, des * es) * ssminv;
  const double den = fma(m, ssm, -bn2);
  if (!star_regular(den, m, su, bn2)) {
    dq.v += g.vs;
    dq.w += g.ws;
    dq.by += g.bys;
    dq.bz += g.bzs;
    return;
  }
  const double r = rcp(den);
  const double cv = bn * d * r;
  const double cb = fma(m, su, -bn2) * r;
  // vs = v - by cv, ws = w - bz cv, bys = by cb, bzs = bz cb
  dq.v += g.vs;
  dq.w += g.ws;
  dq.by += fma(g.bys, cb, -(g.vs * cv));
  dq.bz += fma(g.bzs, cb, -(g.ws * cv));
  const double dcv = -fma(g.vs, q.by, g.ws * q.bz);
  const double dcb = fma(g.bys, q.by, g.bzs * q.bz);
  // cb = (m su - bn2) r, cv = bn d r, r = 1 / den
  const double dnum = dcb * r;
  const double t = dcv * r;
  dbn += t * d;
  dd += t * bn;
  const double dden = -fma(dcb, cb, dcv * cv) * r;
  dm += fma(dnum, su, dden * ssm);
  dsu += dnum * m;
  dssm += dden * m;
  dbn2 -= dnum + dden;
}

// Reverse sweep of hlld(), in terms of the side `a` whose state the face takes and the other side
// `o` (left: a is the left one), so that no operation is doubled for the two choices: with
// du = u_o - u_a and dp = pt_a - pt_o, S_M = u_a + d and d = (m_o du + dp) / (m_o - m_a) for both.
// Like hlld it has one flux formula, that of the state at x/t = 0, whose reverse all lanes take
// together; inside the fan the reverse of the double-star and star states follows.
struct HlldAdj {
  bool left;
  FaceState qa, qo;             // adjoints of the two states (o: 0 outside the fan)
  double pta, pto, b2a, Sa, So;  // of pt, b2 and the outer wave speeds
};
__device__ __forceinline__ void hlld_rev(const FaceState& sl, const FaceState& sr, double bn, double bn2,
                                         double gm1inv, const PhysFlux& L, const PhysFlux& R, double SL, double SR,
                                         const double* dF, HlldAdj& G, double& dbn, double& dbn2) {
  // ---- forward values (as in hlld) ----
  const bool supL = gt0(SL);
  const bool fan = !supL && !lt0(SR);
  double suL = 0.0, suR = 0.0, mL = 0.0, mR = 0.0, du = 0.0, dpt = 0.0, nL = 0.0, dinv = 0.0, SM = 0.0;
  if (fan) {
    suL = SL - sl.u;
    suR = SR - sr.u;
    mL = mul_rn(suL, sl.rho);
    mR = mul_rn(suR, sr.rho);
    dinv = rcp(mR - mL);
    du = sr.u - sl.u;
    dpt = L.pt - R.pt;
    nL = fma(mR, du, dpt);
    SM = fma(nL, dinv, sl.u);
  }
  const bool left = fan ? ge0(SM) : supL;
  const FaceState q = pick(left, sl, sr);
  const double b2 = left ? L.b2 : R.b2;
  const double qpt = left ? L.pt : R.pt;
  const double u2 = fma(q.u, q.u, fma(q.v, q.v, q.w * q.w));
  const double qe = fma(q.p, gm1inv, halve(fma(q.rho, u2, b2)));
  const double qub = fma(q.u, bn, fma(q.v, q.by, q.w * q.bz));
  double rho = q.rho, un = q.u, v = q.v, w = q.w, by = q.by, bz = q.bz, pt = qpt, e = qe, ub = qub;
  double su = 0.0, m = 0.0, nS = 0.0, d = 0.0, ssm = 0.0, ssminv = 0.0, vbs = 0.0, es = 0.0;
  StarT<double> a = {0, 0, 0, 0, 0};
  // the double-star state's pieces
  bool dstar = false;
  FaceState qo = {0, 0, 0, 0, 0, 0, 0};
  double suo = 0.0, mo = 0.0, d_o = 0.0, ssmo = 0.0, oinv = 0.0, isq = 0.0, isqo = 0.0, sqo = 0.0, inv = 0.0;
  double xv = 0.0, xw = 0.0, ssq = 0.0;
  bool neg = false;
  StarT<double> o = {0, 0, 0, 0, 0};
  if (fan) {
    su = left ? suL : suR;
    m = left ? mL : mR;
    nS = left ? nL : fma(mL, du, dpt);
    d = mul_rn(nS, dinv);
    pt = fma(m, d, qpt);
    ssm = su - d;
    star_state(q, m, su, d, ssm, bn, bn2, ssminv, a);
    vbs = fma(SM, bn, fma(a.vs, a.bys, a.ws * a.bzs));
    es = fma(bn, qub - vbs, fma(pt, SM, fma(su, qe, -(qpt * q.u)))) * ssminv;
    rho = a.rs;
    un = SM;
    v = a.vs;
    w = a.ws;
    by = a.bys;
    bz = a.bzs;
    e = es;
    ub = vbs;
    dstar = hlld_in_rotational(left, SM, a.rs, bn2);
    if (dstar) {
      qo = pick(!left, sl, sr);
      suo = left ? suR : suL;
      mo = left ? mR : mL;
      d_o = SM - qo.u;
      ssmo = suo - d_o;
      star_state(qo, mo, suo, d_o, ssmo, bn, bn2, oinv, o);
      isq = rsqrt_(a.rs);
      isqo = rsqrt_(o.rs);
      const double sq = a.rs * isq;
      sqo = o.rs * isqo;
      inv = rcp(sq + sqo);
      neg = lt0(bn) == left;
      xv = fma(sqo, o.vs - a.vs, neg_if(neg, o.bys - a.bys)) * inv;
      xw = fma(sqo, o.ws - a.ws, neg_if(neg, o.bzs - a.bzs)) * inv;
      ssq = neg_if(neg, sq);
      v = a.vs + xv;
      w = a.ws + xw;
      by = fma(ssq, xv, a.bys);
      bz = fma(ssq, xw, a.bzs);
      ub = fma(SM, bn, fma(v, by, w * bz));
      e = fma(ssq, ub - vbs, es);
    }
  }
  // ---- reverse of the flux of the state at x/t = 0 ----
  const double mu = rho * un;
  const double dmu = fma(dF[1], un, fma(dF[2], v, fma(dF[3], w, dF[0])));
  double drho = dmu * un;
  double dun = fma(dmu, rho, fma(dF[1], mu, dF[4] * (e + pt)));
  double dP = fma(dF[4], un, dF[1]);
  dbn2 -= dF[1];
  double dv = dF[2] * mu, dw = dF[3] * mu;
  dbn -= fma(dF[2], by, fma(dF[3], bz, dF[4] * ub));
  double dby = -(dF[2] * bn), dbz = -(dF[3] * bn);
  double de = dF[4] * un, dub = -(dF[4] * bn);
  FaceState dq = {0, 0, 0, 0, 0, 0, 0}, dqo = {0, 0, 0, 0, 0, 0, 0};
  double dqpt = dP;
  G.pto = G.Sa = G.So = 0.0;
  if (fan) {
    // so far dP is the adjoint of p_t*, dun that of S_M, drho that of rho_a*
    double dSM = dun, dvbs = dub, dsu = 0.0, dm = 0.0, dd = 0.0, dssm = 0.0;
    StarAdj da = {drho, dv, dw, dby, dbz};
    double dmo = 0.0, dsuo = 0.0;
    if (dstar) {
      // e = es + ssq (ub - vbs)
      double dssq = de * (ub - vbs);
      dub = fma(de, ssq, dub);
      dvbs = -(de * ssq);
      // ub = SM bn + v by + w bz
      dSM = fma(dub, bn, dSM);
      dbn = fma(dub, SM, dbn);
      dv = fma(dub, by, dv);
      dby = fma(dub, v, dby);
      dw = fma(dub, bz, dw);
      dbz = fma(dub, w, dbz);
      // by = bys + ssq xv, v = vs + xv (and z)
      dssq = fma(dby, xv, fma(dbz, xw, dssq));
      const double dxv = fma(dby, ssq, dv), dxw = fma(dbz, ssq, dw);
      // xv = (sqo (vs_o - vs_a) + s (bys_o - bys_a)) inv, inv = 1 / (sq + sqo)
      const double dnv = dxv * inv, dnw = dxw * inv;
      const double dsum = -fma(dnv, xv, dnw * xw);
      const double dsqo = fma(dnv, o.vs - a.vs, fma(dnw, o.ws - a.ws, dsum));
      const double dsq = dsum + neg_if(neg, dssq);
      const double gv = dnv * sqo, gw = dnw * sqo, gy = neg_if(neg, dnv), gz = neg_if(neg, dnw);
      // sqrt(rs): derivative 1 / (2 sqrt(rs))
      const StarAdj dob = {0.5 * isqo * dsqo, gv, gw, gy, gz};
      da.rs = fma(0.5 * isq, dsq, da.rs);
      da.vs = dv - gv;
      da.ws = dw - gw;
      da.bys = dby - gy;
      da.bzs = dbz - gz;
      double ddo = 0.0, dssmo = 0.0;
      star_state_rev(qo, mo, suo, d_o, ssmo, bn, bn2, oinv, o, dob, 0.0, 0.0, dqo, dmo, dsuo, ddo, dssmo, dbn, dbn2);
      // ssmo = suo - d_o, d_o = SM - u_o
      dsuo += dssmo;
      ddo -= dssmo;
      dSM += ddo;
      dqo.u -= ddo;
    }
    // es = (bn (ub_q - vbs) + p_t* SM + su e_q - pt_q u_q) ssminv
    const double des = de;
    const double dX = des * ssminv;
    dbn = fma(dX, qub - vbs, dbn);
    dub = dX * bn;  // of u . b of the side
    dvbs -= dub;
    dP = fma(dX, SM, dP);
    dSM = fma(dX, pt, dSM);
    dsu = dX * qe;
    de = dX * su;   // of the side's energy
    dqpt = -(dX * q.u);
    dq.u -= dX * qpt;
    // vbs = SM bn + vs bys + ws bzs
    dSM = fma(dvbs, bn, dSM);
    dbn = fma(dvbs, SM, dbn);
    da.vs = fma(dvbs, a.bys, da.vs);
    da.bys = fma(dvbs, a.vs, da.bys);
    da.ws = fma(dvbs, a.bzs, da.ws);
    da.bzs = fma(dvbs, a.ws, da.bzs);
    star_state_rev(q, m, su, d, ssm, bn, bn2, ssminv, a, da, es, des, dq, dm, dsu, dd, dssm, dbn, dbn2);
    // ssm = su - d, p_t* = pt + m d, S_M = u_a + d
    dsu += dssm;
    dd = fma(dP, m, dd - dssm) + dSM;
    dm = fma(dP, d, dm);
    dqpt += dP;
    // d = (m_o du + dp) / (m_o - m_a)
    const double dn = dd * (left ? dinv : neg_if(true, dinv)), dD = dn * d;
    const double mot = left ? mR : mL, suot = left ? suR : suL;
    const FaceState qt = pick(!left, sl, sr);
    dmo += fma(dn, left ? du : neg_if(true, du), -dD);
    dm += dD;
    const double ddu = dn * mot;
    dqpt += dn;
    G.pto = -dn;
    // m = su rho, su = S - u on both sides
    G.Sa = fma(dm, q.rho, dsu);
    dq.rho = fma(dm, su, dq.rho);
    dq.u += dSM - ddu - G.Sa;
    G.So = fma(dmo, qt.rho, dsuo);
    dqo.rho = fma(dmo, suot, dqo.rho);
    dqo.u += ddu - G.So;
  } else {
    dq.rho = drho;
    dq.u = dun;
    dq.v = dv;
    dq.w = dw;
    dq.by = dby;
    dq.bz = dbz;
  }
  // ---- reverse of the side's energy and u . b ----
  const double deh = halve(de), dru = de * q.rho;
  dq.p = de * gm1inv;
  dq.rho = fma(deh, u2, dq.rho);
  dq.u = fma(dub, bn, fma(dru, q.u, dq.u));
  dq.v = fma(dub, q.by, fma(dru, q.v, dq.v));
  dq.w = fma(dub, q.bz, fma(dru, q.w, dq.w));
  dq.by = fma(dub, q.v, dq.by);
  dq.bz = fma(dub, q.w, dq.bz);
  dbn = fma(dub, q.u, dbn);
  G.left = left;
  G.qa = dq;
  G.qo = dqo;
  G.pta = dqpt;
  G.b2a = deh;
}

// Gradient of g = sum_v lf[v] F[v] + lap ap + lam am + lus u* of riemann<RS>(sl, sr, bn) in
// (sl, sr, bn), written into dsl, dsr, dbn.
template <int RS>
__device__ __forceinline__ void riemann_vjp(const FaceState& sl, const FaceState& sr, double bn, double gam,
                                            double gm1inv, const double* lf, double lap, double lam, double lus,
                                            FaceState& dsl, FaceState& dsr, double& dbn) {
  dbn = 0.0;
  const double bn2 = bn * bn;
  double dbn2 = 0.0;
  // ---- forward (as in riemann) ----
  PhysFlux L, R;
  double SL = 0.0, SR = 0.0, ap, am, icmax = 0.0;
  bool llf_left = true, cmax_left = true, umax_left = true, umin_left = true, ap_pos = true, am_pos = true;
  if (RS == RS_LLF) {
    phys_speed(sl, bn, gam, L);
    phys_speed(sr, bn, gam, R);
    const double aL = vabs(sl.u) + sqrt_(L.cf2), aR = vabs(sr.u) + sqrt_(R.cf2);
    llf_left = dbits(aL) >= dbits(aR);
    ap = am = llf_left ? aL : aR;
  } else {
    phys_speed_a(sl, bn2, gam, L);
    phys_speed_a(sr, bn2, gam, R);
    bool plain;
    double ah, x, cmax;
    cmax_left = fast_left(sl, sr, L, R, ah, x, plain);
    // fast_max, and 1 / c from the same reciprocal root (0 where c is 0)
    if (plain) {
      const double y = rsqrt_(x);
      cmax = mul_rn(vabs(ah), y);
      icmax = vabs(cmax_left ? sl.rho : sr.rho) * y;
    } else {
      cmax = fast_max_any(sl.rho, sr.rho, L.A, R.A, cmax_left);
      icmax = is_zero(cmax) ? 0.0 : rcp(cmax);
    }
    umax_left = okey(sl.u) >= okey(sr.u);
    umin_left = okey(sl.u) <= okey(sr.u);
    const double umax = umax_left ? sl.u : sr.u, umin = umin_left ? sl.u : sr.u;
    SR = umax + cmax;
    SL = umin - cmax;
    ap_pos = !(okey(0.0) >= okey(SR));  // vmax(0, SR) picks SR
    am_pos = !((unsigned long long)dbits(SL) <= 0x7ff0000000000000ULL);
    ap = ap_pos ? SR : 0.0;
    am = am_pos ? neg_if(dbits(SL) < 0, SL) : 0.0;
  }
  const double sum = ap + am;
  const bool zero = is_zero(sum);
  const double inv = zero ? 0.0 : rcp(sum);

  // ---- reverse ----
  double dap = lap, dam = lam;
  double dLb2 = 0.0, dLpt = 0.0, dRb2 = 0.0, dRpt = 0.0;
  double dSL = 0.0, dSR = 0.0;
  if (RS == RS_HLLD) {
    HlldAdj G;
    hlld_rev(sl, sr, bn, bn2, gm1inv, L, R, SL, SR, lf, G, dbn, dbn2);
    const bool l = G.left;
    dsl = pick(l, G.qa, G.qo);
    dsr = pick(l, G.qo, G.qa);
    dLpt = l ? G.pta : G.pto;
    dRpt = l ? G.pto : G.pta;
    dLb2 = l ? G.b2a : 0.0;
    dRb2 = l ? 0.0 : G.b2a;
    dSL = l ? G.Sa : G.So;
    dSR = l ? G.So : G.Sa;
  } else {
    dsl = {0, 0, 0, 0, 0, 0, 0};
    dsr = {0, 0, 0, 0, 0, 0, 0};
    phys_flux(sl, bn, gm1inv, L);
    phys_flux(sr, bn, gm1inv, R);
    double dUL[5], dFL[5], dUR[5], dFR[5];
    if (zero) {
      for (int v = 0; v < 5; ++v) { dFL[v] = lf[v]; dUL[v] = 0.0; dFR[v] = 0.0; dUR[v] = 0.0; }
    } else {
      // F = wl FL + wr FR - wd (UR - UL), wl = ap inv, wr = am inv, wd = ap am inv
      const double wl = ap * inv, wr = am * inv, wd = ap * am * inv;
      double dwl = 0.0, dwr = 0.0, dwd = 0.0;
      for (int v = 0; v < 5; ++v) {
        dwl += lf[v] * L.F[v];
        dwr += lf[v] * R.F[v];
        dwd -= lf[v] * (R.U[v] - L.U[v]);
        dFL[v] = lf[v] * wl;
        dFR[v] = lf[v] * wr;
        dUR[v] = -lf[v] * wd;
        dUL[v] = lf[v] * wd;
      }
      dap += dwl * inv + dwd * am * inv;
      dam += dwr * inv + dwd * ap * inv;
      const double dinv = dwl * ap + dwr * am + dwd * ap * am;
      const double ds = -dinv * inv * inv;
      dap += ds;
      dam += ds;
    }
    phys_flux_rev(sl, bn, gm1inv, L, dUL, dFL, 0.0, dsl, dbn, dLb2, dLpt);
    phys_flux_rev(sr, bn, gm1inv, R, dUR, dFR, 0.0, dsr, dbn, dRb2, dRpt);
  }
  // u* = (ap uL + am uR) inv, or uL when ap + am = 0
  if (zero) {
    dsl.u += lus;
  } else {
    const double dn = lus * inv;
    const double ds = -(dn * fma(ap, sl.u, am * sr.u)) * inv;
    dap += fma(dn, sl.u, ds);
    dsl.u = fma(dn, ap, dsl.u);
    dam += fma(dn, sr.u, ds);
    dsr.u = fma(dn, am, dsr.u);
  }
  // wave speeds
  if (RS == RS_LLF) {
    const double da = dap + dam;
    const double du = neg_if(dbits(llf_left ? sl.u : sr.u) < 0, da);
    dsl.u += llf_left ? du : 0.0;
    dsr.u += llf_left ? 0.0 : du;
    // c = sqrt(cf2): derivative rsqrt / 2, taken as 0 at 0
    const FaceState& q = llf_left ? sl : sr;
    FaceState dq = {0, 0, 0, 0, 0, 0, 0};
    const double cf2 = llf_left ? L.cf2 : R.cf2;
    const double dcf2 = is_zero(cf2) ? 0.0 : 0.5 * rsqrt_(cf2) * da;
    const double db2 = speed_rev(q, bn2, llf_left ? L.b2 : R.b2, llf_left ? L.A : R.A, gam, dcf2, dq, dbn2);
    (llf_left ? dLb2 : dRb2) += db2;
    (llf_left ? dsl : dsr).rho += dq.rho;
    (llf_left ? dsl : dsr).p += dq.p;
  } else {
    // ap = max(0, SR), am = max(0, -SL), SR = umax + cmax, SL = umin - cmax
    dSR += ap_pos ? dap : 0.0;
    dSL -= am_pos ? dam : 0.0;
    dsl.u += (umax_left ? dSR : 0.0) + (umin_left ? dSL : 0.0);
    dsr.u += (umax_left ? 0.0 : dSR) + (umin_left ? 0.0 : dSL);
    // the larger speed's side only: dcf2 = dc / (2 c)
    const FaceState q = pick(cmax_left, sl, sr);
    FaceState dq = {0, 0, 0, 0, 0, 0, 0};
    const double db2 = speed_rev(q, bn2, cmax_left ? L.b2 : R.b2, cmax_left ? L.A : R.A, gam,
                                 halve(icmax) * (dSR - dSL), dq, dbn2);
    dLb2 += cmax_left ? db2 : 0.0;
    dRb2 += cmax_left ? 0.0 : db2;
    dsl.rho += cmax_left ? dq.rho : 0.0;
    dsr.rho += cmax_left ? 0.0 : dq.rho;
    dsl.p += cmax_left ? dq.p : 0.0;
    dsr.p += cmax_left ? 0.0 : dq.p;
  }
  pt_rev(sl, dLb2, dLpt, dsl, dbn2);
  pt_rev(sr, dRb2, dRpt, dsr, dbn2);
  dbn = fma(2.0 * bn, dbn2, dbn);
}

}  // namespace mhd
