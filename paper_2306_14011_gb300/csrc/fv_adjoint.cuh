// Reverse mode (vector-Jacobian products) of the face flux and of the MUSCL
// reconstruction, for the discrete adjoint of the residual (paper Eq. (5) with
// the fluxes of Eq. (2) and states of Eq. (6)).
//
// roe_F_vjp recomputes the forward quantities of roe_F_fp64 (fv_device.cuh), with
// its products, reciprocals and roots on the integer pipes: the
// upwind physical flux plus the one acoustic wave that crosses from downwind,
// which equals the central Roe flux (F(QL) + F(QR))/2 - sum |lambda| alpha r/2
// as a function; it propagates a cotangent Gb of F back to the two states,
// line by line in reverse.  Conventions at the non-differentiable points
// follow the forward-mode reference: |x| has derivative sign(x) with
// sign(+0) = +1 (the upwind side of u~_n = +0 is the left one, where the
// contact and shear waves drop out, as sign(+0) = +1 gives), the entropy fix
// applies where |lambda| < delta, and the limited slope minmod(a, b)
// passes the derivative of the argument it returned (b on ties) and none when
// the arguments do not have one strict sign.
#pragma once
#include "fv_device.cuh"

namespace fvk {

// x with the sign of x flipped when s < 0 (or s is -0): x * sign(s), exact, integer pipe.
__device__ __forceinline__ double mul_sign(double x, double s) {
  return __hiloint2double(__double2hiint(x) ^ (__double2hiint(s) & (int)0x80000000u), __double2loint(x));
}

// FX: products, reciprocals and roots run on the integer pipes (fx_mul and its
// kin, fv_roe.h) and bad's sign bit reports an operand or result they do not
// take; the wrapper below then evaluates that lane's face in FP64.
template <int NT, bool FX>
__device__ __forceinline__ void roe_F_vjp_impl(const double (&QL)[NT + 3], const double (&QR)[NT + 3], double g1,
                                               double efix, double inv2efix, const double (&Gb)[NT + 3],
                                               double (&QLb)[NT + 3], double (&QRb)[NT + 3], int &bad) {
  constexpr int E = NT + 2;
  auto M = [&bad](double a, double b) { return FX ? fx_mul(a, b, bad) : a * b; };
  auto rsqrt = [&bad](double x) { return FX ? fx_rsqrt64(x, bad) : rsqrt_fp64(x); };
  auto rcp = [&bad](double x) { return FX ? fx_rcp64(x, bad) : rcp_fp64(x); };
  // ---------------- forward: the quantities of roe_F
  const double tL = rsqrt(QL[0]);
  const double rL = M(tL, tL);
  const double sL = M(QL[0], tL);
  const double unL = M(QL[1], rL);
  double utL[NT];
  double kL = M(QL[1], unL);
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    utL[t] = M(QL[2 + t], rL);
    kL = fma(QL[2 + t], utL[t], kL);
  }
  const double pL = M(g1, fma(-0.5, kL, QL[E]));
  const double eL = QL[E] + pL;
  const double tR = rsqrt(QR[0]);
  const double rR = M(tR, tR);
  const double sR = M(QR[0], tR);
  const double unR = M(QR[1], rR);
  double utR[NT];
  double kR = M(QR[1], unR);
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    utR[t] = M(QR[2 + t], rR);
    kR = fma(QR[2 + t], utR[t], kR);
  }
  const double pR = M(g1, fma(-0.5, kR, QR[E]));
  const double eR = QR[E] + pR;
  const double inv = rcp(sL + sR);
  const double wL = M(sL, inv), wR = M(sR, inv);
  const double dun = unR - unL;
  const double un = fma(-wL, dun, unR);
  double ut[NT], dut[NT];
  double q2 = M(un, un);
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    dut[t] = utR[t] - utL[t];
    ut[t] = fma(-wL, dut[t], utR[t]);
    q2 = fma(ut[t], ut[t], q2);
  }
  const double Hn = fma(eL, tL, M(eR, tR));
  const double H = M(Hn, inv);
  const double rho = M(sL, sR);
  const double c2 = M(g1, H - half_nonneg(q2));
  const double tc = rsqrt(c2);
  const double c = M(c2, tc);
  const bool up_left = __double2hiint(un) >= 0;
  const double aun = iabs(un);
  const double sc = isel(up_left, c, ineg(c));
  const double dp = pR - pL;
  const double rsc = M(rho, sc);
  const double num = fma(-rsc, dun, dp);
  const double tc2h = M(tc, half_nonneg(tc));  // 1 / (2 c~^2)
  const double alpha = M(num, tc2h);
  const double x = aun - c;
  const bool neg = __double2hiint(x) < 0 && !izero(x);
  double k = isel(neg, x, 0.0);
  // The entropy fix where |x| < delta = efix c, decided in FP64 (the forward flux
  // decides in FP64 or 64-bit integers).  FP32 copies that never miss such a face say
  // whether a warp has any.
  const float efix_hi = __fadd_ru(__fmul_ru(f32_trunc(efix), 1.000001f), 0x1p-126f);
  const bool near = f32_trunc(iabs(x)) <= __fmul_ru(efix_hi, f32_trunc(c));
  const bool anyfix = __any_sync(__activemask(), near);
  bool fix = false;
  double delta = 0.0, s2 = 0.0;
  if (anyfix) {
    delta = __dmul_rn(efix, c);
    fix = near && ilt_nonneg(iabs(x), delta);
    s2 = __dmul_rn(tc, inv2efix);  // 1 / (2 delta)
    k = isel(fix, fma(-fma(x, x, __dmul_rn(delta, delta)), __dmul_rn(0.5, s2), __dmul_rn(0.5, x)), k);
  }
  const double g = M(k, alpha);
  const double lam = un - sc;
  const double hr = fma(-c, aun, H);
  const double m = isel(up_left, QL[1], QR[1]);
  const double u_n = isel(up_left, unL, unR);
  const double e = isel(up_left, eL, eR);

  // ---------------- reverse
  // G0 = m + g; G1 = m u_n + p_up + g lam; G2+t = m ut_up + g ut; GE = u_n e + g hr
  double mb = fma(Gb[1], u_n, Gb[0]);
  double u_nb = fma(Gb[E], e, M(Gb[1], m));
  const double pupb = Gb[1];
  const double eupb = M(Gb[E], u_n);
  double gb = fma(Gb[E], hr, fma(Gb[1], lam, Gb[0]));
  double utupb[NT], utb[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    mb = fma(Gb[2 + t], isel(up_left, utL[t], utR[t]), mb);
    utupb[t] = M(Gb[2 + t], m);
    gb = fma(Gb[2 + t], ut[t], gb);
    utb[t] = M(Gb[2 + t], g);
  }
  const double lamb = M(Gb[1], g);
  const double hrb = M(Gb[E], g);
  // hr = H - c aun ; lam = un - sc
  double Hb = hrb;
  double cb = M(-hrb, aun);
  double aunb = M(-hrb, c);
  double unb = lamb;
  double scb = -lamb;
  // g = k alpha
  const double kb = M(gb, alpha);
  const double alphab = M(gb, k);
  // k = min(x, 0), or with the fix x/2 - (x^2 + delta^2) / (4 delta)
  double xb = isel(neg, kb, 0.0);
  if (anyfix) {
    const double xs = __dmul_rn(x, s2);  // x / (2 delta)
    xb = isel(fix, __dmul_rn(kb, 0.5 - xs), xb);
    cb = fma(isel(fix, __dmul_rn(kb, fma(xs, xs, -0.25)), 0.0), efix, cb);  // delta = efix c
  }
  // x = aun - c ; aun = |un|
  aunb += xb;
  cb -= xb;
  unb += mul_sign(aunb, un);
  // alpha = num tc2h ; num = dp - rsc dun ; rsc = rho sc ; tc2h = tc^2 / 2 ; sc = +-c
  const double numb = M(alphab, tc2h);
  double tcb = M(M(alphab, num), tc);
  const double dpb = numb;
  const double rscb = M(-numb, dun);
  const double dunb = M(-numb, rsc);
  const double rhob = M(rscb, sc);
  scb = fma(rscb, rho, scb);
  cb += isel(up_left, scb, ineg(scb));
  // c = c2 tc ; tc = c2^(-1/2)
  tcb = fma(cb, c2, tcb);
  double c2b = M(cb, tc);
  c2b = fma(tcb, -M(half_nonneg(tc), M(tc, tc)), c2b);
  // c2 = g1 (H - q2/2) ; q2 = un^2 + sum ut^2
  Hb = fma(c2b, g1, Hb);
  const double q2b2 = M(-g1, c2b);  // 2 q2b
  unb = fma(q2b2, un, unb);
  // H = Hn inv ; Hn = eL tL + eR tR
  double invb = M(Hb, Hn);
  const double Hnb = M(Hb, inv);
  double eLb = M(Hnb, tL), eRb = M(Hnb, tR);
  double tLb = M(Hnb, eL), tRb = M(Hnb, eR);
  // rho = sL sR
  double sLb = M(rhob, sR), sRb = M(rhob, sL);
  // ut = utR - wL dut = wL utL + wR utR ; un = unR - wL dun ; dun = unR - unL
  double wLb = M(-unb, dun);
  double utLb[NT], utRb[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    utb[t] = fma(q2b2, ut[t], utb[t]);
    wLb = fma(-utb[t], dut[t], wLb);
    utLb[t] = fma(utb[t], wL, isel(up_left, utupb[t], 0.0));
    utRb[t] = fma(utb[t], wR, isel(up_left, 0.0, utupb[t]));
  }
  double unLb = fma(unb, wL, isel(up_left, u_nb, 0.0)) - dunb;
  double unRb = fma(unb, wR, isel(up_left, 0.0, u_nb)) + dunb;
  // wL = sL inv (wR = 1 - wL) ; inv = 1 / (sL + sR)
  sLb = fma(wLb, inv, sLb);
  invb = fma(wLb, sL, invb);
  const double Sb = M(M(-invb, inv), inv);
  sLb += Sb;
  sRb += Sb;
  // dp = pR - pL ; the upwind side's m, p, e
  double pLb = isel(up_left, pupb - dpb, -dpb), pRb = isel(up_left, dpb, pupb + dpb);
  eLb += isel(up_left, eupb, 0.0);
  eRb += isel(up_left, 0.0, eupb);
  double mnLb = isel(up_left, mb, 0.0), mnRb = isel(up_left, 0.0, mb);

  // left side: eL = E + pL ; pL = g1 (E - kL/2) ; kL = mn unL + sum mt utL ;
  // unL = mn rL ; utL = mt rL ; sL = rho tL ; rL = tL^2 ; tL = rho^(-1/2)
  double ELb = eLb;
  pLb += eLb;
  ELb = fma(pLb, g1, ELb);
  const double kLb = M(M(-0.5, g1), pLb);
  mnLb = fma(kLb, unL, mnLb);
  unLb = fma(kLb, QL[1], unLb);
  double rLb = 0.0;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    double mtb = M(kLb, utL[t]);
    utLb[t] = fma(kLb, QL[2 + t], utLb[t]);
    mtb = fma(utLb[t], rL, mtb);
    rLb = fma(utLb[t], QL[2 + t], rLb);
    QLb[2 + t] = mtb;
  }
  mnLb = fma(unLb, rL, mnLb);
  rLb = fma(unLb, QL[1], rLb);
  tLb = fma(sLb, QL[0], tLb);
  double rhoLb = M(sLb, tL);
  tLb = fma(rLb, scale_pow2<1>(tL), tLb);
  rhoLb = fma(tLb, -M(half_nonneg(tL), rL), rhoLb);
  QLb[0] = rhoLb;
  QLb[1] = mnLb;
  QLb[E] = ELb;

  // right side
  double ERb = eRb;
  pRb += eRb;
  ERb = fma(pRb, g1, ERb);
  const double kRb = M(M(-0.5, g1), pRb);
  mnRb = fma(kRb, unR, mnRb);
  unRb = fma(kRb, QR[1], unRb);
  double rRb = 0.0;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    double mtb = M(kRb, utR[t]);
    utRb[t] = fma(kRb, QR[2 + t], utRb[t]);
    mtb = fma(utRb[t], rR, mtb);
    rRb = fma(utRb[t], QR[2 + t], rRb);
    QRb[2 + t] = mtb;
  }
  mnRb = fma(unRb, rR, mnRb);
  rRb = fma(unRb, QR[1], rRb);
  tRb = fma(sRb, QR[0], tRb);
  double rhoRb = M(sRb, tR);
  tRb = fma(rRb, scale_pow2<1>(tR), tRb);
  rhoRb = fma(tRb, -M(half_nonneg(tR), rR), rhoRb);
  QRb[0] = rhoRb;
  QRb[1] = mnRb;
  QRb[E] = ERb;
}

template <int NT>
static __device__ __noinline__ void roe_F_vjp_fp64(const double (&QL)[NT + 3], const double (&QR)[NT + 3], double g1,
                                                   double efix, double inv2efix, const double (&Gb)[NT + 3],
                                                   double (&QLb)[NT + 3], double (&QRb)[NT + 3]) {
  int bad = 0;
  roe_F_vjp_impl<NT, false>(QL, QR, g1, efix, inv2efix, Gb, QLb, QRb, bad);
}

// The face flux VJP.  Only the lanes whose faces the integer operations do not
// take get the FP64 evaluation, so results do not depend on how faces fall
// into warps.  fx_mul has no subnormal numbers: a face whose results all come out
// below 2^-511, from cotangents so small that products with them may have been
// lost, is left to FP64 too (the VJP is linear in them, to the end of the range).
template <int NT>
__device__ __forceinline__ void roe_F_vjp(const double (&QL)[NT + 3], const double (&QR)[NT + 3], double g1,
                                          double efix, double inv2efix, const double (&Gb)[NT + 3],
                                          double (&QLb)[NT + 3], double (&QRb)[NT + 3]) {
  int bad = 0, high = 0;
  roe_F_vjp_impl<NT, true>(QL, QR, g1, efix, inv2efix, Gb, QLb, QRb, bad);
#pragma unroll
  for (int v = 0; v < NT + 3; ++v) high |= __double2hiint(QLb[v]) | __double2hiint(QRb[v]);
  if ((bad | ((high & 0x60000000) - 1)) < 0) {  // no exponent field of 512 or more
    bool any = false;                           // (no cotangent at all: zeros stand)
#pragma unroll
    for (int v = 0; v < NT + 3; ++v) any |= !izero(Gb[v]);
    if (bad < 0 || any) roe_F_vjp_fp64<NT>(QL, QR, g1, efix, inv2efix, Gb, QLb, QRb);
  }
}

// Which argument the limited slope minmod(a, b) passes a derivative through:
// 1 = a, 2 = b, 0 = none (signs differ or an argument is zero; ties -> b).
__device__ __forceinline__ int minmod_pick(double a, double b) {
  const int ha = __double2hiint(a), hb = __double2hiint(b);
  const unsigned la = (unsigned)__double2loint(a), lb = (unsigned)__double2loint(b);
  const unsigned ma = (unsigned)ha & 0x7fffffffu, mb = (unsigned)hb & 0x7fffffffu;
  if (((ha ^ hb) < 0) || (ma | la) == 0u || (mb | lb) == 0u) return 0;
  return (ma < mb || (ma == mb && la < lb)) ? 1 : 2;
}

}  // namespace fvk
