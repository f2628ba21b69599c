// lbcad_coefs.h -- the coefficients of one instance in the compute type, formed in FP64 from its
// parameters (shared by every entry point that launches a step).
#pragma once

#include "lbcad.h"
#include "lbcad_internal.h"

namespace lbcad {

template <typename T>
inline Coef<T> coefs(const lbcad_params& p) {
  Coef<T> c;
  c.tau_inv = (T)(1.0 / p.tau);
  c.guo = (T)(1.0 - 0.5 / p.tau);
  c.rho0 = (T)p.rho0;
  c.A0 = (T)p.A0; c.chi0 = (T)p.chi0; c.chis = (T)p.chis; c.K = (T)p.K; c.q0 = (T)p.q0;
  c.gammaQ = (T)p.gammaQ; c.xi = (T)p.xi; c.a = (T)p.a; c.b = (T)p.b; c.kphi = (T)p.kphi;
  c.M = (T)p.M; c.W = (T)p.W; c.zeta = (T)p.zeta;
  c.A0chi1 = (T)(p.A0 * (p.chi0 + p.chis));
  c.A0chis = (T)(p.A0 * p.chis);
  const double Kqq = p.K * p.q0 * p.q0;
  c.cL = (T)(p.A0 + 4.0 * Kqq);
  c.fQ2 = (T)(0.5 * p.A0 + 2.0 * Kqq);
  c.K2 = (T)(2.0 * p.K); c.Kq = (T)(2.0 * p.K * p.q0); c.W2 = (T)(2.0 * p.W);
  c.ah = (T)(0.5 * p.a); c.bq = (T)(0.25 * p.b); c.kh = (T)(0.5 * p.kphi); c.zh = (T)(0.5 * p.zeta);
  c.xi2 = (T)(2.0 * p.xi); c.xi23 = (T)(2.0 * p.xi / 3.0); c.xi29 = (T)(2.0 * p.xi / 9.0);
  c.xip = (T)(1.0 + p.xi); c.xim = (T)(1.0 - p.xi);
  c.omc = (T)(1.0 - 1.0 / p.tau);
  const int first[3] = {0, 1, 7};  // a velocity of each weight class
  for (int k = 0; k < 3; ++k) {
    const double w = p.lattice == LBCAD_D3Q15 ? lat15_w(first[k]) : lat_w(first[k]), guo = 1.0 - 0.5 / p.tau;
    c.omw[k] = (T)(w / p.tau);
    c.gw3[k] = (T)(3.0 * w * guo);
    c.gw9[k] = (T)(9.0 * w * guo);
  }
  return c;
}

}  // namespace lbcad
