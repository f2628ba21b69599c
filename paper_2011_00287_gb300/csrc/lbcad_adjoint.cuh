// lbcad_adjoint.cuh -- reverse mode (vector-Jacobian products) of one hybrid step.
//
// The step maps the stored state s_t = (g*, Q, psi, u) to s_{t+1}.  Given the cotangent
// lam_{t+1} of s_{t+1}, four gather-form kernels produce lam_t:
//   RK1 k_adj_update : per site, VJP of the update (upwind/co-rotation Q update, Cahn-Hilliard psi
//                      update, BGK + Guo collision) by a hand-written reverse sweep;
//   RK2 k_adj_spread : transposes of the stencils that fed the update (div sigma -> sigma, lap mu -> mu,
//                      grad u -> u, face reads -> Q/psi/u, the pull -> g*);
//   RK3 k_adj_fields : per site the VJP of local_fields (H, mu, sigma of Eqs. 2-5) with respect to its
//                      inputs and to zeta and q0, by a hand-written reverse sweep;
//   RK4 k_adj_gather : transposes of the Q/psi stencils (gradient, Laplacian, Hessian).
// The per-site reverse sweeps recompute the forward intermediates of the site and take
// every branch (upwind sides) as the forward takes it.  Stencil transposes use the negated offsets on the
// periodic lattice, so no site is written by two threads.
//
// What bounds them is the traffic between them: a site's full input cotangents are 88 values of the update and 36
// of local_fields.  Most of these are a factor known at the reading site times a cotangent it can read anyway
// (populations: (1 - 1/tau) lam_g plus a linear form of four values; upwind faces: the face velocity times lam_Q
// or lam_psi; lap mu and H: a coefficient times lam; lap Q, lap psi and the Hessian of psi: K lH, and lmu times
// Q), so only 16 values of the first and 24 of the second are passed, in quads and pairs (and the 10 cotangents of
// sigma and mu, at the site only).  The force F of
// each replayed step is kept by the replay (3 values per site and state), so that no stress is needed here.
#pragma once

#include "lbcad_march.cuh"

namespace lbcad {

// Buffers of one reverse step.
template <typename T>
struct AdjDesc {
  InstDesc<T> I;      // state s_t in I.*_in; the rest unused
  const T* F;         // force of the step from s_t [3][site]
  const T* lg;        // cotangent of s_{t+1}: g* (19), Q (5), psi (1), u (3), [component][site]
  const T* lq;
  const T* lp;
  const T* lu;
  T* A;               // RK1 -> RK2, quads [5][site][4]: (lF, lm0), (lj, -), (lW_ab over a, -) for b = x, y, z
  T* L;               // RK2 -> RK3: quads [2][site][4]: cotangents of sigma 0-3, 4-7; pairs [site][2]: (sigma 8, mu)
  T* B;               // RK3 -> RK4: quads [4][site][4]: ldQ_a components 0-3 for a = x, y, z, lH 0-3; then
                      // pairs [4][site][2]: (ldQ_a component 4, ldpsi_a) for a = x, y, z, (lH 4, lmu)
  T* og;              // cotangent of s_t: g* (19), Q (5), psi (1), u (3); RK1 leaves the site-local parts of Q, psi, u
  T* oq;
  T* op;
  T* ou;
  double* pgrad;      // per block: sums over the reverse steps of d/dzeta, d/dq0 (2 per block)
};

using AdjTile = Tile<32, 4>;
constexpr int kAdjBlock = AdjTile::NT;

template <typename T>
struct Quad {
  T x, y, z, w;
};
template <typename T>
__device__ __forceinline__ Quad<T> ld_quad(const T* base, long long s) {
  if constexpr (sizeof(T) == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(base) + s);
    return Quad<T>{v.x, v.y, v.z, v.w};
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(base) + 2 * s), w = __ldg(reinterpret_cast<const double2*>(base) + 2 * s + 1);
    return Quad<T>{v.x, v.y, w.x, w.y};
  }
}
template <typename T>
__device__ __forceinline__ void st_quad_at(T* base, long long s, T a, T b, T c, T d) {
  if constexpr (sizeof(T) == 4) {
    reinterpret_cast<float4*>(base)[s] = make_float4(a, b, c, d);
  } else {
    reinterpret_cast<double2*>(base)[2 * s] = make_double2(a, b);
    reinterpret_cast<double2*>(base)[2 * s + 1] = make_double2(c, d);
  }
}
template <typename T>
__device__ __forceinline__ Vec2<T> ld_pair(const T* base, long long s) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(base) + s);
    return Vec2<T>{v.x, v.y};
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(base) + s);
    return Vec2<T>{v.x, v.y};
  }
}
template <typename T>
__device__ __forceinline__ void st_pair_at(T* base, long long s, T a, T b) {
  if constexpr (sizeof(T) == 4) reinterpret_cast<float2*>(base)[s] = make_float2(a, b);
  else reinterpret_cast<double2*>(base)[s] = make_double2(a, b);
}

// ---------------------------------------------------------------- reverse mode of update_math
// Vector-Jacobian product of update_math (D3Q19 body-force collision, Euler update) at one
// site, by a hand-written reverse sweep over the forward arithmetic: lo = the cotangents of the 28 outputs
// (qn 0-4, pn 5, u 6-8, g 9-27).  Results: lF, lW (grad u), the site-local parts of the cotangents of Q, psi and
// u (lq0, lp0, lu0), and lm0, lj, in which the cotangent of pulled population i is
// (1 - 1/tau) lo[9 + i] + lm0 + c_i . lj.  The cotangents of lap mu (M lo[5]), H (Gamma lo[k]) and of the face
// values are formed where they are read (k_adj_fields).  qu: Q at the upwind neighbours.  The branches (upwind
// selection, face fluxes) take the side the forward takes, as forward-mode differentiation of the same
// code would.
template <typename T, bool SHIFT>
__device__ __forceinline__ void update_math_vjp(const Coef<T>& c, const T F[3], const T W[3][3], const T q0[5],
                                                const T qu[3][5], T p0, const T pf[6], const T u0[3], const T uf[6],
                                                const T g[19], const T lo[28], T lF[3], T lW[3][3], T lq0[5], T& lp0,
                                                T lu0v[3], T& lm0, T lj[3]) {
  // ---- LB collision (outputs u 6-8, g 9-27)
  T m0 = g[0];
  T jm[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int i = 1; i < 19; i += 2) {
    m0 += g[i] + g[i + 1];
    const T dg = g[i] - g[i + 1];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (lat_c(i, a)) jm[a] += lat_c(i, a) > 0 ? dg : -dg;
  }
  const T rho = SHIFT ? (c.rho0 + m0) : m0;
  const T rinv = T(1) / rho;
  T u[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) u[a] = (jm[a] + T(0.5) * F[a]) * rinv;
  const T u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const T r45 = T(4.5) * rho, r3 = T(3) * rho, om = c.tau_inv;
  T lu[3] = {lo[6], lo[7], lo[8]};
  lF[0] = lF[1] = lF[2] = T(0);
  T lbase = T(0), lr45 = T(0), lr3 = T(0), luF = T(0);
  {
    const T w = T(lat_w(0));
    const T l0 = lo[9];
    lbase += om * w * l0;
    luF += -T(3) * c.guo * w * l0;
  }
#pragma unroll
  for (int i = 1; i < 19; i += 2) {
    const T w = T(lat_w(i)), gw = c.guo * w;
    const T cu = T(lat_c(i, 0)) * u[0] + T(lat_c(i, 1)) * u[1] + T(lat_c(i, 2)) * u[2];
    const T cF = T(lat_c(i, 0)) * F[0] + T(lat_c(i, 1)) * F[1] + T(lat_c(i, 2)) * F[2];
    const T lp = lo[9 + i], lm = lo[10 + i];
    const T lA = om * (lp + lm), lB = om * (lp - lm), lC = lp + lm, lE = lp - lm;
    lbase += w * lA;
    lr45 += w * cu * cu * lA;
    lr3 += w * cu * lB;
    luF += -T(3) * gw * lC;
    const T lcu = T(2) * w * r45 * cu * lA + w * r3 * lB + T(9) * gw * cF * lC;
    const T lcF = T(9) * gw * cu * lC + T(3) * gw * lE;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (lat_c(i, a)) {
        lu[a] += T(lat_c(i, a)) * lcu;
        lF[a] += T(lat_c(i, a)) * lcF;
      }
    }
  }
  // base = m0 - 1.5 rho u2 (shifted) or rho - 1.5 rho u2; r45 = 4.5 rho; r3 = 3 rho
  T lrho = T(0), lu2 = T(0);
  lm0 = T(0);
  if (SHIFT) lm0 += lbase; else lrho += lbase;
  lrho += -T(1.5) * u2 * lbase + T(4.5) * lr45 + T(3) * lr3;
  lu2 += -T(1.5) * rho * lbase;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lu[a] += T(2) * u[a] * lu2 + F[a] * luF;
    lF[a] += u[a] * luF;
  }
  // u = (j + F/2) / rho
  T lrinv = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lrinv += (jm[a] + T(0.5) * F[a]) * lu[a];
    lj[a] = rinv * lu[a];
    lF[a] += T(0.5) * rinv * lu[a];
  }
  lrho += -rinv * rinv * lrinv;
  lm0 += lrho;

  // ---- order-parameter update (outputs qn 0-4, pn 5)
  const T xi = c.xi;
#pragma unroll
  for (int k = 0; k < 5; ++k) lq0[k] = lo[k];
  lp0 = lo[5];
  const T ldivJ = -lo[5];
  // co-rotation S of the five stored components
  T Q[3][3];
  full3(q0, Q);
  T Dm[3][3], Om[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Dm[i][j] = T(0.5) * (W[i][j] + W[j][i]);
      Om[i][j] = T(0.5) * (W[i][j] - W[j][i]);
    }
  T trQW = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) trQW += Q[i][j] * W[j][i];
  const T cq = -T(2) * xi * trQW;
  const T c23 = c.xi23;
  T lQ[3][3], lD[3][3], lO[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) lQ[i][j] = lD[i][j] = lO[i][j] = T(0);
  T lcq = T(0), lcdiag = T(0);
  const int I5[5] = {0, 0, 0, 1, 1};
  const int J5[5] = {0, 1, 2, 1, 2};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int i = I5[k], j = J5[k];
    const T L = lo[k];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      lD[i][m] += xi * L * Q[m][j];
      lQ[m][j] += xi * L * Dm[i][m];
      lQ[i][m] += xi * L * Dm[m][j];
      lD[m][j] += xi * L * Q[i][m];
      lO[i][m] += L * Q[m][j];
      lQ[m][j] += L * Om[i][m];
      lQ[i][m] -= L * Om[m][j];
      lO[m][j] -= L * Q[i][m];
    }
    lD[i][j] += c23 * L;
    lcq += L * Q[i][j];
    lQ[i][j] += cq * L;
    if (i == j) lcdiag += L;
  }
  // cdiag = cq/3 - (2 xi/9) trD; cq = -2 xi tr(QW)
  lcq += lcdiag * T(1.0 / 3.0);
  const T ltrD = -c.xi29 * lcdiag;
  const T ltrQW = -T(2) * xi * lcq;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) lW[i][j] = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    lD[i][i] += ltrD;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      lQ[i][j] += W[j][i] * ltrQW;
      lW[j][i] += Q[i][j] * ltrQW;
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      lW[i][j] += T(0.5) * (lD[i][j] + lO[i][j]);
      lW[j][i] += T(0.5) * (lD[i][j] - lO[i][j]);
    }
  lq0[0] += lQ[0][0] - lQ[2][2];
  lq0[1] += lQ[0][1] + lQ[1][0];
  lq0[2] += lQ[0][2] + lQ[2][0];
  lq0[3] += lQ[1][1] - lQ[2][2];
  lq0[4] += lQ[1][2] + lQ[2][1];
  // upwind advection of Q, -|u| (q0 - qu), and the psi face fluxes
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int ip = 2 * a, im = 2 * a + 1;
    const T ua = fabs(u0[a]);
    T d = T(0);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      d += (q0[k] - qu[a][k]) * lo[k];
      lq0[k] -= ua * lo[k];
    }
    T lu0 = u0[a] > T(0) ? -d : (u0[a] < T(0) ? d : T(0));
    const T ubp = T(0.5) * (u0[a] + uf[ip]);
    if (ubp > T(0)) lp0 += ubp * ldivJ;
    lu0 += T(0.5) * ((ubp > T(0) ? p0 : pf[ip]) * ldivJ);
    const T ubm = T(0.5) * (uf[im] + u0[a]);
    if (!(ubm > T(0))) lp0 -= ubm * ldivJ;
    lu0 -= T(0.5) * ((ubm > T(0) ? pf[im] : p0) * ldivJ);
    lu0v[a] = lu0;
  }
}

// ---------------------------------------------------------------- reverse mode of local_fields
// Vector-Jacobian product of local_fields at one site by a hand-written reverse sweep: in =
// the 36 inputs (q0 0-4, psi 5, dq 6-20 as 6 + 5a + k, lapq 21-25, dp 26-28, lapp 29,
// hp 30-35), lo = the cotangents of its outputs (H 0-4, mu 5, sigma 6-14), out = the
// cotangents of inputs 0-20 and, at 21-23, of dp; lH and lmu_out, in which those of lapq, lapp and hp are K lH,
// -kphi lmu and -2 W lmu (Q_aa on the diagonal, 2 Q_ab off it); lzeta and lq0 receive the derivatives with respect
// to the parameters zeta and q0.  Full 3x3 cotangents of Q and dQ_a are accumulated entry by entry
// as the forward reads them and folded onto the five stored components at the end.
template <typename T>
__device__ __forceinline__ void local_fields_vjp(const Coef<T>& c, const T in[36], const T lo[15], T out[24],
                                                 T lH[5], T& lmu_out, T& lzeta, T& lq0) {
  // ---- forward intermediates
  const T* q = in;
  const T psi = in[5];
  T Q[3][3];
  full3(q, Q);
  T dQ[3][3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) full3(in + 6 + 5 * a, dQ[a]);
  const T* dp = in + 26;
  const T* hp = in + 30;
  const T third = T(1.0 / 3.0);
  const T chi = c.chi0 + c.chis * (T(1) + psi);
  T QQ[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      QQ[i][j] = Q[i][0] * Q[0][j] + Q[i][1] * Q[1][j] + Q[i][2] * Q[2][j];
      QQ[j][i] = QQ[i][j];
    }
  const T trQ2 = QQ[0][0] + QQ[1][1] + QQ[2][2];
  const T trQ3 = QQ[0][0] * Q[0][0] + QQ[1][1] * Q[1][1] + QQ[2][2] * Q[2][2] +
                 T(2) * (QQ[0][1] * Q[0][1] + QQ[0][2] * Q[0][2] + QQ[1][2] * Q[1][2]);
  T C[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    C[0][b] = dQ[1][2][b] - dQ[2][1][b];
    C[1][b] = dQ[2][0][b] - dQ[0][2][b];
    C[2][b] = dQ[0][1][b] - dQ[1][0][b];
  }
  T CC[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) CC[i][j] = C[i][j] + C[j][i];
  const T g2 = dp[0] * dp[0] + dp[1] * dp[1] + dp[2] * dp[2];
  const T Ac = c.A0 * chi;
  const T Kq = T(2) * c.K * c.q0;
  const T lin = -c.A0 * (T(1) - third * chi) - Ac * trQ2 - Kq * T(2) * c.q0;
  const T iso = third * (Ac * trQ2 - c.W * g2);
  const int I5[5] = {0, 0, 0, 1, 1};
  const int J5[5] = {0, 1, 2, 1, 2};
  T H[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int i = I5[k], j = J5[k];
    T h = lin * Q[i][j] + Ac * QQ[i][j] + c.K * in[21 + k] - Kq * CC[i][j] - c.W * dp[i] * dp[j];
    if (i == j) h -= iso;
    H[k] = h;
  }
  T Hf[3][3];
  full3(H, Hf);
  const T Qh = Q[0][0] * hp[0] + Q[1][1] * hp[1] + Q[2][2] * hp[2] +
               T(2) * (Q[0][1] * hp[3] + Q[0][2] * hp[4] + Q[1][2] * hp[5]);
  T divQdp = T(0);
#pragma unroll
  for (int b = 0; b < 3; ++b) divQdp += (dQ[0][0][b] + dQ[1][1][b] + dQ[2][2][b]) * dp[b];
  const T psi2 = psi * psi;
  const T mu = psi * (c.b * psi2 - c.a) - c.kphi * in[29] +
               c.A0 * c.chis * (trQ2 * (T(0.25) * trQ2 - T(1.0 / 6.0)) - third * trQ3) - T(2) * c.W * (divQdp + Qh);
  T Qdp[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) Qdp[i] = Q[i][0] * dp[0] + Q[i][1] * dp[1] + Q[i][2] * dp[2];
  const T QC = Q[0][0] * C[0][0] + Q[1][1] * C[1][1] + Q[2][2] * C[2][2] + Q[0][1] * CC[0][1] +
               Q[0][2] * CC[0][2] + Q[1][2] * CC[1][2];
  T QH[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) QH[i][j] = Q[i][0] * Hf[0][j] + Q[i][1] * Hf[1][j] + Q[i][2] * Hf[2][j];
  const T phic = T(0.5) * (T(1) + psi);
  const T trQH = QH[0][0] + QH[1][1] + QH[2][2];
  const T cQ = T(2) * c.xi * trQH - c.zeta * phic;
  const T cH = -c.xi23;
  const T cP = T(1) - c.xi, cM = -(T(1) + c.xi);
  T wv[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) wv[b] = c.kphi * dp[b] + T(2) * c.W * Qdp[b];
  T v[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int g = (b + 1) % 3, m = (b + 2) % 3;
      v[a][b] = dQ[a][g][0] * Q[0][m] + dQ[a][g][1] * Q[1][m] + dQ[a][g][2] * Q[2][m] -
                (dQ[a][m][0] * Q[0][g] + dQ[a][m][1] * Q[1][g] + dQ[a][m][2] * Q[2][g]);
    }

  // ---- reverse sweep
  T lQ[3][3], ldQ[3][3][3], lHf[3][3], lQH[3][3], lG[3][3], lCC[3][3], lC[3][3], lQQ[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      lQ[i][j] = lHf[i][j] = lQH[i][j] = lG[i][j] = lCC[i][j] = lC[i][j] = lQQ[i][j] = T(0);
#pragma unroll
      for (int a = 0; a < 3; ++a) ldQ[a][i][j] = T(0);
    }
  T ldp[3] = {T(0), T(0), T(0)}, lwv[3] = {T(0), T(0), T(0)}, lQdp[3] = {T(0), T(0), T(0)};
  T lpsi = T(0), lcQ = T(0), lcI = T(0), lKq = T(0), ltrQH = T(0), lP0 = T(0), lphic = T(0);
  lzeta = T(0);
  lq0 = T(0);
  // sigma
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const T L = lo[6 + 3 * a + b];
      lcQ += L * Q[a][b];
      lQ[a][b] += cQ * L;
      lQH[a][b] += cP * L;
      lQH[b][a] += cM * L;
      lHf[a][b] += cH * L;
      lG[a][b] += -c.K * L;
      lKq += -v[a][b] * L;
      const T lv = -Kq * L;
      ldp[a] += -wv[b] * L;
      lwv[b] += -dp[a] * L;
      if (a == b) lcI += L;
      const int g = (b + 1) % 3, m = (b + 2) % 3;
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        ldQ[a][g][n] += lv * Q[n][m];
        lQ[n][m] += lv * dQ[a][g][n];
        ldQ[a][m][n] -= lv * Q[n][g];
        lQ[n][g] -= lv * dQ[a][m][n];
      }
    }
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    ldp[b] += c.kphi * lwv[b];
    lQdp[b] += T(2) * c.W * lwv[b];
  }
  // cQ = 2 xi trQH - zeta phic; cI = (2 xi/3) trQH - P0
  ltrQH += T(2) * c.xi * lcQ + c.xi23 * lcI;
  lzeta += -phic * lcQ;
  lphic += -c.zeta * lcQ;
  lP0 += -lcI;
  lpsi += T(0.5) * lphic;
#pragma unroll
  for (int i = 0; i < 3; ++i) lQH[i][i] += ltrQH;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        lQ[i][m] += lQH[i][j] * Hf[m][j];
        lHf[m][j] += Q[i][m] * lQH[i][j];
      }
  // P0 = psi mu - fden
  const T lmu = lo[5] + psi * lP0;
  lpsi += mu * lP0;
  const T lf = -lP0;
  // fden
  T lpsi2 = (T(0.5) * c.b * psi2 - T(0.5) * c.a) * lf;
  T lg2 = T(0.5) * c.kphi * lf;
  T lchi = c.A0 * (-T(0.5 / 3.0) * trQ2 - third * trQ3 + T(0.25) * trQ2 * trQ2) * lf;
  T ltrQ2 = c.A0 * (T(0.5) * (T(1) - third * chi) + T(0.5) * chi * trQ2) * lf + Kq * c.q0 * lf;
  T ltrQ3 = -c.A0 * third * chi * lf;
#pragma unroll
  for (int a = 0; a < 3; ++a) lG[a][a] += T(0.5) * c.K * lf;
  lKq += QC * lf + c.q0 * trQ2 * lf;
  const T lQC = Kq * lf;
  lq0 += Kq * trQ2 * lf;
  const T lanch = c.W * lf;
  // anch = dp . Qdp; Qdp = Q dp
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    ldp[i] += Qdp[i] * lanch;
    lQdp[i] += dp[i] * lanch;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      lQ[i][m] += lQdp[i] * dp[m];
      ldp[m] += Q[i][m] * lQdp[i];
    }
  // QC
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    lQ[i][i] += C[i][i] * lQC;
    lC[i][i] += Q[i][i] * lQC;
  }
  lQ[0][1] += CC[0][1] * lQC;
  lCC[0][1] += Q[0][1] * lQC;
  lQ[0][2] += CC[0][2] * lQC;
  lCC[0][2] += Q[0][2] * lQC;
  lQ[1][2] += CC[1][2] * lQC;
  lCC[1][2] += Q[1][2] * lQC;
  // mu
  lpsi += (c.b * psi2 - c.a) * lmu;
  lpsi2 += psi * c.b * lmu;
  lmu_out = lmu;
  ltrQ2 += c.A0 * c.chis * (T(0.5) * trQ2 - T(1.0 / 6.0)) * lmu;
  ltrQ3 += -c.A0chis * third * lmu;
  const T ldiv = -T(2) * c.W * lmu, lQh = -T(2) * c.W * lmu;
  // Qh
  lQ[0][0] += hp[0] * lQh;
  lQ[1][1] += hp[1] * lQh;
  lQ[2][2] += hp[2] * lQh;
  lQ[0][1] += T(2) * hp[3] * lQh;
  lQ[0][2] += T(2) * hp[4] * lQh;
  lQ[1][2] += T(2) * hp[5] * lQh;
  // divQdp
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    ldQ[0][0][b] += dp[b] * ldiv;
    ldQ[1][1][b] += dp[b] * ldiv;
    ldQ[2][2][b] += dp[b] * ldiv;
    ldp[b] += (dQ[0][0][b] + dQ[1][1][b] + dQ[2][2][b]) * ldiv;
  }
  lpsi += T(2) * psi * lpsi2;
  // G (symmetric): the computed value s_ab serves G[a][b] and G[b][a]
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      const T ls = (a == b) ? lG[a][a] : lG[a][b] + lG[b][a];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          const T w = (i == j) ? T(1) : T(2);
          ldQ[a][i][j] += w * ls * dQ[b][i][j];
          ldQ[b][i][j] += w * ls * dQ[a][i][j];
        }
    }
  // H (outputs and the uses of Hf)
  lH[0] = lo[0] + lHf[0][0] - lHf[2][2];
  lH[1] = lo[1] + lHf[0][1] + lHf[1][0];
  lH[2] = lo[2] + lHf[0][2] + lHf[2][0];
  lH[3] = lo[3] + lHf[1][1] - lHf[2][2];
  lH[4] = lo[4] + lHf[1][2] + lHf[2][1];
  T llin = T(0), lAc = T(0), liso = T(0);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int i = I5[k], j = J5[k];
    const T L = lH[k];
    llin += Q[i][j] * L;
    lQ[i][j] += lin * L;
    lAc += QQ[i][j] * L;
    lQQ[i][j] += Ac * L;
    lKq += -CC[i][j] * L;
    lCC[i][j] += -Kq * L;
    ldp[i] += -c.W * dp[j] * L;
    ldp[j] += -c.W * dp[i] * L;
    if (i == j) liso += -L;
  }
  // iso, lin, Kq, Ac, g2
  lAc += third * trQ2 * liso;
  ltrQ2 += third * Ac * liso;
  lg2 += -c.W * third * liso;
  lchi += c.A0 * third * llin;
  lAc += -trQ2 * llin;
  ltrQ2 += -Ac * llin;
  lKq += -T(2) * c.q0 * llin;
  lq0 += -T(2) * Kq * llin;
  lq0 += T(2) * c.K * lKq;
  lchi += c.A0 * lAc;
#pragma unroll
  for (int b = 0; b < 3; ++b) ldp[b] += T(2) * dp[b] * lg2;
  // CC (symmetric value per unordered pair) and C
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      if (i == j) {
        lC[i][i] += T(2) * lCC[i][i];
      } else {
        const T l = lCC[i][j] + lCC[j][i];
        lC[i][j] += l;
        lC[j][i] += l;
      }
    }
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    ldQ[1][2][b] += lC[0][b];
    ldQ[2][1][b] -= lC[0][b];
    ldQ[2][0][b] += lC[1][b];
    ldQ[0][2][b] -= lC[1][b];
    ldQ[0][1][b] += lC[2][b];
    ldQ[1][0][b] -= lC[2][b];
  }
  // trQ3, trQ2, QQ
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    lQQ[i][i] += Q[i][i] * ltrQ3 + ltrQ2;
    lQ[i][i] += QQ[i][i] * ltrQ3;
  }
  lQQ[0][1] += T(2) * Q[0][1] * ltrQ3;
  lQ[0][1] += T(2) * QQ[0][1] * ltrQ3;
  lQQ[0][2] += T(2) * Q[0][2] * ltrQ3;
  lQ[0][2] += T(2) * QQ[0][2] * ltrQ3;
  lQQ[1][2] += T(2) * Q[1][2] * ltrQ3;
  lQ[1][2] += T(2) * QQ[1][2] * ltrQ3;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const T l = (i == j) ? lQQ[i][i] : lQQ[i][j] + lQQ[j][i];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        lQ[i][m] += l * Q[m][j];
        lQ[m][j] += l * Q[i][m];
      }
    }
  // chi = chi0 + chis (1 + psi)
  lpsi += c.chis * lchi;
  // fold the full-matrix cotangents onto the stored components (full3 transposed)
  out[0] = lQ[0][0] - lQ[2][2];
  out[1] = lQ[0][1] + lQ[1][0];
  out[2] = lQ[0][2] + lQ[2][0];
  out[3] = lQ[1][1] - lQ[2][2];
  out[4] = lQ[1][2] + lQ[2][1];
  out[5] = lpsi;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    out[6 + 5 * a + 0] = ldQ[a][0][0] - ldQ[a][2][2];
    out[6 + 5 * a + 1] = ldQ[a][0][1] + ldQ[a][1][0];
    out[6 + 5 * a + 2] = ldQ[a][0][2] + ldQ[a][2][0];
    out[6 + 5 * a + 3] = ldQ[a][1][1] - ldQ[a][2][2];
    out[6 + 5 * a + 4] = ldQ[a][1][2] + ldQ[a][2][1];
  }
#pragma unroll
  for (int b = 0; b < 3; ++b) out[21 + b] = ldp[b];
}

// ---------------------------------------------------------------- RK1
// The site of a thread and its neighbour offsets; false past the last site.  (Blocks that march on tiles, as k_adj_fields
// does, find more of their neighbours in L1 but run fewer warps: 37 us for k_adj_spread either way, 25 against 20 for
// k_adj_gather, 64^3.)
__device__ __forceinline__ bool adj_site(int nx, int ny, int nz, long long N, long long& s, Nbr& nb) {
  s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= N) return false;
  const unsigned r = (unsigned)s, t = r / (unsigned)nx;  // a box has at most 2^31 sites
  nb = make_nbr((int)(r % (unsigned)nx), (int)(t % (unsigned)ny), (int)(t / (unsigned)ny), nx, ny, nz);
  return true;
}

template <typename T, bool SHIFT>
__global__ void __launch_bounds__(kAdjBlock) k_adj_update(AdjDesc<T> A) {
  const InstDesc<T>& I = A.I;
  const long long N = I.N;
  long long s;
  GlobalAcc<T> acc;
  if (!adj_site(I.nx, I.ny, I.nz, N, s, acc.nb)) return;
  acc.q_ = I.q_in; acc.ps = I.psi_in; acc.u_ = I.u_in;
  acc.N = N;
  T F[3], W[3][3], q0[5], qu[3][5], pf[6], u0[3], uf[6], g[19];
#pragma unroll
  for (int a = 0; a < 3; ++a) F[a] = A.F[a * N + s];
  gather_velocity<T>(acc, W, u0, uf);
#pragma unroll
  for (int k = 0; k < 5; ++k) q0[k] = ld(I.q_in + k * N + s);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int d = u0[a] > T(0) ? -1 : 1;
    const long long o = acc.nb.off(a == 0 ? d : 0, a == 1 ? d : 0, a == 2 ? d : 0);
#pragma unroll
    for (int k = 0; k < 5; ++k) qu[a][k] = ld(I.q_in + k * N + o);
  }
#pragma unroll
  for (int f = 0; f < 6; ++f) pf[f] = acc.psi(lat_c(f + 1, 0), lat_c(f + 1, 1), lat_c(f + 1, 2));
  const T p0 = ld(I.psi_in + s);
#pragma unroll
  for (int i = 0; i < 19; ++i) g[i] = ld(I.g_in + i * N + acc.nb.off(-lat_c(i, 0), -lat_c(i, 1), -lat_c(i, 2)));
  // output cotangents: qn 0-4, pn 5, u 6-8, g 9-27
  T lo[28];
#pragma unroll
  for (int k = 0; k < 5; ++k) lo[k] = A.lq[k * N + s];
  lo[5] = A.lp[s];
#pragma unroll
  for (int a = 0; a < 3; ++a) lo[6 + a] = A.lu[a * N + s];
#pragma unroll
  for (int i = 0; i < 19; ++i) lo[9 + i] = A.lg[i * N + s];
  T lF[3], lW[3][3], lq0[5], lp0, lu0[3], lm0, lj[3];
  update_math_vjp<T, SHIFT>(I.c, F, W, q0, qu, p0, pf, u0, uf, g, lo, lF, lW, lq0, lp0, lu0, lm0, lj);
  st_quad_at(A.A, s, lF[0], lF[1], lF[2], lm0);
  st_quad_at(A.A + 4 * N, s, lj[0], lj[1], lj[2], T(0));
#pragma unroll
  for (int b = 0; b < 3; ++b) st_quad_at(A.A + (8 + 4 * b) * N, s, lW[0][b], lW[1][b], lW[2][b], T(0));
#pragma unroll
  for (int k = 0; k < 5; ++k) A.oq[k * N + s] = lq0[k];
  A.op[s] = lp0;
#pragma unroll
  for (int a = 0; a < 3; ++a) A.ou[a * N + s] = lu0[a];
}

// ---------------------------------------------------------------- RK2
// Transposes of the stencils of the update and of the pull, gathered at the site.
// (Four blocks per SM: at the 102 registers the compiler takes by itself 37 us, with up to 128 32 us, 64^3.)
template <typename T>
__global__ void __launch_bounds__(kAdjBlock, sizeof(T) == 4 ? 4 : 2) k_adj_spread(AdjDesc<T> A) {
  const InstDesc<T>& I = A.I;
  const long long N = I.N;
  long long s;
  Nbr nb;
  if (!adj_site(I.nx, I.ny, I.nz, N, s, nb)) return;
  {
    const Coef<T>& c = I.c;
    // pull: g[i](x) = g*_i(x - c_i)  =>  lam g*_i(y) = lam g[i](y + c_i).  F_a(x) = sum_b sum_{i odd, c_ib != 0}
    // sgn(c_ib) wt_i (sigma_ab(x + c_i) - sigma_ab(x - c_i)), and grad u the same, so both transposes take
    // the difference of the values at y - c_i and y + c_i.
    T ls[9], lu[3];
#pragma unroll
    for (int k = 0; k < 9; ++k) ls[k] = T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) lu[a] = A.ou[a * N + s];
    {
      const Quad<T> f = ld_quad(A.A, s);
      A.og[s] = c.omc * ld(A.lg + s) + f.w;
    }
#pragma unroll
    for (int i = 1; i < 19; i += 2) {
      const int cx = lat_c(i, 0), cy = lat_c(i, 1), cz = lat_c(i, 2);
      const T wt = lat_c2(i) == 1 ? T(2.0 / 12.0) : T(1.0 / 12.0);
      const long long m = nb.off(-cx, -cy, -cz), p = nb.off(cx, cy, cz);
      const Quad<T> fm = ld_quad(A.A, m), fp = ld_quad(A.A, p);
      const Quad<T> jm = ld_quad(A.A + 4 * N, m), jp = ld_quad(A.A + 4 * N, p);
      A.og[i * N + s] = c.omc * ld(A.lg + i * N + p) + fp.w + (T(cx) * jp.x + T(cy) * jp.y + T(cz) * jp.z);
      A.og[(i + 1) * N + s] = c.omc * ld(A.lg + (i + 1) * N + m) + fm.w - (T(cx) * jm.x + T(cy) * jm.y + T(cz) * jm.z);
      const T df[3] = {fm.x - fp.x, fm.y - fp.y, fm.z - fp.z};
      const int cc[3] = {cx, cy, cz};
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (cc[b] == 0) continue;
        const T w = cc[b] > 0 ? wt : -wt;
#pragma unroll
        for (int a = 0; a < 3; ++a) ls[3 * a + b] += w * df[a];
        const Quad<T> wm = ld_quad(A.A + (8 + 4 * b) * N, m), wp = ld_quad(A.A + (8 + 4 * b) * N, p);
        lu[0] += w * (wm.x - wp.x);
        lu[1] += w * (wm.y - wp.y);
        lu[2] += w * (wm.z - wp.z);
      }
    }
    // lap mu(x) = sum_i lw_i mu(x + c_i) - 4 mu(x): symmetric; its cotangent is M lam_psi
    const T lpc = ld(A.lp + s);
    T lmu = -T(4) * lpc;
#pragma unroll
    for (int i = 1; i < 19; ++i)
      lmu += (lat_c2(i) == 1 ? T(1.0 / 3.0) : T(1.0 / 6.0)) * ld(A.lp + nb.off(-lat_c(i, 0), -lat_c(i, 1), -lat_c(i, 2)));
    lmu *= c.M;
    // face reads of the sites at y - e_a (their upper face) and y + e_a (their lower face)
    T lq[5], lp = A.op[s];
#pragma unroll
    for (int k = 0; k < 5; ++k) lq[k] = A.oq[k * N + s];
    const T p0 = ld(I.psi_in + s);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int ex = a == 0, ey = a == 1, ez = a == 2;
      const long long m = nb.off(-ex, -ey, -ez), p = nb.off(ex, ey, ez);
      const T uc = ld(I.u_in + a * N + s), um = ld(I.u_in + a * N + m), up = ld(I.u_in + a * N + p);
      // Q: the site below takes this one as its upwind neighbour if its velocity is negative, the one above if positive
      const T wm = um < T(0) ? -um : T(0), wp = up > T(0) ? up : T(0);
#pragma unroll
      for (int k = 0; k < 5; ++k) lq[k] += wm * ld(A.lq + k * N + m) + wp * ld(A.lq + k * N + p);
      // psi fluxes: upper face of the site below, cotangent -lam_psi; lower face of the site above, +lam_psi
      const T lm = -ld(A.lp + m), lpp = ld(A.lp + p);
      const T ubp = T(0.5) * (um + uc), ubm = T(0.5) * (uc + up);
      if (!(ubp > T(0))) lp += ubp * lm;
      if (ubm > T(0)) lp += ubm * lpp;
      lu[a] += T(0.5) * ((ubp > T(0) ? ld(I.psi_in + m) : p0) * lm + (ubm > T(0) ? p0 : ld(I.psi_in + p)) * lpp);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) A.ou[a * N + s] = lu[a];
#pragma unroll
    for (int k = 0; k < 5; ++k) A.oq[k * N + s] = lq[k];
    A.op[s] = lp;
    st_quad_at(A.L, s, ls[0], ls[1], ls[2], ls[3]);
    st_quad_at(A.L + 4 * N, s, ls[4], ls[5], ls[6], ls[7]);
    st_pair_at(A.L + 8 * N, s, ls[8], lmu);
  }
}

// ---------------------------------------------------------------- RK3
// The VJP of local_fields (inputs packed: q0 0-4, p0 5, dq 6-20 (a*5 + k), lapq 21-25, dp 26-28, lapp 29, hp 30-35).
// Marches up z on tiles like the step's kernels, with planes of Q and psi in shared memory; without the carry of
// the stencils, whose 54 registers the reverse sweep needs.
constexpr int kAdjRing = 4;

template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 3 : 2)
    k_adj_fields(AdjDesc<T> A, const MarchItem* __restrict__ items, int nitems) {
  using G = AdjTile;
  constexpr int QSL = 6 * G::SP;
  __shared__ __align__(16) T sQ[kAdjRing * QSL];
  const InstDesc<T>& I = A.I;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const long long N = I.N;
  const unsigned plane = (unsigned)(nx * ny);
  const Coef<T>& c = I.c;
  const int tid = threadIdx.x, tx = tid % G::TX, ty = tid / G::TX;
  double pz = 0.0, pq = 0.0;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const MarchItem tl = items[item];
    const int zb = tl.zb, ze = tl.ze;
    unsigned off[G::LD];
    tile_offsets<G>(tl, nx, ny, off);
    auto issue = [&](int p) {
      const unsigned gz = (unsigned)wrap_plane(p, nz) * plane;
      T* dq = sQ + ((p + 4) & 3) * QSL;
#pragma unroll
      for (int r = 0; r < G::LD; ++r) {
        const int k = tid + r * G::NT;
        if (k < G::SP) {
          const unsigned o = gz + off[r];
#pragma unroll
          for (int f = 0; f < 5; ++f) cp_async_elem(dq + qidx<G::SP>(f, k), I.q_in + f * N + o);
          cp_async_elem(dq + qidx<G::SP>(5, k), I.psi_in + o);
        }
      }
    };
    __syncthreads();  // the previous item is done with the tiles
    issue(zb - 1);
    issue(zb);
    issue(zb + 1);
    cp_async_commit_wait_all();
    __syncthreads();
    const bool inside = tl.x0 + tx < nx && tl.y0 + ty < ny;
    const unsigned soff = (unsigned)((tl.y0 + ty) * nx + (tl.x0 + tx));
    TileAcc<T, G> acc;
    acc.sc = (ty + 1) * G::SW + (tx + 1);
#pragma unroll 1
    for (int z = zb; z < ze; ++z) {
      if (z + 1 < ze) issue(z + 2);
      if (inside) {
        const long long s = (unsigned)z * plane + soff;
#pragma unroll
        for (int j = 0; j < 3; ++j) acc.qpl[j] = sQ + ((z + 3 + j) & 3) * QSL;
        // output cotangents: H 0-4, mu 5, sigma 6-14
        T lo[15];
        const Quad<T> l0 = ld_quad(A.L, s), l1 = ld_quad(A.L + 4 * N, s);
        const Vec2<T> l2 = ld_pair(A.L + 8 * N, s);
        lo[6] = l0.x, lo[7] = l0.y, lo[8] = l0.z, lo[9] = l0.w;
        lo[10] = l1.x, lo[11] = l1.y, lo[12] = l1.z, lo[13] = l1.w;
        lo[14] = l2.x, lo[5] = l2.y;
#pragma unroll
        for (int k = 0; k < 5; ++k) lo[k] = c.gammaQ * ld(A.lq + k * N + s);
        T in[36];
        {
          T q0[5], pc, dq[3][5], lapq[5], dp[3], lapp, hp[6];
          gather_fields<T>(acc, q0, pc, dq, lapq, dp, lapp, hp);
#pragma unroll
          for (int k = 0; k < 5; ++k) in[k] = q0[k];
          in[5] = pc;
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int k = 0; k < 5; ++k) in[6 + 5 * a + k] = dq[a][k];
#pragma unroll
          for (int k = 0; k < 5; ++k) in[21 + k] = lapq[k];
#pragma unroll
          for (int a = 0; a < 3; ++a) in[26 + a] = dp[a];
          in[29] = lapp;
#pragma unroll
          for (int k = 0; k < 6; ++k) in[30 + k] = hp[k];
        }
        T ci[24], lH[5], lmo, lz, lq0;
        local_fields_vjp<T>(c, in, lo, ci, lH, lmo, lz, lq0);
#pragma unroll
        for (int k = 0; k < 5; ++k) A.oq[k * N + s] += ci[k];
        A.op[s] += ci[5];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          st_quad_at(A.B + 4 * a * N, s, ci[6 + 5 * a], ci[7 + 5 * a], ci[8 + 5 * a], ci[9 + 5 * a]);
          st_pair_at(A.B + (16 + 2 * a) * N, s, ci[10 + 5 * a], ci[21 + a]);
        }
        st_quad_at(A.B + 12 * N, s, lH[0], lH[1], lH[2], lH[3]);
        st_pair_at(A.B + 22 * N, s, lH[4], lmo);
        pz += (double)lz;
        pq += (double)lq0;
      }
      cp_async_commit_wait_all();
      __syncthreads();
    }
  }
  // per-block FP64 sums of the parameter gradients (fixed order: deterministic), added to the block's own over the
  // reverse steps; one pass over the blocks at the end sums them
  __shared__ double sh[2][G::NT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    pz += __shfl_down_sync(0xffffffffu, pz, o);
    pq += __shfl_down_sync(0xffffffffu, pq, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { sh[0][wid] = pz; sh[1][wid] = pq; }
  __syncthreads();
  if (threadIdx.x < 2) {
    double a0 = 0.0;
    for (int w = 0; w < G::NT / 32; ++w) a0 += sh[threadIdx.x][w];
    A.pgrad[2 * blockIdx.x + threadIdx.x] += a0;
  }
}

// ---------------------------------------------------------------- RK4
// Transposes of gather_fields, added to the partial cotangents of Q and psi:
//   d_a f(x) = sum_i 3 w_i c_ia f(x + c_i),  lap f(x) = sum_i lw_i f(x + c_i) - 4 f(x),
//   hess_aa f(x) = f(x + e_a) + f(x - e_a) - 2 f(x),
//   hess_ab f(x) = 1/4 sum_{edges in the ab plane} c_a c_b f(x + c),
// with the cotangents K lH of lap Q, -kphi lmu of lap psi and -2 W lmu (Q_aa; 2 Q_ab) of the Hessian.
template <typename T>
__global__ void __launch_bounds__(kAdjBlock) k_adj_gather(AdjDesc<T> A) {
  const InstDesc<T>& I = A.I;
  const long long N = I.N;
  long long s;
  Nbr nb;
  if (!adj_site(I.nx, I.ny, I.nz, N, s, nb)) return;
  const Coef<T>& c = I.c;
  const T* __restrict__ q = I.q_in;
  T dq[5], lapH[5], dps = T(0), lapm, hess;
  {
    const Quad<T> h = ld_quad(A.B + 12 * N, s);
    const Vec2<T> h4 = ld_pair(A.B + 22 * N, s);
    lapH[0] = -T(4) * h.x;
    lapH[1] = -T(4) * h.y;
    lapH[2] = -T(4) * h.z;
    lapH[3] = -T(4) * h.w;
    lapH[4] = -T(4) * h4.x;
    lapm = -T(4) * h4.y;
    hess = T(0);  // -2 (Q_xx + Q_yy + Q_zz) lmu = 0: Q is traceless
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) dq[k] = T(0);
#pragma unroll
  for (int i = 1; i < 19; ++i) {
    const int cx = lat_c(i, 0), cy = lat_c(i, 1), cz = lat_c(i, 2);
    const long long m = nb.off(-cx, -cy, -cz);  // x = y - c_i reads f(y) through c_i
    const bool face = lat_c2(i) == 1;
    const T gw = face ? T(1.0 / 6.0) : T(1.0 / 12.0);
    const T lw = face ? T(1.0 / 3.0) : T(1.0 / 6.0);
    const int cc[3] = {cx, cy, cz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (cc[a] == 0) continue;
      const T w = cc[a] > 0 ? gw : -gw;
      const Quad<T> d = ld_quad(A.B + 4 * a * N, m);
      const Vec2<T> e = ld_pair(A.B + (16 + 2 * a) * N, m);
      dq[0] += w * d.x;
      dq[1] += w * d.y;
      dq[2] += w * d.z;
      dq[3] += w * d.w;
      dq[4] += w * e.x;
      dps += w * e.y;
    }
    const Quad<T> h = ld_quad(A.B + 12 * N, m);
    const Vec2<T> h4 = ld_pair(A.B + 22 * N, m);
    lapH[0] += lw * h.x;
    lapH[1] += lw * h.y;
    lapH[2] += lw * h.z;
    lapH[3] += lw * h.w;
    lapH[4] += lw * h4.x;
    lapm += lw * h4.y;
    if (face) {
      const T Qaa = cx ? ld(q + m) : (cy ? ld(q + 3 * N + m) : -ld(q + m) - ld(q + 3 * N + m));
      hess += Qaa * h4.y;
    } else {
      const int k = cz == 0 ? 1 : (cy == 0 ? 2 : 4);  // Q_xy, Q_xz, Q_yz
      hess += (T(0.5) * T(cx * cy + cx * cz + cy * cz)) * (ld(q + k * N + m) * h4.y);
    }
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) A.oq[k * N + s] += dq[k] + c.K * lapH[k];
  A.op[s] += dps - c.kphi * lapm - c.W2 * hess;
}

// ---------------------------------------------------------------- objective seed
// J = |X(T) - X(0)|^2 / 2 with X_a = (L_a / 2 pi) atan2(S_a, C_a), S_a = sum phi_c sin,
// C_a = sum phi_c cos, phi_c = (1 + psi)/2.  dJ/dpsi(x) = sum_a dX_a coef_a
// (C_a sin th_a(x) - S_a cos th_a(x)) / 2, coef_a = (L_a / 2 pi) / (C_a^2 + S_a^2).
template <typename T>
__global__ void k_adj_seed(InstDesc<T> I, double dX0, double dX1, double dX2, double k0s, double k0c, double k1s,
                           double k1c, double k2s, double k2c, T* lp) {
  const long long N = I.N;
  const double two_pi = 6.283185307179586476925286766559;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(s % I.nx);
    const long long t = s / I.nx;
    const int y = (int)(t % I.ny), z = (int)(t / I.ny);
    double sx, cx, sy, cy, sz, cz;
    sincos(two_pi * x / I.nx, &sx, &cx);
    sincos(two_pi * y / I.ny, &sy, &cy);
    sincos(two_pi * z / I.nz, &sz, &cz);
    const double v = 0.5 * (dX0 * (k0s * sx - k0c * cx) + dX1 * (k1s * sy - k1c * cy) + dX2 * (k2s * sz - k2c * cz));
    lp[s] = (T)v;
  }
}

// Cotangent of a stored state, written in the lbcad_get_fields layout: populations as the
// pre-collision f_i(x) = g*_i(x - c_i) (so lam f_i(x) = lam g*_i(x - c_i)), then U, Q, PSI.
template <typename T>
__global__ void k_adj_export(InstDesc<T> I, const T* __restrict__ lg, const T* __restrict__ lq,
                             const T* __restrict__ lp, const T* __restrict__ lu, long long oG, long long oU,
                             long long oQ, long long oP, double* __restrict__ dst) {
  const long long N = I.N;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(s % I.nx);
    const long long t = s / I.nx;
    const int y = (int)(t % I.ny), z = (int)(t / I.ny);
    if (oG >= 0) {
      const Nbr nb = make_nbr(x, y, z, I.nx, I.ny, I.nz);
#pragma unroll
      for (int i = 0; i < 19; ++i)
        dst[oG + i * N + s] = (double)lg[i * N + nb.off(-lat_c(i, 0), -lat_c(i, 1), -lat_c(i, 2))];
    }
    if (oU >= 0)
      for (int a = 0; a < 3; ++a) dst[oU + a * N + s] = (double)lu[a * N + s];
    if (oQ >= 0)
      for (int k = 0; k < 5; ++k) dst[oQ + k * N + s] = (double)lq[k * N + s];
    if (oP >= 0) dst[oP + s] = (double)lp[s];
  }
}

// ---------------------------------------------------------------- launchers
template <typename T, bool SHIFT>
cudaError_t LaunchAdj<T, SHIFT>::export_fields(const InstDesc<T>& I, const T* lam, uint32_t mask, double* dst,
                                               cudaStream_t s) {
  const long long N = I.N;
  long long o = 0, oG = -1, oU = -1, oQ = -1, oP = -1;
  if (mask & 1u) { oG = o; o += 19 * N; }
  if (mask & 4u) { oU = o; o += 3 * N; }
  if (mask & 8u) { oQ = o; o += 5 * N; }
  if (mask & 16u) { oP = o; o += N; }
  k_adj_export<T><<<grid_for(N, 256), 256, 0, s>>>(I, lam, lam + 19 * N, lam + 24 * N, lam + 25 * N, oG, oU, oQ, oP,
                                                     dst);
  return cudaGetLastError();
}
template <typename T, bool SHIFT>
cudaError_t LaunchAdj<T, SHIFT>::reverse_step(const AdjDescHost<T>& h, cudaStream_t s) {
  AdjDesc<T> A;
  A.I = h.I;
  A.F = h.F;
  A.lg = h.lg; A.lq = h.lq; A.lp = h.lp; A.lu = h.lu;
  A.A = h.A; A.L = h.L; A.B = h.B;
  A.og = h.og; A.oq = h.oq; A.op = h.op; A.ou = h.ou;
  A.pgrad = h.pgrad;
  const unsigned nb = (unsigned)((h.I.N + kAdjBlock - 1) / kAdjBlock);
  k_adj_update<T, SHIFT><<<nb, kAdjBlock, 0, s>>>(A);
  k_adj_spread<T><<<nb, kAdjBlock, 0, s>>>(A);
  k_adj_fields<T><<<h.work.grid, kAdjBlock, 0, s>>>(A, h.work.items, h.work.nitems);
  k_adj_gather<T><<<nb, kAdjBlock, 0, s>>>(A);
  return cudaGetLastError();
}

template <typename T, bool SHIFT>
cudaError_t LaunchAdj<T, SHIFT>::fields_shape(int* tx, int* ty, int* per_sm) {
  *tx = AdjTile::TX;
  *ty = AdjTile::TY;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_adj_fields<T>, kAdjBlock, 0);
}

template <typename T, bool SHIFT>
cudaError_t LaunchAdj<T, SHIFT>::seed(const InstDesc<T>& I, const double dX[3], const double ks[3],
                                      const double kc[3], T* lp, cudaStream_t s) {
  k_adj_seed<T><<<grid_for(I.N, 256), 256, 0, s>>>(I, dX[0], dX[1], dX[2], ks[0], kc[0], ks[1], kc[1], ks[2], kc[2], lp);
  return cudaGetLastError();
}

}  // namespace lbcad
