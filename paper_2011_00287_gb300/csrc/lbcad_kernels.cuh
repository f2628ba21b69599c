// lbcad_kernels.cuh -- CUDA kernels of the hybrid LB step, templated on the compute
// type T (float or double) and on SHIFT (populations stored as f_i - w_i rho0).
//
// The per-site device functions every path shares (stencils, local fields, order-parameter
// update, collision), the a6 pass, and the per-site kernels of the two cross-check paths.
// On the two-kernel path one step (Sec. 3 of Carenza, Gonnella & Negro) runs as:
//   k_fields : isotropic D3Q19 stencils of Q and psi -> molecular field H (Eq. 2, 5),
//              chemical potential mu (Eq. 1, 5) and total stress sigma (Eq. 3, 4)
//              into scratch;
//   k_update : F = div sigma, BGK + Guo collision of the pulled populations (Eqs. 6-8),
//              Beris-Edwards update of Q with upwind advection and co-rotation (Eq. 2),
//              Cahn-Hilliard update of psi in upwind flux form (Eq. 1).
// Layout: every field is [component][z][y][x] (x fastest) per instance; neighbour reads
// are coalesced along x and served by L1/L2.
#pragma once

#include "lbcad_internal.h"

namespace lbcad {

template <typename T>
__device__ __forceinline__ T ld(const T* p) {
  return __ldg(p);
}

template <typename T>
__device__ __forceinline__ int find_inst(const InstDesc<T>* __restrict__ D, int n, long long b) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (D[mid].blk0 <= b) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Periodic neighbour offsets of one site: off(dx, dy, dz) for dx, dy, dz in {-1, 0, 1}.
struct Nbr {
  int xo[3];
  int yo[3];
  long long zo[3];
  __device__ __forceinline__ long long off(int dx, int dy, int dz) const {
    return (long long)xo[dx + 1] + yo[dy + 1] + zo[dz + 1];
  }
};

__device__ __forceinline__ Nbr make_nbr(int x, int y, int z, int nx, int ny, int nz) {
  Nbr n;
  n.xo[0] = x ? x - 1 : nx - 1;
  n.xo[1] = x;
  n.xo[2] = (x + 1 < nx) ? x + 1 : 0;
  n.yo[0] = (y ? y - 1 : ny - 1) * nx;
  n.yo[1] = y * nx;
  n.yo[2] = ((y + 1 < ny) ? y + 1 : 0) * nx;
  const long long pl = (long long)nx * ny;
  n.zo[0] = (z ? z - 1 : nz - 1) * pl;
  n.zo[1] = z * pl;
  n.zo[2] = ((z + 1 < nz) ? z + 1 : 0) * pl;
  return n;
}

// Periodic offsets of the sites at distance up to 2 along each axis (radius-2 stencils;
// every edge is >= 4, so one wrap suffices).
struct NbrR2 {
  int xo[5];
  int yo[5];
  long long zo[5];
  __device__ __forceinline__ long long off(int dx, int dy, int dz) const {
    return (long long)xo[dx + 2] + yo[dy + 2] + zo[dz + 2];
  }
};

__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

__device__ __forceinline__ NbrR2 make_nbr_r2(int x, int y, int z, int nx, int ny, int nz) {
  NbrR2 n;
  const long long pl = (long long)nx * ny;
#pragma unroll
  for (int d = -2; d <= 2; ++d) {
    n.xo[d + 2] = wrap1(x + d, nx);
    n.yo[d + 2] = wrap1(y + d, ny) * nx;
    n.zo[d + 2] = wrap1(z + d, nz) * pl;
  }
  return n;
}

// Neighbour map of stencil set ST: 0 = isotropic D3Q19 (radius 1), 1 = fourth order (radius 2).
template <int ST>
__device__ __forceinline__ auto make_nbr_st(int x, int y, int z, int nx, int ny, int nz) {
  if constexpr (ST == 1) return make_nbr_r2(x, y, z, nx, ny, nz);
  else return make_nbr(x, y, z, nx, ny, nz);
}

// Full symmetric traceless tensor from the five stored components xx, xy, xz, yy, yz.
template <typename T>
__device__ __forceinline__ void full3(const T q[5], T Q[3][3]) {
  Q[0][0] = q[0]; Q[0][1] = q[1]; Q[0][2] = q[2];
  Q[1][0] = q[1]; Q[1][1] = q[3]; Q[1][2] = q[4];
  Q[2][0] = q[2]; Q[2][1] = q[4]; Q[2][2] = -q[0] - q[3];
}

// Two-lane values for packed arithmetic: float2 uses the f32x2 instructions (one issue
// slot for two lanes); other types fall back to two scalar operations.
template <typename T>
struct Vec2 {
  T x, y;
};
template <typename T>
__device__ __forceinline__ Vec2<T> v2(T a, T b) { return Vec2<T>{a, b}; }
// Every multiply-add is an explicit fma and every lone product is rounded on its own, so the
// stencils round identically in every kernel that inlines them, whatever the compiler would
// contract.  Scalar overloads let one stencil serve single fields and pairs.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add2(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add2(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub2(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub2(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float fma2(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma2(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mul2(float a, float b) { return mul_rn(a, b); }
__device__ __forceinline__ double mul2(double a, double b) { return mul_rn(a, b); }
__device__ __forceinline__ float2 f2(Vec2<float> a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ Vec2<float> v2f(float2 a) { return Vec2<float>{a.x, a.y}; }
__device__ __forceinline__ Vec2<float> add2(Vec2<float> a, Vec2<float> b) { return v2f(__fadd2_rn(f2(a), f2(b))); }
__device__ __forceinline__ Vec2<float> sub2(Vec2<float> a, Vec2<float> b) {
  return v2f(__ffma2_rn(f2(b), make_float2(-1.f, -1.f), f2(a)));  // a - b, one rounding
}
__device__ __forceinline__ Vec2<float> fma2(Vec2<float> a, Vec2<float> b, Vec2<float> c) {
  return v2f(__ffma2_rn(f2(a), f2(b), f2(c)));
}
__device__ __forceinline__ Vec2<float> mul2(Vec2<float> a, Vec2<float> b) { return v2f(__fmul2_rn(f2(a), f2(b))); }
__device__ __forceinline__ Vec2<double> add2(Vec2<double> a, Vec2<double> b) {
  return Vec2<double>{add2(a.x, b.x), add2(a.y, b.y)};
}
__device__ __forceinline__ Vec2<double> sub2(Vec2<double> a, Vec2<double> b) {
  return Vec2<double>{sub2(a.x, b.x), sub2(a.y, b.y)};
}
__device__ __forceinline__ Vec2<double> fma2(Vec2<double> a, Vec2<double> b, Vec2<double> c) {
  return Vec2<double>{fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}
__device__ __forceinline__ Vec2<double> mul2(Vec2<double> a, Vec2<double> b) {
  return Vec2<double>{mul_rn(a.x, b.x), mul_rn(a.y, b.y)};
}
// The constant k in every lane of a value of type V.
template <class V>
struct Bcast {
  __device__ __forceinline__ static V of(double k) { return V(k); }
};
template <typename T>
struct Bcast<Vec2<T>> {
  __device__ __forceinline__ static Vec2<T> of(double k) { return Vec2<T>{T(k), T(k)}; }
};

// Gradient (1/12)[2 D_face + signed edge pairs] from opposite-pair differences D[i] =
// f(c_i) - f(c_{i+1}) of one field or two (V = T or Vec2<T>).
template <class V>
__device__ __forceinline__ void grad_from_pairs(const V D[19], V g[3]) {
  const V k2 = Bcast<V>::of(2.0), k12 = Bcast<V>::of(1.0 / 12.0);
  g[0] = mul2(fma2(D[1], k2, add2(add2(D[7], D[9]), add2(D[11], D[13]))), k12);
  g[1] = mul2(fma2(D[3], k2, add2(sub2(D[7], D[9]), add2(D[15], D[17]))), k12);
  g[2] = mul2(fma2(D[5], k2, add2(sub2(D[11], D[13]), sub2(D[15], D[17]))), k12);
}

// Stress and chemical potential as five pairs, the unit of the tiles in shared memory:
// pair j of a site holds (sigma_xb, sigma_yb) for j = b = 0, 1, 2, (sigma_zx, sigma_zy) for
// j = 3 and (sigma_zz, mu) for j = 4.  sig_pair(c) = j and sig_lane(c) = lane of sigma_c
// (c = 3a + b); mu sits in pair 4, lane 1.
__host__ __device__ constexpr int sig_pair(int c) { return c < 6 ? c % 3 : (c < 8 ? 3 : 4); }
__host__ __device__ constexpr int sig_lane(int c) { return c < 6 ? c / 3 : (c < 8 ? c - 6 : 0); }
// the two stress components of pair j (the second is -1 for mu)
__host__ __device__ constexpr int pair_c0(int j) { return j < 3 ? j : (j == 3 ? 6 : 8); }
__host__ __device__ constexpr int pair_c1(int j) { return j < 3 ? j + 3 : (j == 3 ? 7 : -1); }

// H (5), mu and the total stress sigma (9, row-major a*3+b) at one site from Q, psi and
// their stencils: dq[a][k] = d_a of stored component k, lapq[k], dp[a] = d_a psi,
// lapp, hp = Hessian of psi (xx, yy, zz, xy, xz, yz).
template <typename T>
__device__ __forceinline__ void local_fields(const Coef<T>& c, const T q[5], T psi, const T dq[3][5],
                                             const T lapq[5], const T dp[3], T lapp, const T hp[6], T H[5],
                                             T& mu, T sig[9]) {
  T Q[3][3];
  full3(q, Q);
  T dQ[3][3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) full3(dq[a], dQ[a]);
  const T third = T(1.0 / 3.0);
  // Q.Q is symmetric: six products
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
  // curl: C_ab = eps_amn d_m Q_nb, and its symmetric part CC = C + C^T
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
    for (int j = i; j < 3; ++j) {
      CC[i][j] = C[i][j] + C[j][i];
      CC[j][i] = CC[i][j];
    }
  const T g2 = dp[0] * dp[0] + dp[1] * dp[1] + dp[2] * dp[2];
  const T Ac = c.A0chis * psi + c.A0chi1;  // A0 chi
  const T lin = Ac * (third - trQ2) - c.cL;
  const T iso = third * (Ac * trQ2 - c.W * g2);
  const T Wdp[3] = {c.W * dp[0], c.W * dp[1], c.W * dp[2]};
  // H = -dF/dQ (traceless symmetric by construction: tr CC = 0 for symmetric Q)
  const int I5[5] = {0, 0, 0, 1, 1};
  const int J5[5] = {0, 1, 2, 1, 2};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int i = I5[k], j = J5[k];
    T h = lin * Q[i][j] + Ac * QQ[i][j] + c.K * lapq[k] - c.Kq * CC[i][j] - Wdp[i] * dp[j];
    if (i == j) h -= iso;
    H[k] = h;
  }
  T Hf[3][3];
  full3(H, Hf);

  // mu = dF/dpsi
  const T Qh = Q[0][0] * hp[0] + Q[1][1] * hp[1] + Q[2][2] * hp[2] +
               T(2) * (Q[0][1] * hp[3] + Q[0][2] * hp[4] + Q[1][2] * hp[5]);
  T divQdp = T(0);
#pragma unroll
  for (int b = 0; b < 3; ++b) divQdp += (dQ[0][0][b] + dQ[1][1][b] + dQ[2][2][b]) * dp[b];
  const T psi2 = psi * psi;
  const T bulk = trQ2 * (T(0.25) * trQ2 - T(1.0 / 6.0)) - third * trQ3;
  mu = psi * (c.b * psi2 - c.a) - c.kphi * lapp + c.A0chis * bulk - c.W2 * (divQdp + Qh);

  // Elastic stress E_ab = K dQ_a : dQ_b + Kq v_b(dQ_a), v_b(M) = eps_bgm (M Q)_gm the axial vector
  // of M Q.  Both are linear in dQ_a, so E_ab = dQ_a : t_b with one symmetric t_b = K dQ_b +
  // Kq n_b per b; on the five stored components of the traceless dQ_a it takes five products
  // (off-diagonal entries of t doubled, t_zz subtracted from the diagonal).
  const T kxy = c.Kq * Q[0][1], kxz = c.Kq * Q[0][2], kyz = c.Kq * Q[1][2];
  const T kzy = c.Kq * (Q[2][2] - Q[1][1]), kxx = c.Kq * (Q[0][0] - Q[2][2]), kyx = c.Kq * (Q[1][1] - Q[0][0]);
  T t[3][5];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const T ax = T(2) * dq[b][0] + dq[b][3], ay = dq[b][0] + T(2) * dq[b][3];
    t[b][0] = c.K * ax + (b == 0 ? kyz : b == 1 ? -T(2) * kxz : kxy);
    t[b][3] = c.K * ay + (b == 0 ? T(2) * kyz : b == 1 ? -kxz : -kxy);
    t[b][1] = c.K2 * dq[b][1] + (b == 0 ? kxz : b == 1 ? -kyz : kyx);
    t[b][2] = c.K2 * dq[b][2] + (b == 0 ? -kxy : b == 1 ? kxx : kyz);
    t[b][4] = c.K2 * dq[b][4] + (b == 0 ? kzy : b == 1 ? kxy : -kxz);
  }
  T E[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      E[a][b] = dq[a][0] * t[b][0] + dq[a][1] * t[b][1] + dq[a][2] * t[b][2] + dq[a][3] * t[b][3] + dq[a][4] * t[b][4];
  // Q:curl Q (= sum_a v_a(dQ_a)), Q.grad psi
  const T QC = Q[0][0] * C[0][0] + Q[1][1] * C[1][1] + Q[2][2] * C[2][2] + Q[0][1] * CC[0][1] +
               Q[0][2] * CC[0][2] + Q[1][2] * CC[1][2];
  T Qdp[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) Qdp[i] = Q[i][0] * dp[0] + Q[i][1] * dp[1] + Q[i][2] * dp[2];
  const T anch = dp[0] * Qdp[0] + dp[1] * Qdp[1] + dp[2] * Qdp[2];
  // K/2 dQ:dQ + Kq Q:curl Q = (tr E + Kq Q:curl Q)/2; the A0 terms are A0/2 trQ2 + A0 chi bulk
  const T fden = psi2 * (c.bq * psi2 - c.ah) + c.kh * g2 + c.fQ2 * trQ2 + Ac * bulk +
                 T(0.5) * (E[0][0] + E[1][1] + E[2][2] + c.Kq * QC) + c.W * anch;
  const T P0 = psi * mu - fden;

  // reactive and active parts: with (HQ)_ab = (QH)_ba,
  //   -xi (HQ~ + Q~H) + 2 xi Q~ tr(QH) + QH - HQ - zeta phi_c Q
  //   = (1 - xi) QH - (1 + xi) HQ - (2 xi/3) H + (2 xi tr(QH) - zeta phi_c) Q + (2 xi/3) tr(QH) I
  T QH[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) QH[i][j] = Q[i][0] * Hf[0][j] + Q[i][1] * Hf[1][j] + Q[i][2] * Hf[2][j];
  const T trQH = QH[0][0] + QH[1][1] + QH[2][2];
  const T cQ = c.xi2 * trQH - (c.zh * psi + c.zh);  // zeta phi_c = zeta (1 + psi)/2
  const T cI = c.xi23 * trQH - P0;
  T wv[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) wv[b] = c.kphi * dp[b] + c.W2 * Qdp[b];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      const T sb = cQ * Q[a][b] - c.xi23 * Hf[a][b];  // the part symmetric in a, b
      if (a == b) {
        sig[4 * a] = sb + cI - c.xi2 * QH[a][a] - E[a][a] - dp[a] * wv[a];
      } else {
        sig[3 * a + b] = sb + c.xim * QH[a][b] - c.xip * QH[b][a] - E[a][b] - dp[a] * wv[b];
        sig[3 * b + a] = sb + c.xim * QH[b][a] - c.xip * QH[a][b] - E[b][a] - dp[b] * wv[a];
      }
    }
}

// ---------------------------------------------------------------- shared per-site pieces
// Every step path evaluates its stencils with the functions below, in the same order and with
// the same arithmetic, through an accessor A that returns neighbour values: pairs of fields
// A::pair(j, ...) (see gather_fields), pairs of stresses A::spair(j, ...) (see sig_pair) and
// the velocity A::u3(...).
//
// The 19-point stencils (rest, six faces, twelve edges) are sums over three planes z-1, z, z+1
// of in-plane sums, and the in-plane sums of a plane serve three output planes.  So the
// stencils are written as carries: advance() takes the nine points of one new plane, finishes
// the output of the plane before it and keeps what the next plane needs.  A kernel that
// marches up z reads nine points per field and plane instead of 19 and adds 38 instead of 63
// times; a per-site kernel runs the same carry over its three planes, so that all paths round
// alike.  With D f the in-plane difference f(+1) - f(-1), S the sum of the four in-plane
// neighbours' differences to the centre, S2 that of the four diagonal ones, and f+- the
// plane's centre value above and below:
//   d_x f = [2 D_x + D_x(y+1) + D_x(y-1) + D_x(z+1) + D_x(z-1)] / 12,   d_y likewise,
//   d_z f = [(6 (f+ - f) + S(z+1)) - (6 (f- - f) + S(z-1))] / 12,
//   lap f = [2 S + S2 + (6 (f+ - f) + S(z+1)) + (6 (f- - f) + S(z-1))] / 6.
// Sums are taken of differences to a centre value, which keeps them free of cancellation in
// FP32.

// a1: gradient and Laplacian of the five Q components and psi, and the Hessian of psi
// (three-point differences on the diagonal, four corners off it).  The six fields are
// taken in pairs (Q_xx, Q_xy), (Q_xz, Q_yy), (Q_yz, psi), so one two-lane operation advances
// two fields.
template <typename T>
struct FieldsCarry {
  using V = Vec2<T>;
  V c[3], dx[3], dy[3], s4[3];  // of the last plane: value, differences, sum over the neighbours
  V A[3], B[3];                 // its own part of 12 d_x, 12 d_y and that of the plane below
  V L[3], Z[3];                 // ... of 6 lap, and the part of the plane below of 12 d_z
  T hxx, hyy, hxy;              // psi: in-plane second differences of the last plane
  T px, py, fm;                 // psi: dx, dy of the plane below, and psi there minus psi
  __device__ __forceinline__ FieldsCarry() {
#pragma unroll
    for (int j = 0; j < 3; ++j) c[j] = dx[j] = dy[j] = s4[j] = A[j] = B[j] = L[j] = Z[j] = V{T(0), T(0)};
    hxx = hyy = hxy = px = py = fm = T(0);
  }
  // pl(j, cx, cy): pair j of the new plane.  Outputs: the plane before it.
  template <class P>
  __device__ __forceinline__ void advance(const P& pl, T q0[5], T& p0, T dq[3][5], T lapq[5], T dp[3], T& lapp,
                                          T hp[6]) {
    const V k2 = Bcast<V>::of(2.0), k6 = Bcast<V>::of(6.0), m6 = Bcast<V>::of(-6.0);
    const V k12i = Bcast<V>::of(1.0 / 12.0), k6i = Bcast<V>::of(1.0 / 6.0);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const V f0 = pl(j, 0, 0), fe = pl(j, 1, 0), fw = pl(j, -1, 0), fn = pl(j, 0, 1), fs = pl(j, 0, -1);
      const V ne = pl(j, 1, 1), sw = pl(j, -1, -1), se = pl(j, 1, -1), nw = pl(j, -1, 1);
      const V ndx = sub2(fe, fw), ndy = sub2(fn, fs);
      const V sx = add2(sub2(fe, f0), sub2(fw, f0)), sy = add2(sub2(fn, f0), sub2(fs, f0));
      const V ns4 = add2(sx, sy);
      const V s1 = add2(sub2(ne, f0), sub2(sw, f0)), s2 = add2(sub2(se, f0), sub2(nw, f0));
      const V p = sub2(ne, sw), m = sub2(se, nw);
      const V gx = fma2(k2, ndx, add2(p, m)), gy = fma2(k2, ndy, sub2(p, m));
      const V lp = fma2(k2, ns4, add2(s1, s2));
      // the plane before
      const V fp = sub2(f0, c[j]);
      const V e = fma2(k6, fp, ns4);
      const V ox = mul2(add2(A[j], ndx), k12i), oy = mul2(add2(B[j], ndy), k12i);
      const V oz = mul2(sub2(e, Z[j]), k12i), ol = mul2(add2(L[j], e), k6i);
      const int k0 = 2 * j;
      q0[k0] = c[j].x;
      dq[0][k0] = ox.x;
      dq[1][k0] = oy.x;
      dq[2][k0] = oz.x;
      lapq[k0] = ol.x;
      if (j < 2) {
        q0[k0 + 1] = c[j].y;
        dq[0][k0 + 1] = ox.y;
        dq[1][k0 + 1] = oy.y;
        dq[2][k0 + 1] = oz.y;
        lapq[k0 + 1] = ol.y;
      } else {
        p0 = c[j].y;
        dp[0] = ox.y;
        dp[1] = oy.y;
        dp[2] = oz.y;
        lapp = ol.y;
        hp[0] = hxx;
        hp[1] = hyy;
        hp[2] = add2(fp.y, fm);
        hp[3] = hxy;
        hp[4] = mul_rn(T(0.25), sub2(ndx.y, px));
        hp[5] = mul_rn(T(0.25), sub2(ndy.y, py));
        hxx = sx.y;
        hyy = sy.y;
        hxy = mul_rn(T(0.25), sub2(s1.y, s2.y));
        px = dx[j].y;
        py = dy[j].y;
        fm = -fp.y;
      }
      // this plane
      Z[j] = fma2(m6, fp, s4[j]);
      A[j] = add2(gx, dx[j]);
      B[j] = add2(gy, dy[j]);
      L[j] = add2(lp, Z[j]);
      c[j] = f0;
      dx[j] = ndx;
      dy[j] = ndy;
      s4[j] = ns4;
    }
  }
};

// The same at one site, from its three planes.
template <typename T, class A>
__device__ __forceinline__ void gather_fields(const A& acc, T q0[5], T& p0, T dq[3][5], T lapq[5], T dp[3],
                                              T& lapp, T hp[6]) {
  FieldsCarry<T> car;
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
    car.advance([&](int j, int cx, int cy) { return acc.pair(j, cx, cy, cz); }, q0, p0, dq, lapq, dp, lapp, hp);
}

// a3 (divergence): F_a = d_b sigma_ab, through the stress pairs of a plane: (F_x, F_y) from
// pairs 0-2 two lanes at a time, F_z from pair 3 (sigma_zx, sigma_zy) and lane 0 of pair 4
// (sigma_zz).
template <class V>
struct DivCarry {
  V P, A1, s4, c;  // the last plane's sum so far; its in-plane differences; of sigma_az: neighbours, value
  __device__ __forceinline__ DivCarry() { P = A1 = s4 = c = Bcast<V>::of(0.0); }
  // x(cx, cy), y(cx, cy), z(cx, cy): sigma_ax, sigma_ay, sigma_az of the new plane; returns F of
  // the plane before it.
  template <class X, class Y, class Zf>
  __device__ __forceinline__ V advance(const X& x, const Y& y, const Zf& z) {
    const V k2 = Bcast<V>::of(2.0), k6 = Bcast<V>::of(6.0), m6 = Bcast<V>::of(-6.0), k12i = Bcast<V>::of(1.0 / 12.0);
    const V a1 = add2(sub2(x(1, 0), x(-1, 0)), sub2(y(0, 1), y(0, -1)));
    const V d = add2(add2(sub2(x(1, 1), x(-1, -1)), sub2(x(1, -1), x(-1, 1))),
                     sub2(sub2(y(1, 1), y(-1, -1)), sub2(y(1, -1), y(-1, 1))));
    const V z0 = z(0, 0);
    const V ns4 = add2(add2(sub2(z(1, 0), z0), sub2(z(-1, 0), z0)), add2(sub2(z(0, 1), z0), sub2(z(0, -1), z0)));
    const V e = sub2(z0, c);
    const V F = mul2(add2(P, add2(a1, fma2(k6, e, ns4))), k12i);
    P = sub2(add2(fma2(k2, a1, d), A1), fma2(m6, e, s4));
    A1 = a1;
    s4 = ns4;
    c = z0;
    return F;
  }
};
template <typename T>
struct ForceCarry {
  DivCarry<Vec2<T>> xy;
  DivCarry<T> z;
  template <class P>
  __device__ __forceinline__ void advance(const P& sp, T F[3]) {
    const Vec2<T> f = xy.advance([&](int cx, int cy) { return sp(0, cx, cy); },
                                 [&](int cx, int cy) { return sp(1, cx, cy); },
                                 [&](int cx, int cy) { return sp(2, cx, cy); });
    F[0] = f.x;
    F[1] = f.y;
    F[2] = z.advance([&](int cx, int cy) { return sp(3, cx, cy).x; }, [&](int cx, int cy) { return sp(3, cx, cy).y; },
                     [&](int cx, int cy) { return sp(4, cx, cy).x; });
  }
};

// Laplacian of one field; f(cx, cy): the new plane.
template <typename T>
struct LapCarry {
  T c = T(0), s4 = T(0), L = T(0), fm = T(0);
  template <class P>
  __device__ __forceinline__ T advance(const P& f) {
    const T f0 = f(0, 0);
    const T ns4 = add2(add2(sub2(f(1, 0), f0), sub2(f(-1, 0), f0)), add2(sub2(f(0, 1), f0), sub2(f(0, -1), f0)));
    const T s2 = add2(add2(sub2(f(1, 1), f0), sub2(f(-1, -1), f0)), add2(sub2(f(1, -1), f0), sub2(f(-1, 1), f0)));
    const T fp = sub2(f0, c);
    const T lap = mul2(fma2(T(6), add2(fp, fm), add2(L, ns4)), T(1.0 / 6.0));
    L = add2(fma2(T(2), ns4, s2), s4);
    c = f0;
    s4 = ns4;
    fm = -fp;
    return lap;
  }
};

template <typename T, class A>
__device__ __forceinline__ void gather_force(const A& acc, T F[3]) {
  ForceCarry<T> car;
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
    car.advance([&](int j, int cx, int cy) { return acc.spair(j, cx, cy, cz); }, F);
}

// lap mu (lane 1 of stress pair 4).
template <typename T, class A>
__device__ __forceinline__ T gather_lapmu(const A& acc) {
  LapCarry<T> car;
  T l = T(0);
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz) l = car.advance([&](int cx, int cy) { return acc.spair(4, cx, cy, cz).y; });
  return l;
}

// The velocity of one site as (u_x, u_y) and u_z.
template <typename T>
struct Vel3 {
  Vec2<T> xy;
  T z;
};

// W_ab = d_b u_a and the axial face velocities (face slot 2a: u_a at +e_a, 2a+1: at -e_a).
template <typename T, class A>
__device__ __forceinline__ void gather_velocity(const A& acc, T Wg[3][3], T u0[3], T uf[6]) {
  using V = Vec2<T>;
  V f[19], D[19], g[3];
  T fz[19], Dz[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const Vel3<T> v = acc.u3(lat_c(i, 0), lat_c(i, 1), lat_c(i, 2));
    f[i] = v.xy;
    fz[i] = v.z;
  }
#pragma unroll
  for (int i = 1; i < 19; i += 2) {
    D[i] = sub2(f[i], f[i + 1]);
    Dz[i] = sub2(fz[i], fz[i + 1]);
  }
  grad_from_pairs(D, g);
  grad_from_pairs(Dz, Wg[2]);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    Wg[0][b] = g[b].x;
    Wg[1][b] = g[b].y;
  }
  u0[0] = f[0].x;
  u0[1] = f[0].y;
  u0[2] = fz[0];
  uf[0] = f[1].x;
  uf[1] = f[2].x;
  uf[2] = f[3].y;
  uf[3] = f[4].y;
  uf[4] = fz[5];
  uf[5] = fz[6];
}

// Q at the upwind neighbours (side by the sign of u0 along each axis) as the field pairs of
// A::pair, and psi at the six faces.
template <typename T, class A>
__device__ __forceinline__ void gather_upwind(const A& acc, const T u0[3], Vec2<T> qu[3][3], T pf[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int j = 0; j < 3; ++j) qu[a][j] = acc.pair_upwind(j, a, u0[a] > T(0));
#pragma unroll
  for (int i = 1; i < 7; ++i) pf[i - 1] = acc.psi(lat_c(i, 0), lat_c(i, 1), lat_c(i, 2));
}

// The stencils of a4 at one site: W_ab = d_b u_a, Q and psi at the centre, Q at the upwind neighbours, psi and
// the axial velocities at the faces; gather_op: and lap mu.
template <typename T, class A>
__device__ __forceinline__ void gather_advection(const A& acc, T Wg[3][3], T q0[5], Vec2<T> qu[3][3], T& p0, T pf[6],
                                                 T u0[3], T uf[6]) {
  gather_velocity<T>(acc, Wg, u0, uf);
  gather_upwind<T>(acc, u0, qu, pf);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const Vec2<T> v = acc.pair(j, 0, 0, 0);
    q0[2 * j] = v.x;
    if (j < 2) q0[2 * j + 1] = v.y;
    else p0 = v.y;
  }
}
template <typename T, class A>
__device__ __forceinline__ void gather_op(const A& acc, T& lapmu, T Wg[3][3], T q0[5], Vec2<T> qu[3][3], T& p0,
                                          T pf[6], T u0[3], T uf[6]) {
  lapmu = gather_lapmu<T>(acc);
  gather_advection<T>(acc, Wg, q0, qu, p0, pf, u0, uf);
}

// a4, psi: the divergence of the upwind flux of psi.
template <typename T>
__device__ __forceinline__ T flux_divergence(T p0, const T pf[6], const T u0[3], const T uf[6]) {
  T divJ = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int ip = 2 * a, im = 2 * a + 1;
    const T ubp = mul_rn(T(0.5), add2(u0[a], uf[ip]));
    const T ubm = mul_rn(T(0.5), add2(uf[im], u0[a]));
    const T Jm = mul_rn(ubm, ubm > T(0) ? pf[im] : p0);
    divJ = add2(divJ, fma2(ubp, ubp > T(0) ? p0 : pf[ip], -Jm));
  }
  return divJ;
}

// a4, Q: the increment of Q in one step (Eq. 2): co-rotation, Gamma_Q H, and upwind advection
// with the velocity u0.  up (q0 - q_-) + um (q_+ - q0) with up = max(u, 0), um = min(u, 0) is
// |u| (q0 - q_upwind), so only the upwind neighbour qu[a] (field pairs) is read.
template <typename T>
__device__ __forceinline__ void q_increment(const Coef<T>& c, const T Wg[3][3], const T q0[5],
                                            const Vec2<T> qu[3][3], const T u0[3], const T Hs[5], T inc[5]) {
  using V = Vec2<T>;
  V a01 = v2(T(0), T(0)), a23 = v2(T(0), T(0));
  T a4 = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T ua = fabs(u0[a]);
    a01 = fma2(v2(ua, ua), sub2(v2(q0[0], q0[1]), qu[a][0]), a01);
    a23 = fma2(v2(ua, ua), sub2(v2(q0[2], q0[3]), qu[a][1]), a23);
    a4 = fma2(ua, sub2(q0[4], qu[a][2].x), a4);
  }
  const T adv[5] = {a01.x, a01.y, a23.x, a23.y, a4};
  T Q[3][3];
  full3(q0, Q);
  // co-rotation S = (xi D + Om)(Q + I/3) + (Q + I/3)(xi D - Om) - 2 xi tr(QW)(Q + I/3), with
  // D, Om the symmetric and antisymmetric parts of W.  With M = xi D + Om, (xi D - Om) = M^T, so
  // S = P + P^T - 2 xi tr(QW)(Q + I/3) for P = M (Q + I/3); it is projected to its traceless part
  // (its trace is 2 xi tr(D)/3).  M_ij = (xi + 1)/2 W_ij + (xi - 1)/2 W_ji.
  T M[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) M[i][j] = T(0.5) * (c.xip * Wg[i][j] - c.xim * Wg[j][i]);
  T Qt[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Qt[i][j] = i == j ? Q[i][j] + T(1.0 / 3.0) : Q[i][j];
  T trQW = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) trQW += Q[i][j] * Wg[j][i];
  const T trD = Wg[0][0] + Wg[1][1] + Wg[2][2];
  const T cq = -c.xi2 * trQW;
  const T cdiag = -c.xi29 * trD;
  auto P = [&](int i, int j) { return M[i][0] * Qt[0][j] + M[i][1] * Qt[1][j] + M[i][2] * Qt[2][j]; };
  const int I5[5] = {0, 0, 0, 1, 1};
  const int J5[5] = {0, 1, 2, 1, 2};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int i = I5[k], j = J5[k];
    T S = (i == j ? T(2) * P(i, i) : P(i, j) + P(j, i)) + cq * Qt[i][j];
    if (i == j) S += cdiag;
    inc[k] = fma(c.gammaQ, Hs[k], S) - adv[k];
  }
}

// a4 at one site: Beris-Edwards update of Q (Eq. 2) and Cahn-Hilliard update of psi
// (Eq. 1) with the advecting velocity u0/uf (and its gradient Wg).  RHS = false gives the
// Euler step Q + R(Q), RHS = true the right-hand side R(Q) alone (for the Heun stages).
// The increments are summed first and added to Q and psi once: every addition at the
// magnitude of the field rounds to its storage resolution, and three of them per step
// (Q - adv, + S, + Gamma H) added half again to the error that FP32 storage alone causes.
template <typename T, bool RHS>
__device__ __forceinline__ void op_update(const Coef<T>& c, T lapmu, const T Wg[3][3], const T q0[5],
                                          const Vec2<T> qu[3][3], T p0, const T pf[6], const T u0[3], const T uf[6],
                                          const T Hs[5], T qn[5], T& pn) {
  T inc[5];
  q_increment<T>(c, Wg, q0, qu, u0, Hs, inc);
#pragma unroll
  for (int k = 0; k < 5; ++k) qn[k] = RHS ? inc[k] : q0[k] + inc[k];
  const T pinc = fma(c.M, lapmu, -flux_divergence(p0, pf, u0, uf));
  pn = RHS ? pinc : p0 + pinc;
}

// c_i . a of velocity i (components 0, +1, -1).
template <typename T, class V>
__device__ __forceinline__ T dot_c(int i, const T a[3]) {
  T s = T(0);
  bool first = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int ck = V::c(i, k);
    if (ck == 0) continue;
    s = first ? (ck > 0 ? a[k] : -a[k]) : (ck > 0 ? add2(s, a[k]) : sub2(s, a[k]));
    first = false;
  }
  return s;
}

// New values of the velocity pair (i, i+1) of the collision below and, if `two`, of (i+2, i+3), whose weight is
// the same (class k: 1 faces, 2 the others).
template <typename T, class V>
__device__ __forceinline__ void lb_pair_update(const Coef<T>& c, bool two, int i, int k, const T u[3], const T F[3],
                                               T r45, T r3, T base, T uF, T g[V::Q]) {
  using W = Vec2<T>;
  const int j = two ? i + 2 : i;
  const W cu{dot_c<T, V>(i, u), dot_c<T, V>(j, u)}, cF{dot_c<T, V>(i, F), dot_c<T, V>(j, F)};
  auto b = [](T v) { return W{v, v}; };
  const T rest = fma(c.omw[k], base, -mul_rn(c.gw3[k], uF));
  const W X = fma2(b(mul_rn(c.omw[k], r45)), mul2(cu, cu), fma2(mul2(b(c.gw9[k]), cu), cF, b(rest)));
  const W Y = fma2(b(mul_rn(c.omw[k], r3)), cu, mul2(b(c.gw3[k]), cF));
  const W p = fma2(b(c.omc), W{g[i], g[j]}, add2(X, Y)), m = fma2(b(c.omc), W{g[i + 1], g[j + 1]}, sub2(X, Y));
  g[i] = p.x;
  g[i + 1] = m.x;
  if (two) {
    g[j] = p.y;
    g[j + 1] = m.y;
  }
}

// a5 at one site: moments of the pulled populations g and the force F, then BGK + Guo
// collision (Eqs. 6-8); g is overwritten with the post-collision values, u = velocity.
// The equilibrium and forcing terms of opposite velocities c and -c share their even part.
// mom (optional): the site's share of the conserved sums of the new state, mom[0] = mass
// (minus rho0 when SHIFT) and mom[1..3] = post-collision momentum j + F.
template <typename T, bool SHIFT, class V = VelD3Q19>
__device__ __forceinline__ void lb_collide(const Coef<T>& c, const T F[3], T g[V::Q], T u[3], T* mom = nullptr) {
  // moments from opposite pairs
  T m0 = g[0];
  T j[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int i = 1; i < V::Q; i += 2) {
    m0 += g[i] + g[i + 1];
    const T dg = g[i] - g[i + 1];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (V::c(i, a)) j[a] += V::c(i, a) > 0 ? dg : -dg;
  }
  const T rho = SHIFT ? (c.rho0 + m0) : m0;
  const T rinv = T(1) / rho;
  // every product-sum below is an explicit fma: the collision then rounds identically in every
  // kernel that inlines it, whatever the compiler would contract
#pragma unroll
  for (int a = 0; a < 3; ++a) u[a] = fma(T(0.5), F[a], j[a]) * rinv;
  if (mom) {
    mom[0] = m0;
#pragma unroll
    for (int a = 0; a < 3; ++a) mom[1 + a] = j[a] + F[a];
  }
  const T u2 = fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]));
  const T uF = fma(u[2], F[2], fma(u[1], F[1], u[0] * F[0]));
  // BGK + Guo as g' = (1 - om) g + om f_eq + F_i, with the equilibrium
  // w rho (1 + 3 cu + 4.5 cu^2 - 1.5 u^2) (shifted: minus w rho0) and the Guo term
  // guo w (3 (c - u).F + 9 (c.u)(c.F)).  For the pair (c, -c) the new values are
  // (1 - om) g_(+-) + (X +- Y), with the even part X = om w (base + 4.5 rho cu^2) + guo w
  // (9 cu cF - 3 uF) and the odd part Y = 3 om w rho cu + 3 guo w cF; their coefficients depend
  // on the weight class only, so each class forms them once.
  const T base = fma(T(-1.5) * rho, u2, SHIFT ? m0 : rho);
  const T r45 = T(4.5) * rho;
  const T r3 = T(3) * rho;
  g[0] = fma(c.omc, g[0], fma(c.omw[0], base, -mul_rn(c.gw3[0], uF)));
  // two velocity pairs of one weight class at a time, the first of each pair in one two-lane value and the
  // opposite ones in another: the faces' pairs 1, 3 and 5, then the others
  lb_pair_update<T, V>(c, true, 1, 1, u, F, r45, r3, base, uF, g);
  lb_pair_update<T, V>(c, false, 5, 1, u, F, r45, r3, base, uF, g);
#pragma unroll
  for (int i = 7; i < V::Q; i += 4) lb_pair_update<T, V>(c, true, i, 2, u, F, r45, r3, base, uF, g);
}

// a5 in the form of Eqs. 9-11 at one site: the equilibrium carries the symmetric stress,
//   f_eq_i = w_i [rho + 3 rho c.u + (9/2)(c c - I/3) : (rho u u - sigma^S)],
// the antisymmetric stress enters as F_i = 3 w_i c . FA with FA = div sigma^A (moments 0, FA,
// 0: Eq. 10), rho u = sum f c (Eq. 8), f* = f - (f - f_eq)/tau + F_i (Eq. 7).  sig is the full
// stress at the site (9, row-major).  Opposite velocities share the even part of f_eq.
template <typename T, bool SHIFT, class V>
__device__ __forceinline__ void lb_collide_stress(const Coef<T>& c, const T FA[3], const T sig[9], T g[V::Q],
                                                  T u[3], T* mom = nullptr) {
  T m0 = g[0];
  T j[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int i = 1; i < V::Q; i += 2) {
    m0 += g[i] + g[i + 1];
    const T dg = g[i] - g[i + 1];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (V::c(i, a)) j[a] += V::c(i, a) > 0 ? dg : -dg;
  }
  const T rho = SHIFT ? (c.rho0 + m0) : m0;
  const T rinv = T(1) / rho;
#pragma unroll
  for (int a = 0; a < 3; ++a) u[a] = j[a] * rinv;
  if (mom) {  // as in lb_collide: the forcing adds FA to the momentum (Eq. 10)
    mom[0] = m0;
#pragma unroll
    for (int a = 0; a < 3; ++a) mom[1 + a] = j[a] + FA[a];
  }
  // Pi = rho u u - sigma^S (symmetric: xx, yy, zz, xy, xz, yz)
  const T Pxx = rho * u[0] * u[0] - sig[0], Pyy = rho * u[1] * u[1] - sig[4], Pzz = rho * u[2] * u[2] - sig[8];
  const T Pxy = rho * u[0] * u[1] - T(0.5) * (sig[1] + sig[3]);
  const T Pxz = rho * u[0] * u[2] - T(0.5) * (sig[2] + sig[6]);
  const T Pyz = rho * u[1] * u[2] - T(0.5) * (sig[5] + sig[7]);
  const T tr3 = (Pxx + Pyy + Pzz) * T(1.0 / 3.0);
  // even part: w (rho + 4.5 (c.Pi.c - tr Pi/3)), minus w rho0 when shifted
  const T base = SHIFT ? m0 : rho;
  const T om = c.tau_inv;
  {
    const T w = T(V::w(0));
    const T geq = w * (base - T(4.5) * tr3);
    g[0] = g[0] - (g[0] - geq) * om;
  }
#pragma unroll
  for (int i = 1; i < V::Q; i += 2) {
    const T w = T(V::w(i));
    const int cx = V::c(i, 0), cy = V::c(i, 1), cz = V::c(i, 2);
    const T cPc = T(cx * cx) * Pxx + T(cy * cy) * Pyy + T(cz * cz) * Pzz +
                  T(2 * cx * cy) * Pxy + T(2 * cx * cz) * Pxz + T(2 * cy * cz) * Pyz;
    const T cu = T(cx) * u[0] + T(cy) * u[1] + T(cz) * u[2];
    const T cF = T(cx) * FA[0] + T(cy) * FA[1] + T(cz) * FA[2];
    const T Aeq = w * (base + T(4.5) * (cPc - tr3));
    const T Beq = w * T(3) * rho * cu;
    const T Ef = T(3) * w * cF;
    const T gp = g[i], gm = g[i + 1];
    g[i] = gp - (gp - (Aeq + Beq)) * om + Ef;
    g[i + 1] = gm - (gm - (Aeq - Beq)) * om - Ef;
  }
}

// a4 + a5 of the one-pass step: Euler update of Q and psi with the velocity of the
// previous step, and the collision of the pulled populations.
template <typename T, bool SHIFT>
__device__ __forceinline__ void update_math(const Coef<T>& c, const T F[3], T lapmu, const T Wg[3][3],
                                            const T q0[5], const Vec2<T> qu[3][3], T p0, const T pf[6], const T u0[3],
                                            const T uf[6], const T Hs[5], T g[19], T qn[5], T& pn, T u[3]) {
  op_update<T, false>(c, lapmu, Wg, q0, qu, p0, pf, u0, uf, Hs, qn, pn);
  lb_collide<T, SHIFT>(c, F, g, u);
}

// Neighbour reads straight from global memory with periodic wrap (two-kernel path).
template <typename T, class NB = Nbr>
struct GlobalAcc {
  const T* q_;
  const T* ps;
  const T* sg;
  const T* mu_;
  const T* u_;
  long long N;
  NB nb;
  __device__ __forceinline__ T q(int k, int cx, int cy, int cz) const { return ld(q_ + k * N + nb.off(cx, cy, cz)); }
  __device__ __forceinline__ T psi(int cx, int cy, int cz) const { return ld(ps + nb.off(cx, cy, cz)); }
  __device__ __forceinline__ T sig(int k, int cx, int cy, int cz) const { return ld(sg + k * N + nb.off(cx, cy, cz)); }
  __device__ __forceinline__ T mu(int cx, int cy, int cz) const { return ld(mu_ + nb.off(cx, cy, cz)); }
  __device__ __forceinline__ T u(int a, int cx, int cy, int cz) const { return ld(u_ + a * N + nb.off(cx, cy, cz)); }
  // fields (2j, 2j+1) of the order (Q_xx, Q_xy, Q_xz, Q_yy, Q_yz, psi)
  __device__ __forceinline__ Vec2<T> pair(int j, int cx, int cy, int cz) const {
    const long long o = nb.off(cx, cy, cz);
    return Vec2<T>{ld(q_ + (2 * j) * N + o), j < 2 ? ld(q_ + (2 * j + 1) * N + o) : ld(ps + o)};
  }
  __device__ __forceinline__ Vec2<T> pair_upwind(int j, int a, bool from_below) const {
    const int d = from_below ? -1 : 1;
    return pair(j, a == 0 ? d : 0, a == 1 ? d : 0, a == 2 ? d : 0);
  }
  __device__ __forceinline__ Vel3<T> u3(int cx, int cy, int cz) const {
    const long long o = nb.off(cx, cy, cz);
    return Vel3<T>{Vec2<T>{ld(u_ + o), ld(u_ + N + o)}, ld(u_ + 2 * N + o)};
  }
  // stress pair j (see sig_pair)
  __device__ __forceinline__ Vec2<T> spair(int j, int cx, int cy, int cz) const {
    const long long o = nb.off(cx, cy, cz);
    return Vec2<T>{ld(sg + pair_c0(j) * N + o), j == 4 ? ld(mu_ + o) : ld(sg + pair_c1(j) * N + o)};
  }
};

// ---------------------------------------------------------------- radius-2 stencils
// Fourth-order central differences along the axes (the other reading of "fourth-order
// accurate stencils", Sec. 3):
//   d_a f = [8 (f(+1) - f(-1)) - (f(+2) - f(-2))] / 12,
//   d_aa f = [16 (f(+1) + f(-1)) - (f(+2) + f(-2)) - 30 f(0)] / 12 (summed as differences to
//   f(0)), d_a d_b f = d_a of d_b f (16 points), the Laplacian = sum of the d_aa.
// F(dx, dy, dz) returns the field at the offset.
template <typename T, class F>
__device__ __forceinline__ void r2_axis(const F& f, T c, int a, T& d1, T& d2) {
  const int ex = a == 0, ey = a == 1, ez = a == 2;
  const T m2 = f(-2 * ex, -2 * ey, -2 * ez), m1 = f(-ex, -ey, -ez), p1 = f(ex, ey, ez), p2 = f(2 * ex, 2 * ey, 2 * ez);
  d1 = (T(8) * (p1 - m1) - (p2 - m2)) * T(1.0 / 12.0);
  // as differences to the centre, so that FP32 does not cancel terms of size 30 f
  d2 = (T(16) * ((p1 - c) + (m1 - c)) - ((p2 - c) + (m2 - c))) * T(1.0 / 12.0);
}

template <typename T, class F>
__device__ __forceinline__ T r2_mixed(const F& f, int a, int b) {
  const T w[5] = {T(1.0 / 12.0), T(-8.0 / 12.0), T(0), T(8.0 / 12.0), T(-1.0 / 12.0)};
  T s = T(0);
#pragma unroll
  for (int i = -2; i <= 2; ++i) {
    if (i == 0) continue;
    T r = T(0);
#pragma unroll
    for (int j = -2; j <= 2; ++j) {
      if (j == 0) continue;
      const int dx = (a == 0 ? i : 0) + (b == 0 ? j : 0);
      const int dy = (a == 1 ? i : 0) + (b == 1 ? j : 0);
      const int dz = (a == 2 ? i : 0) + (b == 2 ? j : 0);
      r += w[j + 2] * f(dx, dy, dz);
    }
    s += w[i + 2] * r;
  }
  return s;
}

// a1 with the radius-2 set: the same outputs as gather_fields.
template <typename T, class A>
__device__ __forceinline__ void gather_fields_r2(const A& acc, T q0[5], T& p0, T dq[3][5], T lapq[5], T dp[3],
                                                 T& lapp, T hp[6]) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    auto f = [&](int dx, int dy, int dz) { return acc.q(k, dx, dy, dz); };
    const T c = f(0, 0, 0);
    q0[k] = c;
    T l = T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T d1, d2;
      r2_axis<T>(f, c, a, d1, d2);
      dq[a][k] = d1;
      l += d2;
    }
    lapq[k] = l;
  }
  auto fp = [&](int dx, int dy, int dz) { return acc.psi(dx, dy, dz); };
  p0 = fp(0, 0, 0);
  T l = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    T d1, d2;
    r2_axis<T>(fp, p0, a, d1, d2);
    dp[a] = d1;
    hp[a] = d2;
    l += d2;
  }
  lapp = l;
  hp[3] = r2_mixed<T>(fp, 0, 1);
  hp[4] = r2_mixed<T>(fp, 0, 2);
  hp[5] = r2_mixed<T>(fp, 1, 2);
}

// a3 with the radius-2 set: F_a = sum_b d_b sigma_ab.
template <typename T, class A>
__device__ __forceinline__ void gather_force_r2(const A& acc, T F[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    T s = T(0);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int k = 3 * a + b;
      auto f = [&](int dx, int dy, int dz) { return acc.sig(k, dx, dy, dz); };
      T d1, d2;
      r2_axis<T>(f, T(0), b, d1, d2);
      s += d1;
    }
    F[a] = s;
  }
}

// The stencils of a4 with the radius-2 set; the upwind faces stay at distance 1.
template <typename T, class A>
__device__ __forceinline__ void gather_op_r2(const A& acc, T& lapmu, T Wg[3][3], T q0[5], Vec2<T> qu[3][3], T& p0,
                                             T pf[6], T u0[3], T uf[6]) {
  {
    auto f = [&](int dx, int dy, int dz) { return acc.mu(dx, dy, dz); };
    const T c = f(0, 0, 0);
    T l = T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T d1, d2;
      r2_axis<T>(f, c, a, d1, d2);
      l += d2;
    }
    lapmu = l;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    auto f = [&](int dx, int dy, int dz) { return acc.u(a, dx, dy, dz); };
    u0[a] = f(0, 0, 0);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      T d1, d2;
      r2_axis<T>(f, u0[a], b, d1, d2);
      Wg[a][b] = d1;
    }
    uf[2 * a] = f(a == 0, a == 1, a == 2);
    uf[2 * a + 1] = f(-(a == 0), -(a == 1), -(a == 2));
  }
  gather_upwind<T>(acc, u0, qu, pf);
#pragma unroll
  for (int k = 0; k < 5; ++k) q0[k] = acc.q(k, 0, 0, 0);
  p0 = acc.psi(0, 0, 0);
}

// ---------------------------------------------------------------- k_fields
// H, mu and sigma of (q_in, psi_in) into the scratch; with PRED, H and mu of the Heun
// predicted state qp into the (then free) sigma scratch: H at sig[0..5N), mu at sig[5N..6N).
template <typename T, bool PRED = false, int ST = 0>
__global__ void __launch_bounds__(kStepBlock) k_fields(const InstDesc<T>* __restrict__ D, int ninst) {
  const int ii = find_inst(D, ninst, (long long)blockIdx.x);
  const InstDesc<T>& I = D[ii];
  const long long N = I.N;
  const long long s = ((long long)blockIdx.x - I.blk0) * blockDim.x + threadIdx.x;
  if (s >= N) return;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int x = (int)(s % nx);
  const long long t = s / nx;
  const int y = (int)(t % ny);
  const int z = (int)(t / ny);
  GlobalAcc<T, decltype(make_nbr_st<ST>(0, 0, 0, 4, 4, 4))> acc;
  acc.q_ = PRED ? I.qp : I.q_in;
  acc.ps = PRED ? I.qp + 5 * N : I.psi_in;
  acc.N = N;
  acc.nb = make_nbr_st<ST>(x, y, z, nx, ny, nz);
  T q0[5], p0, dq[3][5], lapq[5], dp[3], lapp, hp[6];
  if constexpr (ST == 1) gather_fields_r2<T>(acc, q0, p0, dq, lapq, dp, lapp, hp);
  else gather_fields<T>(acc, q0, p0, dq, lapq, dp, lapp, hp);
  T H[5], sig[9], mu;
  local_fields<T>(I.c, q0, p0, dq, lapq, dp, lapp, hp, H, mu, sig);
  if constexpr (PRED) {
#pragma unroll
    for (int k = 0; k < 5; ++k) I.sig[k * N + s] = H[k];
    I.sig[5 * N + s] = mu;
  } else {
#pragma unroll
    for (int k = 0; k < 5; ++k) I.H[k * N + s] = H[k];
    I.mu[s] = mu;
#pragma unroll
    for (int k = 0; k < 9; ++k) I.sig[k * N + s] = sig[k];
  }
}

// ---------------------------------------------------------------- staged path
// The antisymmetric part of the stress scratch, for the force of the form of Eqs. 9-11.
template <typename T, class NB = Nbr>
struct AntiSigAcc {
  const T* sg;
  long long N;
  NB nb;
  __device__ __forceinline__ T sig(int k, int cx, int cy, int cz) const {
    const int a = k / 3, b = k - 3 * a;
    if (a == b) return T(0);
    const long long o = nb.off(cx, cy, cz);
    return T(0.5) * (ld(sg + k * N + o) - ld(sg + (3 * b + a) * N + o));
  }
  // pair 4 holds sigma^A_zz = 0 (and no mu: the force does not read lane 1)
  __device__ __forceinline__ Vec2<T> spair(int j, int cx, int cy, int cz) const {
    if (j == 4) return Vec2<T>{T(0), T(0)};
    return Vec2<T>{sig(pair_c0(j), cx, cy, cz), sig(pair_c1(j), cx, cy, cz)};
  }
};

// k_lb: the force from the stress scratch, pull, moments and collision (a3, a5):
// g_out, u_out = velocity of this step.  FORM 0: F = div sigma, BGK + Guo (Eqs. 6-8).
// FORM 1: FA = div sigma^A and the equilibrium with sigma^S (Eqs. 9-11).
template <typename T, bool SHIFT, class V, int FORM, int ST>
__global__ void __launch_bounds__(kStepBlock) k_lb(const InstDesc<T>* __restrict__ D, int ninst) {
  const int ii = find_inst(D, ninst, (long long)blockIdx.x);
  const InstDesc<T>& I = D[ii];
  const long long N = I.N;
  const long long s = ((long long)blockIdx.x - I.blk0) * blockDim.x + threadIdx.x;
  if (s >= N) return;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int x = (int)(s % nx);
  const long long t = s / nx;
  const int y = (int)(t % ny);
  const int z = (int)(t / ny);
  auto nb = make_nbr_st<ST>(x, y, z, nx, ny, nz);
  using NB = decltype(nb);
  T F[3];
  if (FORM == 0) {
    GlobalAcc<T, NB> acc;
    acc.sg = I.sig;
    acc.N = N;
    acc.nb = nb;
    if constexpr (ST == 1) gather_force_r2<T>(acc, F);
    else gather_force<T>(acc, F);
  } else {
    AntiSigAcc<T, NB> acc{I.sig, N, nb};
    if constexpr (ST == 1) gather_force_r2<T>(acc, F);
    else gather_force<T>(acc, F);
  }
  T g[V::Q];
#pragma unroll
  for (int i = 0; i < V::Q; ++i) g[i] = ld(I.g_in + i * N + nb.off(-V::c(i, 0), -V::c(i, 1), -V::c(i, 2)));
  T u[3];
  if (FORM == 0) {
    lb_collide<T, SHIFT, V>(I.c, F, g, u);
  } else {
    T sg[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) sg[k] = I.sig[k * N + s];
    lb_collide_stress<T, SHIFT, V>(I.c, F, sg, g, u);
  }
#pragma unroll
  for (int i = 0; i < V::Q; ++i) I.g_out[i * N + s] = g[i];
#pragma unroll
  for (int a = 0; a < 3; ++a) I.u_out[a * N + s] = u[a];
}

// k_op: the order-parameter update (a4) of the staged path, advecting with u_in (lagged)
// or u_out (sync, written by k_lb of this step).
//   STAGE 0  Euler:           q_out = Q + R(Q)                        (H, mu from the scratch)
//   STAGE 1  Heun predictor:  rq = R(Q), qp = Q + rq
//   STAGE 2  Heun corrector:  q_out = Q + (rq + R(qp)) / 2            (H, mu of qp in sigma)
template <typename T, int STAGE, int ST>
__global__ void __launch_bounds__(kStepBlock) k_op(const InstDesc<T>* __restrict__ D, int ninst, int sync) {
  const int ii = find_inst(D, ninst, (long long)blockIdx.x);
  const InstDesc<T>& I = D[ii];
  const long long N = I.N;
  const long long s = ((long long)blockIdx.x - I.blk0) * blockDim.x + threadIdx.x;
  if (s >= N) return;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int x = (int)(s % nx);
  const long long t = s / nx;
  const int y = (int)(t % ny);
  const int z = (int)(t / ny);
  GlobalAcc<T, decltype(make_nbr_st<ST>(0, 0, 0, 4, 4, 4))> acc;
  acc.q_ = STAGE == 2 ? I.qp : I.q_in;
  acc.ps = STAGE == 2 ? I.qp + 5 * N : I.psi_in;
  acc.mu_ = STAGE == 2 ? I.sig + 5 * N : I.mu;
  acc.u_ = sync ? I.u_out : I.u_in;
  acc.N = N;
  acc.nb = make_nbr_st<ST>(x, y, z, nx, ny, nz);
  T lapmu, Wg[3][3], q0[5], p0, pf[6], u0[3], uf[6];
  Vec2<T> qu[3][3];
  if constexpr (ST == 1) gather_op_r2<T>(acc, lapmu, Wg, q0, qu, p0, pf, u0, uf);
  else gather_op<T>(acc, lapmu, Wg, q0, qu, p0, pf, u0, uf);
  const T* Hsrc = STAGE == 2 ? I.sig : I.H;
  T Hs[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) Hs[k] = Hsrc[k * N + s];
  T qn[5], pn;
  if (STAGE == 0) {
    op_update<T, false>(I.c, lapmu, Wg, q0, qu, p0, pf, u0, uf, Hs, qn, pn);
#pragma unroll
    for (int k = 0; k < 5; ++k) I.q_out[k * N + s] = qn[k];
    I.psi_out[s] = pn;
  } else if (STAGE == 1) {
    op_update<T, true>(I.c, lapmu, Wg, q0, qu, p0, pf, u0, uf, Hs, qn, pn);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      I.rq[k * N + s] = qn[k];
      I.qp[k * N + s] = q0[k] + qn[k];
    }
    I.rq[5 * N + s] = pn;
    I.qp[5 * N + s] = p0 + pn;
  } else {
    op_update<T, true>(I.c, lapmu, Wg, q0, qu, p0, pf, u0, uf, Hs, qn, pn);
#pragma unroll
    for (int k = 0; k < 5; ++k) I.q_out[k * N + s] = I.q_in[k * N + s] + T(0.5) * (I.rq[k * N + s] + qn[k]);
    I.psi_out[s] = I.psi_in[s] + T(0.5) * (I.rq[5 * N + s] + pn);
  }
}

// ---------------------------------------------------------------- k_update
template <typename T, bool SHIFT>
__global__ void __launch_bounds__(kStepBlock) k_update(const InstDesc<T>* __restrict__ D, int ninst) {
  const int ii = find_inst(D, ninst, (long long)blockIdx.x);
  const InstDesc<T>& I = D[ii];
  const long long N = I.N;
  const long long s = ((long long)blockIdx.x - I.blk0) * blockDim.x + threadIdx.x;
  if (s >= N) return;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int x = (int)(s % nx);
  const long long t = s / nx;
  const int y = (int)(t % ny);
  const int z = (int)(t / ny);
  GlobalAcc<T> acc;
  acc.q_ = I.q_in;
  acc.ps = I.psi_in;
  acc.sg = I.sig;
  acc.mu_ = I.mu;
  acc.u_ = I.u_in;
  acc.N = N;
  acc.nb = make_nbr(x, y, z, nx, ny, nz);
  T F[3], lapmu, Wg[3][3], q0[5], p0, pf[6], u0[3], uf[6];
  Vec2<T> qu[3][3];
  gather_force<T>(acc, F);
  gather_op<T>(acc, lapmu, Wg, q0, qu, p0, pf, u0, uf);
  T Hs[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) Hs[k] = I.H[k * N + s];
  T g[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) g[i] = ld(I.g_in + i * N + acc.nb.off(-lat_c(i, 0), -lat_c(i, 1), -lat_c(i, 2)));
  T qn[5], pn, u[3];
  update_math<T, SHIFT>(I.c, F, lapmu, Wg, q0, qu, p0, pf, u0, uf, Hs, g, qn, pn, u);
#pragma unroll
  for (int k = 0; k < 5; ++k) I.q_out[k * N + s] = qn[k];
  I.psi_out[s] = pn;
#pragma unroll
  for (int i = 0; i < 19; ++i) I.g_out[i * N + s] = g[i];
#pragma unroll
  for (int a = 0; a < 3; ++a) I.u_out[a * N + s] = u[a];
}

// ---------------------------------------------------------------- field exchange
// dst components, in mask order: G(19) RHO(1) U(3) Q(5) PSI(1); offsets given per group
// (-1 = not selected).
template <typename T, bool SHIFT, class V>
__global__ void k_get_fields(InstDesc<T> I, long long oG, long long oR, long long oU, long long oQ,
                             long long oP, double* __restrict__ dst) {
  const long long N = I.N;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const int x = (int)(s % nx);
    const long long t = s / nx;
    const int y = (int)(t % ny);
    const int z = (int)(t / ny);
    if (oG >= 0 || oR >= 0) {
      const Nbr nb = make_nbr(x, y, z, nx, ny, nz);
      double rho = 0.0;
#pragma unroll
      for (int i = 0; i < V::Q; ++i) {
        const long long src = nb.off(-V::c(i, 0), -V::c(i, 1), -V::c(i, 2));
        double fi = (double)I.g_in[i * N + src];
        if (SHIFT) fi += V::w(i) * (double)I.c.rho0;
        rho += fi;
        if (oG >= 0) dst[oG + i * N + s] = fi;
      }
      if (oR >= 0) dst[oR + s] = rho;
    }
    if (oU >= 0)
      for (int a = 0; a < 3; ++a) dst[oU + a * N + s] = (double)I.u_in[a * N + s];
    if (oQ >= 0)
      for (int k = 0; k < 5; ++k) dst[oQ + k * N + s] = (double)I.q_in[k * N + s];
    if (oP >= 0) dst[oP + s] = (double)I.psi_in[s];
  }
}

// Writes pre-collision populations f_i(x) as the stored post-collision array of the
// previous step: stored_i(x - c_i) = f_i(x) (- w_i rho0 when SHIFT).
template <typename T, bool SHIFT, class V>
__global__ void k_set_fields(InstDesc<T> I, long long oG, long long oU, long long oQ, long long oP,
                             const double* __restrict__ src, T* g_t, T* q_t, T* p_t, T* u_t) {
  const long long N = I.N;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const int x = (int)(s % nx);
    const long long t = s / nx;
    const int y = (int)(t % ny);
    const int z = (int)(t / ny);
    if (oG >= 0) {
      const Nbr nb = make_nbr(x, y, z, nx, ny, nz);
#pragma unroll
      for (int i = 0; i < V::Q; ++i) {
        const long long d = nb.off(-V::c(i, 0), -V::c(i, 1), -V::c(i, 2));
        double fi = src[oG + i * N + s];
        if (SHIFT) fi -= V::w(i) * (double)I.c.rho0;
        g_t[i * N + d] = (T)fi;
      }
    }
    if (oU >= 0)
      for (int a = 0; a < 3; ++a) u_t[a * N + s] = (T)src[oU + a * N + s];
    if (oQ >= 0)
      for (int k = 0; k < 5; ++k) q_t[k * N + s] = (T)src[oQ + k * N + s];
    if (oP >= 0) p_t[s] = (T)src[oP + s];
  }
}

// ---------------------------------------------------------------- FP64 reductions
// a6 as a separate pass (state set from outside, or a path without the fused sums): FP64
// mass, sum psi, momentum (3), sum phi_c cos (3), sum phi_c sin (3) and sum phi_c of the
// populations stored at each site (streaming only permutes them, so the sums equal those of
// the pulled populations).  Each warp takes whole x rows (no index division per site); a lane
// adds its sites of a row in T, then into FP64; cos and sin come from the instance's tables.
// (s, c) += x, with s + x split by TwoSum (Knuth, TAOCP vol. 2, 4.2.2) into its rounded sum
// and its exact rounding error, which c gathers: s + c carries about twice T's precision.  The
// a6 sums of the FP32 path are formed this way, so they come out as the FP64 sums of the
// per-site FP32 shares.
// (The shares are products rounded by mul_rn: they must come out as the same T values in every
// pass, so they may not be contracted into a following addition.)

template <typename T>
__device__ __forceinline__ void two_sum_add(T& s, T& c, T x) {
  const T t = s + x;
  const T bp = t - s;
  const T err = (s - (t - bp)) + (x - bp);
  s = t;
  c += err;
}

// k_obs_partial writes partial[block][12]; k_obs_final sums them in a fixed order.  Each
// thread adds the per-site shares (mass and momentum of the site's 19 stored populations, psi,
// phi_c and phi_c times the cos/sin tables, each formed in T as the fused step forms them) into
// error-free (sum, error) pairs, then FP64 takes over.
template <typename T, bool SHIFT, class V>
__global__ void __launch_bounds__(kObsBlock) k_obs_partial(InstDesc<T> I, double* __restrict__ partial) {
  T as[12], ac[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) as[k] = ac[k] = T(0);
  const int nx = I.nx, ny = I.ny;
  const long long N = I.N;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int WPB = kObsBlock / 32;
  const int rows = ny * I.nz;
  for (int r = blockIdx.x * WPB + wid; r < rows; r += gridDim.x * WPB) {
    const int y = r % ny, z = r / ny;
    const long long base = (long long)r * nx;
    const T cy = __ldg(I.trig + 2 * (nx + y)), sy = __ldg(I.trig + 2 * (nx + y) + 1);
    const T cz = __ldg(I.trig + 2 * (nx + ny + z)), sz = __ldg(I.trig + 2 * (nx + ny + z) + 1);
    for (int x = lane; x < nx; x += 32) {
      const long long st = base + x;
      T m = T(0), j0 = T(0), j1 = T(0), j2 = T(0);
#pragma unroll
      for (int i = 0; i < V::Q; ++i) {
        const T f = __ldg(I.g_in + i * N + st);
        m += f;
        if (V::c(i, 0)) j0 += V::c(i, 0) > 0 ? f : -f;
        if (V::c(i, 1)) j1 += V::c(i, 1) > 0 ? f : -f;
        if (V::c(i, 2)) j2 += V::c(i, 2) > 0 ? f : -f;
      }
      const T p = __ldg(I.psi_in + st);
      const T h = T(0.5) * (T(1) + p);
      const T v[12] = {m, p, j0, j1, j2, mul_rn(h, __ldg(I.trig + 2 * x)), mul_rn(h, cy), mul_rn(h, cz),
                       mul_rn(h, __ldg(I.trig + 2 * x + 1)), mul_rn(h, sy), mul_rn(h, sz), h};
#pragma unroll
      for (int k = 0; k < 12; ++k) two_sum_add(as[k], ac[k], v[k]);
    }
  }
  double acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = (double)as[k] + (double)ac[k];
  if (SHIFT && blockIdx.x == 0 && threadIdx.x == 0) acc[0] += (double)N * (double)I.c.rho0;
  __shared__ double sh[WPB][12];
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    double v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wid][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 12) {
    double v = 0.0;
    for (int w = 0; w < WPB; ++w) v += sh[w][threadIdx.x];
    partial[blockIdx.x * 12 + threadIdx.x] = v;
  }
}

// Sums partial[nblocks][12] into out[12]: thread (l, k) adds blocks l, l + 32, ... of value k,
// then the 32 subtotals of each value are added in order.
static __global__ void __launch_bounds__(384) k_obs_final(const double* __restrict__ partial, int nblocks,
                                                          double* __restrict__ out) {
  __shared__ double red[32][12];
  const int k = threadIdx.x % 12, l = threadIdx.x / 12;
  double v = 0.0;
  for (int b = l; b < nblocks; b += 32) v += partial[b * 12 + k];
  red[l][k] = v;
  __syncthreads();
  if (threadIdx.x < 12) {
    double t = 0.0;
    for (int q = 0; q < 32; ++q) t += red[q][threadIdx.x];
    out[threadIdx.x] = t;
  }
}

// ---------------------------------------------------------------- launchers
template <typename T, bool SHIFT>
cudaError_t Launch<T, SHIFT>::step(const InstDesc<T>* d_desc, int ninst, long long total_blocks, int bs,
                                   cudaStream_t s) {
  k_fields<T><<<(unsigned)total_blocks, bs, 0, s>>>(d_desc, ninst);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_update<T, SHIFT><<<(unsigned)total_blocks, bs, 0, s>>>(d_desc, ninst);
  return cudaGetLastError();
}

template <typename T, bool SHIFT, int ST>
cudaError_t staged_st(const InstDesc<T>* d_desc, int ninst, unsigned g, int bs, bool heun, bool sync, int vel,
                      int form, cudaStream_t s) {
  k_fields<T, false, ST><<<g, bs, 0, s>>>(d_desc, ninst);
  if (vel == 0 && form == 0) k_lb<T, SHIFT, VelD3Q19, 0, ST><<<g, bs, 0, s>>>(d_desc, ninst);
  else if (vel == 0) k_lb<T, SHIFT, VelD3Q19, 1, ST><<<g, bs, 0, s>>>(d_desc, ninst);
  else if (form == 0) k_lb<T, SHIFT, VelD3Q15, 0, ST><<<g, bs, 0, s>>>(d_desc, ninst);
  else k_lb<T, SHIFT, VelD3Q15, 1, ST><<<g, bs, 0, s>>>(d_desc, ninst);
  if (!heun) {
    k_op<T, 0, ST><<<g, bs, 0, s>>>(d_desc, ninst, sync ? 1 : 0);
  } else {
    k_op<T, 1, ST><<<g, bs, 0, s>>>(d_desc, ninst, sync ? 1 : 0);
    k_fields<T, true, ST><<<g, bs, 0, s>>>(d_desc, ninst);
    k_op<T, 2, ST><<<g, bs, 0, s>>>(d_desc, ninst, sync ? 1 : 0);
  }
  return cudaGetLastError();
}

template <typename T, bool SHIFT>
cudaError_t Launch<T, SHIFT>::staged(const InstDesc<T>* d_desc, int ninst, long long total_blocks, int bs, bool heun,
                                     bool sync, int vel, int form, int stencil, cudaStream_t s) {
  const unsigned g = (unsigned)total_blocks;
  if (stencil == 1) return staged_st<T, SHIFT, 1>(d_desc, ninst, g, bs, heun, sync, vel, form, s);
  return staged_st<T, SHIFT, 0>(d_desc, ninst, g, bs, heun, sync, vel, form, s);
}

inline unsigned grid_for(long long N, int bs) {
  long long g = (N + bs - 1) / bs;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

template <typename T, bool SHIFT>
cudaError_t Launch<T, SHIFT>::get_fields(const InstDesc<T>& I, uint32_t mask, double* dst, cudaStream_t s) {
  long long o = 0, oG = -1, oR = -1, oU = -1, oQ = -1, oP = -1;
  if (mask & 1u) { oG = o; o += (I.vel ? 15 : 19) * I.N; }
  if (mask & 2u) { oR = o; o += I.N; }
  if (mask & 4u) { oU = o; o += 3 * I.N; }
  if (mask & 8u) { oQ = o; o += 5 * I.N; }
  if (mask & 16u) { oP = o; o += I.N; }
  if (I.vel) k_get_fields<T, SHIFT, VelD3Q15><<<grid_for(I.N, 256), 256, 0, s>>>(I, oG, oR, oU, oQ, oP, dst);
  else k_get_fields<T, SHIFT, VelD3Q19><<<grid_for(I.N, 256), 256, 0, s>>>(I, oG, oR, oU, oQ, oP, dst);
  return cudaGetLastError();
}

template <typename T, bool SHIFT>
cudaError_t Launch<T, SHIFT>::set_fields(const InstDesc<T>& I, uint32_t mask, const double* src, T* g_t, T* q_t,
                                         T* p_t, T* u_t, cudaStream_t s) {
  long long o = 0, oG = -1, oU = -1, oQ = -1, oP = -1;
  if (mask & 1u) { oG = o; o += (I.vel ? 15 : 19) * I.N; }
  if (mask & 4u) { oU = o; o += 3 * I.N; }
  if (mask & 8u) { oQ = o; o += 5 * I.N; }
  if (mask & 16u) { oP = o; o += I.N; }
  if (I.vel)
    k_set_fields<T, SHIFT, VelD3Q15><<<grid_for(I.N, 256), 256, 0, s>>>(I, oG, oU, oQ, oP, src, g_t, q_t, p_t, u_t);
  else
    k_set_fields<T, SHIFT, VelD3Q19><<<grid_for(I.N, 256), 256, 0, s>>>(I, oG, oU, oQ, oP, src, g_t, q_t, p_t, u_t);
  return cudaGetLastError();
}

template <typename T, bool SHIFT>
cudaError_t Launch<T, SHIFT>::observables(const InstDesc<T>& I, double* partial, int nblocks, double* out,
                                          cudaStream_t s) {
  if (I.vel) k_obs_partial<T, SHIFT, VelD3Q15><<<nblocks, kObsBlock, 0, s>>>(I, partial);
  else k_obs_partial<T, SHIFT, VelD3Q19><<<nblocks, kObsBlock, 0, s>>>(I, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_obs_final<<<1, 384, 0, s>>>(partial, nblocks, out);
  return cudaGetLastError();
}

}  // namespace lbcad
