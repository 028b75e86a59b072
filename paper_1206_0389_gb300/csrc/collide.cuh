// Per-cell collision operators and equilibria (device code).
//
// Every function works on the shifted values g_i held in registers:
//   D3Q19 (incompressible, Section 2): g_i = f_i, the fluctuation with sum delta rho;
//   D3Q27 (compressible, Section 2):   g_i = f_i - w_i, with sum rho - 1.
// Keeping the weights out of the registers keeps float32 arithmetic accurate
// relative to the small non-equilibrium parts.
#pragma once
#include <cuda_fp16.h>

#include <type_traits>

#include "lattice.cuh"

namespace lbm {

// ------------------------------------------------------------------ storage
// Storage types: double / float hold g_i; __half holds g_i / w_i.
template <class S>
struct Store;
template <>
struct Store<double> {
  using T = double;
  template <int Q, int i>
  __device__ static __forceinline__ T get(const double* p) { return *p; }
  template <int Q, int i>
  __device__ static __forceinline__ void put(double* p, T v) { *p = v; }
};
template <>
struct Store<float> {
  using T = float;
  template <int Q, int i>
  __device__ static __forceinline__ T get(const float* p) { return __ldg(p); }
  template <int Q, int i>
  __device__ static __forceinline__ void put(float* p, T v) { *p = v; }
};
template <>
struct Store<__half> {
  using T = float;
  template <int Q, int i>
  __device__ static __forceinline__ T get(const __half* p) {
    return __half2float(__ldg(p)) * float(Lattice<Q>::w(i));
  }
  template <int Q, int i>
  __device__ static __forceinline__ void put(__half* p, T v) {
    *p = __float2half_rn(v * float(1.0 / Lattice<Q>::w(i)));
  }
};

// runtime-index variants for the small interface / utility kernels
template <class S, int Q>
__device__ __forceinline__ typename Store<S>::T load_rt(const S* p, int i);
template <class S, int Q>
__device__ __forceinline__ void store_rt(S* p, int i, typename Store<S>::T v);

template <int Q>
__device__ __forceinline__ double weight_rt(int i) {
  double w = 0.0;
  static_for<Q>([&](auto c) {
    if (i == c) w = Lattice<Q>::w(c);
  });
  return w;
}

template <>
__device__ __forceinline__ double load_rt<double, 19>(const double* p, int) { return *p; }
template <>
__device__ __forceinline__ double load_rt<double, 27>(const double* p, int) { return *p; }
template <>
__device__ __forceinline__ float load_rt<float, 19>(const float* p, int) { return *p; }
template <>
__device__ __forceinline__ float load_rt<float, 27>(const float* p, int) { return *p; }
template <>
__device__ __forceinline__ float load_rt<__half, 19>(const __half* p, int i) {
  return __half2float(*p) * float(weight_rt<19>(i));
}
template <>
__device__ __forceinline__ float load_rt<__half, 27>(const __half* p, int i) {
  return __half2float(*p) * float(weight_rt<27>(i));
}
template <>
__device__ __forceinline__ void store_rt<double, 19>(double* p, int, double v) { *p = v; }
template <>
__device__ __forceinline__ void store_rt<double, 27>(double* p, int, double v) { *p = v; }
template <>
__device__ __forceinline__ void store_rt<float, 19>(float* p, int, float v) { *p = v; }
template <>
__device__ __forceinline__ void store_rt<float, 27>(float* p, int, float v) { *p = v; }
template <>
__device__ __forceinline__ void store_rt<__half, 19>(__half* p, int i, float v) {
  *p = __float2half_rn(v / float(weight_rt<19>(i)));
}
template <>
__device__ __forceinline__ void store_rt<__half, 27>(__half* p, int i, float v) {
  *p = __float2half_rn(v / float(weight_rt<27>(i)));
}

// ------------------------------------------------------------------ D3Q19 MRT-LES
// Incompressible equilibrium (Section 2, c = 1): w (drho + 3 e.u + 9/2 (e.u)^2 - 3/2 u^2).
template <class T>
__device__ __forceinline__ void feq19(T drho, T ux, T uy, T uz, T* out) {
  const T uu = T(1.5) * (ux * ux + uy * uy + uz * uz);
  static_for<19>([&](auto i) {
    constexpr int x = D3Q19::ex(i), y = D3Q19::ey(i), z = D3Q19::ez(i);
    const T eu = T(x) * ux + T(y) * uy + T(z) * uz;
    out[i] = T(D3Q19::w(i)) * (drho + T(3) * eu + T(4.5) * eu * eu - uu);
  });
}

template <class T>
__device__ __forceinline__ void moments19(const T* g, T& drho, T& ux, T& uy, T& uz) {
  drho = T(0);
  ux = uy = uz = T(0);
  static_for<19>([&](auto i) {
    drho += g[i];
    if constexpr (D3Q19::ex(i) != 0) ux += T(D3Q19::ex(i)) * g[i];
    if constexpr (D3Q19::ey(i) != 0) uy += T(D3Q19::ey(i)) * g[i];
    if constexpr (D3Q19::ez(i) != 0) uz += T(D3Q19::ez(i)) * g[i];
  });
}

// MRT with every non-shear rate 1 (the paper's choice, Section 2) written in
// closed form: f* = f_eq + (1 - s1) P (f - f_eq).  P keeps the five shear
// moments of Table 1 (s1 group) of the non-equilibrium part and drops all
// others: axis links receive 1/2 (Pi_aa - tr Pi / 3), the diagonal links of
// plane ab receive 1/4 e_a e_b Pi_ab, the rest link 0.  s1 = 1/tau_total with
// tau_total from Eq. eqTauTotFinal and Q from Eq. EqnQ.
// Opposite links (2k-1, 2k) are handled as pairs: their sums carry the even
// moments and their differences the odd ones, and since the D3Q19 set is
// isotropic to fourth order, sum_i e_a e_b f_eq_i = drho/3 delta_ab + u_a u_b,
// so Pi^neq = sum e e f - drho/3 I - u u without forming f - f_eq per link.
// Returns |S| = 3 Q / (2 tau_total) (Eq. eqStrainRate, lattice units).
// Scaled: g holds g_i / w_i on entry and exit (the FP16 storage form); the
// weights then enter as constant factors of the sums and of the output
// terms instead of one multiply per population each way.
template <class T, bool Scaled = false>
__device__ __forceinline__ T collide19(T* g, T tau0, T cs2_18) {
  T sp[9], dp[9];
  static_for<9>([&](auto p) {
    sp[p] = g[2 * p + 1] + g[2 * p + 2];
    dp[p] = g[2 * p + 1] - g[2 * p + 2];
  });
  T drho = Scaled ? T(D3Q19::w(0)) * g[0] : g[0];
  T ux = T(0), uy = T(0), uz = T(0);
  T sxx = T(0), syy = T(0), szz = T(0), sxy = T(0), sxz = T(0), syz = T(0);
  static_for<9>([&](auto p) {
    constexpr int i = 2 * p + 1;
    constexpr int x = D3Q19::ex(i), y = D3Q19::ey(i), z = D3Q19::ez(i);
    constexpr double ws = Scaled ? D3Q19::w(i) : 1.0;
    drho += T(ws) * sp[p];
    if constexpr (x != 0) { ux += T(x * ws) * dp[p]; sxx += T(ws) * sp[p]; }
    if constexpr (y != 0) { uy += T(y * ws) * dp[p]; syy += T(ws) * sp[p]; }
    if constexpr (z != 0) { uz += T(z * ws) * dp[p]; szz += T(ws) * sp[p]; }
    if constexpr (x * y != 0) sxy += T(x * y * ws) * sp[p];
    if constexpr (x * z != 0) sxz += T(x * z * ws) * sp[p];
    if constexpr (y * z != 0) syz += T(y * z * ws) * sp[p];
  });
  const T d3 = drho * T(1.0 / 3.0);
  const T pxx = sxx - d3 - ux * ux, pyy = syy - d3 - uy * uy, pzz = szz - d3 - uz * uz;
  const T pxy = sxy - ux * uy, pxz = sxz - ux * uz, pyz = syz - uy * uz;
  const T qq = T(2) * (pxx * pxx + pyy * pyy + pzz * pzz + T(2) * (pxy * pxy + pxz * pxz + pyz * pyz));
  const T Qn = sqrt(qq);
  const T tau = T(0.5) * (tau0 + sqrt(tau0 * tau0 + cs2_18 * Qn));
  const T k = T(1) - T(1) / tau;
  const T tr3 = (pxx + pyy + pzz) * T(1.0 / 3.0);
  // shear projections 1/2 (axis links) and 1/4 (diagonal links), divided by
  // the link weights 1/18 and 1/36 when scaled
  const T cA = Scaled ? T(9) : T(0.5), cD = Scaled ? T(9) : T(0.25);
  const T ax = cA * k * (pxx - tr3), ay = cA * k * (pyy - tr3), az = cA * k * (pzz - tr3);
  const T dxy = cD * k * pxy, dxz = cD * k * pxz, dyz = cD * k * pyz;
  const T base = drho - T(1.5) * (ux * ux + uy * uy + uz * uz);
  g[0] = Scaled ? base : T(D3Q19::w(0)) * base;
  static_for<9>([&](auto p) {
    constexpr int i = 2 * p + 1;
    constexpr int x = D3Q19::ex(i), y = D3Q19::ey(i), z = D3Q19::ez(i);
    constexpr int nz = (x != 0) + (y != 0) + (z != 0);
    T eu = T(0);
    if constexpr (x != 0) eu += T(x) * ux;
    if constexpr (y != 0) eu += T(y) * uy;
    if constexpr (z != 0) eu += T(z) * uz;
    constexpr T w = T(D3Q19::w(i));
    T proj;
    if constexpr (nz == 1) proj = (x != 0) ? ax : (y != 0) ? ay : az;
    else if constexpr (z == 0) proj = T(x * y) * dxy;
    else if constexpr (y == 0) proj = T(x * z) * dxz;
    else proj = T(y * z) * dyz;
    T sym, asym;
    if constexpr (Scaled) {
      sym = base + T(4.5) * eu * eu + proj;
      asym = T(3) * eu;
    } else {
      sym = w * (base + T(4.5) * eu * eu) + proj;
      asym = (T(3) * w) * eu;
    }
    g[i] = sym + asym;
    g[i + 1] = sym - asym;
  });
  return T(1.5) * Qn / tau;
}

// The same collision in float64, whose pipes bound the update: the sums of the
// two pairs of each plane serve all moments (48 additions instead of 63), the
// squares of u serve every link, and one reciprocal of tau_total serves k and
// |S|.  32^3 D3Q19 FP64 16.8 -> 14.1 us per step.
__device__ __forceinline__ double collide19_f64(double* g, double tau0, double cs2_18) {
  double s[9], d[9];
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    s[p] = g[2 * p + 1] + g[2 * p + 2];
    d[p] = g[2 * p + 1] - g[2 * p + 2];
  }
  // pairs 0..2: x, y, z; (3, 4), (5, 6), (7, 8): the diagonals of xy, xz, yz
  const double Exy = s[3] + s[4], Exz = s[5] + s[6], Eyz = s[7] + s[8];
  const double sxy = s[3] - s[4], sxz = s[5] - s[6], syz = s[7] - s[8];
  const double ux = d[0] + (d[3] + d[4]) + (d[5] + d[6]);
  const double uy = d[1] + (d[3] - d[4]) + (d[7] + d[8]);
  const double uz = d[2] + (d[5] - d[6]) + (d[7] - d[8]);
  const double drho = g[0] + ((s[0] + s[1]) + s[2]) + ((Exy + Exz) + Eyz);
  const double xx = ux * ux, yy = uy * uy, zz = uz * uz, d3 = drho * (1.0 / 3.0);
  const double pxx = s[0] + Exy + Exz - d3 - xx, pyy = s[1] + Exy + Eyz - d3 - yy, pzz = s[2] + Exz + Eyz - d3 - zz;
  const double pxy = sxy - ux * uy, pxz = sxz - ux * uz, pyz = syz - uy * uz;
  const double qq = 2.0 * (pxx * pxx + pyy * pyy + pzz * pzz) + 4.0 * (pxy * pxy + pxz * pxz + pyz * pyz);
  const double Qn = sqrt(qq);
  const double inv = 2.0 / (tau0 + sqrt(tau0 * tau0 + cs2_18 * Qn));  // 1 / tau_total
  const double k = 1.0 - inv, k2 = 0.5 * k, k4 = 0.25 * k;
  const double tr3 = (pxx + pyy + pzz) * (1.0 / 3.0);
  const double base = drho - 1.5 * (xx + yy + zz);
  g[0] = (1.0 / 3.0) * base;
  const double b1 = (1.0 / 18.0) * base, b2 = (1.0 / 36.0) * base;
  // axis links: w (base + 4.5 u_a^2) + k/2 (Pi_aa - tr Pi / 3) +- u_a / 6
  auto axis = [&](int i, double u, double uu, double pi) {
    const double sym = b1 + 0.25 * uu + k2 * (pi - tr3), asym = (1.0 / 6.0) * u;
    g[i] = sym + asym;
    g[i + 1] = sym - asym;
  };
  axis(1, ux, xx, pxx);
  axis(3, uy, yy, pyy);
  axis(5, uz, zz, pzz);
  // diagonals: w (base + 4.5 (u_a +- u_b)^2) +- k/4 Pi_ab +- (u_a +- u_b) / 12
  const double hx = (1.0 / 12.0) * ux, hy = (1.0 / 12.0) * uy, hz = (1.0 / 12.0) * uz;
  auto plane = [&](int i, double ua, double ub, double aa, double bb, double ha, double hb, double pi) {
    const double even = b2 + 0.125 * (aa + bb), odd = 0.25 * ua * ub + k4 * pi;
    const double sp = even + odd, sm = even - odd, ap = ha + hb, am = ha - hb;
    g[i] = sp + ap;
    g[i + 1] = sp - ap;
    g[i + 2] = sm + am;
    g[i + 3] = sm - am;
  };
  plane(7, ux, uy, xx, yy, hx, hy, pxy);
  plane(11, ux, uz, xx, zz, hx, hz, pxz);
  plane(15, uy, uz, yy, zz, hy, hz, pyz);
  return 1.5 * Qn * inv;
}

// ------------------------------------------------------------------ D3Q27 FCLB
// one-dimensional weights (index 0/1/2 means velocity -1/0/+1)
__host__ __device__ constexpr double w1(int k) { return k == 1 ? 2.0 / 3.0 : 1.0 / 6.0; }

template <class T>
__device__ __forceinline__ void moments27(const T* g, T& drho, T& jx, T& jy, T& jz) {
  drho = jx = jy = jz = T(0);
  static_for<27>([&](auto i) {
    drho += g[i];
    if constexpr (D3Q27::ex(i) != 0) jx += T(D3Q27::ex(i)) * g[i];
    if constexpr (D3Q27::ey(i) != 0) jy += T(D3Q27::ey(i)) * g[i];
    if constexpr (D3Q27::ez(i) != 0) jz += T(D3Q27::ez(i)) * g[i];
  });
}

// Factorized cascaded collision (Section 2, Table 2; whole moments recomputed):
// the normal-stress differences and shear moments relax with omega, the
// trace and every higher moment with rate 1 to the Table 2 equilibria built
// from the post-collision second-order moments (third and fifth order 0,
// fourth M_aa M_bb and M_aa M_bc, sixth M11 M22 M33).  With a body force F,
// u = (j + F/2)/rho and the first central moments leave as F/(2 rho).
//
// In closed form, used by the stream-collide kernels with FP32 and FP16 storage.
// Because every moment above second order is relaxed with rate 1, only the
// six pre-collision second-order central moments matter; they follow from
// raw sums: rho kappa_aa = S_aa - 2 u_a j_a + u_a^2 rho (+ const), rho kappa_ab =
// S_ab - u_a j_b - u_b j_a + u_a u_b rho.  The post-collision normalised
// central moments are then a sum of per-axis products: prod_a (1, 0, X_a)
// for the diagonal part (X_a = 1/3 + D_a), plus kappa'_xy (0,1,0)(0,1,0)(1,0,Z)
// and its two permutations, plus F/(2 rho) in the first order.  The 1-D
// inverse transform of (1, 0, X) is phi(0) = 1 - u^2 - X, phi(+-1) =
// (u^2 +- u + X)/2; of (0, 1, 0) psi(0) = -2u, psi(+-1) = u +- 1/2; of
// (1, 0, 0) chi(0) = 1 - u^2, chi(+-1) = (u^2 +- u)/2.  Writing phi = w1 + delta
// keeps f* - w free of cancellation:
//   f*_i - w_i = drho W_i + rho (dx Py Pz... expanded) + k_xy psi_x psi_y phi_z + ...
// (the paper notes that fixed rates remove most of the FCLB flops).
// Scaled: g holds g_i / w_i on entry and exit (the FP16 storage form); the
// product weights w_i = w1_x w1_y w1_z then enter once per z-line on input
// and once per (e_y, e_z) pair and per e_x factor on output.
template <class T, bool Force, bool Scaled = false>
__device__ __forceinline__ void collide27_closed(T* g, T omega, T Fx, T Fy, T Fz) {
  // ---- zeroth, first and second raw moments of g by a z, y, x collapse
  T m0[3][3], dz[3][3], sz[3][3];  // per (ex, ey): sum, difference, sum of ends along z
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const T lo = g[D3Q27::index(a - 1, b - 1, -1)];
      const T mi = g[D3Q27::index(a - 1, b - 1, 0)];
      const T hi = g[D3Q27::index(a - 1, b - 1, 1)];
      if constexpr (Scaled) {
        const T ce = T(w1(a) * w1(b) * w1(0)), cm = T(w1(a) * w1(b) * w1(1));
        sz[a][b] = ce * (hi + lo);
        dz[a][b] = ce * (hi - lo);
        m0[a][b] = sz[a][b] + cm * mi;
      } else {
        sz[a][b] = hi + lo;
        dz[a][b] = hi - lo;
        m0[a][b] = sz[a][b] + mi;
      }
    }
  T M0[3], My[3], Myy[3], Dz[3], Dyz[3], Szz[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T e = m0[a][2] + m0[a][0];
    Myy[a] = e;
    My[a] = m0[a][2] - m0[a][0];
    M0[a] = e + m0[a][1];
    Dz[a] = dz[a][0] + dz[a][1] + dz[a][2];
    Dyz[a] = dz[a][2] - dz[a][0];
    Szz[a] = sz[a][0] + sz[a][1] + sz[a][2];
  }
  const T Sxx = M0[2] + M0[0];
  const T drho = Sxx + M0[1];
  const T jx = M0[2] - M0[0];
  const T jy = My[0] + My[1] + My[2];
  const T Sxy = My[2] - My[0];
  const T Syy = Myy[0] + Myy[1] + Myy[2];
  const T jz = Dz[0] + Dz[1] + Dz[2];
  const T Sxz = Dz[2] - Dz[0];
  const T Syz = Dyz[0] + Dyz[1] + Dyz[2];
  const T Szzt = Szz[0] + Szz[1] + Szz[2];
  // ---- velocity and second-order central moments (deviations from rho/3)
  const T rho = T(1) + drho;
  const T r = T(1) / rho;
  T px = jx, py = jy, pz = jz;
  if constexpr (Force) {
    px += T(0.5) * Fx;
    py += T(0.5) * Fy;
    pz += T(0.5) * Fz;
  }
  const T ux = px * r, uy = py * r, uz = pz * r;
  // rho u_a u_a - 2 u_a j_a = u_a (rho u_a - 2 j_a) = u_a (p_a - 2 j_a)
  const T vxx = Sxx + ux * (px - T(2) * jx);
  const T vyy = Syy + uy * (py - T(2) * jy);
  const T vzz = Szzt + uz * (pz - T(2) * jz);
  const T vxy = Sxy + ux * py - ux * jy - uy * jx;
  const T vxz = Sxz + ux * pz - ux * jz - uz * jx;
  const T vyz = Syz + uy * pz - uy * jz - uz * jy;
  // ---- relaxation: deviatoric part with omega, trace to equilibrium
  const T om1 = T(1) - omega;
  const T mean = (vxx + vyy + vzz) * T(1.0 / 3.0);
  const T Dx = om1 * (vxx - mean) * r, Dy = om1 * (vyy - mean) * r, Dz_ = om1 * (vzz - mean) * r;
  const T kxy = om1 * vxy, kxz = om1 * vxz, kyz = om1 * vyz;  // rho kappa'
  // ---- per-axis factors, index 0/1/2 = velocity -1/0/+1
  T dl[3][3], ph[3][3], ps[3][3], ch[3][3];
  const T uu[3] = {ux, uy, uz};
  const T DD[3] = {Dx, Dy, Dz_};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T u = uu[a], u2 = u * u, D = DD[a];
    dl[a][1] = -u2 - D;
    dl[a][0] = T(0.5) * (u2 - u + D);
    dl[a][2] = T(0.5) * (u2 + u + D);
    ph[a][1] = T(2.0 / 3.0) + dl[a][1];
    ph[a][0] = T(1.0 / 6.0) + dl[a][0];
    ph[a][2] = T(1.0 / 6.0) + dl[a][2];
    ps[a][1] = T(-2) * u;
    ps[a][0] = u - T(0.5);
    ps[a][2] = u + T(0.5);
    if constexpr (Force) {
      ch[a][1] = T(1) - u2;
      ch[a][0] = T(0.5) * (u2 - u);
      ch[a][2] = T(0.5) * (u2 + u);
    }
  }
  // ---- per (e_y, e_z) pair, then per e_x
  if constexpr (Scaled) {
    // the x factors divided by w1_x once
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dl[0][a] *= T(1.0 / w1(a));
      ps[0][a] *= T(1.0 / w1(a));
      ph[0][a] *= T(1.0 / w1(a));
      if constexpr (Force) ch[0][a] *= T(1.0 / w1(a));
    }
  }
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T P = ph[1][b] * ph[2][c];                            // phi_y phi_z
      const T Qd = T(w1(b)) * dl[2][c] + dl[1][b] * ph[2][c];     // phi_y phi_z - w1_y w1_z
      T rP = rho * P, rQ = rho * Qd;
      T R = kxy * ps[1][b] * ph[2][c] + kxz * ph[1][b] * ps[2][c];
      T Sy = kyz * ps[1][b] * ps[2][c];
      T Fp = T(0), Gp = T(0);
      if constexpr (Force) {
        Fp = T(0.5) * Fx * ch[1][b] * ch[2][c];
        Gp = T(0.5) * Fy * ps[1][b] * ch[2][c] + T(0.5) * Fz * ch[1][b] * ps[2][c];
      }
      if constexpr (Scaled) {
        const T ibc = T(1.0 / (w1(b) * w1(c)));
        rP *= ibc;
        R *= ibc;
        Sy *= ibc;
        if constexpr (Force) {
          Fp *= ibc;
          Gp *= ibc;
        }
        const T base = drho + ibc * rQ;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          T v = base + dl[0][a] * rP + ps[0][a] * R + ph[0][a] * Sy;
          if constexpr (Force) v += ps[0][a] * Fp + ch[0][a] * Gp;
          g[D3Q27::index(a - 1, b - 1, c - 1)] = v;
        }
      } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const T W = T(w1(a) * w1(b) * w1(c));
          T v = drho * W + dl[0][a] * rP + T(w1(a)) * rQ + ps[0][a] * R + ph[0][a] * Sy;
          if constexpr (Force) v += ps[0][a] * Fp + ch[0][a] * Gp;
          g[D3Q27::index(a - 1, b - 1, c - 1)] = v;
        }
      }
    }
}

// The collision of collide27_closed as nested one-dimensional lines, for FP64
// storage.  A line is the three values along one axis of
//   c w1(e) + A delta(e) + R psi(e),   delta(+-1) = E +- u/2, delta(0) = -2 E,
//   psi(+-1) = u +- 1/2, psi(0) = -2 u,  E = (u^2 + D) / 2,
// which come in pairs: with t = E A + u R the even part is c/6 + t, the odd
// part u A + R, and the centre c - 2 (c/6 + t), so a line takes 7 operations
// and its sum is c by construction.  Along z the slots are (drho, rho, 0); each
// value c found gives the next axis its A = c + w, and kyz psi_z its R; the
// shear terms kxy phi_z, kxz psi_z make a second line along y that is the R of
// the x lines.  About 245 operations a cell against 400 of collide27_closed,
// and fewer values alive (112 registers against 212 without a cap): 128^3, bound
// by the float64 pipes, 1313 -> 1006 us per step.  The last bits differ, which
// FP32 and FP16 runs show as drifts and flipped roundings of the storage, so
// those, bound by memory, keep the other form.  om1 = 1 - omega.
template <class T>
__device__ __forceinline__ void emit_line(T c, T t, T odd, T& lo, T& mid, T& hi) {
  const T ev = T(1.0 / 6.0) * c + t;
  mid = c - T(2) * ev;
  lo = ev - T(0.5) * odd;
  hi = ev + T(0.5) * odd;
}
template <class T, bool Force>
__device__ __forceinline__ void collide27_lines(T* g, T om1, T Fx, T Fy, T Fz) {
  // ---- raw moments up to second order by a z, y, x collapse
  T m0[3][3], dz[3][3], sz[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const T lo = g[D3Q27::index(a - 1, b - 1, -1)], hi = g[D3Q27::index(a - 1, b - 1, 1)];
      sz[a][b] = hi + lo;
      dz[a][b] = hi - lo;
      m0[a][b] = sz[a][b] + g[D3Q27::index(a - 1, b - 1, 0)];
    }
  T M0[3], My[3], Myy[3], Dz[3], Dyz[3], Szz[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Myy[a] = m0[a][2] + m0[a][0];
    My[a] = m0[a][2] - m0[a][0];
    M0[a] = Myy[a] + m0[a][1];
    Dz[a] = (dz[a][2] + dz[a][0]) + dz[a][1];
    Dyz[a] = dz[a][2] - dz[a][0];
    Szz[a] = (sz[a][2] + sz[a][0]) + sz[a][1];
  }
  T Sxx = M0[2] + M0[0], jx = M0[2] - M0[0];
  T drho = Sxx + M0[1];
  T jy = (My[2] + My[0]) + My[1], Sxy = My[2] - My[0];
  T Syy = (Myy[2] + Myy[0]) + Myy[1];
  T jz = (Dz[2] + Dz[0]) + Dz[1], Sxz = Dz[2] - Dz[0];
  T Syz = (Dyz[2] + Dyz[0]) + Dyz[1];
  T Szzt = (Szz[2] + Szz[0]) + Szz[1];
  // ---- velocity, second-order central moments, relaxation
  const T rho = T(1) + drho;
  const T r = T(1) / rho;
  T px = jx, py = jy, pz = jz;
  if constexpr (Force) {
    px += T(0.5) * Fx;
    py += T(0.5) * Fy;
    pz += T(0.5) * Fz;
  }
  const T ux = px * r, uy = py * r, uz = pz * r;
  T vxx, vyy, vzz, vxy, vxz, vyz;
  if constexpr (Force) {
    vxx = Sxx + ux * (px - T(2) * jx);
    vyy = Syy + uy * (py - T(2) * jy);
    vzz = Szzt + uz * (pz - T(2) * jz);
    vxy = Sxy + ux * (py - jy) - uy * jx;
    vxz = Sxz + ux * (pz - jz) - uz * jx;
    vyz = Syz + uy * (pz - jz) - uz * jy;
  } else {
    vxx = Sxx - ux * jx;
    vyy = Syy - uy * jy;
    vzz = Szzt - uz * jz;
    vxy = Sxy - uy * jx;
    vxz = Sxz - uz * jx;
    vyz = Syz - uz * jy;
  }
  const T mean = (vxx + vyy + vzz) * T(1.0 / 3.0);
  const T hr = T(0.5) * om1 * r;  // E = u^2 / 2 + D / 2, D = om1 (v - mean) / rho
  const T Ex = T(0.5) * ux * ux + hr * (vxx - mean);
  const T Ey = T(0.5) * uy * uy + hr * (vyy - mean);
  const T Ez = T(0.5) * uz * uz + hr * (vzz - mean);
  const T kxy = om1 * vxy, kxz = om1 * vxz, kyz = om1 * vyz;
  // ---- lines along z: rho phi_z - w, kyz psi_z, kxz psi_z, kxy phi_z
  const T zero = T(0);
  T cz[3], rz[3], xz[3], yz[3];
  emit_line<T>(drho, Ez * rho, pz, cz[0], cz[1], cz[2]);
  emit_line<T>(zero, uz * kyz, kyz, rz[0], rz[1], rz[2]);
  emit_line<T>(zero, uz * kxz, kxz, xz[0], xz[1], xz[2]);
  emit_line<T>(kxy, Ez * kxy, uz * kxy, yz[0], yz[1], yz[2]);
  // the force's first-order moments have no second-order part: chi = (1, 0, 0)
  T hz[3], qz[3], Hx = zero, Hy = zero, Hz = zero;
  if constexpr (Force) {
    Hx = T(0.5) * ux * ux - T(1.0 / 6.0);
    Hy = T(0.5) * uy * uy - T(1.0 / 6.0);
    Hz = T(0.5) * uz * uz - T(1.0 / 6.0);
    emit_line<T>(T(1), Hz, uz, hz[0], hz[1], hz[2]);
    const T f = T(0.5) * Fz;
    emit_line<T>(zero, uz * f, f, qz[0], qz[1], qz[2]);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    // ---- lines along y at this e_z
    const T A = cz[k] + T(w1(k));
    T cy[3], ry[3], gy[3];
    emit_line<T>(cz[k], Ey * A + uy * rz[k], uy * A + rz[k], cy[0], cy[1], cy[2]);
    emit_line<T>(xz[k], Ey * xz[k] + uy * yz[k], uy * xz[k] + yz[k], ry[0], ry[1], ry[2]);
    if constexpr (Force) {
      // Fx/2 chi_y chi_z joins the x lines' R; Fy/2 psi_y chi_z + Fz/2 chi_y psi_z
      // is their chi slot
      const T f = T(0.5) * Fx * hz[k], q = T(0.5) * Fy * hz[k];
      T lo, mid, hi;
      emit_line<T>(f, Hy * f, uy * f, lo, mid, hi);
      ry[0] += lo;
      ry[1] += mid;
      ry[2] += hi;
      emit_line<T>(qz[k], Hy * qz[k] + uy * q, uy * qz[k] + q, gy[0], gy[1], gy[2]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      // ---- lines along x
      const T Ax = cy[b] + T(w1(b) * w1(k));
      T& lo = g[D3Q27::index(-1, b - 1, k - 1)];
      T& mid = g[D3Q27::index(0, b - 1, k - 1)];
      T& hi = g[D3Q27::index(1, b - 1, k - 1)];
      if constexpr (Force)
        emit_line<T>(cy[b] + gy[b], Ex * Ax + ux * ry[b] + Hx * gy[b], ux * (Ax + gy[b]) + ry[b], lo, mid, hi);
      else
        emit_line<T>(cy[b], Ex * Ax + ux * ry[b], ux * Ax + ry[b], lo, mid, hi);
    }
  }
}

// the form that a storage's update uses
template <class T, bool Force, bool Scaled>
__device__ __forceinline__ void collide27(T* g, T omega, T Fx, T Fy, T Fz) {
  if constexpr (std::is_same<T, double>::value) collide27_lines<T, Force>(g, T(1) - omega, Fx, Fy, Fz);
  else collide27_closed<T, Force, Scaled>(g, omega, Fx, Fy, Fz);
}

// Product-form D3Q27 equilibrium minus the weights: the distribution whose
// normalised central moments are the Table 2 equilibria at rest shape is
// rho prod_a phi(e_a, u_a), phi(0) = 2/3 - u^2, phi(+-1) = (1/3 + u^2 +- u)/2.
// With phi = w1 + delta it is evaluated without cancellation as
// drho W + rho (delta_x phi_y phi_z + w1_x (delta_y phi_z + w1_y delta_z)).
template <class T>
__device__ __forceinline__ void feq27(T drho, T ux, T uy, T uz, T* out) {
  const T rho = T(1) + drho;
  T dl[3][3], ph[3][3];
  const T uu[3] = {ux, uy, uz};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T u = uu[a], u2 = u * u;
    dl[a][1] = -u2;
    dl[a][0] = T(0.5) * (u2 - u);
    dl[a][2] = T(0.5) * (u2 + u);
    ph[a][1] = T(2.0 / 3.0) + dl[a][1];
    ph[a][0] = T(1.0 / 6.0) + dl[a][0];
    ph[a][2] = T(1.0 / 6.0) + dl[a][2];
  }
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T rP = rho * ph[1][b] * ph[2][c];
      const T rQ = rho * (T(w1(b)) * dl[2][c] + dl[1][b] * ph[2][c]);
#pragma unroll
      for (int a = 0; a < 3; ++a)
        out[D3Q27::index(a - 1, b - 1, c - 1)] = drho * T(w1(a) * w1(b) * w1(c)) + dl[0][a] * rP + T(w1(a)) * rQ;
    }
}

// ------------------------------------------------------------------ model traits
struct MrtLes {
  static constexpr int Q = 19;
  template <class T>
  __device__ static __forceinline__ void moments(const T* g, T& rl, T& ux, T& uy, T& uz) {
    moments19(g, rl, ux, uy, uz);  // rho_0 = 1
  }
  template <class T>
  __device__ static __forceinline__ void feq(T rl, T ux, T uy, T uz, T* out) {
    feq19(rl, ux, uy, uz, out);
  }
};
struct Fclb {
  static constexpr int Q = 27;
  template <class T>
  __device__ static __forceinline__ void moments(const T* g, T& rl, T& ux, T& uy, T& uz) {
    T jx, jy, jz;
    moments27(g, rl, jx, jy, jz);
    const T ir = T(1) / (T(1) + rl);
    ux = jx * ir;
    uy = jy * ir;
    uz = jz * ir;
  }
  template <class T>
  __device__ static __forceinline__ void feq(T rl, T ux, T uy, T uz, T* out) {
    feq27(rl, ux, uy, uz, out);
  }
};

}  // namespace lbm
