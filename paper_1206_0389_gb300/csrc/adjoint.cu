// Discrete adjoint of one D3Q27 FCLB stream-collide step with a body force.
//
// Forward step (single periodic level): f~_{t+1}(x) = C(p(x), F(x)) with the
// pulled pre-collision vector p(x)_i = f~_t(x - e_i)_i.  For a loss L of the
// final state, lambda_t = dL/df~_t obeys
//   mu(x) = J_C(p(x), F(x))^T lambda_{t+1}(x),   lambda_t(x - e_i)_i = mu(x)_i,
// and dL/dF(x) += (dC/dF(p(x), F(x)))^T lambda_{t+1}(x).
// So the adjoint kernel reads f~_t at exactly the addresses the forward pull
// reads, reads lambda_{t+1} at its own cell, and writes mu_i to lambda_t at
// the forward pull addresses (each written once: no races).
//
// J_C^T is hand-derived reverse mode of collide27_lines (collide.cuh): its
// lines along z and y are evaluated again, the lines along x, y and z and the
// relaxation reversed, each z layer of lambda taken down to the layer's line
// inputs before the next is begun.
#include "chained.cuh"
#include "collide.cuh"
#include "kernels.cuh"

namespace lbm {

// adjoint of emit_line (unscaled): from those of its three values to those of
// c, t and odd
template <class T>
struct LineAdj {
  T c, t, odd;
  __device__ __forceinline__ LineAdj(T lo, T mid, T hi) {
    t = (lo + hi) - T(2) * mid;
    odd = T(0.5) * (hi - lo);
    c = mid + T(1.0 / 6.0) * t;
  }
};

// mu = J_C^T lambda for the pre-collision shifted values g; lam holds lambda
// on entry and mu on exit; F-bar (dL/dF of this step) is added to Fb.
// A trailing b marks an adjoint.
template <class T>
__device__ __forceinline__ void collide27_adjoint(const T* g, T* lam, T om1, T Fx, T Fy, T Fz, T& Fbx, T& Fby,
                                                  T& Fbz) {
  // ---- raw moments by a z, y, x collapse (as collide27_lines)
  T drho, jx, jy, jz, Sxx, Syy, Szz, Sxy, Sxz, Syz;
  {
    T M0[3], My[3], Myy[3], Dz[3], Dyz[3], Zz[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T m[3], d[3], e[3];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const T lo = g[D3Q27::index(a - 1, b - 1, -1)], hi = g[D3Q27::index(a - 1, b - 1, 1)];
        e[b] = hi + lo;
        d[b] = hi - lo;
        m[b] = e[b] + g[D3Q27::index(a - 1, b - 1, 0)];
      }
      Myy[a] = m[2] + m[0];
      My[a] = m[2] - m[0];
      M0[a] = Myy[a] + m[1];
      Dz[a] = (d[2] + d[0]) + d[1];
      Dyz[a] = d[2] - d[0];
      Zz[a] = (e[2] + e[0]) + e[1];
    }
    Sxx = M0[2] + M0[0];
    jx = M0[2] - M0[0];
    drho = Sxx + M0[1];
    jy = (My[2] + My[0]) + My[1];
    Sxy = My[2] - My[0];
    Syy = (Myy[2] + Myy[0]) + Myy[1];
    jz = (Dz[2] + Dz[0]) + Dz[1];
    Sxz = Dz[2] - Dz[0];
    Syz = (Dyz[2] + Dyz[0]) + Dyz[1];
    Szz = (Zz[2] + Zz[0]) + Zz[1];
  }
  // ---- velocity, second-order central moments, relaxation
  const T rho = T(1) + drho, r = T(1) / rho;
  const T px = jx + T(0.5) * Fx, py = jy + T(0.5) * Fy, pz = jz + T(0.5) * Fz;
  const T ux = px * r, uy = py * r, uz = pz * r;
  T dxx = Sxx + ux * (px - T(2) * jx), dyy = Syy + uy * (py - T(2) * jy), dzz = Szz + uz * (pz - T(2) * jz);
  {
    const T mean = (dxx + dyy + dzz) * T(1.0 / 3.0);
    dxx -= mean;
    dyy -= mean;
    dzz -= mean;
  }
  const T kxy = om1 * (Sxy + ux * (py - jy) - uy * jx);
  const T kxz = om1 * (Sxz + ux * (pz - jz) - uz * jx);
  const T kyz = om1 * (Syz + uy * (pz - jz) - uz * jy);
  const T hr = T(0.5) * om1 * r;
  const T Ex = T(0.5) * ux * ux + hr * dxx, Ey = T(0.5) * uy * uy + hr * dyy, Ez = T(0.5) * uz * uz + hr * dzz;
  const T Hx = T(0.5) * ux * ux - T(1.0 / 6.0), Hy = T(0.5) * uy * uy - T(1.0 / 6.0);
  const T fx = T(0.5) * Fx, fy = T(0.5) * Fy, fz = T(0.5) * Fz;
  // ---- lines along z
  const T zero = T(0);
  T cz[3], rz[3], xz[3], yz[3], hz[3], qz[3];
  emit_line<T>(drho, Ez * rho, pz, cz[0], cz[1], cz[2]);
  emit_line<T>(zero, uz * kyz, kyz, rz[0], rz[1], rz[2]);
  emit_line<T>(zero, uz * kxz, kxz, xz[0], xz[1], xz[2]);
  emit_line<T>(kxy, Ez * kxy, uz * kxy, yz[0], yz[1], yz[2]);
  emit_line<T>(T(1), T(0.5) * uz * uz - T(1.0 / 6.0), uz, hz[0], hz[1], hz[2]);
  emit_line<T>(zero, uz * fz, fz, qz[0], qz[1], qz[2]);
  // ---- per z layer: lines along y again, then the x and y lines reversed;
  // the adjoint of each z value takes its place
  T Exb = zero, Eyb = zero, Ezb = zero, Hxb = zero, Hyb = zero;
  T uxb = zero, uyb = zero, uzb = zero;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T A = cz[k] + T(w1(k)), f = fx * hz[k], q = fy * hz[k];
    T cy[3], ry[3], gy[3];
    emit_line<T>(cz[k], Ey * A + uy * rz[k], uy * A + rz[k], cy[0], cy[1], cy[2]);
    emit_line<T>(xz[k] + f, Ey * xz[k] + uy * yz[k] + Hy * f, uy * (xz[k] + f) + yz[k], ry[0], ry[1], ry[2]);
    emit_line<T>(qz[k], Hy * qz[k] + uy * q, uy * qz[k] + q, gy[0], gy[1], gy[2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const LineAdj<T> l(lam[D3Q27::index(-1, b - 1, k - 1)], lam[D3Q27::index(0, b - 1, k - 1)],
                         lam[D3Q27::index(1, b - 1, k - 1)]);
      const T Ax = cy[b] + T(w1(b) * w1(k));
      Exb += Ax * l.t;
      Hxb += gy[b] * l.t;
      uxb += ry[b] * l.t + (Ax + gy[b]) * l.odd;
      const T uo = ux * l.odd;
      cy[b] = l.c + (Ex * l.t + uo);
      ry[b] = ux * l.t + l.odd;
      gy[b] = l.c + (Hx * l.t + uo);
    }
    const LineAdj<T> lc(cy[0], cy[1], cy[2]), lr(ry[0], ry[1], ry[2]), lg(gy[0], gy[1], gy[2]);
    Eyb += A * lc.t + xz[k] * lr.t;
    Hyb += f * lr.t + qz[k] * lg.t;
    uyb += rz[k] * lc.t + A * lc.odd + yz[k] * lr.t + (xz[k] + f) * lr.odd + q * lg.t + qz[k] * lg.odd;
    const T ur = uy * lr.odd;
    const T fb = lr.c + (Hy * lr.t + ur), qb = uy * lg.t + lg.odd;
    cz[k] = lc.c + (Ey * lc.t + uy * lc.odd);
    rz[k] = uy * lc.t + lc.odd;
    xz[k] = lr.c + (Ey * lr.t + ur);
    yz[k] = uy * lr.t + lr.odd;
    qz[k] = lg.c + (Hy * lg.t + uy * lg.odd);
    Fbx += T(0.5) * hz[k] * fb;
    Fby += T(0.5) * hz[k] * qb;
    hz[k] = fx * fb + fy * qb;
  }
  // ---- lines along z reversed
  T drb, pbz, kxyb, kxzb, kyzb, rhob;
  {
    const LineAdj<T> lc(cz[0], cz[1], cz[2]), lr(rz[0], rz[1], rz[2]), lx(xz[0], xz[1], xz[2]),
        ly(yz[0], yz[1], yz[2]), lh(hz[0], hz[1], hz[2]), lq(qz[0], qz[1], qz[2]);
    drb = lc.c;
    pbz = lc.odd;
    rhob = Ez * lc.t;
    kyzb = uz * lr.t + lr.odd;
    kxzb = uz * lx.t + lx.odd;
    kxyb = ly.c + Ez * ly.t + uz * ly.odd;
    Ezb = rho * lc.t + kxy * ly.t;
    uzb = kyz * lr.t + kxz * lx.t + kxy * ly.odd + lh.odd + fz * lq.t;
    uzb += uz * (Ezb + lh.t);  // E_z and H_z hold u_z^2 / 2
    Fbz += T(0.5) * (uz * lq.t + lq.odd);
  }
  uxb += ux * (Exb + Hxb);
  uyb += uy * (Eyb + Hyb);
  // ---- relaxation
  const T Sb = hr * (Exb + Eyb + Ezb) * T(1.0 / 3.0);
  const T vxxb = hr * Exb - Sb, vyyb = hr * Eyb - Sb, vzzb = hr * Ezb - Sb;
  const T vxyb = om1 * kxyb, vxzb = om1 * kxzb, vyzb = om1 * kyzb;
  T rb = T(0.5) * om1 * (Exb * dxx + Eyb * dyy + Ezb * dzz);
  // ---- second-order central moments from raw moments
  T jbx = T(-2) * vxxb * ux - vxyb * uy - vxzb * uz;
  T jby = T(-2) * vyyb * uy - vxyb * ux - vyzb * uz;
  T jbz = T(-2) * vzzb * uz - vxzb * ux - vyzb * uy;
  // (v_ab is written with u_a p_b, so p_x enters only v_xx and p_y only v_yy, v_xy)
  T pbx = vxxb * ux;
  T pby = vyyb * uy + vxyb * ux;
  pbz += vzzb * uz + vxzb * ux + vyzb * uy;
  uxb += vxxb * (px - T(2) * jx) + vxyb * (py - jy) + vxzb * (pz - jz);
  uyb += vyyb * (py - T(2) * jy) - vxyb * jx + vyzb * (pz - jz);
  uzb += vzzb * (pz - T(2) * jz) - vxzb * jx - vyzb * jy;
  // ---- u = p r, p = j + F/2, r = 1/rho, rho = 1 + drho
  pbx += uxb * r;
  pby += uyb * r;
  pbz += uzb * r;
  rb += uxb * px + uyb * py + uzb * pz;
  jbx += pbx;
  jby += pby;
  jbz += pbz;
  Fbx += T(0.5) * pbx;
  Fby += T(0.5) * pby;
  Fbz += T(0.5) * pbz;
  drb += rhob - rb * r * r;
  // ---- back to the populations: mu_i = drb + e.jb + e_a e_b Sb_ab, along x
  // base and base + vxxb +- slope
#pragma unroll
  for (int b = -1; b <= 1; ++b)
#pragma unroll
    for (int c = -1; c <= 1; ++c) {
      T base = drb, slope = jbx;
      if (b != 0) base += vyyb + T(b) * jby;
      if (c != 0) base += vzzb + T(c) * jbz;
      if (b * c != 0) base += T(b * c) * vyzb;
      if (b != 0) slope += T(b) * vxyb;
      if (c != 0) slope += T(c) * vxzb;
      const T ends = base + vxxb;
      lam[D3Q27::index(0, b, c)] = base;
      lam[D3Q27::index(1, b, c)] = ends + slope;
      lam[D3Q27::index(-1, b, c)] = ends - slope;
    }
}

// One adjoint step over all blocks of a periodic single level, a cell per
// thread and four CTAs per block.  An FP32 step reads f_t, lambda and the force
// and writes lambda and dL/dF, 360 bytes a cell, and is bound by HBM on large
// grids, by the latency of its 54 scattered loads per thread on small ones: the
// reverse of the lines (half the instructions of a pass-by-pass reverse) fits 96
// registers, 20 warps per SM instead of 16, and CTAs of one cell per thread
// chain and even out better than four cells in a row.  us per step, pass by
// pass -> lines -> also chained, 5 CTAs per SM, a cell per thread -> loads of
// dL/dF before the stores of lambda: 96^3 FP32 76.4 -> 64.1 -> 58.3 -> 50.9
// (0.92 of the copy peak), 128^3 165 -> 140 -> 131 -> 114 (0.97), 32^3 12.4 ->
// 11.3 -> 5.3 -> 5.3.  FP64 is bound by the float64 pipes: 64^3 639 -> 420 -> 369
// -> 367.
constexpr int kAdjTPB = 128, kAdjCtas = kCells / kAdjTPB;
template <class T>
__global__ void __launch_bounds__(kAdjTPB, sizeof(T) == 4 ? 5 : 2) k_adjoint(const AdjointArgs a) {
  begin_chained();
  constexpr int Q = 27;
  constexpr int QS = Q * kCells;
  // (no __restrict__: lambda, f_t and dL/dF are written by kernels that may
  // still run when this one comes up, so none of them may be read as data
  // that stays unchanged; chained.cuh)
  const T* fsrc = reinterpret_cast<const T*>(a.f_t);
  const T* lin = reinterpret_cast<const T*>(a.lam_in);
  T* lout = reinterpret_cast<T*>(a.lam_out);
  T* gF = reinterpret_cast<T*>(a.dLdF);
  const int64_t ncell = int64_t(a.BX) * a.BY * a.BZ * kCells;
  const int b = int(blockIdx.x) / kAdjCtas;
  const int c = int(blockIdx.x) % kAdjCtas * kAdjTPB + int(threadIdx.x);
  const int bx = b % a.BX, by = (b / a.BX) % a.BY, bz = b / (a.BX * a.BY);
  const int BXY = a.BX * a.BY;
  // x / y block offsets fit an int (the planner keeps BX * BY * 27 * 512
  // below 2^31); a periodic z wrap moves by up to nblocks * 27 * 512
  // elements, so the z neighbours enter through 64-bit base indices
  const int dxm = bx == 0 ? a.BX - 1 : -1, dxp = bx == a.BX - 1 ? -(a.BX - 1) : 1;
  const int dym = by == 0 ? a.BX * (a.BY - 1) : -a.BX, dyp = by == a.BY - 1 ? -a.BX * (a.BY - 1) : a.BX;
  const int64_t dzm = bz == 0 ? int64_t(BXY) * (a.BZ - 1) : -int64_t(BXY);
  const int64_t dzp = bz == a.BZ - 1 ? -int64_t(BXY) * (a.BZ - 1) : int64_t(BXY);
  const int x = c & 7, y = (c >> 3) & 7, z = c >> 6;
  const int Xm = (x == 0) ? dxm * QS + 8 : 0, Xp = (x == 7) ? dxp * QS - 8 : 0;
  const int Ym = (y == 0) ? dym * QS + 64 : 0, Yp = (y == 7) ? dyp * QS - 64 : 0;
  const int64_t own = int64_t(b) * QS + c;
  const int64_t B1 = z == 0 ? own + dzm * QS + 512 : own;   // base of e_z = +1 pulls
  const int64_t Bm = z == 7 ? own + dzp * QS - 512 : own;   // base of e_z = -1 pulls
  // element index of population i's pull source (= its adjoint target)
  auto pull = [&](auto i) {
    constexpr int ex = D3Q27::ex(i), ey = D3Q27::ey(i), ez = D3Q27::ez(i);
    int o = int(i) * kCells - (ex + 8 * ey + 64 * ez);
    if constexpr (ex == 1) o += Xm;
    if constexpr (ex == -1) o += Xp;
    if constexpr (ey == 1) o += Ym;
    if constexpr (ey == -1) o += Yp;
    return (ez == 1 ? B1 : ez == -1 ? Bm : own) + o;
  };
  T g[Q], lam[Q];
  static_for<Q>([&](auto i) {
    g[i] = fsrc[pull(i)];
    lam[i] = lin[own + int(i) * kCells];
  });
  const int64_t j = int64_t(b) * kCells + c;
  T Fx = T(0), Fy = T(0), Fz = T(0);
  if (a.force != nullptr) {
    const T* F = reinterpret_cast<const T*>(a.force);
    Fx = F[j];
    Fy = F[ncell + j];
    Fz = F[2 * ncell + j];
  }
  T Fbx = T(0), Fby = T(0), Fbz = T(0);
  collide27_adjoint<T>(g, lam, T(1) - T(a.omega), Fx, Fy, Fz, Fbx, Fby, Fbz);
  Fbx += gF[j];
  Fby += gF[ncell + j];
  Fbz += gF[2 * ncell + j];
  static_for<Q>([&](auto i) { lout[pull(i)] = lam[i]; });
  gF[j] = Fbx;
  gF[ncell + j] = Fby;
  gF[2 * ncell + j] = Fbz;
}

cudaError_t launch_adjoint(int storage, const AdjointArgs& a, cudaStream_t st) {
  if (a.nblocks == 0) return cudaSuccess;
  const int grid = a.nblocks * kAdjCtas;
  if (storage == LBM_F64) return launch_chained(k_adjoint<double>, grid, kAdjTPB, a, false, st);
  if (storage == LBM_F32) return launch_chained(k_adjoint<float>, grid, kAdjTPB, a, true, st);
  return cudaErrorInvalidValue;
}

}  // namespace lbm
