// Fused pull-stream + collide kernel (one launch covers the work of every
// level that takes a substep at that time).
//
// f(x, t+1) = f~(x - e_i, t) (the streaming on the left of Eqs. lbgk / MRT),
// then the local collision of Section 2, then f~(x, t+1) is stored.
// Storage per level: a dense box of 8^3 blocks, [block][i][512 cells], cell
// index x + 8 y + 64 z.  A warp covers four x-rows of one block, so loads of
// one population are 128-byte (F32) contiguous runs, shifted by one cell for
// populations with e_x != 0.
//
// Neighbour blocks are found arithmetically in the level box: per thread the
// extra element offset for leaving the block along -x is Xm (non-zero only
// for cells with x == 0), along +x Xp (x == 7), likewise Ym/Yp/Zm/Zp, so the
// source of population i is own_block + i*512 + cell - (e_x + 8 e_y + 64 e_z)
// + X(e_x) + Y(e_y) + Z(e_z) with X(+1) = Xm, X(-1) = Xp, X(0) = 0.  On the
// zero-gradient outflow face (Xp = -1 for x == 7) the ghost copy of cell
// (NX - 1, y', z') is read from that cell directly.
//
// Walls (instances with W = true): a pull of a level-0 cell that would cross
// a wall face of the domain (y, z, or the no-slip x faces) is replaced after
// the periodic pull, for the cells next to a wall only.  No-slip (half-way
// bounce-back): f_i(x) = f~_opp(i)(x), the opposite population of the cell
// itself.  Free-slip (specular reflection): the population with the
// wall-normal components flipped, pulled along the axes not crossed only,
// f_i(x) = f~_m(i)(x - e_i + (e_i . n) n).  A no-slip crossing wins over a
// free-slip one; two free-slip crossings flip both components.  Opposite and
// mirrored populations have the same weight, so the storage decode of i
// applies to them unchanged.
#pragma once
#include <algorithm>
#include <type_traits>

#include "chained.cuh"
#include "collide.cuh"
#include "kernels.cuh"
#include "pair.cuh"

namespace lbm {

// Loads of the state that ask L2 to fetch the surrounding 256 bytes (the pulls
// of a warp's next rows then find their sectors in L2: 0.5225 -> 0.5203 ms per
// 256^3 D3Q27 FP32 step).  Ordinary coherent loads, kept after the wait of a
// chained launch: the kernel before writes this state while this one is
// already resident (chained.cuh).
__device__ __forceinline__ __half load_state(const __half* p) {
  unsigned short v;
  asm volatile("ld.global.L2::256B.b16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
  return __ushort_as_half(v);
}
__device__ __forceinline__ float load_state(const float* p) {
  float v;
  asm volatile("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double load_state(const double* p) { return *p; }

// Start of an update kernel (chained.cuh).  With the graphs of 16 steps: 96^3
// D3Q27 FP32 36.9 -> 31.3 us per step, 256^3 520 -> 515 us.
__device__ __forceinline__ void begin_update(const UpdateArgs& a) {
  begin_chained();
  if (a.step_inc != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *a.step_inc += 1;
}

template <class M, class S, int TPB, int MINB, bool W>
__global__ void __launch_bounds__(TPB, MINB) k_update(const UpdateArgs a) {
  begin_update(a);
  using St = Store<S>;
  using T = typename St::T;
  constexpr int Q = M::Q;
  constexpr int QS = Q * kCells;
  // a unit of work is one of 2^split equal runs of a block's cells
  // (a.run_mask = cells per run - 1; a thread ends its run when its cell
  // index wraps to the run's first TPB cells, which needs no register for
  // the run's end)
  for (int it = blockIdx.x; it < (a.nitems << a.split); it += gridDim.x) {
    const WorkItem w = a.items[it >> a.split];
    const int c0 = int(unsigned(it) * unsigned(a.run_mask + 1) % kCells) + threadIdx.x;
    const LevelPtrs& L = a.lv[w.level];
    const int BX = L.BX, BXY = L.BX * L.BY;
    // block deltas towards -x, +x, -y, +y (periodic wrap on box faces); the
    // planner keeps BX * BY * Q * 512 below 2^31, so x and y offsets fit an
    // int.  A wrap across z moves by up to nblocks * Q * 512 elements, past
    // the int range on large boxes: the blocks below and above are reached
    // through 64-bit base pointers instead (the source bases of e_z = +1 pulls
    // of the cells z == 0 and of e_z = -1 pulls of the cells z == 7).
    const int dxm = (w.edges & 1) ? (L.BX - 1) : -1;
    const int dxp = (w.edges & 2) ? -(L.BX - 1) : 1;
    const int dym = (w.edges & 4) ? BX * (L.BY - 1) : -BX;
    const int dyp = (w.edges & 8) ? -BX * (L.BY - 1) : BX;
    // (z block deltas in blocks fit an int: the box holds fewer than 2^31
    // blocks; the element offset is widened per cell)
    const int dzm = (w.edges & 16) ? BXY * (L.BZ - 1) : -BXY;
    const int dzp = (w.edges & 32) ? -BXY * (L.BZ - 1) : BXY;
    // wall faces this block touches (bit 0/1 low/high y, 2/3 low/high z):
    // the level-0 box spans the domain in y and z, so its wrapping faces
    // are the walls; the x faces come from edges bits 7 (x = 0) and 6 (the
    // face x = NX, whose fused outflow read the fix-up then replaces)
    const int wf = (W && w.level == 0)
                       ? (a.walls & (((w.edges >> 2) & 15) | ((w.edges & 128) ? 16 : 0) | ((w.edges & 64) ? 32 : 0)))
                       : 0;
    const T tau0 = T(L.tau0);
    const S* src = reinterpret_cast<const S*>(L.src) + int64_t(w.block) * QS;
    S* dst = reinterpret_cast<S*>(L.dst) + int64_t(w.block) * QS;
    // source of population i for cell c: base(e_z) + c + i*512 - (e_x + 8 e_y
    // + 64 e_z) + the x / y block offsets of the faces the pull crosses, with
    // base(0) = src, base(+1) = the block below for z == 0 (else src),
    // base(-1) = the block above for z == 7 (else src)
    auto offsets = [&](int c, int& Xm, int& Xp, int& Ym, int& Yp) {
      const int x = c & 7, y = (c >> 3) & 7;
      Xm = (x == 0) ? dxm * QS + 8 : 0;
      Xp = (x == 7) ? ((w.edges & 64) ? -1 : dxp * QS - 8) : 0;
      Ym = (y == 0) ? dym * QS + 64 : 0;
      Yp = (y == 7) ? dyp * QS - 64 : 0;
    };
    auto zbase = [&](int c, const S*& b1, const S*& bm) {
      const int z = c >> 6;
      b1 = src + c + (z == 0 ? int64_t(dzm) * QS + 512 : int64_t(0));
      bm = src + c + (z == 7 ? int64_t(dzp) * QS - 512 : int64_t(0));
    };
    auto pull = [&](int c, auto&& load) {
      int Xm, Xp, Ym, Yp;
      offsets(c, Xm, Xp, Ym, Yp);
      const S *b1, *bm;
      zbase(c, b1, bm);
      const S* p = src + c;
      static_for<Q>([&](auto i) {
        constexpr int ex = Lattice<Q>::ex(i), ey = Lattice<Q>::ey(i), ez = Lattice<Q>::ez(i);
        constexpr int k = int(i) * kCells - (ex + 8 * ey + 64 * ez);
        int o = 0;
        if constexpr (ex == 1) o += Xm;
        if constexpr (ex == -1) o += Xp;
        if constexpr (ey == 1) o += Ym;
        if constexpr (ey == -1) o += Yp;
        if constexpr (ez == 1) load(i, b1 + o + k);
        else if constexpr (ez == -1) load(i, bm + o + k);
        else load(i, p + o + k);
      });
    };
    auto active = [&](int c) {
      if (w.mask < 0) return true;
      const uint32_t m = __ldg(a.masks + w.mask * 16 + (c >> 5));
      return bool((m >> (c & 31)) & 1u);
    };
    // replaces, for a cell next to a wall face, the populations whose pull
    // crossed it (the periodic pull above read a valid but unused value)
    auto wall_fix = [&](int c, T (&g)[Q]) {
      const int x = c & 7, y = (c >> 3) & 7, z = c >> 6;
      const bool yl = (wf & 1) && y == 0, yh = (wf & 2) && y == 7;
      const bool zl = (wf & 4) && z == 0, zh = (wf & 8) && z == 7;
      const bool xl = (wf & 16) && x == 0, xh = (wf & 32) && x == 7;
      if (!(yl || yh || zl || zh || xl || xh)) return;
      int Xm, Xp, Ym, Yp;
      offsets(c, Xm, Xp, Ym, Yp);
      const S *b1, *bm;
      zbase(c, b1, bm);
      const S* p = src + c;
      static_for<Q>([&](auto i) {
        constexpr int ex = Lattice<Q>::ex(i), ey = Lattice<Q>::ey(i), ez = Lattice<Q>::ez(i);
        if constexpr (ex != 0 || ey != 0 || ez != 0) {
          const bool cy = ey == 1 ? yl : ey == -1 ? yh : false;
          const bool cz = ez == 1 ? zl : ez == -1 ? zh : false;
          const bool cx = ex == 1 ? xl : ex == -1 ? xh : false;  // x walls are no-slip
          if (cy || cz || cx) {
            const bool sy = a.slip & (ey == 1 ? 1 : 2), sz = a.slip & (ez == 1 ? 4 : 8);
            const int X = ex == 1 ? Xm : ex == -1 ? Xp : 0;
            const int Y = ey == 1 ? Ym : ey == -1 ? Yp : 0;
            constexpr int ib = Lattice<Q>::index(-ex, -ey, -ez);
            constexpr int iy = Lattice<Q>::index(ex, -ey, ez);
            constexpr int iz = Lattice<Q>::index(ex, ey, -ez);
            constexpr int iyz = Lattice<Q>::index(ex, -ey, -ez);
            // the reflected source: the cell itself (bounce-back), or the
            // pull along the axes not crossed (z pulls from the z base)
            const S* q;
            if (cx || (cy && !sy) || (cz && !sz)) q = p + ib * kCells;
            else if (cy && cz) q = p + (iyz * kCells - ex + X);
            else if (cy) q = (ez == 1 ? b1 : ez == -1 ? bm : p) + (iy * kCells - (ex + 64 * ez) + X);
            else q = p + (iz * kCells - (ex + 8 * ey) + X + Y);
            g[i] = *q;
          }
        }
      });
    };
    auto collide_store = [&](int c, T (&g)[Q]) {
      if constexpr (Q == 19) {
        T S_;
        if constexpr (std::is_same<T, double>::value) S_ = collide19_f64(g, tau0, T(a.cs2_18));
        else S_ = collide19<T>(g, tau0, T(a.cs2_18));
        if (L.aux_dst) reinterpret_cast<T*>(L.aux_dst)[int64_t(w.block) * kCells + c] = S_;
      } else {
        if (a.force != nullptr && w.level == 0) {
          const int64_t n = int64_t(L.BX) * L.BY * L.BZ * kCells;
          const int64_t j = int64_t(w.block) * kCells + c;
          const T* F = reinterpret_cast<const T*>(a.force);
          collide27<T, true, false>(g, T(L.omega), F[j], F[n + j], F[2 * n + j]);
        } else {
          collide27<T, false, false>(g, T(L.omega), T(0), T(0), T(0));
        }
      }
      S* q = dst + c;
      static_for<Q>([&](auto i) { St::template put<Q, i>(q + int(i) * kCells, g[i]); });
    };
    int c = c0;
#pragma unroll 1
    do {
      if (active(c)) {
        T g[Q];
        pull(c, [&](auto i, const S* p) { g[i] = load_state(p); });
        if constexpr (W) if (wf) wall_fix(c, g);
        collide_store(c, g);
      }
      c += TPB;
    } while ((c & a.run_mask) >= TPB);
  }
}

// collision of FP16 storage values (one cell or a pair)
template <int Q, class T>
__device__ __forceinline__ void collide_scaled(T* g, T tau0, T omega, T cs2_18, bool forced, T Fx, T Fy, T Fz, T& strain) {
  if constexpr (Q == 19) {
    strain = collide19<T, true>(g, tau0, cs2_18);
  } else {
    if (forced) collide27<T, true, true>(g, omega, Fx, Fy, Fz);
    else collide27<T, false, true>(g, omega, T(0), T(0), T(0));
  }
}

// FP16 storage: each thread updates an x-adjacent pair of cells (c, c + 1),
// c even, through the two-cell arithmetic of pair.cuh.  Packed FP32x2
// instructions run the two collisions for about the instruction count of
// one (the single-cell FP16 kernel was close to issue-bound), populations
// with e_x = 0 come in as one aligned half2 load for both cells, and every
// population leaves as one half2 store.  Pulls with e_x != 0 are two scalar
// loads (their sources straddle the pair alignment).  Mixed pairs (one cell
// masked out) store only the active cell.  Storage holds (f_i - w_i) / w_i,
// which the collision takes and returns.  W = true: walls as in k_update; both
// cells of a pair share their y and z faces, an x face has one of them.
// 192 x 80 x 112 D3Q19 with walls: 29.1 us per step (a cell per thread: 33.2).
template <class M, int TPB, int MINB, bool W>
__global__ void __launch_bounds__(TPB, MINB) k_update_pair(const UpdateArgs a) {
  using S = __half;
  constexpr int Q = M::Q;
  constexpr int QS = Q * kCells;
  constexpr int NP = kCells / 2;  // pairs per block
  begin_update(a);
  // runs as in k_update, in pairs (a.run_mask = pairs per run - 1)
  for (int it = blockIdx.x; it < (a.nitems << a.split); it += gridDim.x) {
    const WorkItem w = a.items[it >> a.split];
    const LevelPtrs& L = a.lv[w.level];
    const int BX = L.BX, BXY = L.BX * L.BY;
    if (threadIdx.x == 0 && a.pf_ahead > 0 && it + a.pf_ahead < a.nitems) {
      // the block that a CTA pf_ahead items later takes: its whole [Q][512] run
      // (contiguous, 16-byte aligned) into L2 by one bulk prefetch of the
      // TMA unit, so that CTA's loads find L2 instead of DRAM
      const WorkItem wn = a.items[it + a.pf_ahead];
      const char* pb = reinterpret_cast<const char*>(a.lv[wn.level].src) + int64_t(wn.block) * QS * int64_t(sizeof(S));
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(pb), "r"(int(QS * sizeof(S))) : "memory");
    }
    // block deltas as in k_update (x / y offsets 32-bit, z widened per pair)
    const int dxm = (w.edges & 1) ? (L.BX - 1) : -1;
    const int dxp = (w.edges & 2) ? -(L.BX - 1) : 1;
    const int dym = (w.edges & 4) ? BX * (L.BY - 1) : -BX;
    const int dyp = (w.edges & 8) ? -BX * (L.BY - 1) : BX;
    const int dzm = (w.edges & 16) ? BXY * (L.BZ - 1) : -BXY;
    const int dzp = (w.edges & 32) ? -BXY * (L.BZ - 1) : BXY;
    const int wf = (W && w.level == 0)
                       ? (a.walls & (((w.edges >> 2) & 15) | ((w.edges & 128) ? 16 : 0) | ((w.edges & 64) ? 32 : 0)))
                       : 0;  // as in k_update
    const V2 tau0 = V2(float(L.tau0), float(L.tau0)), omega = V2(float(L.omega), float(L.omega));
    const S* src = reinterpret_cast<const S*>(L.src) + int64_t(w.block) * QS;
    S* dst = reinterpret_cast<S*>(L.dst) + int64_t(w.block) * QS;
    auto active = [&](int c) {
      if (w.mask < 0) return true;
      const uint32_t m = __ldg(a.masks + w.mask * 16 + (c >> 5));
      return bool((m >> (c & 31)) & 1u);
    };
    bool more = true;
#pragma unroll 1
    for (int p = int(unsigned(it) * unsigned(a.run_mask + 1) % NP) + threadIdx.x; more; p += TPB, more = (p & a.run_mask) >= TPB) {
      const int c0 = 2 * p;
      const bool a0 = active(c0), a1 = active(c0 + 1);
      if (!a0 && !a1) continue;
      const int x0 = c0 & 7, y = (c0 >> 3) & 7, z = c0 >> 6;
      // cell c0 pulls e_x = +1 across the -x face when x0 == 0; cell c0 + 1
      // pulls e_x = -1 across the +x face when x0 == 6 (from that cell itself
      // on the zero-gradient outflow face)
      const int Xm0 = (x0 == 0) ? dxm * QS + 8 : 0;
      const int Xp1 = (x0 == 6) ? ((w.edges & 64) ? -1 : dxp * QS - 8) : 0;
      const int Ym = (y == 0) ? dym * QS + 64 : 0;
      const int Yp = (y == 7) ? dyp * QS - 64 : 0;
      const S* p0 = src + c0;
      const S* b1 = p0 + (z == 0 ? int64_t(dzm) * QS + 512 : int64_t(0));
      const S* bm = p0 + (z == 7 ? int64_t(dzp) * QS - 512 : int64_t(0));
      V2 g[Q];
      static_for<Q>([&](auto i) {
        constexpr int ex = Lattice<Q>::ex(i), ey = Lattice<Q>::ey(i), ez = Lattice<Q>::ez(i);
        constexpr int k = int(i) * kCells - (ex + 8 * ey + 64 * ez);
        int o = 0;
        if constexpr (ey == 1) o += Ym;
        if constexpr (ey == -1) o += Yp;
        const S* b = ez == 1 ? b1 : ez == -1 ? bm : p0;
        if constexpr (ex == 0) {
          // both sources adjacent at an even element offset: one half2 load
          const __half2 h = *reinterpret_cast<const __half2*>(b + o + k);
          g[i] = V2(__low2float(h), __high2float(h));
        } else if constexpr (ex == 1) {
          g[i] = V2(__half2float(load_state(b + o + k + Xm0)), __half2float(load_state(b + o + k + 1)));
        } else {
          g[i] = V2(__half2float(load_state(b + o + k)), __half2float(load_state(b + o + k + 1 + Xp1)));
        }
      });
      if constexpr (W) {
        const bool yl = (wf & 1) && y == 0, yh = (wf & 2) && y == 7;
        const bool zl = (wf & 4) && z == 0, zh = (wf & 8) && z == 7;
        const bool xl = (wf & 16) && x0 == 0, xh = (wf & 32) && x0 == 6;
        if (yl || yh || zl || zh || xl || xh) {
          static_for<Q>([&](auto i) {
            constexpr int ex = Lattice<Q>::ex(i), ey = Lattice<Q>::ey(i), ez = Lattice<Q>::ez(i);
            if constexpr (ex != 0 || ey != 0 || ez != 0) {
              const bool cy = ey == 1 ? yl : ey == -1 ? yh : false;
              const bool cz = ez == 1 ? zl : ez == -1 ? zh : false;
              const bool cx = ex == 1 ? xl : ex == -1 ? xh : false;  // of the one cell at the x face
              if (cy || cz || cx) {
                const bool sy = a.slip & (ey == 1 ? 1 : 2), sz = a.slip & (ez == 1 ? 4 : 8);
                constexpr int ib = Lattice<Q>::index(-ex, -ey, -ez);
                constexpr int iy = Lattice<Q>::index(ex, -ey, ez);
                constexpr int iz = Lattice<Q>::index(ex, ey, -ez);
                constexpr int iyz = Lattice<Q>::index(ex, -ey, -ez);
                const __half2 back = *reinterpret_cast<const __half2*>(p0 + ib * kCells);
                V2 v = g[i];
                if ((cy && !sy) || (cz && !sz)) {
                  v = V2(__low2float(back), __high2float(back));
                } else if (cy || cz) {
                  const S* q;
                  if (cy && cz) q = p0 + (iyz * kCells - ex);
                  else if (cy) q = (ez == 1 ? b1 : ez == -1 ? bm : p0) + (iy * kCells - (ex + 64 * ez));
                  else q = p0 + (iz * kCells - (ex + 8 * ey) + (ey == 1 ? Ym : ey == -1 ? Yp : 0));
                  v = V2(__half2float(q[ex == 1 ? Xm0 : 0]), __half2float(q[1 + (ex == -1 ? Xp1 : 0)]));
                }
                if (cx && ex == 1) v.x = __low2float(back);
                if (cx && ex == -1) v.y = __high2float(back);
                g[i] = v;
              }
            }
          });
        }
      }
      // body force of the pair (level 0 of a forced D3Q27 grid)
      const bool forced = Q == 27 && a.force != nullptr && w.level == 0;
      V2 F[3] = {V2(0.0), V2(0.0), V2(0.0)};
      if (forced) {
        const int64_t n = int64_t(L.BX) * L.BY * L.BZ * kCells;
        const float* f = reinterpret_cast<const float*>(a.force) + int64_t(w.block) * kCells + c0;
#pragma unroll
        for (int k = 0; k < 3; ++k) F[k] = V2(f[k * n], f[k * n + 1]);
      }
      V2 strain;
      if constexpr (W) {
        // walled grids collide the two cells one after the other in scalar
        // code (the compiler's contractions, so the bits of those runs, are
        // those of a cell per thread)
        float h0[Q], h1[Q];
        static_for<Q>([&](auto i) {
          h0[i] = g[i].x;
          h1[i] = g[i].y;
        });
        collide_scaled<Q>(h0, tau0.x, omega.x, float(a.cs2_18), forced, F[0].x, F[1].x, F[2].x, strain.x);
        collide_scaled<Q>(h1, tau0.x, omega.x, float(a.cs2_18), forced, F[0].y, F[1].y, F[2].y, strain.y);
        static_for<Q>([&](auto i) { g[i] = V2(h0[i], h1[i]); });
      } else {
        collide_scaled<Q>(g, tau0, omega, V2(float(a.cs2_18), float(a.cs2_18)), forced, F[0], F[1], F[2], strain);
      }
      if (Q == 19 && L.aux_dst) {
        float* ad = reinterpret_cast<float*>(L.aux_dst) + int64_t(w.block) * kCells + c0;
        if (a0) ad[0] = strain.x;
        if (a1) ad[1] = strain.y;
      }
      S* q = dst + c0;
      if (a0 && a1) {
        // streaming stores: the new state is not read again before the next
        // step, so its lines go first when L2 needs room for prefetched blocks
        static_for<Q>([&](auto i) {
          __stcs(reinterpret_cast<__half2*>(q + int(i) * kCells), __floats2half2_rn(g[i].x, g[i].y));
        });
      } else if (a0) {
        static_for<Q>([&](auto i) { q[int(i) * kCells] = __float2half_rn(g[i].x); });
      } else {
        static_for<Q>([&](auto i) { q[int(i) * kCells + 1] = __float2half_rn(g[i].y); });
      }
    }
  }
}

// Launch shapes the autotuner chooses from: threads per CTA, and a minimum
// number of resident CTAs per SM that caps the registers (higher occupancy).
// FP16 storage runs the cell-pair kernel, whose bytes in flight come from its
// residency: D3Q19 takes the listed caps as they are (256^3, 8 or 7 CTAs, both
// of 64 registers: 194 and 193 us per step, 6: 203, 5: 217); D3Q27, whose
// packed collision holds 126 registers, takes 4, 5 or 2 CTAs.

// Splitting the blocks of short work lists: a launch with fewer blocks than
// the part holds CTAs leaves SMs idle (64 blocks of a 32^3 grid on 152 SMs)
// and walks 2-4 cells per thread one after the other.  A block is cut into
// up to kCells / TPB (pairs: kCells / 2 / TPB) runs of cells as long as all of
// them stay resident at once; beyond that a cut only repeats the per-block
// address set-up.  FP64 storage is bound by the float64 pipes, whose work is
// long against that set-up, so its blocks are always cut: shorter CTAs even
// out the last wave.  32^3 D3Q19 FP64 (64 blocks, now 256 CTAs): 36 -> 21.5 us
// per step; 128^3 D3Q27 FP64 and the 105-block FP32 grid unchanged within 1 %.
inline int split_for(int nitems, int max_runs, int resident, bool always) {
  int s = 0;
  while ((2 << s) <= max_runs && (always || (int64_t(nitems) << (s + 1)) <= resident)) ++s;
  return s;
}

// CTAs per SM that the cell-pair kernel is compiled for in place of a listed
// shape's
template <class M>
constexpr int pair_ctas(int listed) {
  return M::Q == 19 ? listed : listed == 8 ? 4 : listed == 7 ? 5 : 2;
}
template <class M, bool W, int TPB, int MINB>
cudaError_t launch_pair_shape(UpdateArgs a, int ctas, cudaStream_t st) {
  a.split = split_for(a.nitems, kCells / 2 / TPB, a.resident, false);
  a.run_mask = ((kCells / 2) >> a.split) - 1;
  const int units = a.nitems << a.split, grid = ctas > 0 ? std::min(ctas, units) : units;
  // prefetch distance: three eighths of the CTAs resident at once, or the grid
  // (persistent CTAs take items grid apart); a list short enough to be split is
  // resident as a whole.  256^3, one CTA per block, us per step at a distance
  // of none, 1/8, 1/4, 3/8, 1/2, 3/4 and all of the residents: D3Q19 (8 CTAs
  // per SM) 215, 202, 197, 195, 195, 203, 216; D3Q27 (4) 329, 311, 304, 300,
  // 301, 303, 308
  a.pf_ahead = a.split > 0 ? 0 : ctas > 0 ? grid : a.resident * 3 / 8;
  return launch_chained(k_update_pair<M, TPB, MINB, W>, grid, TPB, a, a.chained, st);
}
template <class M, bool W>
cudaError_t launch_pair(const UpdateArgs& a, int threads, int minb, int ctas, cudaStream_t st) {
  if (threads == 128 && minb == 7) return launch_pair_shape<M, W, 128, pair_ctas<M>(7)>(a, ctas, st);
  if (threads == 128 && minb == 1) return launch_pair_shape<M, W, 128, 1>(a, ctas, st);
  if (threads == 256 && minb == 1) return launch_pair_shape<M, W, 256, 1>(a, ctas, st);
  if (threads == 128 && minb == 8) return launch_pair_shape<M, W, 128, pair_ctas<M>(8)>(a, ctas, st);
  if (threads == 256 && minb == 4) return launch_pair_shape<M, W, 256, pair_ctas<M>(4)>(a, ctas, st);
  return cudaErrorInvalidValue;
}
template <class M, bool W>
cudaError_t occ_pair(int threads, int minb, int* n) {
  if (threads == 128 && minb == 7) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update_pair<M, 128, pair_ctas<M>(7), W>, 128, 0);
  if (threads == 128 && minb == 1) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update_pair<M, 128, 1, W>, 128, 0);
  if (threads == 256 && minb == 1) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update_pair<M, 256, 1, W>, 256, 0);
  if (threads == 128 && minb == 8) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update_pair<M, 128, pair_ctas<M>(8), W>, 128, 0);
  if (threads == 256 && minb == 4) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update_pair<M, 256, pair_ctas<M>(4), W>, 256, 0);
  return cudaErrorInvalidValue;
}

template <class M, class S, bool W, int TPB, int MINB>
cudaError_t launch_shape(UpdateArgs a, int ctas, cudaStream_t st) {
  a.split = split_for(a.nitems, kCells / TPB, a.resident, std::is_same<S, double>::value);
  a.run_mask = (kCells >> a.split) - 1;
  const int units = a.nitems << a.split, grid = ctas > 0 ? std::min(ctas, units) : units;
  return launch_chained(k_update<M, S, TPB, MINB, W>, grid, TPB, a, a.chained, st);
}

template <class M, class S, bool W>
cudaError_t launch_ms(const UpdateArgs& a, int threads, int minb, int ctas, cudaStream_t st) {
  if (a.nitems == 0) return cudaSuccess;
  if constexpr (std::is_same<S, __half>::value) {
    return launch_pair<M, W>(a, threads, minb, ctas, st);
  } else {
    if (threads == 128 && minb == 7) return launch_shape<M, S, W, 128, 7>(a, ctas, st);
    if (threads == 128 && minb == 1) return launch_shape<M, S, W, 128, 1>(a, ctas, st);
    if (threads == 256 && minb == 1) return launch_shape<M, S, W, 256, 1>(a, ctas, st);
    if (threads == 128 && minb == 8) return launch_shape<M, S, W, 128, 8>(a, ctas, st);
    if (threads == 256 && minb == 4) return launch_shape<M, S, W, 256, 4>(a, ctas, st);
    return cudaErrorInvalidValue;
  }
}

template <class M, class S, bool W>
cudaError_t occ_ms(int threads, int minb, int* n) {
  if constexpr (std::is_same<S, __half>::value) {
    return occ_pair<M, W>(threads, minb, n);
  } else {
    if (threads == 128 && minb == 7) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update<M, S, 128, 7, W>, 128, 0);
    if (threads == 128 && minb == 1) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update<M, S, 128, 1, W>, 128, 0);
    if (threads == 256 && minb == 1) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update<M, S, 256, 1, W>, 256, 0);
    if (threads == 128 && minb == 8) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update<M, S, 128, 8, W>, 128, 0);
    if (threads == 256 && minb == 4) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_update<M, S, 256, 4, W>, 256, 0);
    return cudaErrorInvalidValue;
  }
}

// one translation unit per (model, storage) instantiates the periodic
// kernels, another the wall kernels (update_walls_<model>_<storage>.cu)
#define LBM_UPDATE_INSTANCE(M, S, NAME)                                                               \
  cudaError_t launch_update_##NAME(const UpdateArgs& a, int threads, int minb, int ctas, cudaStream_t st) { \
    return launch_ms<M, S, false>(a, threads, minb, ctas, st);                                       \
  }                                                                                                  \
  cudaError_t occupancy_update_##NAME(int threads, int minb, int* n) { return occ_ms<M, S, false>(threads, minb, n); }

#define LBM_UPDATE_WALL_INSTANCE(M, S, NAME)                                                          \
  cudaError_t launch_update_walls_##NAME(const UpdateArgs& a, int threads, int minb, int ctas,        \
                                         cudaStream_t st) {                                          \
    return launch_ms<M, S, true>(a, threads, minb, ctas, st);                                        \
  }                                                                                                  \
  cudaError_t occupancy_update_walls_##NAME(int threads, int minb, int* n) {                         \
    return occ_ms<M, S, true>(threads, minb, n);                                                     \
  }

#define LBM_UPDATE_DECL(NAME)                                                                          \
  cudaError_t launch_update_##NAME(const UpdateArgs& a, int threads, int minb, int ctas, cudaStream_t st); \
  cudaError_t occupancy_update_##NAME(int threads, int minb, int* n);                                   \
  cudaError_t launch_update_walls_##NAME(const UpdateArgs& a, int threads, int minb, int ctas,          \
                                         cudaStream_t st);                                             \
  cudaError_t occupancy_update_walls_##NAME(int threads, int minb, int* n);

LBM_UPDATE_DECL(d3q19_f64)
LBM_UPDATE_DECL(d3q19_f32)
LBM_UPDATE_DECL(d3q19_f16)
LBM_UPDATE_DECL(d3q27_f64)
LBM_UPDATE_DECL(d3q27_f32)
LBM_UPDATE_DECL(d3q27_f16)

}  // namespace lbm
