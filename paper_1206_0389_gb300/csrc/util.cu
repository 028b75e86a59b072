// Utility kernels: dense <-> block staging (state, equilibrium initialisation,
// macroscopic fields, body force), sampled gathers and the float64
// mass/momentum audit.
#include <cmath>

#include "collide.cuh"
#include "kernels.cuh"

namespace lbm {

template <int Q>
__device__ __forceinline__ double shift_of(int i) {
  return Q == 27 ? weight_rt<27>(i) : 0.0;  // D3Q19 stores the incompressible f itself
}

// locate dense level cell (x, y, z) in the level box; -1 if outside
__device__ __forceinline__ int64_t box_index(int x, int y, int z, int ox, int oy, int oz, int BX,
                                             int BY, int BZ) {
  const int bx = (x >> 3) - ox, by = (y >> 3) - oy, bz = (z >> 3) - oz;
  if (bx < 0 || bx >= BX || by < 0 || by >= BY || bz < 0 || bz >= BZ) return -1;
  return (int64_t(bx) + int64_t(BX) * (by + int64_t(BY) * bz)) * kCells + (x & 7) + 8 * (y & 7) +
         64 * (z & 7);
}

// delta rho and momentum of one cell's shifted populations by a z, y, x
// collapse (D3Q27, 49 additions) or over opposite pairs (D3Q19, 39) instead
// of one addition per non-zero term (81 and 49)
template <int Q, class T>
__device__ __forceinline__ void raw_moments(const T (&g)[Q], T& r, T& jx, T& jy, T& jz) {
  if constexpr (Q == 27) {
    T M0[3], My[3], Dz[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T m[3], d[3];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const T lo = g[D3Q27::index(a - 1, b - 1, -1)], hi = g[D3Q27::index(a - 1, b - 1, 1)];
        m[b] = (hi + lo) + g[D3Q27::index(a - 1, b - 1, 0)];
        d[b] = hi - lo;
      }
      M0[a] = (m[2] + m[0]) + m[1];
      My[a] = m[2] - m[0];
      Dz[a] = (d[2] + d[0]) + d[1];
    }
    r = (M0[2] + M0[0]) + M0[1];
    jx = M0[2] - M0[0];
    jy = (My[2] + My[0]) + My[1];
    jz = (Dz[2] + Dz[0]) + Dz[1];
  } else {
    r = g[0];
    jx = jy = jz = T(0);
    static_for<9>([&](auto p) {
      constexpr int i = 2 * p + 1;
      constexpr int x = D3Q19::ex(i), y = D3Q19::ey(i), z = D3Q19::ez(i);
      const T d = g[i] - g[i + 1];
      r += g[i] + g[i + 1];
      if constexpr (x != 0) jx += x > 0 ? d : -d;
      if constexpr (y != 0) jy += y > 0 ? d : -d;
      if constexpr (z != 0) jz += z > 0 ? d : -d;
    });
  }
}

// The same sums in float64.  GB300 issues 2 float64 operations per clock and
// SM against 128 float32 ones, so for FP32 and FP16 storage the sums run in
// float32 without losing a bit that float64 would keep: each value is cut
// into g = h + h' + h'' on two grids common to the cell, 2^-19 and 2^-39 of the
// power of two above its largest population (adding and subtracting 1.5 times
// 2^23 grid units rounds to the grid; both cuts are exact).  Sums of up to 27
// terms with factors 0, +-1 on a grid are exact in 24 bits, and those of the
// rests h'' (below 2^-40 of the largest) are off by less than 2^-54 of it,
// less than the roundings of a plain float64 sum.  Only the three partial sums
// of each moment are added in float64.  Values from 2^100 up, infinite ones
// among them, take the plain sum; NaN spreads through either.  Macroscopic
// fields of 256^3 D3Q27 FP32 into device memory 6.0 -> 1.24 ms, a statistics
// sample of the 40 M-cell FP16 jet 13.4 -> 3.5 ms, of a 3 M-cell D3Q19 FP32
// jet 0.64 -> 0.22 ms; still bound by float64 issue (about 45 operations).
template <class S, int Q>
__device__ __forceinline__ void moments64(const S* f, double& r, double& jx, double& jy, double& jz) {
  if constexpr (std::is_same<S, double>::value) {
    double g[Q];
    static_for<Q>([&](auto i) { g[i] = f[int(i) * kCells]; });
    raw_moments<Q>(g, r, jx, jy, jz);
  } else {
    float g[Q], top = 0.f;
    static_for<Q>([&](auto i) {
      if constexpr (std::is_same<S, __half>::value)
        g[i] = __fmul_rn(__half2float(f[int(i) * kCells]), float(Lattice<Q>::w(i)));  // as the collision sees it
      else
        g[i] = f[int(i) * kCells];
      top = fmaxf(top, fabsf(g[i]));
    });
    if (top < 0x1p100f) {
      // biased exponent of the largest value; cells below 2^-79 (the front of a
      // disturbance in fluid at rest) are lifted by 2^100, so that the grids
      // and the rests stay clear of the smallest floats
      int e = __float_as_int(top) >> 23;
      const bool lift = e < 48;
      if (lift) {
        static_for<Q>([&](auto i) { g[i] *= 0x1p100f; });
        e = max(__float_as_int(top * 0x1p100f) >> 23, 48);
      }
      double sum[4] = {0, 0, 0, 0};
#pragma unroll
      for (int cut = 0; cut < 3; ++cut) {
        float h[Q], m[4];
        if (cut < 2) {
          const float c = __int_as_float(((e + (cut == 0 ? 5 : -15)) << 23) | 0x400000);
          static_for<Q>([&](auto i) {
            h[i] = __fsub_rn(__fadd_rn(g[i], c), c);
            g[i] = __fsub_rn(g[i], h[i]);
          });
        } else {
          static_for<Q>([&](auto i) { h[i] = g[i]; });
        }
        raw_moments<Q>(h, m[0], m[1], m[2], m[3]);
#pragma unroll
        for (int k = 0; k < 4; ++k) sum[k] = cut == 0 ? double(m[k]) : sum[k] + double(m[k]);
      }
      if (lift) {
#pragma unroll
        for (int k = 0; k < 4; ++k) sum[k] *= 0x1p-100;
      }
      r = sum[0];
      jx = sum[1];
      jy = sum[2];
      jz = sum[3];
    } else {
      r = jx = jy = jz = 0;
#pragma unroll 1
      for (int i = 0; i < Q; ++i) {
        const double v = double(load_rt<S, Q>(f + i * kCells, i));
        r += v;
        if (ex27(i)) jx += ex27(i) * v;
        if (ey27(i)) jy += ey27(i) * v;
        if (ez27(i)) jz += ez27(i) * v;
      }
    }
  }
}

// a / b for three numerators: one reciprocal, each quotient corrected by its
// residual.  Where that is not finite (b zero or infinite, a infinite, an
// overflow on the way) the quotient is taken by itself.
__device__ __forceinline__ void divide3(double b, double& x, double& y, double& z) {
  const double r = 1.0 / b;
  auto q = [&](double a) {
    const double v = a * r, c = fma(fma(-v, b, a), r, v);
    return (__double2hiint(c) & 0x7ff00000) != 0x7ff00000 ? c : a / b;
  };
  x = q(x);
  y = q(y);
  z = q(z);
}

template <class M, class S>
__global__ void k_slab(const SlabArgs a) {
  using T = typename Store<S>::T;
  constexpr int Q = M::Q;
  const int64_t n = int64_t(a.NX) * a.NY * a.nz;
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int x = int(t % a.NX), y = int((t / a.NX) % a.NY), z = a.z0 + int(t / (int64_t(a.NX) * a.NY));
  const int64_t j = box_index(x, y, z, a.ox, a.oy, a.oz, a.BX, a.BY, a.BZ);
  const int64_t blk = j >= 0 ? j / kCells : 0, cell = j >= 0 ? j % kCells : 0;
  S* f = reinterpret_cast<S*>(a.f) + blk * Q * kCells + cell;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  switch (a.mode) {
    case SLAB_SET_STATE: {
      if (j < 0) return;
      for (int i = 0; i < Q; ++i) {
        const double v = a.in[i][t];
        if (isnan(v)) continue;
        store_rt<S, Q>(f + i * kCells, i, T(v - shift_of<Q>(i)));
      }
      return;
    }
    case SLAB_GET_STATE: {
      for (int i = 0; i < Q; ++i)
        a.out[i][t] = j < 0 ? nan : double(load_rt<S, Q>(f + i * kCells, i)) + shift_of<Q>(i);
      return;
    }
    case SLAB_INIT_EQ: {
      if (j < 0) return;
      auto in = [&](int c) { return a.in[c] != nullptr ? a.in[c][t] : a.fill[c]; };
      const T rl = T(in(0) - 1.0);  // delta rho for both shifted models
      const T ux = T(in(1)), uy = T(in(2)), uz = T(in(3));
      T feq[Q];
      M::feq(rl, ux, uy, uz, feq);
      for (int i = 0; i < Q; ++i) store_rt<S, Q>(f + i * kCells, i, feq[i]);
      return;
    }
    case SLAB_MACRO: {
      const uint8_t k = j < 0 ? uint8_t(K_NONE) : a.kind[j];
      if (k != K_ACTIVE && k != K_HIDDEN1 && k != K_HIDDEN2) {
        for (int c = 0; c < 4; ++c) a.out[c][t] = nan;
        return;
      }
      double rl, ux, uy, uz;
      moments64<S, Q>(f, rl, ux, uy, uz);
      const double rho = 1.0 + rl;
      if (Q == 27) {
        if (a.force != nullptr) {
          const int64_t nn = int64_t(a.BX) * a.BY * a.BZ * kCells;
          ux += 0.5 * a.force[j];
          uy += 0.5 * a.force[nn + j];
          uz += 0.5 * a.force[2 * nn + j];
        }
        divide3(rho, ux, uy, uz);
      }
      a.out[0][t] = rho;
      a.out[1][t] = ux;
      a.out[2][t] = uy;
      a.out[3][t] = uz;
      return;
    }
    case SLAB_SET_LAMBDA: {
      if (j < 0) return;
      T* r = reinterpret_cast<T*>(a.raw) + blk * Q * kCells + cell;
      for (int i = 0; i < Q; ++i) r[i * kCells] = T(a.in[i][t]);
      return;
    }
    case SLAB_GET_FIELD3: {
      const int64_t nn = int64_t(a.BX) * a.BY * a.BZ * kCells;
      const T* r = reinterpret_cast<const T*>(a.raw);
      for (int c = 0; c < 3; ++c) a.out[c][t] = j < 0 ? nan : double(r[c * nn + j]);
      return;
    }
    case SLAB_GET_STATS: {
      // mean rho, u_x, u_y, u_z, then the variances <u_a^2> - <u_a>^2
      const uint8_t k = j < 0 ? uint8_t(K_NONE) : a.kind[j];
      const bool ok = k == K_ACTIVE || k == K_HIDDEN1 || k == K_HIDDEN2;
      const int64_t nn = int64_t(a.BX) * a.BY * a.BZ * kCells;
      const double* r = reinterpret_cast<const double*>(a.raw);
      for (int c = 0; c < 4; ++c) a.out[c][t] = ok ? r[c * nn + j] * a.scale : nan;
      for (int c = 0; c < 3; ++c) {
        const double m = ok ? r[(1 + c) * nn + j] * a.scale : 0.0;
        a.out[4 + c][t] = ok ? r[(4 + c) * nn + j] * a.scale - m * m : nan;
      }
      return;
    }
    case SLAB_GET_AUX: {
      a.out[0][t] = j < 0 ? nan : double(reinterpret_cast<const T*>(a.raw)[j]);
      return;
    }
    case SLAB_SET_AUX: {
      if (j < 0 || isnan(a.in[0][t])) return;
      reinterpret_cast<T*>(a.raw)[j] = T(a.in[0][t]);
      return;
    }
    case SLAB_SET_FORCE: {
      if (j < 0) return;
      const int64_t nn = int64_t(a.BX) * a.BY * a.BZ * kCells;
      for (int c = 0; c < 3; ++c) a.force[c * nn + j] = a.in[c][t];
      return;
    }
  }
}

// one thread per (cell, population): a thread per cell chained Q loads of a
// few cells one after the other, and its results lay Q apart
template <class M, class S>
__global__ void k_gather(const GatherArgs a) {
  constexpr int Q = M::Q;
  const int64_t o = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, t = o / Q;
  if (t >= a.n) return;
  const int i = int(o - t * Q);
  const long long c = a.cells[t];
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  const long long ncell = (long long)a.NX * a.NY * a.NZ;
  int64_t j = -1;
  if (c >= 0 && c < ncell) {
    const int x = int(c % a.NX), y = int((c / a.NX) % a.NY), z = int(c / ((long long)a.NX * a.NY));
    j = box_index(x, y, z, a.ox, a.oy, a.oz, a.BX, a.BY, a.BZ);
  }
  if (j < 0) {
    a.out[o] = nan;
    return;
  }
  const S* f = reinterpret_cast<const S*>(a.f) + ((j / kCells) * Q + i) * kCells + j % kCells;
  a.out[o] = double(load_rt<S, Q>(f, i)) + shift_of<Q>(i);
}

// Float64 sums over active cells: (delta rho, j_x, j_y, j_z) times vol.
//
// Each thread first sums every population separately over its cells,
// S_i = sum_cells g_i, and forms delta rho = sum_i S_i and j_a = sum_i e_ia S_i
// only at the end: Q float64 additions per cell instead of one per non-zero
// term of the four sums (81 for D3Q27), which matters on a part whose
// float64 rate is a small fraction of its float32 rate.  For float32 and
// float16 storage the per-population sums run in float32 pairs (s, e) by
// Knuth's TwoSum, s + e being the sum of up to kFlush values with the
// rounding of each addition kept in e, and every kFlush cells (inactive
// ones adding zeros) both are added to the float64 sum.  The pair's error
// over m values is below about m^2 u^2 sum |g| (u = 2^-24), 4e-12 of sum |g|
// for m = 32, the order of the bound of plain float64 recursive summation
// over a thread's values; the float64 work (two conversions and two
// additions per population and flush) is what limits the kernel on GB300.
// The populations are taken in chunks (registers), each chunk one pass over
// the thread's cells.
constexpr int kFlush = 32;
constexpr int kReduceUnroll = 4;  // cells per iteration, their loads issued together

template <class M, class S>
__global__ void __launch_bounds__(256, reduce_ctas_per_sm(std::is_same<S, __half>::value ? LBM_F16 : LBM_F32))
    k_reduce(const ReduceArgs a) {
  constexpr int Q = M::Q;
  constexpr int P = Q == 19 ? 10 : 9;  // populations per pass
  constexpr int NP = (Q + P - 1) / P;
  constexpr int U = kReduceUnroll;
  constexpr bool kPair = !std::is_same<S, double>::value;
  using V = typename std::conditional<kPair, float, double>::type;
  double s[4] = {0, 0, 0, 0};
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  const int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  static_for<NP>([&](auto pass) {
    constexpr int i0 = int(pass) * P;
    constexpr int n = (Q - i0) < P ? (Q - i0) : P;
    double D[n];
    float hs[n], he[n];
    static_for<n>([&](auto k) {
      D[k] = 0.0;
      hs[k] = 0.f;
      he[k] = 0.f;
    });
    [[maybe_unused]] int m = 0;  // cells since the last flush (float pairs only)
    for (int64_t t = t0; t < a.ncells; t += U * stride) {
      // U cells t, t + stride, ...: every value and kind loaded at once (the
      // values unconditionally: every cell of the box has storage, so no
      // load waits for a kind), then inactive cells select zeros
      S raw[U][n];
      bool on[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t tt = t + u * stride;
        const int64_t tc = tt < a.ncells ? tt : a.ncells - 1;
        const S* f = reinterpret_cast<const S*>(a.f) + (tc / kCells) * Q * kCells + tc % kCells;
        static_for<n>([&](auto k) { raw[u][k] = f[(i0 + int(k)) * kCells]; });
        on[u] = tt < a.ncells && a.kind[tc] == K_ACTIVE;
      }
      V v[U][n];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        static_for<n>([&](auto k) {
          [[maybe_unused]] constexpr int i = i0 + int(k);
          if constexpr (std::is_same<S, __half>::value)
            // the stored value as the collision sees it: the product h w
            // rounded to float (__fmul_rn keeps it from being fused into
            // the addition below, which would sum unrounded products)
            v[u][k] = on[u] ? __fmul_rn(__half2float(raw[u][k]), float(Lattice<Q>::w(i))) : 0.f;
          else
            v[u][k] = on[u] ? V(raw[u][k]) : V(0);
        });
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        static_for<n>([&](auto k) {
          if constexpr (!kPair) {
            D[k] += v[u][k];
          } else {
            // TwoSum: x = hs + g exactly equals x + r
            const float g = v[u][k];
            const float x = hs[k] + g;
            const float b = x - hs[k];
            const float r = (hs[k] - (x - b)) + (g - b);
            hs[k] = x;
            he[k] += r;
          }
        });
      }
      if constexpr (kPair) {
        m += U;
        if (m >= kFlush) {
          static_for<n>([&](auto k) {
            D[k] += double(hs[k]);
            D[k] += double(he[k]);
            hs[k] = 0.f;
            he[k] = 0.f;
          });
          m = 0;
        }
      }
    }
    static_for<n>([&](auto k) {
      constexpr int i = i0 + int(k);
      const double Si = kPair ? (D[k] + double(hs[k])) + double(he[k]) : D[k];
      s[0] += Si;
      if constexpr (Lattice<Q>::ex(i) != 0) s[1] += Lattice<Q>::ex(i) > 0 ? Si : -Si;
      if constexpr (Lattice<Q>::ey(i) != 0) s[2] += Lattice<Q>::ey(i) > 0 ? Si : -Si;
      if constexpr (Lattice<Q>::ez(i) != 0) s[3] += Lattice<Q>::ez(i) > 0 ? Si : -Si;
    });
  });
  __shared__ double sh[4][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    double v = s[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[c][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double v = 0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) v += sh[threadIdx.x][w];
    a.partial[blockIdx.x * 4 + threadIdx.x] = v * a.vol;
  }
}

// one warp per sum; out may be registered host memory
__global__ void k_reduce_final(const double* partial, int n, double* out) {
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double v = 0;
  for (int i = lane; i < n; i += 32) v += partial[i * 4 + c];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) out[c] = v;
}

template <class M, class S>
static cudaError_t slab_ms(const SlabArgs& a, cudaStream_t st) {
  const int64_t n = int64_t(a.NX) * a.NY * a.nz;
  if (n == 0) return cudaSuccess;
  k_slab<M, S><<<unsigned((n + 255) / 256), 256, 0, st>>>(a);
  return cudaGetLastError();
}
template <class M, class S>
static cudaError_t gather_ms(const GatherArgs& a, cudaStream_t st) {
  if (a.n == 0) return cudaSuccess;
  k_gather<M, S><<<unsigned((a.n * M::Q + 127) / 128), 128, 0, st>>>(a);
  return cudaGetLastError();
}
template <class M, class S>
static cudaError_t reduce_ms(const ReduceArgs& a, int ctas, cudaStream_t st) {
  k_reduce<M, S><<<ctas, 256, 0, st>>>(a);
  return cudaGetLastError();
}

#define LBM_DISPATCH(FN, ...)                                       \
  if (model == LBM_D3Q19_MRT_LES) {                                 \
    if (storage == LBM_F64) return FN<MrtLes, double>(__VA_ARGS__); \
    if (storage == LBM_F32) return FN<MrtLes, float>(__VA_ARGS__);  \
    return FN<MrtLes, __half>(__VA_ARGS__);                         \
  }                                                                 \
  if (storage == LBM_F64) return FN<Fclb, double>(__VA_ARGS__);     \
  if (storage == LBM_F32) return FN<Fclb, float>(__VA_ARGS__);      \
  return FN<Fclb, __half>(__VA_ARGS__);

cudaError_t launch_slab(int model, int storage, const SlabArgs& a, cudaStream_t st) { LBM_DISPATCH(slab_ms, a, st) }
cudaError_t launch_gather(int model, int storage, const GatherArgs& a, cudaStream_t st) { LBM_DISPATCH(gather_ms, a, st) }
cudaError_t launch_reduce(int model, int storage, const ReduceArgs& a, int ctas, cudaStream_t st) {
  LBM_DISPATCH(reduce_ms, a, ctas, st)
}
// input checks: four loads in flight per thread (the values may lie in host
// memory, a link away)
__global__ void __launch_bounds__(256) k_check(const double* p, long long n, int shift, int* flags) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  int f = 0;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += 4 * stride) {
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = t + k * stride < n ? p[t + k * stride] : 1.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) f |= (isnan(v[k]) ? 1 : 0) | (isinf(v[k]) ? 2 : 0) | (v[k] > 0 ? 0 : 4);
  }
  f = __reduce_or_sync(0xffffffffu, unsigned(f));
  if (f && (threadIdx.x & 31) == 0) atomicOr(flags, f << shift);
}
// one sample of the time statistics: rho and u of every cell holding a value
// of the level (the same moments as the macroscopic output), accumulated in
// float64
template <class M, class S>
__global__ void k_stats(const StatsArgs a) {
  constexpr int Q = M::Q;
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= a.ncells) return;
  const uint8_t k = a.kind[j];
  if (k != K_ACTIVE && k != K_HIDDEN1 && k != K_HIDDEN2) return;
  const S* f = reinterpret_cast<const S*>(a.f) + (j / kCells) * Q * kCells + (j % kCells);
  double rl, ux, uy, uz;
  moments64<S, Q>(f, rl, ux, uy, uz);
  const double rho = 1.0 + rl;
  if (Q == 27) divide3(rho, ux, uy, uz);
  const double v[3] = {ux, uy, uz};
  double old[7];
#pragma unroll
  for (int c = 0; c < 7; ++c) old[c] = a.sums[c * a.ncells + j];
  a.sums[j] = old[0] + rho;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a.sums[(1 + c) * a.ncells + j] = old[1 + c] + v[c];
    a.sums[(4 + c) * a.ncells + j] = fma(v[c], v[c], old[4 + c]);
  }
}

__global__ void k_radial(const RadialArgs a) {
  const int64_t per = int64_t(a.NY) * a.NZ;
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= per * a.nst) return;
  const int s = int(t / per);
  const int y = int(t % a.NY), z = int((t % per) / a.NY);
  const int64_t j = box_index(a.xs[s], y, z, a.ox, a.oy, a.oz, a.BX, a.BY, a.BZ);
  if (j < 0) return;
  const uint8_t k = a.kind[j];
  if (k != K_ACTIVE && (a.active_only || (k != K_HIDDEN1 && k != K_HIDDEN2))) return;
  const double dy = (y + 0.5) * a.inv_scale - a.y0, dz = (z + 0.5) * a.inv_scale - a.z0;
  const double r = sqrt(__dadd_rn(__dmul_rn(dy, dy), __dmul_rn(dz, dz)));
  // compare before converting: r / dr may exceed the int range (tiny dr)
  const double rb = floor(r / a.dr);
  if (!(rb < double(a.nbins))) return;
  const int b = int(rb);
  const int64_t nn = int64_t(a.BX) * a.BY * a.BZ * kCells;
  const double m = a.sums[nn + j] * a.scale;
  const double v = a.sums[4 * nn + j] * a.scale - m * m;
  const int64_t o = int64_t(s) * a.nbins + b;
  atomicAdd(a.acc + 3 * o, a.weight * m);
  atomicAdd(a.acc + 3 * o + 1, a.weight * v);
  atomicAdd(a.acc + 3 * o + 2, a.weight);
  atomicAdd(a.cnt + o, 1ull);
}

cudaError_t launch_radial(const RadialArgs& a, cudaStream_t st) {
  const int64_t n = int64_t(a.NY) * a.NZ * a.nst;
  if (n == 0) return cudaSuccess;
  k_radial<<<unsigned((n + 255) / 256), 256, 0, st>>>(a);
  return cudaGetLastError();
}

template <class M, class S>
static cudaError_t stats_ms(const StatsArgs& a, cudaStream_t st) {
  if (a.ncells == 0) return cudaSuccess;
  k_stats<M, S><<<unsigned((a.ncells + 255) / 256), 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_stats(int model, int storage, const StatsArgs& a, cudaStream_t st) {
  if (model == LBM_D3Q19_MRT_LES) {
    if (storage == LBM_F64) return stats_ms<MrtLes, double>(a, st);
    if (storage == LBM_F32) return stats_ms<MrtLes, float>(a, st);
    return stats_ms<MrtLes, __half>(a, st);
  }
  if (storage == LBM_F64) return stats_ms<Fclb, double>(a, st);
  if (storage == LBM_F32) return stats_ms<Fclb, float>(a, st);
  return stats_ms<Fclb, __half>(a, st);
}

__global__ void k_to_float(const double* in, float* out, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = float(in[i]);
}

cudaError_t launch_to_float(const double* in, float* out, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_to_float<<<unsigned((n + 255) / 256), 256, 0, st>>>(in, out, n);
  return cudaGetLastError();
}

cudaError_t launch_check(const double* p, long long n, int shift, int* flags, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const long long ctas = (n + 1023) / 1024;
  k_check<<<unsigned(ctas < 4096 ? ctas : 4096), 256, 0, st>>>(p, n, shift, flags);
  return cudaGetLastError();
}

cudaError_t launch_reduce_final(const double* partial, int n, double* out, cudaStream_t st) {
  k_reduce_final<<<1, 128, 0, st>>>(partial, n, out);
  return cudaGetLastError();
}

}  // namespace lbm
