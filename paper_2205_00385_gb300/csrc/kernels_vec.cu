// Float64-accurate long-vector kernels: the CG recursion of the mixed path,
// the PARM/CARM Gram matrices and combinations, and Gram-Schmidt.
//
// A vector is stored either as float64 (the FP64 path: float64 arithmetic)
// or as double-float pairs float2 {hi, lo} (the mixed path: every operation
// in double-float on the FP32 pipe, ~2^-48 relative).  GB300 executes one
// float64 FMA per clock per SM against 128 float32 FMAs, so the mixed path
// keeps its float64-accurate vectors in the pair format: loads and stores
// need no conversion and the FP64 pipe is left idle.  Reductions use a
// fixed grid and fixed summation orders, so results do not depend on
// scheduling.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "dfmath.cuh"
#include "kernels.h"

namespace topo {

// Arithmetic of a storage type: T is the register type.
template <typename S>
struct Ar;
template <>
struct Ar<double> {
  using T = double;
  __device__ static T ld(const double* p, long long i) { return p[i]; }
  __device__ static void st(double* p, long long i, T v) { p[i] = v; }
  __device__ static T zero() { return 0.0; }
  __device__ static T from_d(double x) { return x; }
  __device__ static T add(T a, T b) { return a + b; }
  __device__ static T fma3(T a, T b, T c) { return fma(a, b, c); }
  __device__ static T mulf(T a, float b) { return a * (double)b; }
  __device__ static double to_d(T a) { return a; }
  __device__ static T shfl_down(T a, int o) { return __shfl_down_sync(0xffffffffu, a, o); }
  // dot-product accumulation (acc += a b) and its final normalisation
  __device__ static void dacc(T& acc, T a, T b) { acc = fma(a, b, acc); }
  __device__ static T dfin(T a) { return a; }
};
template <>
struct Ar<float2> {
  using T = dfl;
  __device__ static T ld(const float2* p, long long i) {
    const float2 v = p[i];
    return {v.x, v.y};
  }
  __device__ static void st(float2* p, long long i, T v) { p[i] = make_float2(v.h, v.l); }
  __device__ static T zero() { return {0.f, 0.f}; }
  __device__ static T from_d(double x) { return split_d(x); }
  __device__ static T add(T a, T b) { return df_add(a, b); }
  __device__ static T fma3(T a, T b, T c) { return df_fma(a, b, c); }
  // a * b for a float b (b exact): TwoProduct on hi plus the lo term
  __device__ static T mulf(T a, float b) {
    const float p = a.h * b;
    float e = fmaf(a.h, b, -p);
    e = fmaf(a.l, b, e);
    const float h = p + e;
    return {h, e - (h - p)};
  }
  __device__ static double to_d(T a) { return df_to_d(a); }
  __device__ static T shfl_down(T a, int o) {
    return {__shfl_down_sync(0xffffffffu, a.h, o), __shfl_down_sync(0xffffffffu, a.l, o)};
  }
  __device__ static void dacc(T& acc, T a, T b) { df_dot_acc(acc, a, b); }
  __device__ static T dfin(T a) { return df_norm(a); }
};

// store a register value into a (possibly different) storage type
__device__ __forceinline__ void st_any(double* p, long long i, double v) { p[i] = v; }
__device__ __forceinline__ void st_any(double* p, long long i, dfl v) { p[i] = df_to_d(v); }
__device__ __forceinline__ void st_any(float2* p, long long i, dfl v) { p[i] = make_float2(v.h, v.l); }

// grid_sum of NV per-thread values; warps reduce in the storage's arithmetic
template <typename S, int NV, int NW>
__device__ __forceinline__ bool grid_sum_v(const typename Ar<S>::T (&v)[NV], double (&sh)[NV][NW],
                                           double (&out)[NV], double* partials,
                                           unsigned* counter) {
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    typename Ar<S>::T x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = Ar<S>::add(x, Ar<S>::shfl_down(x, o));
    if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = Ar<S>::to_d(x);
  }
  return grid_sum<NV, NW>(sh, out, partials, counter);
}

// single-value reduction finished by the last block, *out = sum: all its threads
// read the blocks' sums (one warp, as for several values, took 2 us more of a PARM
// update's 16 at 64 x 32 x 32 in float64 and of its 18 at 96 x 48 x 48 in pairs)
template <typename S>
__device__ __forceinline__ void reduce_to(typename Ar<S>::T v, double* out, double* partials,
                                          unsigned* counter) {
  __shared__ double sh[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = Ar<S>::add(v, Ar<S>::shfl_down(v, o));
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (lane == 0) sh[threadIdx.x >> 5] = Ar<S>::to_d(v);
  __syncthreads();
  double o1[1] = {0.0};
  if (threadIdx.x < 32) {
    o1[0] = lane < nw ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) o1[0] += __shfl_down_sync(0xffffffffu, o1[0], o);
  }
  __syncthreads();
  if (publish_partials<1>(o1, partials, counter)) {
    double t[1];
    finish_sum<1>(partials, counter, t, sh);
    if (threadIdx.x == 0) *out = t[0];
  }
}

#define GRID_LOOP(k, n)                                                 \
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; \
       k < (n); k += (long long)gridDim.x * blockDim.x)

// ---------------------------------------------------------------------------
// Basic vector operations
// ---------------------------------------------------------------------------
template <typename S>
__global__ void __launch_bounds__(RED_THREADS)
    k_vdot(long long n, const S* __restrict__ a, const S* __restrict__ b, double* partials,
           unsigned* counter, double* out) {
  using A = Ar<S>;
  typename A::T v[2] = {A::zero(), A::zero()};
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; k + 3 * stride < n; k += 4 * stride) {
    typename A::T av[4], bv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      av[u] = A::ld(a, k + u * stride);
      bv[u] = A::ld(b, k + u * stride);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) A::dacc(v[u & 1], av[u], bv[u]);
  }
  for (; k < n; k += stride) A::dacc(v[0], A::ld(a, k), A::ld(b, k));
  reduce_to<S>(A::add(A::dfin(v[0]), A::dfin(v[1])), out, partials, counter);
}

__global__ void __launch_bounds__(256) k_split(long long n, const double* __restrict__ in,
                                               float2* __restrict__ out) {
  GRID_LOOP(k, n) {
    const dfl v = split_d(in[k]);
    out[k] = make_float2(v.h, v.l);
  }
}

__global__ void __launch_bounds__(256) k_join(long long n, const float2* __restrict__ in,
                                              double* __restrict__ out) {
  GRID_LOOP(k, n) {
    const float2 v = in[k];
    out[k] = df_to_d({v.x, v.y});
  }
}

template <typename S>
__global__ void __launch_bounds__(256) k_vcopy(long long n, const S* __restrict__ a,
                                               S* __restrict__ b) {
  GRID_LOOP(k, n) b[k] = a[k];
}

// a *= 1/sqrt(*s2) (0 when *s2 <= 0); the scale is formed once per block
template <typename S>
__global__ void __launch_bounds__(256) k_vscale_inv_sqrt(long long n, S* __restrict__ a,
                                                         const double* __restrict__ s2) {
  using A = Ar<S>;
  __shared__ double s_sc;
  if (threadIdx.x == 0) s_sc = (*s2 > 0.0) ? 1.0 / sqrt(*s2) : 0.0;
  __syncthreads();
  const typename A::T sc = A::from_d(s_sc);
  GRID_LOOP(k, n) A::st(a, k, A::fma3(A::ld(a, k), sc, A::zero()));
}

// ---------------------------------------------------------------------------
// Gram matrix G[i + ldg*j] = sum_k A[k + i*n] B[k + j*n] (i < na, j < nb,
// both <= MAXB) in one pass over the data: a block stages a chunk of MD_CH
// indices of every column in shared memory, then its threads accumulate
// 2 x 2 tiles of G over interleaved index subsets.  Per-block partials are
// summed by the last block in block order.
// ---------------------------------------------------------------------------
constexpr int MD_CH = 128;   // indices per chunk = threads per block

__device__ __forceinline__ void cp_async8(void* dst, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src),
               "r"(valid ? 8 : 0)
               : "memory");
}

template <typename S>
__global__ void __launch_bounds__(MD_CH)
    k_gram(long long n, const S* __restrict__ A, int na, const int* na_dev,
           const S* __restrict__ B, int nb, const int* nb_dev, double* G, int ldg,
           double* partials, unsigned* counter, bool sym) {
  using Rg = Ar<S>;
  using V = typename Rg::T;
  static_assert(sizeof(V) == sizeof(S), "staged values keep the storage layout");
  extern __shared__ unsigned char md_smem[];
  V* sv = reinterpret_cast<V*>(md_smem);   // [2][nv][MD_CH]
  __shared__ bool s_last;
  const int ma = na_dev ? min(max(*na_dev, 0), na) : na;
  const int mb = nb_dev ? min(max(*nb_dev, 0), nb) : nb;
  const int nv = ma + mb;
  const int tr = (ma + 1) / 2, tc = (mb + 1) / 2;
  // sym (a symmetric product, ma == mb): only the 2 x 2 tiles on or above
  // the diagonal, numbered column by column (tile = tj (tj+1)/2 + ti)
  const int ntt = sym ? tr * (tr + 1) / 2 : tr * tc;
  const int ntile = ntt > 0 ? ntt : 1;
  const int S_ = MD_CH / ntile;   // index subsets per tile (>= 2)
  const int t = threadIdx.x;
  const int tile = t % ntile, sub = t / ntile;
  const bool active = ntt > 0 && sub < S_;
  int ti = tile % (tr > 0 ? tr : 1), tj = tile / (tr > 0 ? tr : 1);
  if (sym) {
    tj = 0;
    while ((tj + 1) * (tj + 2) / 2 <= tile) ++tj;
    ti = tile - tj * (tj + 1) / 2;
  }
  const int i0 = active ? 2 * ti : 0, j0 = active ? 2 * tj : 0;
  V acc[2][2];
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 2; ++q) acc[p][q] = Rg::zero();
  const long long cstride = (long long)gridDim.x * MD_CH;
  // chunk k0 -> stage buffer st: thread t copies index k0 + t of every column
  auto issue = [&](long long k0, int st) {
    const long long k = k0 + t;
    const bool ok = k < n;
    for (int v = 0; v < nv; ++v) {
      const S* col = v < ma ? A + (size_t)v * n : B + (size_t)(v - ma) * n;
      cp_async8(sv + ((size_t)st * nv + v) * MD_CH + t, ok ? col + k : col, ok);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  long long k0 = (long long)blockIdx.x * MD_CH;
  int st = 0;
  if (k0 < n) issue(k0, 0);
  for (; k0 < n; k0 += cstride) {
    if (k0 + cstride < n) {
      issue(k0 + cstride, st ^ 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    if (active) {
      const V* base = sv + (size_t)st * nv * MD_CH;
      const V* a0 = base + i0 * MD_CH;
      const V* a1 = base + (i0 + 1 < ma ? i0 + 1 : i0) * MD_CH;
      const V* b0 = base + (ma + j0) * MD_CH;
      const V* b1 = base + (ma + (j0 + 1 < mb ? j0 + 1 : j0)) * MD_CH;
      for (int idx = sub; idx < MD_CH; idx += S_) {
        const V x0 = a0[idx], x1 = a1[idx], y0 = b0[idx], y1 = b1[idx];
        Rg::dacc(acc[0][0], x0, y0);
        Rg::dacc(acc[1][0], x1, y0);
        Rg::dacc(acc[0][1], x0, y1);
        Rg::dacc(acc[1][1], x1, y1);
      }
      // renormalise the double-float accumulators once per chunk, so that
      // their error terms never grow over more than one chunk's products
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) acc[p][q] = Rg::dfin(acc[p][q]);
    }
    __syncthreads();
    st ^= 1;
  }
  double* red = reinterpret_cast<double*>(md_smem);   // ntile * 4 * S_ <= 4 * MD_CH doubles
  if (active) {
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q)
        red[(tile * 4 + p + 2 * q) * S_ + sub] = Rg::to_d(Rg::dfin(acc[p][q]));
  }
  __syncthreads();
  const int np = ma * mb;
  double* part = partials + (size_t)blockIdx.x * (MAXB * MAXB);
  for (int e = t; e < np; e += MD_CH) {
    const int i = e % ma, j = e / ma;
    if (sym && i > j) continue;
    const int tl = sym ? (j / 2) * (j / 2 + 1) / 2 + i / 2 : (i / 2) + tr * (j / 2);
    const int qq = (i & 1) + 2 * (j & 1);
    double sum = 0.0;
    for (int u = 0; u < S_; ++u) sum += red[(tl * 4 + qq) * S_ + u];
    part[e] = sum;
  }
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the blocks' sums: with few entries several threads share one, each an
  // interleaved part of the blocks
  const int ng = np > 0 && np <= MD_CH / 2 ? MD_CH / np : 1;
  for (int e0 = 0; e0 < np; e0 += MD_CH) {
    const int e = ng > 1 ? t % np : e0 + t, gi = ng > 1 ? t / np : 0;
    const int i = e < np ? e % ma : 0, j = e < np ? e / ma : 0;
    const bool mine = e < np && gi < ng && !(sym && i > j);
    double sum = 0.0;
    if (mine) {
#pragma unroll 8
      for (int bl = gi; bl < (int)gridDim.x; bl += ng)
        sum += partials[(size_t)bl * (MAXB * MAXB) + e];
    }
    if (ng > 1) {
      __syncthreads();
      red[t] = sum;
      __syncthreads();
      if (gi == 0)
        for (int u = 1; u < ng; ++u) sum += red[u * np + e];
    }
    if (mine && gi == 0) {
      G[i + (size_t)ldg * j] = sum;
      if (sym) G[j + (size_t)ldg * i] = sum;
    }
  }
  if (t == 0) *counter = 0u;
}

// Column case: g[i] = sum_k A[k + i*n] b[k].  Warp w of a block
// accumulates column w % na over its own share of the indices, wpc = blockDim
// / (32 na) warps per column (more warps for few columns, so that a launch
// with one or two columns still keeps enough loads outstanding); one
// accumulator set per lane, four indices in flight.  Lanes, the warps of a
// column, and blocks are summed in a fixed order.
template <typename S>
__global__ void __launch_bounds__(32 * MAXB)
    k_gram_col(long long n, const S* __restrict__ A, int na, const int* na_dev,
               const S* __restrict__ b, double* g, double* partials, unsigned* counter) {
  using Rg = Ar<S>;
  using V = typename Rg::T;
  __shared__ double sh[32 * MAXB / 32];
  __shared__ bool s_last;
  const int ma = na_dev ? min(max(*na_dev, 0), na) : na;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int wpc = nw / na, ci = wi % na, sub = wi / na;
  V acc = Rg::zero(), acc2 = Rg::zero();
  if (ci < ma) {
    const S* col = A + (size_t)ci * n;
    const long long stride = (long long)gridDim.x * wpc * 32;
    long long k = ((long long)blockIdx.x * wpc + sub) * 32 + lane;
    V acc3 = Rg::zero(), acc4 = Rg::zero();
    for (; k + 3 * stride < n; k += 4 * stride) {
      const V a0 = Rg::ld(col, k), b0 = Rg::ld(b, k);
      const V a1 = Rg::ld(col, k + stride), b1 = Rg::ld(b, k + stride);
      const V a2 = Rg::ld(col, k + 2 * stride), b2 = Rg::ld(b, k + 2 * stride);
      const V a3 = Rg::ld(col, k + 3 * stride), b3 = Rg::ld(b, k + 3 * stride);
      Rg::dacc(acc, a0, b0);
      Rg::dacc(acc2, a1, b1);
      Rg::dacc(acc3, a2, b2);
      Rg::dacc(acc4, a3, b3);
    }
    for (; k < n; k += stride) Rg::dacc(acc, Rg::ld(col, k), Rg::ld(b, k));
    acc = Rg::add(Rg::add(Rg::dfin(acc), Rg::dfin(acc2)), Rg::add(Rg::dfin(acc3), Rg::dfin(acc4)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = Rg::add(acc, Rg::shfl_down(acc, o));
  }
  if (lane == 0) sh[wi] = ci < ma ? Rg::to_d(acc) : 0.0;
  __syncthreads();
  if ((int)threadIdx.x < MAXB) {
    double v = 0.0;
    if ((int)threadIdx.x < na)
      for (int u = 0; u < wpc; ++u) v += sh[u * na + threadIdx.x];
    partials[(size_t)blockIdx.x * MAXB + threadIdx.x] = v;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the blocks' sums, a warp per column (one thread per column took 608 loads
  // and additions in a row)
  for (int i = wi; i < ma; i += nw) {
    const double sum = warp_sum_strided(partials + i, (int)gridDim.x, MAXB);
    if (lane == 0) g[i] = sum;
  }
  if (threadIdx.x == 0) *counter = 0u;
}

// y = beta*y + sign*sum_i c[i] A[:, i] (i < m <= MMAX); optional
// |y - w|^2 -> *rr.  A, w (and y when SY = S) in storage S; y may be
// float64 when S is the pair format (one float64 add per stored value).
// The coefficients sit in shared memory; each thread keeps two indices in
// flight so that enough loads are outstanding to cover DRAM latency.
template <typename S, typename SY, int MMAX>
__global__ void __launch_bounds__(RED_THREADS, 4)
    k_combine(long long n, const S* __restrict__ A, int m, const int* m_dev,
              const double* __restrict__ c, double sign, double beta, SY* __restrict__ y,
              const S* __restrict__ w, double* rr, double* partials, unsigned* counter) {
  using Rg = Ar<S>;
  using V = typename Rg::T;
  __shared__ V scc[MMAX];
  const int mm = m_dev ? min(max(*m_dev, 0), m) : m;
  if (threadIdx.x < MMAX) {
    const double ci = (int)threadIdx.x < mm ? c[threadIdx.x] : 0.0;
    scc[threadIdx.x] = Rg::from_d(sign == 1.0 ? ci : sign == -1.0 ? -ci : sign * ci);
  }
  __syncthreads();
  const V bb = Rg::from_d(beta);
  auto start = [&](long long k) -> V {
    if (beta == 0.0) return Rg::zero();
    V yk;
    if constexpr (std::is_same<SY, S>::value) yk = Rg::ld(y, k);
    else yk = Rg::from_d((double)y[k]);
    return (beta == 1.0) ? yk : Rg::fma3(bb, yk, Rg::zero());
  };
  auto resid = [&](V s, long long k, V& acc) {
    V d = s;
    if (w) d = Rg::add(s, Rg::fma3(Rg::ld(w, k), Rg::from_d(-1.0), Rg::zero()));
    acc = Rg::fma3(d, d, acc);
  };
  V v = Rg::zero();
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; k + stride < n; k += 2 * stride) {
    const long long k1 = k + stride;
    V s0 = start(k), s1 = start(k1);
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < mm) {
        const V ci = scc[i];
        const S* col = A + (size_t)i * n;
        s0 = Rg::fma3(ci, Rg::ld(col, k), s0);
        s1 = Rg::fma3(ci, Rg::ld(col, k1), s1);
      }
    st_any(y, k, s0);
    st_any(y, k1, s1);
    if (rr) {
      resid(s0, k, v);
      resid(s1, k1, v);
    }
  }
  if (k < n) {
    V s0 = start(k);
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < mm) s0 = Rg::fma3(scc[i], Rg::ld(A + (size_t)i * n, k), s0);
    st_any(y, k, s0);
    if (rr) resid(s0, k, v);
  }
  if (!rr) return;
  reduce_to<S>(v, rr, partials, counter);
}

// One classical Gram-Schmidt pass fused with the next pass's projections:
// y <- y - sum_{i<m} c[i] A[:, i], then h[i] = A[:, i] . y for the new y
// (m = *m_dev when given).  The columns are read once for both; the dots
// are double-float, summed per block and then over blocks in order.
template <typename S, int MMAX>
__global__ void __launch_bounds__(RED_THREADS, 2)
    k_combine_dots(long long n, const S* __restrict__ A, int m, const int* m_dev,
                   const double* __restrict__ c, S* __restrict__ y, double* h,
                   double* partials, unsigned* counter) {
  using Rg = Ar<S>;
  using V = typename Rg::T;
  __shared__ double sh[MMAX][RED_THREADS / 32], tot[MMAX];
  __shared__ V scc[MMAX];
  pdl_wait();
  const int mm = m_dev ? min(max(*m_dev, 0), m) : m;
  if (threadIdx.x < MMAX)
    scc[threadIdx.x] = Rg::from_d((int)threadIdx.x < mm ? -c[threadIdx.x] : 0.0);
  __syncthreads();
  V hacc[MMAX];
#pragma unroll
  for (int i = 0; i < MMAX; ++i) hacc[i] = Rg::zero();
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    V a[MMAX];
    V sv = Rg::ld(y, k);
#pragma unroll
    for (int i = 0; i < MMAX; ++i) a[i] = i < mm ? Rg::ld(A + (size_t)i * n, k) : Rg::zero();
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < mm) sv = Rg::fma3(scc[i], a[i], sv);
    Rg::st(y, k, sv);
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < mm) Rg::dacc(hacc[i], a[i], sv);
  }
#pragma unroll
  for (int i = 0; i < MMAX; ++i) hacc[i] = Rg::dfin(hacc[i]);
  pdl_launch_dependents();
  if (grid_sum_v<S>(hacc, sh, tot, partials, counter) && (int)threadIdx.x < mm)
    h[threadIdx.x] = tot[threadIdx.x];
}

// Gram-Schmidt acceptance: if |r_src|^2 after orthogonalisation exceeds
// tol^2 times its value before, R[:, k] = r_src / |r_src| with k the
// current count (the count itself is advanced by k_gs_count afterwards)
template <typename S>
__global__ void __launch_bounds__(256)
    k_gs_accept(long long n, S* R, int src, const double* scal, int n0, int n1, double tol,
                const int* ints) {
  using Rg = Ar<S>;
  __shared__ double s_scale;
  const double before = scal[n0], after = scal[n1];
  const bool keep = after > tol * tol * before && after > 0.0;
  if (!keep) return;
  const int k = ints[I_KCOUNT];
  if (threadIdx.x == 0) s_scale = 1.0 / sqrt(after);   // once per block
  __syncthreads();
  const typename Rg::T sc = Rg::from_d(s_scale);
  const S* a = R + (size_t)src * n;
  S* b = R + (size_t)k * n;
  GRID_LOOP(i, n) Rg::st(b, i, Rg::fma3(Rg::ld(a, i), sc, Rg::zero()));
}

// Records column src of the QR factor of the basis, Rt[:, src] (ld MAXB):
// its projections h1 + h2 on the k columns accepted before it and, when it
// is accepted, its remaining norm at row k; then advances the count.  Also
// stores the column's norm before orthogonalisation in rn[src].
__global__ void k_gs_record(const double* scal, int n0, int n1, double tol, int src,
                            const double* h1, const double* h2, double* Rt, double* rn,
                            int* ints) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double before = scal[n0], after = scal[n1];
  const bool keep = after > tol * tol * before && after > 0.0;
  const int k = ints[I_KCOUNT];
  double* col = Rt + (size_t)MAXB * src;
  for (int j = 0; j < MAXB; ++j) col[j] = j < k ? h1[j] + h2[j] : 0.0;
  if (keep) col[k] = sqrt(after);
  rn[src] = sqrt(fmax(before, 0.0));
  if (keep) ints[I_KCOUNT] = k + 1;
}

// ---------------------------------------------------------------------------
// CG recursion of the mixed path: x, r, p in the pair format; the operator
// works on the float32 shadow p32 -> q32 and the V-cycle returns z32.
// alpha and beta are formed once per block from the float64 scalars.
// ---------------------------------------------------------------------------
// Grids cover short vectors once (a reduction's last block bounds those: at
// 27 k DOFs 608 blocks took 7.5 us a dot product and 9.6 us an update), with
// at most RED_BLOCKS blocks.  In the two updates a thread takes two
// neighbouring indices per 16- or 8-byte load (the vectors are the workspace's
// own, 256-byte aligned; a last odd index goes to one thread): at n = 5.4 M
// 45.8 and 17.0 us instead of 46.5 and 19.0, which is the copy bandwidth.
constexpr int VEC_T = 256, VEC_W = VEC_T / 32;

struct Pair2 {
  dfl v[2];
};
__device__ __forceinline__ Pair2 ld_pair2(const float2* p, long long q) {
  const float4 t = reinterpret_cast<const float4*>(p)[q];
  return {{{t.x, t.y}, {t.z, t.w}}};
}
__device__ __forceinline__ void st_pair2(float2* p, long long q, const Pair2& a) {
  reinterpret_cast<float4*>(p)[q] = make_float4(a.v[0].h, a.v[0].l, a.v[1].h, a.v[1].l);
}
__device__ __forceinline__ float2 ld_two(const float* p, long long q) {
  return reinterpret_cast<const float2*>(p)[q];
}

// body(q) for the pairs of indices (2 q, 2 q + 1) below n of this thread, U at
// a time (load(q, u) first for all of them, then use(q, u)); odd(k) for a last
// odd index.
template <int U, typename Load, typename Use, typename Odd>
__device__ __forceinline__ void pair_loop2(long long n, Load load, Use use, Odd odd) {
  const long long m = n >> 1, stride = (long long)gridDim.x * VEC_T;
  long long q = (long long)blockIdx.x * VEC_T + threadIdx.x;
  if (q == 0 && (n & 1)) odd(n - 1);
  for (; q + (U - 1) * stride < m; q += U * stride) {
#pragma unroll
    for (int u = 0; u < U; ++u) load(q + u * stride, u);
#pragma unroll
    for (int u = 0; u < U; ++u) use(q + u * stride, u);
  }
  for (; q < m; q += stride) {
    load(q, 0);
    use(q, 0);
  }
}

// out = sum_k a[k] b[k], a pairs, b float32.  Twelve bytes per index, one index
// per load and eight in flight: two indices per load measured 19 us instead of
// 17 at n = 5.4 M.
constexpr int DOT_U = 8;
__global__ void __launch_bounds__(VEC_T)
    k_dot_d2f(long long n, const float2* __restrict__ a, const float* __restrict__ b,
              double* partials, unsigned* counter, double* out) {
  __shared__ double sh[1][VEC_W], tot[1];
  pdl_wait();
  dfl v[2] = {{0.f, 0.f}, {0.f, 0.f}};
  const long long stride = (long long)gridDim.x * VEC_T;
  long long k = (long long)blockIdx.x * VEC_T + threadIdx.x;
  for (; k + (DOT_U - 1) * stride < n; k += DOT_U * stride) {
    dfl av[DOT_U];
    float bv[DOT_U];
#pragma unroll
    for (int u = 0; u < DOT_U; ++u) {
      av[u] = ld_df(a, k + u * stride);
      bv[u] = b[k + u * stride];
    }
#pragma unroll
    for (int u = 0; u < DOT_U; ++u) df_dot_acc(v[u & 1], av[u], dfl{bv[u], 0.f});
  }
  for (; k < n; k += stride) df_dot_acc(v[0], ld_df(a, k), dfl{b[k], 0.f});
  pdl_launch_dependents();
  const dfl w[1] = {df_add(df_norm(v[0]), df_norm(v[1]))};
  if (grid_sum_df(w, sh, tot, partials, counter) && threadIdx.x == 0) *out = tot[0];
}

// The CG update of kernels_blas.cu (k_cg_xr) on pairs.  It also starts the
// next V-cycle: b = r rounded to float32 and zpre = omega dinv b (its
// pre-smoothing from a zero guess), the values the V-cycle's first kernel
// would compute.
constexpr int CG_U = 2;
__global__ void __launch_bounds__(VEC_T)
    k_cg_xr_d2(long long n, float2* __restrict__ x, float2* __restrict__ r,
               const float2* __restrict__ p, const float* __restrict__ q, double* scal,
               double* partials, unsigned* counter, float* __restrict__ b,
               float* __restrict__ zpre, const float* __restrict__ dinv, float omega,
               double* host_rr) {
  using Rg = Ar<float2>;
  __shared__ double sh[1][VEC_W], tot[1];
  __shared__ dfl s_alpha;
  pdl_wait();
  if (threadIdx.x == 0) s_alpha = split_d(scal[S_RZ1] / scal[S_PQ]);
  __syncthreads();
  const dfl al = s_alpha, mal = {-al.h, -al.l};
  dfl v[2] = {{0.f, 0.f}, {0.f, 0.f}};
  // one index: updates xk and rk, returns b
  auto step = [&](dfl& xk, dfl& rk, dfl pk, float qk, dfl& acc) {
    xk = df_fma(al, pk, xk);
    rk = df_add(Rg::mulf(mal, qk), rk);
    df_dot_acc(acc, rk, rk);
    return __fadd_rn(rk.h, rk.l);
  };
  Pair2 xv[CG_U], rv[CG_U], pv[CG_U];
  float2 qv[CG_U], dv[CG_U];
  pair_loop2<CG_U>(
      n,
      [&](long long k, int u) {
        xv[u] = ld_pair2(x, k);
        rv[u] = ld_pair2(r, k);
        pv[u] = ld_pair2(p, k);
        qv[u] = ld_two(q, k);
        dv[u] = ld_two(dinv, k);
      },
      [&](long long k, int u) {
        const float b0 = step(xv[u].v[0], rv[u].v[0], pv[u].v[0], qv[u].x, v[0]);
        const float b1 = step(xv[u].v[1], rv[u].v[1], pv[u].v[1], qv[u].y, v[1]);
        st_pair2(x, k, xv[u]);
        st_pair2(r, k, rv[u]);
        reinterpret_cast<float2*>(b)[k] = make_float2(b0, b1);
        reinterpret_cast<float2*>(zpre)[k] =
            make_float2(omega * dv[u].x * b0, omega * dv[u].y * b1);
      },
      [&](long long k) {
        dfl xk = ld_df(x, k), rk = ld_df(r, k);
        const float bk = step(xk, rk, ld_df(p, k), q[k], v[0]);
        st_df(x, k, xk);
        st_df(r, k, rk);
        b[k] = bk;
        zpre[k] = omega * dinv[k] * bk;
      });
  pdl_launch_dependents();
  const dfl w[1] = {df_add(df_norm(v[0]), df_norm(v[1]))};
  if (grid_sum_df(w, sh, tot, partials, counter) && threadIdx.x == 0)
    cg_publish(scal, tot[0], host_rr);
}

// p = z + beta p (beta = scal[num]/scal[den], or p = z when num < 0);
// p32 = p rounded to float32
constexpr int CGP_U = 4;
__global__ void __launch_bounds__(VEC_T)
    k_cg_p_d2(long long n, float2* __restrict__ p, float* __restrict__ p32,
              const float* __restrict__ z, const double* __restrict__ scal, int num, int den) {
  __shared__ dfl s_beta;
  pdl_wait();
  const bool restart = num < 0;
  if (threadIdx.x == 0) s_beta = split_d(restart ? 0.0 : scal[num] / scal[den]);
  __syncthreads();
  const dfl be = s_beta;
  auto step = [&](float zv, dfl pold) {
    const dfl zk = {zv, 0.f};
    return restart ? zk : df_add(df_mul(be, pold), zk);
  };
  Pair2 pv[CGP_U];
  float2 zv[CGP_U];
  pair_loop2<CGP_U>(
      n,
      [&](long long k, int u) {
        if (!restart) pv[u] = ld_pair2(p, k);
        zv[u] = ld_two(z, k);
      },
      [&](long long k, int u) {
        const Pair2 o = {{step(zv[u].x, pv[u].v[0]), step(zv[u].y, pv[u].v[1])}};
        st_pair2(p, k, o);
        reinterpret_cast<float2*>(p32)[k] =
            make_float2(__fadd_rn(o.v[0].h, o.v[0].l), __fadd_rn(o.v[1].h, o.v[1].l));
      },
      [&](long long k) {
        const dfl o = step(z[k], restart ? dfl{0.f, 0.f} : ld_df(p, k));
        st_df(p, k, o);
        p32[k] = __fadd_rn(o.h, o.l);
      });
  pdl_launch_dependents();
}

#undef GRID_LOOP

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
static inline int vgrid(long long n) {
  long long b = (n + 255) / 256;
  if (b > RED_BLOCKS) b = RED_BLOCKS;
  return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_vdot(long long n, int vt, const void* a, const void* b, double* partials,
                        unsigned* counter, double* out, cudaStream_t s) {
  if (vt == V_DF2)
    k_vdot<float2><<<vgrid(n), RED_THREADS, 0, s>>>(n, (const float2*)a, (const float2*)b,
                                                      partials, counter, out);
  else
    k_vdot<double><<<vgrid(n), RED_THREADS, 0, s>>>(n, (const double*)a, (const double*)b,
                                                      partials, counter, out);
  return cudaGetLastError();
}

cudaError_t launch_vconvert(long long n, int tin, const void* in, int tout, void* out,
                            cudaStream_t s) {
  if (tin == tout) {
    if (in == out) return cudaSuccess;
    if (tin == V_DF2)
      k_vcopy<float2><<<vgrid(n), 256, 0, s>>>(n, (const float2*)in, (float2*)out);
    else
      k_vcopy<double><<<vgrid(n), 256, 0, s>>>(n, (const double*)in, (double*)out);
  } else if (tin == V_F64) {
    k_split<<<vgrid(n), 256, 0, s>>>(n, (const double*)in, (float2*)out);
  } else {
    k_join<<<vgrid(n), 256, 0, s>>>(n, (const float2*)in, (double*)out);
  }
  return cudaGetLastError();
}

// x[dim node + c] = 0 where DOF c of the node is fixed; one thread per node
template <typename S>
__global__ void __launch_bounds__(256)
    k_zero_fixed(long long nn, int dim, const uint8_t* __restrict__ mask, S* __restrict__ x) {
  const long long node = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (node >= nn) return;
  const unsigned m = mask[node];
  if (!m) return;
  for (int c = 0; c < dim; ++c)
    if ((m >> c) & 1u) x[dim * node + c] = S{};
}

cudaError_t launch_zero_fixed(long long nn, int dim, const uint8_t* mask, int vt, void* x,
                              cudaStream_t s) {
  if (nn <= 0) return cudaSuccess;
  if (vt == V_DF2)
    k_zero_fixed<float2><<<nblocks(nn, 256), 256, 0, s>>>(nn, dim, mask, (float2*)x);
  else
    k_zero_fixed<double><<<nblocks(nn, 256), 256, 0, s>>>(nn, dim, mask, (double*)x);
  return cudaGetLastError();
}

cudaError_t launch_vscale_inv_sqrt(long long n, int vt, void* a, const double* s2,
                                   cudaStream_t s) {
  if (vt == V_DF2)
    k_vscale_inv_sqrt<float2><<<vgrid(n), 256, 0, s>>>(n, (float2*)a, s2);
  else
    k_vscale_inv_sqrt<double><<<vgrid(n), 256, 0, s>>>(n, (double*)a, s2);
  return cudaGetLastError();
}

template <typename S>
static void gram_t(long long n, const void* A, int na, const int* na_dev, const void* B, int nb,
                   const int* nb_dev, double* G, int ldg, double* partials, unsigned* counter,
                   cudaStream_t s, bool sym = false) {
  // up to 2 stages x 2*MAXB columns x MD_CH values; set once, before any
  // launch of any host thread
  static std::once_flag smem_once;
  std::call_once(smem_once, [] {
    cudaFuncSetAttribute(k_gram<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(2 * 2 * MAXB * MD_CH * sizeof(S)));
  });
  if (nb == 1 && nb_dev == nullptr && !sym) {
    const int wpc = na >= 8 ? 1 : 8 / na;   // warps per column
    // (four to eight indices a lane at least)
    const int gb = (int)std::min<long long>((n + 256LL * wpc - 1) / (256LL * wpc), RED_BLOCKS);
    k_gram_col<S><<<gb, 32 * na * wpc, 0, s>>>(n, (const S*)A, na, na_dev,
                                                       (const S*)B, G, partials, counter);
  } else
    k_gram<S><<<(int)std::min<long long>((n + 2 * MD_CH - 1) / (2 * MD_CH), RED_BLOCKS), MD_CH,
                (size_t)2 * (na + nb) * MD_CH * sizeof(S), s>>>(
        n, (const S*)A, na, na_dev, (const S*)B, nb, nb_dev, G, ldg, partials, counter, sym);
}

cudaError_t launch_gram_sym(long long n, int vt, const void* A, const void* B, int m, double* G,
                            int ldg, double* partials, unsigned* counter, cudaStream_t s) {
  if (m > MAXB || m < 1) return cudaErrorInvalidValue;
  if (vt == V_DF2)
    gram_t<float2>(n, A, m, nullptr, B, m, nullptr, G, ldg, partials, counter, s, true);
  else
    gram_t<double>(n, A, m, nullptr, B, m, nullptr, G, ldg, partials, counter, s, true);
  return cudaGetLastError();
}

cudaError_t launch_gram(long long n, int vt, const void* A, int na, const int* na_dev,
                        const void* B, int nb, const int* nb_dev, double* G, int ldg,
                        double* partials, unsigned* counter, cudaStream_t s) {
  if (na > MAXB || nb > MAXB || na < 1 || nb < 1) return cudaErrorInvalidValue;
  if (vt == V_DF2)
    gram_t<float2>(n, A, na, na_dev, B, nb, nb_dev, G, ldg, partials, counter, s);
  else
    gram_t<double>(n, A, na, na_dev, B, nb, nb_dev, G, ldg, partials, counter, s);
  return cudaGetLastError();
}

template <typename S, typename SY>
static void combine_t(long long n, const void* A, int m, const int* m_dev, const double* c,
                      double sign, double beta, void* y, const void* w, double* rr,
                      double* partials, unsigned* counter, cudaStream_t s) {
  const S* a = (const S*)A;
  const S* ww = (const S*)w;
  SY* yy = (SY*)y;
  if (m <= 4)
    k_combine<S, SY, 4><<<vgrid(n), RED_THREADS, 0, s>>>(n, a, m, m_dev, c, sign, beta, yy, ww,
                                                           rr, partials, counter);
  else if (m <= 8)
    k_combine<S, SY, 8><<<vgrid(n), RED_THREADS, 0, s>>>(n, a, m, m_dev, c, sign, beta, yy, ww,
                                                           rr, partials, counter);
  else if (m <= 12)
    k_combine<S, SY, 12><<<vgrid(n), RED_THREADS, 0, s>>>(n, a, m, m_dev, c, sign, beta, yy,
                                                            ww, rr, partials, counter);
  else
    k_combine<S, SY, MAXB><<<vgrid(n), RED_THREADS, 0, s>>>(n, a, m, m_dev, c, sign, beta, yy,
                                                              ww, rr, partials, counter);
}

template <typename S>
static cudaError_t combine_dots_t(long long n, const void* A, int m, const int* m_dev,
                                  const double* c, void* y, double* h, double* partials,
                                  unsigned* counter, cudaStream_t s) {
  auto kern = m <= 4 ? k_combine_dots<S, 4> : m <= 12 ? k_combine_dots<S, 12> : k_combine_dots<S, MAXB>;
  return launch_pdl(kern, dim3(vgrid(n)), dim3(RED_THREADS), 0, s, n, (const S*)A, m, m_dev, c, (S*)y,
                    h, partials, counter);
}

cudaError_t launch_combine_dots(long long n, int vt, const void* A, int m, const int* m_dev,
                                const double* c, void* y, double* h, double* partials,
                                unsigned* counter, cudaStream_t s) {
  if (m > MAXB || m < 0) return cudaErrorInvalidValue;
  return vt == V_DF2 ? combine_dots_t<float2>(n, A, m, m_dev, c, y, h, partials, counter, s)
                     : combine_dots_t<double>(n, A, m, m_dev, c, y, h, partials, counter, s);
}

cudaError_t launch_combine(long long n, int vt, const void* A, int m, const int* m_dev,
                           const double* c, double sign, double beta, void* y, int yt,
                           const void* w, double* rr, double* partials, unsigned* counter,
                           cudaStream_t s) {
  if (m > MAXB || m < 0) return cudaErrorInvalidValue;
  if (vt == V_DF2 && yt == V_DF2)
    combine_t<float2, float2>(n, A, m, m_dev, c, sign, beta, y, w, rr, partials, counter, s);
  else if (vt == V_DF2 && yt == V_F64)
    combine_t<float2, double>(n, A, m, m_dev, c, sign, beta, y, w, rr, partials, counter, s);
  else if (vt == V_F64 && yt == V_F64)
    combine_t<double, double>(n, A, m, m_dev, c, sign, beta, y, w, rr, partials, counter, s);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_gs_accept(long long n, int vt, void* R, int src, const double* scal, int n0,
                             int n1, double tol, const double* h1, const double* h2, double* Rt,
                             double* rn, int* ints, cudaStream_t s) {
  if (src < 0 || src >= MAXB) return cudaErrorInvalidValue;
  if (vt == V_DF2)
    k_gs_accept<float2><<<vgrid(n), 256, 0, s>>>(n, (float2*)R, src, scal, n0, n1, tol, ints);
  else
    k_gs_accept<double><<<vgrid(n), 256, 0, s>>>(n, (double*)R, src, scal, n0, n1, tol, ints);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_gs_record<<<1, 32, 0, s>>>(scal, n0, n1, tol, src, h1, h2, Rt, rn, ints);
  return cudaGetLastError();
}

// Y[:, j] = sum_{i < kq} U[i + MAXB j] Q[:, i] for j < k: the kept left
// singular directions of the basis expressed in its orthonormal QR factor.
// Each thread loads the kq entries of one index once and forms all k
// outputs; U sits in shared memory.
template <typename S, int KQ>
__global__ void __launch_bounds__(256)
    k_combine_multi(long long n, const S* __restrict__ Q, int kq, const double* __restrict__ U,
                    int k, S* __restrict__ Y) {
  using Rg = Ar<S>;
  using V = typename Rg::T;
  __shared__ V su[KQ * MAXB];
  for (int e = threadIdx.x; e < KQ * MAXB; e += blockDim.x) {
    const int i = e % KQ, j = e / KQ;
    su[e] = Rg::from_d(i < kq && j < k ? U[i + (size_t)MAXB * j] : 0.0);
  }
  __syncthreads();
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    V q[KQ];
#pragma unroll
    for (int i = 0; i < KQ; ++i) q[i] = i < kq ? Rg::ld(Q + (size_t)i * n, idx) : Rg::zero();
    for (int j = 0; j < k; ++j) {
      V acc = Rg::zero();
#pragma unroll
      for (int i = 0; i < KQ; ++i)
        if (i < kq) acc = Rg::fma3(su[i + KQ * j], q[i], acc);
      Rg::st(Y + (size_t)j * n, idx, acc);
    }
  }
}

template <typename S>
static void combine_multi_t(long long n, const void* Q, int kq, const double* U, int k, void* Y,
                            cudaStream_t s) {
  const int g = vgrid(n);
  if (kq <= 4)
    k_combine_multi<S, 4><<<g, 256, 0, s>>>(n, (const S*)Q, kq, U, k, (S*)Y);
  else if (kq <= 8)
    k_combine_multi<S, 8><<<g, 256, 0, s>>>(n, (const S*)Q, kq, U, k, (S*)Y);
  else if (kq <= 12)
    k_combine_multi<S, 12><<<g, 256, 0, s>>>(n, (const S*)Q, kq, U, k, (S*)Y);
  else
    k_combine_multi<S, MAXB><<<g, 256, 0, s>>>(n, (const S*)Q, kq, U, k, (S*)Y);
}

cudaError_t launch_combine_multi(long long n, int vt, const void* Q, int kq, const double* U,
                                 int k, void* Y, cudaStream_t s) {
  if (kq < 1 || kq > MAXB || k < 0 || k > kq || Q == Y) return cudaErrorInvalidValue;
  if (k == 0) return cudaSuccess;
  if (vt == V_DF2)
    combine_multi_t<float2>(n, Q, kq, U, k, Y, s);
  else
    combine_multi_t<double>(n, Q, kq, U, k, Y, s);
  return cudaGetLastError();
}

static dim3 pair2_grid(long long n, int per_thread) {
  const long long b = (n + 2LL * per_thread * VEC_T - 1) / (2LL * per_thread * VEC_T);
  return dim3((unsigned)std::min<long long>(std::max<long long>(b, 1), RED_BLOCKS));
}

cudaError_t launch_dot_d2f(long long n, const void* a, const float* b, double* partials,
                           unsigned* counter, double* out, cudaStream_t s) {
  return launch_pdl(k_dot_d2f, pair2_grid(n, 1), dim3(VEC_T), 0, s, n, (const float2*)a, b, partials,
                    counter, out);
}

cudaError_t launch_cg_xr_d2(long long n, void* x, void* r, const void* p, const float* q,
                            double* scal, double* partials, unsigned* counter, float* b,
                            float* zpre, const float* dinv, double omega, cudaStream_t s,
                            double* host_rr) {
  return launch_pdl(k_cg_xr_d2, pair2_grid(n, 1), dim3(VEC_T), 0, s, n, (float2*)x, (float2*)r,
                    (const float2*)p, q, scal, partials, counter, b, zpre, dinv,
                    (float)omega, host_rr);
}

cudaError_t launch_cg_p_d2(long long n, void* p, float* p32, const float* z, const double* scal,
                           int num, int den, cudaStream_t s) {
  return launch_pdl(k_cg_p_d2, pair2_grid(n, 1), dim3(VEC_T), 0, s, n, (float2*)p, p32, z, scal, num,
                    den);
}

}  // namespace topo
