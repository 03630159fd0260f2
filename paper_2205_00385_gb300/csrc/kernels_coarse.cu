// Explicit inverse of the coarsest grid's matrix (Algorithm 2's exact
// coarsest solve): A = L L^T, X = L^{-1}, A^{-1} = X^T X.
//
// GB300 runs one float64 FMA per clock per SM, so the ~n^3/2 operations must
// be spread over the whole chip: one block takes 3.8 ms at n = 336.  Here
// every NB-column step of a right-looking elimination of [A | I] is two
// launches over all SMs.  Block row i > k of the working matrix W (in place
// of A) holds, left of column block k, the rows of X in progress and, right
// of it, the remaining Schur complement:
//   panel k:  P_i = A_ik X_kk^T (= L_ik, kept beside W),  X_kj = X_kk B_kj
//   update k: A_ij -= P_i P_j^T (j > k),  B_ij -= P_i X_kj (j <= k),
//             and the first block factors the next diagonal block and inverts
//             the factor (X_kk), while the others update the rest.
// The chain of diagonal blocks bounds it (one warp, reciprocal square roots
// and rank-1 updates in registers), so NB is 16 in float64, where a 32-wide
// block costs four times the FMAs on one SM, and 32 in float32, where the
// launches cost more than the chain.  Launches overlap by programmatic
// stream serialization.  Whole inverse, one block before / now: float64
// n = 186 1.23 / 0.31 ms and n = 336 3.83 / 0.49 ms; float32 n = 336 0.71 /
// 0.21 ms.
#include "kernels.h"

namespace topo {
namespace {

constexpr int CT = 16;   // output tile and thread block side (CT x CT threads)

template <typename T>
struct CoarseNB {
  static constexpr int NB = sizeof(T) == 8 ? 16 : 32;
};

__device__ __forceinline__ float inv_sqrt(float d) { return 1.0f / sqrtf(d); }

// Newton's iteration y <- y + y (1 - m y^2) / 2 for m^{-1/2} from a float32
// starting value (22 -> 44 -> over 53 bits), m = d scaled by an even power
// of two into [1, 4); subnormal and non-finite d take the library functions.
__device__ __forceinline__ double inv_sqrt(double d) {
  const int hi = __double2hiint(d), ex = ((hi >> 20) & 0x7FF) - 1023;
  if (ex == -1023 || ex == 1024) return 1.0 / sqrt(d);
  const int e2 = ex & ~1;
  const double m = __hiloint2double(hi - (e2 << 20), __double2loint(d));
  double y = (double)rsqrtf((float)m);
#pragma unroll
  for (int it = 0; it < 2; ++it) y = fma(0.5 * y, fma(-m * y, y, 1.0), y);
  return __hiloint2double(__double2hiint(y) - ((e2 >> 1) << 20), __double2loint(y));
}

// Cholesky factor of the NB x NB block D and its inverse X (zero above the
// diagonal), by one warp: lane r holds row r of D, then column r of X.
// Returns false when a pivot is not positive (the pivot is then taken as 1).
template <typename T, int NB>
__device__ __forceinline__ bool factor_invert(T (&D)[NB][NB + 1], T (&X)[NB][NB + 1]) {
  const int lane = threadIdx.x & 31, r = lane < NB ? lane : NB - 1;
  T a[NB], rs[NB];
  bool ok = true;
#pragma unroll
  for (int c = 0; c < NB; ++c) a[c] = D[r][c];
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    T d = __shfl_sync(0xffffffffu, a[j], j);
    if (!(d > T(0))) {
      ok = false;
      d = T(1);
    }
    rs[j] = inv_sqrt(d);
    a[j] = r == j ? d * rs[j] : a[j] * rs[j];
#pragma unroll
    for (int c = j + 1; c < NB; ++c) a[c] -= a[j] * __shfl_sync(0xffffffffu, a[j], c);
  }
#pragma unroll
  for (int c = 0; c < NB; ++c)
    if (lane < NB) D[r][c] = a[c];
  __syncwarp();
  T x[NB];
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    T s = i == r ? T(1) : T(0);
#pragma unroll
    for (int m = 0; m < i; ++m) s -= D[i][m] * x[m];
    x[i] = s * rs[i];
    if (lane < NB) X[i][r] = i >= r ? x[i] : T(0);
  }
  return ok;
}

// Running sum of products.  In float32 it is compensated (products exact,
// the additions' errors in a second word), so that an entry is rounded once per
// panel: subtracting NB products one by one rounds it NB times, which a long
// elimination adds up.  Error of the inverse in a two-level V-cycle, rms of 12
// densities, one by one / compensated (LAPACK's float32 inverse): n = 336 1.8e-5 /
// 5.4e-6 (4.8e-6), n = 480 3.7e-5 / 6.9e-6 (6.5e-6); n = 1188, products summed first /
// compensated 1.6e-5 / 1.5e-5 (1.7e-5).  Whole inverse 0.19 -> 0.21 ms at n = 336.
template <typename T>
struct Sum {
  T v = T(0);
  __device__ __forceinline__ void add(T a, T b) { v += a * b; }
  __device__ __forceinline__ T get() const { return v; }
};
template <>
struct Sum<float> {
  float v = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b), t = __fadd_rn(v, p), w = __fsub_rn(t, v);
    const float e = __fadd_rn(__fsub_rn(v, __fsub_rn(t, w)), __fsub_rn(p, w));
    lo = __fadd_rn(lo, __fadd_rn(e, __fmaf_rn(a, b, -p)));
    v = t;
  }
  __device__ __forceinline__ float get() const { return v + lo; }
};

// v - sum a_q b_q
template <int NB, typename T>
__device__ __forceinline__ T take_products(T v, const T* a, const T* b) {
  Sum<T> s;
  s.v = v;
#pragma unroll
  for (int q = 0; q < NB; ++q) s.add(-a[q], b[q]);
  return s.get();
}

// Update with panel k (rows k0 .. k0 + NB), or, with k0 < 0, only the
// factorisation of the first diagonal block.  Block 0 owns the next diagonal
// block: it updates, factors and inverts it into Dx (NB x NB).  Block b > 0
// owns one CT x CT tile of the rows below panel k.
template <typename T, int NB>
__global__ void __launch_bounds__(CT * CT)
    k_coarse_update(int n, int k0, T* __restrict__ W, const T* __restrict__ P,
                    T* __restrict__ Dx, int* status) {
  pdl_wait();
  const int tx = threadIdx.x % CT, ty = threadIdx.x / CT;
  const int k1 = k0 < 0 ? 0 : k0 + NB;   // first row of the next block
  if (blockIdx.x == 0) {
    __shared__ T D[NB][NB + 1], X[NB][NB + 1], Ps[NB][NB + 1];
    if (k0 >= 0)
      for (int q = threadIdx.x; q < NB * NB; q += CT * CT) {
        const int i = q / NB, c = q % NB;
        Ps[i][c] = k1 + i < n ? P[(size_t)(k1 + i) * NB + c] : T(0);
      }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < NB; a += CT)
#pragma unroll
      for (int b = 0; b <= a; b += CT) {
        const int i = a + ty, j = b + tx;
        // identity beyond n, so that the padding factors to itself
        T v = k1 + i < n && k1 + j < n ? W[(size_t)(k1 + i) * n + k1 + j] : T(i == j);
        if (k0 >= 0) v = take_products<NB>(v, Ps[i], Ps[j]);
        D[i][j] = v;
        if (a != b) D[j][i] = v;
      }
    __syncthreads();
    if (threadIdx.x < 32 && !factor_invert<T, NB>(D, X) && threadIdx.x == 0)
      *status = TO_E_SINGULAR;
    __syncthreads();
    for (int q = threadIdx.x; q < NB * NB; q += CT * CT) Dx[q] = X[q / NB][q % NB];
  } else {
    // tile (rt, ct): rows k1 + CT rt .., columns CT ct .. up to the diagonal
    const int kt = k1 / CT;
    int rt = 0, t = (int)blockIdx.x - 1;
    // row rt has kt + rt + 1 tiles: invert the triangular count
    {
      const float h = kt + 0.5f;
      rt = max((int)(sqrtf(h * h + 2.0f * t) - h), 0);
      while ((long long)rt * kt + (long long)rt * (rt + 1) / 2 > t) --rt;
      while ((long long)(rt + 1) * kt + (long long)(rt + 1) * (rt + 2) / 2 <= t) ++rt;
    }
    const int ct = t - (rt * kt + rt * (rt + 1) / 2);
    const int i0 = k1 + CT * rt, j0 = CT * ct;
    if (!(rt < NB / CT && j0 >= k1)) {   // (the next diagonal block is block 0's)
      __shared__ T a[CT][NB + 1], b[CT][NB + 1];
      const bool schur = j0 >= k1;
      for (int q = threadIdx.x; q < CT * NB; q += CT * CT) {
        const int i = q / NB, c = q % NB;
        a[i][c] = i0 + i < n ? P[(size_t)(i0 + i) * NB + c] : T(0);
        if (schur) b[i][c] = j0 + i < n ? P[(size_t)(j0 + i) * NB + c] : T(0);
      }
      if (!schur)
        for (int q = threadIdx.x; q < CT * NB; q += CT * CT) {
          const int c = q / CT, j = q % CT;
          b[j][c] = W[(size_t)(k0 + c) * n + j0 + j];
        }
      __syncthreads();
      const int i = i0 + ty, j = j0 + tx;
      if (i < n && j < n) {
        // column block k of X starts here: what W holds there is A_ik
        const T v = schur || j0 < k0 ? W[(size_t)i * n + j] : T(0);
        W[(size_t)i * n + j] = take_products<NB>(v, a[ty], b[tx]);
      }
    }
  }
  pdl_launch_dependents();
}

// Panel k: blocks 0 .. nr - 1 form P_i = A_ik X_kk^T for CT rows below the
// block each; the others multiply CT columns of block row k by X_kk in place
// (the last of them writes X_kk itself).
template <typename T, int NB>
__global__ void __launch_bounds__(CT * CT)
    k_coarse_panel(int n, int k0, int nr, T* __restrict__ W, T* __restrict__ P,
                   const T* __restrict__ Dx) {
  __shared__ T X[NB][NB + 1], s[NB][NB + 1];
  pdl_wait();
  const int tx = threadIdx.x % CT, ty = threadIdx.x / CT, b = blockIdx.x;
  for (int q = threadIdx.x; q < NB * NB; q += CT * CT) X[q / NB][q % NB] = Dx[q];
  if (b < nr) {
    const int i0 = k0 + NB + CT * b;
    for (int q = threadIdx.x; q < CT * NB; q += CT * CT) {
      const int i = q / NB, c = q % NB;
      s[i][c] = i0 + i < n ? W[(size_t)(i0 + i) * n + k0 + c] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int cb = 0; cb < NB; cb += CT) {
      const int c = cb + tx;
      Sum<T> v;
#pragma unroll
      for (int q = 0; q < cb + CT; ++q) v.add(s[ty][q], X[c][q]);
      if (i0 + ty < n) P[(size_t)(i0 + ty) * NB + c] = v.get();
    }
  } else {
    const int j0 = CT * (b - nr);
    if (j0 < k0) {
      for (int q = threadIdx.x; q < CT * NB; q += CT * CT) {
        const int c = q / CT, j = q % CT;
        s[c][j] = k0 + c < n ? W[(size_t)(k0 + c) * n + j0 + j] : T(0);
      }
      __syncthreads();
#pragma unroll
      for (int rb = 0; rb < NB; rb += CT) {
        const int r = rb + ty;
        Sum<T> v;
#pragma unroll
        for (int q = 0; q < rb + CT; ++q) v.add(X[r][q], s[q][tx]);
        if (k0 + r < n) W[(size_t)(k0 + r) * n + j0 + tx] = v.get();
      }
    } else {
      __syncthreads();
      for (int q = threadIdx.x; q < NB * NB; q += CT * CT) {
        const int r = q / NB, c = q % NB;
        if (k0 + r < n && k0 + c < n) W[(size_t)(k0 + r) * n + k0 + c] = X[r][c];
      }
    }
  }
  pdl_launch_dependents();
}

// Ainv = X^T X, X lower triangular: entry (i, j) sums over m >= max(i, j).
// A block forms one GT x GT tile of the lower triangle and its mirror image,
// its GK thread groups taking interleaved m: the longest sum (the first
// tile, all n rows) sets the time, so tiles are small and the sum is split.
constexpr int GT = 8, GK = 4;
template <typename T>
__global__ void __launch_bounds__(GT * GT * GK)
    k_coarse_gram(int n, const T* __restrict__ X, T* __restrict__ Ainv) {
  __shared__ T xi[32][GT + 1], xj[32][GT + 1], red[GK][GT * GT];
  pdl_wait();
  int ti = (int)((sqrtf(8.0f * blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while ((long long)ti * (ti + 1) / 2 > blockIdx.x) --ti;
  while ((long long)(ti + 1) * (ti + 2) / 2 <= blockIdx.x) ++ti;
  const int tj = (int)(blockIdx.x - (long long)ti * (ti + 1) / 2);
  const int e = threadIdx.x % (GT * GT), g = threadIdx.x / (GT * GT);
  const int li = e / GT, lj = e % GT;
  T acc = T(0);
  for (int m0 = GT * ti; m0 < n; m0 += 32) {
    const int m = threadIdx.x / GT, c = threadIdx.x % GT;   // 32 rows x GT columns
    const int row = m0 + m, ci = GT * ti + c, cj = GT * tj + c;
    // above the diagonal W still holds other values
    xi[m][c] = row < n && ci <= row ? X[(size_t)row * n + ci] : T(0);
    xj[m][c] = row < n && cj <= row ? X[(size_t)row * n + cj] : T(0);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 32 / GK; ++q) acc += xi[GK * q + g][li] * xj[GK * q + g][lj];
    __syncthreads();
  }
  red[g][e] = acc;
  __syncthreads();
  if (g == 0) {
    const T v = (red[0][e] + red[1][e]) + (red[2][e] + red[3][e]);
    const int i = GT * ti + li, j = GT * tj + lj;
    // on the diagonal tile only the lower entries are kept, so that the
    // result is symmetric bit for bit
    if (i < n && j <= i) {
      Ainv[(size_t)i * n + j] = v;
      Ainv[(size_t)j * n + i] = v;
    }
  }
  pdl_launch_dependents();
}

template <typename T>
cudaError_t inverse_t(int n, T* W, T* Ainv, T* scratch, int* status, cudaStream_t s) {
  constexpr int NB = CoarseNB<T>::NB;
  T* Dx = scratch;
  T* P = scratch + NB * NB;
  const dim3 th(CT * CT);
  cudaError_t e = launch_pdl(k_coarse_update<T, NB>, dim3(1), th, 0, s, n, -1, W, P, Dx, status);
  for (int k0 = 0; k0 < n && e == cudaSuccess; k0 += NB) {
    const int m = n - k0 - NB;                       // rows below the block
    const int nr = m > 0 ? (m + CT - 1) / CT : 0;
    e = launch_pdl(k_coarse_panel<T, NB>, dim3(nr + k0 / CT + 1), th, 0, s, n, k0, nr, W, P, Dx);
    if (nr == 0 || e != cudaSuccess) continue;
    const int kt = (k0 + NB) / CT;
    const int tiles = nr * kt + nr * (nr + 1) / 2;
    e = launch_pdl(k_coarse_update<T, NB>, dim3(1 + tiles), th, 0, s, n, k0, W, P, Dx, status);
  }
  if (e != cudaSuccess) return e;
  const int gt = (n + GT - 1) / GT;
  return launch_pdl(k_coarse_gram<T>, dim3(gt * (gt + 1) / 2), dim3(GT * GT * GK), 0, s, n, W,
                    Ainv);
}

}  // namespace

long long coarse_scratch_values(long long n) { return 32 * 32 + 32 * n; }

cudaError_t launch_cholesky_inverse(int t, int n, void* A, void* Ainv, void* scratch, int* status,
                                    cudaStream_t s) {
  return t == T_F64 ? inverse_t<double>(n, (double*)A, (double*)Ainv, (double*)scratch, status, s)
                    : inverse_t<float>(n, (float*)A, (float*)Ainv, (float*)scratch, status, s);
}

}  // namespace topo
