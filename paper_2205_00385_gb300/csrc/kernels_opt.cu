// Design-side kernels: SIMP modulus (Eq. 1), density filter and its
// transpose (Eq. 31-33), compliance and sensitivity (Eq. 3, 6, 34) and the
// optimality-criteria update with a device-side search for the volume
// multiplier.  float64, but for the mixed path's 3D sensitivity and the search,
// which sum in double-float.
#include <math.h>

#include <algorithm>
#include <cstdlib>

#include "dfmath.cuh"
#include "kernels.h"

namespace topo {

__device__ __forceinline__ double ipow(double x, double p) {
  if (p == 3.0) return x * x * x;
  if (p == 2.0) return x * x;
  if (p == 1.0) return x;
  if (p == 4.0) return (x * x) * (x * x);
  return pow(x, p);
}

__global__ void __launch_bounds__(256)
    k_simp(long long nel, const double* __restrict__ rho, double E0, double Emin, double penal,
           double* __restrict__ E64, float* __restrict__ E32) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nel) return;
  const double E = Emin + (E0 - Emin) * ipow(rho[e], penal);
  E64[e] = E;
  E32[e] = (float)E;
}

__global__ void __launch_bounds__(256)
    k_delta(long long nel, const double* __restrict__ E, const double* __restrict__ Ep,
            double* __restrict__ dE64, float* __restrict__ dE32, float* __restrict__ Ep32) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nel) return;
  const double d = E[e] - Ep[e];
  dE64[e] = d;
  dE32[e] = (float)d;
  Ep32[e] = (float)Ep[e];
}

// invHs_i = 1 / sum_j w_ij (precomputed, so no float64 division per term)
// mode 0: out_i = invHs_i sum_j w_ij in_j ; mode 1: out_e = sum_i w_ie in_i invHs_i
// mode 2: out_i = invHs_i (in ignored)
template <int DIM>
__global__ void __launch_bounds__(256)
    k_filter(GridP g, StencilP st, int mode, const double* __restrict__ invHs,
             const double* __restrict__ in, double* __restrict__ out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= g.nel) return;
  const int ex = (int)(e % g.nx);
  const long long rest = e / g.nx;
  const int ey = (int)(rest % g.ny);
  const int ez = DIM == 3 ? (int)(rest / g.ny) : 0;
  double acc = 0.0;
  for (int q = 0; q < st.count; ++q) {
    const int jx = ex + st.d[q][0], jy = ey + st.d[q][1], jz = ez + st.d[q][2];
    bool in_range = jx >= 0 && jx < g.nx && jy >= 0 && jy < g.ny;
    if (DIM == 3) in_range = in_range && jz >= 0 && jz < g.nz;
    if (!in_range) continue;
    const long long j = jx + (long long)g.nx * (jy + (long long)g.ny * (DIM == 3 ? jz : 0));
    const double w = st.w[q];
    if (mode == 0)
      acc = fma(w, in[j], acc);
    else if (mode == 1)
      acc = fma(w, in[j] * invHs[j], acc);
    else
      acc += w;
  }
  if (mode == 0)
    out[e] = acc * invHs[e];
  else if (mode == 1)
    out[e] = acc;
  else
    out[e] = 1.0 / acc;
}

// 3D filter with offsets of at most R elements per axis (1 < rmin <= R + 1).
// The weight depends on dx^2 + dy^2 + dz^2 alone, so a layer's values are first
// summed over the offsets of equal dx^2 + dy^2 (s = 0, 1, 2 and, for R = 2, 4, 5,
// 8), and each sum enters the 2R + 1 layers around it with one FMA: 15 (R = 1) or
// at most 45 (R = 2) float64 instructions per element instead of two per
// offset (27 to 93 offsets), on a pipe that does two per clock per SM.  A block
// owns 32 x 4 columns of FLZ elements; their values with a halo (zero outside
// the grid) are all requested at once and staged in shared memory, where the
// factor invHs of the transpose is applied once, and a thread then runs up its
// column.  Transpose at 192 x 96 x 96, offset list / this: rmin 1.5 131 / 62 us,
// 2.0 184 / 74 us, 2.5 542 / 186 us; 64 x 32 x 32, 1.5: 10 / 8 us.  (One layer
// staged at a time: 110 us at rmin 2.0, 24 us on small grids; 8 rows instead of
// 4: 2 to 4 us more on small grids; weights of 0 tested at run time: float64
// comparisons, as dear as the FMAs.)  Small grids take the offset list
// (filter3_small).
constexpr int FLX = 32, FLY = 4, FLZ = 4;

template <int R>
struct FilterW {
  static constexpr int NS = R == 1 ? 3 : 6;   // classes of dx^2 + dy^2
  double w[NS][R + 1];                        // weight of class s at |dz| = m
};
// dx^2 + dy^2 of class q
__host__ __device__ constexpr int filter_class(int q) {
  return q < 3 ? q : q == 3 ? 4 : q == 4 ? 5 : 8;
}

// D: the largest dx^2 + dy^2 + dz^2 inside the radius
template <int R, int D>
__global__ void __launch_bounds__(FLX * FLY)
    k_filter3(GridP g, FilterW<R> fw, bool sens, const double* __restrict__ invHs,
              const double* __restrict__ in, double* __restrict__ out) {
  constexpr int NS = FilterW<R>::NS, SX = FLX + 2 * R, SY = FLY + 2 * R, SZ = FLZ + 2 * R;
  __shared__ double t[SZ][SY][SX];
  const int tid = threadIdx.x, tx = tid % FLX, ty = tid / FLX;
  const int x0 = blockIdx.x * FLX, y0 = blockIdx.y * FLY, z0 = blockIdx.z * FLZ;
  const long long plane = (long long)g.nx * g.ny;
#pragma unroll 8
  for (int q = tid; q < SX * SY * SZ; q += FLX * FLY) {
    const int c = q % SX, r = q / SX % SY, l = q / (SX * SY);
    const int jx = x0 - R + c, jy = y0 - R + r, jz = z0 - R + l;
    const bool ok = jx >= 0 && jx < g.nx && jy >= 0 && jy < g.ny && jz >= 0 && jz < g.nz;
    const long long j = ok ? jx + (long long)g.nx * jy + plane * jz : 0;
    t[l][r][c] = ok ? (sens ? in[j] * invHs[j] : in[j]) : 0.0;
  }
  __syncthreads();
  if (x0 + tx >= g.nx || y0 + ty >= g.ny) return;
  double acc[2 * R + 1];   // acc[i]: the output of layer l - 2 R + i so far
#pragma unroll
  for (int i = 0; i < 2 * R + 1; ++i) acc[i] = 0.0;
#pragma unroll
  for (int l = 0; l < SZ; ++l) {
    auto at = [&](int dx, int dy) { return t[l][ty + R + dy][tx + R + dx]; };
    double v[NS];
    v[0] = at(0, 0);
    v[1] = (at(-1, 0) + at(1, 0)) + (at(0, -1) + at(0, 1));
    if constexpr (D >= 2) v[2] = (at(-1, -1) + at(1, -1)) + (at(-1, 1) + at(1, 1));
    if constexpr (R == 2) {
      v[3] = (at(-2, 0) + at(2, 0)) + (at(0, -2) + at(0, 2));
      if constexpr (D >= 5)
        v[4] = ((at(-2, -1) + at(2, -1)) + (at(-2, 1) + at(2, 1))) +
               ((at(-1, -2) + at(1, -2)) + (at(-1, 2) + at(1, 2)));
      if constexpr (D >= 8) v[5] = (at(-2, -2) + at(2, -2)) + (at(-2, 2) + at(2, 2));
    }
#pragma unroll
    for (int i = 0; i < 2 * R + 1; ++i) {
      const int zo = l - 2 * R + i, m = i < R ? R - i : i - R;   // output layer, |dz|
      if (zo < 0 || zo >= FLZ) continue;
#pragma unroll
      for (int q = 0; q < NS; ++q)
        if (filter_class(q) + m * m <= D) acc[i] = fma(fw.w[q][m], v[q], acc[i]);
    }
    const int zo = l - 2 * R;
    if (zo >= 0 && z0 + zo < g.nz) {
      const long long e = x0 + tx + (long long)g.nx * (y0 + ty) + plane * (z0 + zo);
      out[e] = sens ? acc[0] : acc[0] * invHs[e];
    }
#pragma unroll
    for (int i = 0; i < 2 * R; ++i) acc[i] = acc[i + 1];
    acc[2 * R] = 0.0;
  }
}

template <int R, int D>
static cudaError_t run_filter3(const GridP& g, const StencilP& st, bool sens, const double* invHs,
                               const double* in, double* out, cudaStream_t s) {
  FilterW<R> fw = {};
  for (int q = 0; q < st.count; ++q) {
    const int d2 = st.d[q][0] * st.d[q][0] + st.d[q][1] * st.d[q][1];
    for (int c = 0; c < FilterW<R>::NS; ++c)
      if (filter_class(c) == d2) fw.w[c][std::abs(st.d[q][2])] = st.w[q];
  }
  k_filter3<R, D><<<dim3((g.nx + FLX - 1) / FLX, (g.ny + FLY - 1) / FLY, (g.nz + FLZ - 1) / FLZ),
                    FLX * FLY, 0, s>>>(g, fw, sens, invHs, in, out);
  return cudaGetLastError();
}

// Double-float Walsh blocks of KE (hi and lo parts of each float64 entry), the
// entries above the diagonal doubled: X^T B X = sum of the upper triangles
struct WhtDf {
  float h[8][3][3], l[8][3][3];
};

__device__ __forceinline__ void wht4_dfl(dfl (&v)[4]) {
  const dfl s0 = df_add(v[0], v[1]), d0 = df_add(v[0], df_neg(v[1]));
  const dfl s1 = df_add(v[2], v[3]), d1 = df_add(v[2], df_neg(v[3]));
  v[0] = df_add(s0, s1);
  v[1] = df_add(d0, d1);
  v[2] = df_add(s0, df_neg(s1));
  v[3] = df_add(d0, df_neg(d1));
}

// 3D compliance and sensitivity of k_sensitivity3_wht in double-float
// arithmetic (mixed path), for an integer penalisation exponent:
// dc_e = pfac rho_e^ipen ce_e with pfac = -penal (E0 - Emin), ipen = penal - 1.
// A thread streams one element column in z: a face's twelve displacements are
// loaded, split and xy-transformed once for the element below and the one
// above (one element per thread read, split and transformed 24: 334 us at
// 192 x 96 x 96, now 158), and the quadratic form takes the 33 non-zero entries of the
// blocks' upper triangles instead of all 72.
__global__ void __launch_bounds__(SN_X * SN_Y, 6)
    k_sensitivity3_df(GridP g, const uint8_t* __restrict__ mask, WhtDf kb, int zc,
                      const double* __restrict__ u, const double* __restrict__ E,
                      const double* __restrict__ rho, double pfac, int ipen,
                      double* __restrict__ dc, double* compliance, double* partials,
                      unsigned* counter) {
  __shared__ double sh[1][SN_X * SN_Y / 32], tot[1];
  const int ex = blockIdx.x * SN_X + threadIdx.x % SN_X, ey = blockIdx.y * SN_Y + threadIdx.x / SN_X;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, g.nz);
  const long long plane = (long long)g.nnx * g.nny;
  const dfl pf = split_d(pfac);
  dfl v[1] = {{0.f, 0.f}};
  if (ex < g.nx && ey < g.ny) {
    auto face = [&](int kz, dfl (&W)[3][4]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long nd = ex + (q & 1) + (long long)g.nnx * (ey + (q >> 1)) + plane * kz;
        const unsigned m = mask[nd];
#pragma unroll
        for (int c = 0; c < 3; ++c)
          W[c][q] = ((m >> c) & 1u) ? dfl{0.f, 0.f} : split_d(u[3 * nd + c]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) wht4_dfl(W[c]);
    };
    dfl Wb[3][4], Wt[3][4];
    face(z0, Wb);
    for (int ez = z0; ez < z1; ++ez) {
      const long long e = ex + (long long)g.nx * (ey + (long long)g.ny * ez);
      const double re64 = rho[e], e64 = E[e];
      face(ez + 1, Wt);
      dfl X[3][8];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          X[c][t] = df_add(Wb[c][t], Wt[c][t]);
          X[c][t + 4] = df_add(Wb[c][t], df_neg(Wt[c][t]));
          Wb[c][t] = Wt[c][t];
        }
      dfl ce = {0.f, 0.f};
#pragma unroll
      for (int tau = 0; tau < 8; ++tau)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (wht_zero(tau, c, c)) continue;   // (its row and column are zero too)
          const dfl z = X[c][tau ^ (1 << c)];
          dfl s = df_mul(dfl{kb.h[tau][c][c], kb.l[tau][c][c]}, z);
#pragma unroll
          for (int cp = c + 1; cp < 3; ++cp)
            if (!wht_zero(tau, c, cp))
              s = df_add(df_mul(dfl{kb.h[tau][c][cp], kb.l[tau][c][cp]}, X[cp][tau ^ (1 << cp)]),
                         s);
          ce = df_add(df_mul(z, s), ce);
        }
      const dfl re = split_d(re64);
      dfl f = pf;
      for (int q = 0; q < ipen; ++q) f = df_mul(f, re);
      dc[e] = df_to_d(df_mul(f, ce));
      v[0] = df_add(df_mul(split_d(e64), ce), v[0]);
    }
  }
  if (grid_sum_df(v, sh, tot, partials, counter) && threadIdx.x == 0) *compliance = tot[0];
}

// ce_e = u_e^T KE u_e; dc_e = -penal (E0-Emin) rho_e^(penal-1) ce_e;
// compliance = sum_e E_e ce_e (deterministic reduction).
// 3D: u_e^T KE u_e = X^T B X with X the Walsh transform of u_e (KE = T B T),
// ~170 float64 operations per element instead of ~600.
__global__ void __launch_bounds__(RED_THREADS)
    k_sensitivity3_wht(GridP g, const uint8_t* __restrict__ mask, WhtBlocks<double> kb,
                       const double* __restrict__ u, const double* __restrict__ E,
                       const double* __restrict__ rho, double penal, double E0, double Emin,
                       double* __restrict__ dc, double* compliance, double* partials,
                       unsigned* counter) {
  __shared__ double sh[32];
  double v[1] = {0.0};
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < g.nel;
       e += (long long)gridDim.x * blockDim.x) {
    const int ex = (int)(e % g.nx);
    const long long rest = e / g.nx;
    const int ey = (int)(rest % g.ny);
    const int ez = (int)(rest / g.ny);
    double X[3][8];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int i = ex + (a & 1), j = ey + ((a >> 1) & 1), k = ez + ((a >> 2) & 1);
      const long long nd = i + (long long)g.nnx * (j + (long long)g.nny * k);
      const unsigned m = mask[nd];
#pragma unroll
      for (int c = 0; c < 3; ++c) X[c][a] = ((m >> c) & 1u) ? 0.0 : u[3 * nd + c];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) fwht8<double>(X[c]);
    double ce = 0.0;
#pragma unroll
    for (int tau = 0; tau < 8; ++tau) {
      double z[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) z[c] = X[c][tau ^ (1 << c)];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        double s = kb.b[tau][c][0] * z[0];
        s = fma(kb.b[tau][c][1], z[1], s);
        s = fma(kb.b[tau][c][2], z[2], s);
        ce = fma(z[c], s, ce);
      }
    }
    const double re = rho[e];
    dc[e] = -penal * (E0 - Emin) * ipow(re, penal - 1.0) * ce;
    v[0] = fma(E[e], ce, v[0]);
  }
  block_sum<1>(v, sh);
  if (publish_partials<1>(v, partials, counter)) {
    double o[1];
    finish_sum<1>(partials, counter, o, sh);
    if (threadIdx.x == 0) *compliance = o[0];
  }
}

template <int DIM>
__global__ void __launch_bounds__(RED_THREADS)
    k_sensitivity(GridP g, const uint8_t* __restrict__ mask, KEP<double, Geo<DIM>::ND> ke,
                  const double* __restrict__ u, const double* __restrict__ E,
                  const double* __restrict__ rho, double penal, double E0, double Emin,
                  double* __restrict__ dc, double* compliance, double* partials,
                  unsigned* counter, const double* __restrict__ adj) {
  constexpr int ND = Geo<DIM>::ND, NPE = Geo<DIM>::NPE;
  __shared__ double sh[32];
  double v[1] = {0.0};
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < g.nel;
       e += (long long)gridDim.x * blockDim.x) {
    const int ex = (int)(e % g.nx);
    const long long rest = e / g.nx;
    const int ey = (int)(rest % g.ny);
    const int ez = DIM == 3 ? (int)(rest / g.ny) : 0;
    // ue: the field; ve: the adjoint field (the field itself for compliance)
    double ue[ND], ve[ND];
#pragma unroll
    for (int a = 0; a < NPE; ++a) {
      const int i = ex + (a & 1), j = ey + ((a >> 1) & 1), k = ez + ((a >> 2) & 1);
      const long long nd = i + (long long)g.nnx * (j + (long long)g.nny * (DIM == 3 ? k : 0));
      const unsigned m = mask[nd];
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        const bool fx = (m >> c) & 1u;
        ue[DIM * a + c] = fx ? 0.0 : u[DIM * nd + c];
        ve[DIM * a + c] = fx ? 0.0 : (adj ? adj[DIM * nd + c] : u[DIM * nd + c]);
      }
    }
    double ce = 0.0;
#pragma unroll
    for (int r = 0; r < ND; ++r) {
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < ND; ++c) s = fma(ke.v[r * ND + c], ue[c], s);
      ce = fma(ve[r], s, ce);
    }
    const double re = rho[e];
    dc[e] = -penal * (E0 - Emin) * ipow(re, penal - 1.0) * ce;
    v[0] = fma(E[e], ce, v[0]);
  }
  block_sum<1>(v, sh);
  if (publish_partials<1>(v, partials, counter)) {
    double o[1];
    finish_sum<1>(partials, counter, o, sh);
    if (threadIdx.x == 0) *compliance = o[0];
  }
}

// a_e = rho_e sqrt(max(0, -dc_e / dv_e)); bracket [0, 1e9]
__global__ void __launch_bounds__(256)
    k_oc_prep(long long nel, const double* __restrict__ rho, const double* __restrict__ dc,
              const double* __restrict__ dv, double* __restrict__ a, double* scal) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e == 0) {
    scal[S_OC_L1] = 0.0;
    scal[S_OC_L2] = 1e9;
  }
  if (e >= nel) return;
  a[e] = rho[e] * sqrt(fmax(0.0, -dc[e] / dv[e]));
}

__device__ __forceinline__ double oc_new(double a, double s, double r, double move) {
  const double lo = fmax(0.0, r - move), hi = fmin(1.0, r + move);
  return fmin(hi, fmax(lo, a * s));
}

// One bisection step: lmid = (l1+l2)/2; the filtered volume of rho_new(lmid)
// decides which half is kept (as in the oracle).  No-op once the bracket is
// within a relative 1e-13.
__global__ void __launch_bounds__(RED_THREADS)
    k_oc_step(long long nel, const double* __restrict__ rho, const double* __restrict__ a,
              const double* __restrict__ dv, double move, double target, double* scal,
              double* partials, unsigned* counter) {
  __shared__ double sh[32];
  const double l1 = scal[S_OC_L1], l2 = scal[S_OC_L2];
  if (!((l2 - l1) > 1e-13 * (l1 + l2))) return;
  const double lmid = 0.5 * (l1 + l2);
  const double s = 1.0 / sqrt(lmid);
  double v[1] = {0.0};
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nel;
       e += (long long)gridDim.x * blockDim.x)
    v[0] = fma(dv[e], oc_new(a[e], s, rho[e], move), v[0]);
  block_sum<1>(v, sh);
  if (publish_partials<1>(v, partials, counter)) {
    double o[1];
    finish_sum<1>(partials, counter, o, sh);
    if (threadIdx.x == 0) {
      if (o[0] > target)
        scal[S_OC_L1] = lmid;
      else
        scal[S_OC_L2] = lmid;
      scal[S_OC_VOL] = o[0];
    }
  }
}

// Context path of the mixed and float64 solvers alike: the search for the
// multiplier lambda.  The volume is a non-decreasing, piecewise linear
// function of s = lambda^-eta, so after a bracket [l1, l2] with
// V(l1) > target >= V(l2) is narrow, the secant point of the bracket is off by
// about the square of its width.  A sweep sums the volume at OC_NP points of
// the bracket in double-float; its last block keeps the sub-interval that
// holds the root and writes the next points:
//   first sweep      around the multiplier that no limit would clamp, l0 8^j
//   lower end 0      l2 / 8^7 .. l2 / 8
//   ratio above 4    geometric
//   narrow           the secant point, +- guards of half the squared width and
//                    1/32 of that, and the bracket's thirds
//   no slope (the volume changes by its own rounding), or the last narrow
//   sweep left more than a fifth    equal sections
// Six or seven sweeps reach the relative bracket of 1e-13 on most designs (equal
// sections of the bracket took 17 to 23), up to 20 where the volume is nearly flat
// in lambda.  A sweep after that is a no-op.  Where OC_SWEEPS were not enough one
// launch goes on by itself (k_oc_rest), so that nothing waits for the host and a
// captured update needs no more launches.  A sweep reads 32 bytes per element (57
// MB at 192 x 96 x 96, which stays in L2): 24 us there, of which the arithmetic
// of the seven points is 8.
constexpr int OC_NP = 7, OC_T = 512, OC_BLOCKS = 304, OC_SWEEPS = 9;
constexpr double OC_LAM_MAX = 1e9;
static_assert(OC_NP <= S_OC_NPT && OC_NP <= OC_T / 32, "one warp per point");

// x^eta of the OC rule (sqrt for the compliance rule's eta = 1/2) and the
// multiplier's factor lambda^-eta
__device__ __forceinline__ double oc_damp(double x, double eta) {
  return eta == 0.5 ? sqrt(x) : pow(x, eta);
}
__device__ __forceinline__ double oc_lam_factor(double lam, double eta) {
  return eta == 0.5 ? 1.0 / sqrt(lam) : pow(lam, -eta);
}
__device__ __forceinline__ double oc_lam_of(double s, double eta) {
  return eta == 0.5 ? 1.0 / (s * s) : pow(s, -1.0 / eta);
}

// bracket within its final width (also when both ends are 0)
__device__ __forceinline__ bool oc_done(double l1, double l2) {
  return !((l2 - l1) > 1e-13 * (l1 + l2));
}

// Writes the bracket and its next points; called by one whole warp.
// v1, v2 and s1, s2: the volumes and factors lambda^-eta at the bracket's ends
// (of the lower end unknown, and not used, while it is 0).  missed: the last
// secant points did not narrow the bracket.
__device__ __forceinline__ void oc_next_points(double l1, double l2, double v1, double v2,
                                               double s1, double s2, double target, double eta,
                                               double l0, bool missed, volatile double* scal) {
  const int j = threadIdx.x & 31;
  double lam;
  if (l0 > 0.0) {
    lam = fmin(ldexp(l0, 3 * (j - OC_NP / 2)), l2);
  } else if (l1 == 0.0) {
    lam = ldexp(l2, -3 * (OC_NP - j));
  } else if (l2 > 4.0 * l1) {
    const double q = sqrt(sqrt(sqrt(l2 / l1)));
    lam = l1;
    for (int i = 0; i <= j && i < OC_NP; ++i) lam *= q;
  } else if (missed || !(v1 - v2 > 1e-13 * target)) {
    lam = l1 + (j + 1) * ((l2 - l1) / (OC_NP + 1));
  } else {
    const double mid = oc_lam_of(s2 + (target - v2) * ((s1 - s2) / (v1 - v2)), eta);
    const double w = (l2 - l1) / l2, d = mid * fmax(0.5 * w * w, 6.4e-13);
    lam = j == 0 ? mid - d
        : j == 1 ? mid - d / 32
        : j == 2 ? mid
        : j == 3 ? mid + d / 32
        : j == 4 ? mid + d
                 : l1 + (j - 4) * ((l2 - l1) / 3);
  }
  lam = fmin(fmax(lam, l1), l2);
  // ascending order: the rank of each point among the OC_NP
  int rank = 0;
#pragma unroll
  for (int i = 0; i < OC_NP; ++i) {
    const double o = __shfl_sync(0xffffffffu, lam, i);
    rank += o < lam || (o == lam && i < j);
  }
  if (j < OC_NP) {
    scal[S_OC_PT + rank] = lam;
    scal[S_OC_SP + rank] = oc_lam_factor(lam, eta);
  }
  if (j == 0) {
    scal[S_OC_L1] = l1;
    scal[S_OC_L2] = l2;
    scal[S_OC_V1] = v1;
    scal[S_OC_V2] = v2;
    scal[S_OC_S1] = s1;
    scal[S_OC_S2] = s2;
  }
}

// a_e = rho_e max(0, -dc_e / dv_e)^eta, the move limits and the weights as
// pairs, the search's bracket [0, 1e9] and its first points.  When even the
// upper limits hold no more than the target volume the bracket is 0, and
// when its upper end still holds more, that end.
__global__ void __launch_bounds__(OC_T)
    k_oc_prep_d(long long nel, const double* __restrict__ rho, const double* __restrict__ dc,
                const double* __restrict__ dv, double move, double target,
                double* __restrict__ a64, float2* __restrict__ a, float2* __restrict__ lo,
                float2* __restrict__ hi, float2* __restrict__ dvd, double* scal, double eta,
                double* partials, unsigned* counter) {
  __shared__ double sh[3][OC_T / 32], tot[3];
  __shared__ dfl s_top;
  if (threadIdx.x == 0) s_top = split_d(oc_lam_factor(OC_LAM_MAX, eta));
  __syncthreads();
  const dfl top = s_top;
  dfl v[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  for (long long e = (long long)blockIdx.x * OC_T + threadIdx.x; e < nel;
       e += (long long)gridDim.x * OC_T) {
    const double r = rho[e], d = dv[e];
    const double ae = r * oc_damp(fmax(0.0, -dc[e] / d), eta);
    a64[e] = ae;
    const dfl av = split_d(ae);
    const dfl lv = split_d(fmax(0.0, r - move)), hv = split_d(fmin(1.0, r + move));
    const dfl dd = split_d(d);
    a[e] = make_float2(av.h, av.l);
    lo[e] = make_float2(lv.h, lv.l);
    hi[e] = make_float2(hv.h, hv.l);
    dvd[e] = make_float2(dd.h, dd.l);
    df_dot_acc(v[0], dd, av);
    df_dot_acc(v[1], dd, av.h > 0.f ? hv : lv);
    const dfl x = df_mul(av, top);
    df_dot_acc(v[2], dd, df_gt(x, hv) ? hv : (df_gt(lv, x) ? lv : x));
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) v[q] = df_norm(v[q]);
  if (!grid_sum_df(v, sh, tot, partials, counter) || threadIdx.x >= 32) return;
  const double l0 = oc_lam_of(target / tot[0], eta);
  const double l1 = tot[1] > target && tot[2] > target ? OC_LAM_MAX : 0.0;
  const double l2 = tot[1] > target ? OC_LAM_MAX : 0.0;
  const double st = oc_lam_factor(OC_LAM_MAX, eta);
  oc_next_points(l1, l2, tot[1], tot[2], st, st, target, eta,
                 l0 > 1e-60 && l0 < OC_LAM_MAX ? l0 : 0.0, false, scal);
}

struct OcFields {   // the elements' factors, limits and weights, two per float4
  const float4 *a, *lo, *hi, *dv;
};

// The volumes at the sweep's points over the grid; true in the last block, where
// tot holds them.
template <typename Sh>
__device__ __forceinline__ bool oc_volumes(long long nel, const OcFields& f, volatile double* scal,
                                           Sh& sh, double (&tot)[OC_NP], double* partials,
                                           unsigned* counter, bool trigger) {
  dfl sv[OC_NP], v[OC_NP];
#pragma unroll
  for (int j = 0; j < OC_NP; ++j) {
    sv[j] = split_d(scal[S_OC_SP + j]);
    v[j] = {0.f, 0.f};
  }
  auto element = [&](dfl av, dfl lv, dfl hv, dfl dd) {
#pragma unroll
    for (int j = 0; j < OC_NP; ++j) {
      dfl x = df_mul(av, sv[j]);
      x = df_gt(x, hv) ? hv : (df_gt(lv, x) ? lv : x);
      df_dot_acc(v[j], dd, x);
    }
  };
  // two elements per 16-byte load (nel is even: every grid coarsens once)
  for (long long q = (long long)blockIdx.x * OC_T + threadIdx.x; 2 * q < nel;
       q += (long long)gridDim.x * OC_T) {
    const float4 a4 = __ldg(f.a + q), l4 = __ldg(f.lo + q), h4 = __ldg(f.hi + q), d4 = __ldg(f.dv + q);
    element({a4.x, a4.y}, {l4.x, l4.y}, {h4.x, h4.y}, {d4.x, d4.y});
    element({a4.z, a4.w}, {l4.z, l4.w}, {h4.z, h4.w}, {d4.z, d4.w});
  }
#pragma unroll
  for (int j = 0; j < OC_NP; ++j) v[j] = df_norm(v[j]);
  if (trigger) pdl_launch_dependents();
  return grid_sum_df(v, sh, tot, partials, counter);
}

// The sub-interval that holds the root, and its points; by one warp.  The volume
// decreases with lambda: the last point above target and the first at or below it.
__device__ __forceinline__ void oc_narrow(const double (&tot)[OC_NP], double target, double eta,
                                          volatile double* scal) {
  const double l1 = scal[S_OC_L1], l2 = scal[S_OC_L2];
  int k = 0;
  while (k < OC_NP && tot[k] > target) ++k;
  const double n1 = k > 0 ? scal[S_OC_PT + k - 1] : l1;
  const double w1 = k > 0 ? tot[k - 1] : scal[S_OC_V1];
  const double f1 = scal[k > 0 ? S_OC_SP + k - 1 : S_OC_S1];
  const double n2 = k < OC_NP ? scal[S_OC_PT + k] : l2;
  const double w2 = k < OC_NP ? tot[k] : scal[S_OC_V2];
  const double f2 = scal[k < OC_NP ? S_OC_SP + k : S_OC_S2];
  const bool missed = l2 <= 4.0 * l1 && n2 - n1 > 0.2 * (l2 - l1);
  __syncwarp();
  oc_next_points(n1, n2, w1, w2, f1, f2, target, eta, 0.0, missed, scal);
}

// one sweep
__global__ void __launch_bounds__(OC_T, 2)
    k_oc_sweep(long long nel, OcFields f, double target, volatile double* scal, double* partials,
               unsigned* counter, double eta) {
  __shared__ double sh[OC_NP][OC_T / 32], tot[OC_NP];
  pdl_wait();
  if (oc_done(scal[S_OC_L1], scal[S_OC_L2])) return;
  if (oc_volumes(nel, f, scal, sh, tot, partials, counter, true) && threadIdx.x < 32)
    oc_narrow(tot, target, eta, scal);
}

// Sweeps until the bracket is done: blocks that are all resident (one cluster, or a
// cooperative launch) wait for the last one's points, so the wait ends; its limit
// of a few seconds sets *status.  A sweep at least thirds a bracket that does not start at
// 0 and takes one that does down by 8^7, so the loop's limit is not met.
constexpr int OC_WAIT = 1 << 22, OC_CLUSTER = 16;
__global__ void __launch_bounds__(OC_T, 2)
    k_oc_rest(long long nel, OcFields f, double target, volatile double* scal, double* partials,
              unsigned* counter, volatile unsigned* turn, int* status, double eta) {
  __shared__ double sh[OC_NP][OC_T / 32], tot[OC_NP];
  __shared__ bool s_go;
  pdl_wait();
  unsigned t0 = 0;
  if (threadIdx.x == 0) {
    t0 = *turn;
    __threadfence();   // (read before this block's first partial sums are counted)
  }
  for (int it = 0; it < 160; ++it) {
    if (oc_done(scal[S_OC_L1], scal[S_OC_L2])) return;
    const bool last = oc_volumes(nel, f, scal, sh, tot, partials, counter, false);
    if (last && threadIdx.x < 32) oc_narrow(tot, target, eta, scal);
    __syncthreads();
    if (threadIdx.x == 0) {
      s_go = true;
      if (last) {
        __threadfence();
        *turn = t0 + 1;
      } else {
        for (int w = 0; *turn == t0; ++w) {
          if (w == OC_WAIT) {
            *status = TO_E_TIMEOUT;
            s_go = false;
            break;
          }
          __nanosleep(40);
        }
        __threadfence();
      }
      ++t0;
    }
    __syncthreads();
    if (!s_go) return;
  }
}

// rho <- clamp(a lambda^-eta) and max |rho_new - rho|.  The limits are
// selected by comparing bit patterns as integers (doubles of one sign order as
// their bits do), which leaves four FP64 instructions per element; a product
// that is not a number (0 x infinity) takes the lower limit, as fmax does.
__global__ void __launch_bounds__(RED_THREADS)
    k_oc_final(long long nel, double* __restrict__ rho, const double* __restrict__ a,
               double move, double* scal, double* change_dev, double* partials,
               unsigned* counter, double eta) {
  __shared__ double sh[32];
  const double lam = 0.5 * (scal[S_OC_L1] + scal[S_OC_L2]);
  const double s = oc_lam_factor(lam, eta);
  const long long inf = 0x7ff0000000000000LL, minus_inf = (long long)0xfff0000000000000ULL;
  const long long one = __double_as_longlong(1.0);
  long long most = 0;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nel;
       e += (long long)gridDim.x * blockDim.x) {
    const double r = rho[e];
    long long lo = __double_as_longlong(r - move), hi = __double_as_longlong(r + move);
    long long t = __double_as_longlong(a[e] * s);
    lo = lo < 0 || lo > inf ? 0 : lo;
    hi = hi > one || (hi < 0 && hi > minus_inf) ? one : hi;   // (NaN of either sign: 1)
    t = t < lo || t > inf ? lo : t;
    t = t > hi ? hi : t;
    const double rn = __longlong_as_double(t);
    rho[e] = rn;
    const long long d = __double_as_longlong(rn - r) & 0x7fffffffffffffffLL;
    if (d <= inf && d > most) most = d;
  }
  double v[1] = {__longlong_as_double(most)};
  block_max<1>(v, sh);
  if (publish_partials<1>(v, partials, counter)) {
    double o[1];
    finish_max<1>(partials, counter, o, sh);
    if (threadIdx.x == 0) {
      scal[S_CHANGE] = o[0];
      if (change_dev) *change_dev = o[0];
    }
  }
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
cudaError_t launch_simp(long long nel, const double* rho, double E0, double Emin, double penal,
                        double* E64, float* E32, cudaStream_t s) {
  k_simp<<<nblocks(nel, 256), 256, 0, s>>>(nel, rho, E0, Emin, penal, E64, E32);
  return cudaGetLastError();
}

cudaError_t launch_delta(long long nel, const double* E, const double* Eprev, double* dE64,
                         float* dE32, float* Eprev32, cudaStream_t s) {
  k_delta<<<nblocks(nel, 256), 256, 0, s>>>(nel, E, Eprev, dE64, dE32, Eprev32);
  return cudaGetLastError();
}

// Grids on which the offset list is the faster filter: a thread per element hides
// its loads better than a block's staging while the chip is not full.  Offset list /
// staged, us: density filter at 16 x 8 x 8 5.2 / 6.2 (rmin 1.5), 10.3 / 12.3 (2.5), at
// 32 x 16 x 16 6.2 / 6.2 (1.5), 6.2 / 8.2 (2.0), 10.4 / 12.3 (2.5), at 48 x 24 x 24 6.2 /
// 6.2, 6.2 / 8.2 and 11.7 / 12.3, at 64 x 32 x 32 8.2 / 8.2 (2.0) and 14.8 / 12.3
// (2.5).  The transpose has two values per offset: at 16 x 8 x 8 6.2 / 7.2 (1.5), 14.6 /
// 12.3 (2.5), at 32 x 16 x 16 6.2 / 8.2 (1.5), at 48 x 24 x 24 8.2 / 8.2.
static bool filter3_small(const GridP& g, const StencilP& st, int mode) {
  if (mode == 1) return st.reach == 1 && g.nel <= 8192;
  return g.nel <= (st.d2max > 2 ? 32768 : 4096);
}

cudaError_t launch_filter(int dim, const GridP& g, const StencilP& st, int mode,
                          const double* Hs, const double* in, double* out, cudaStream_t s) {
  if (dim == 2)
    k_filter<2><<<nblocks(g.nel, 256), 256, 0, s>>>(g, st, mode, Hs, in, out);
  else if (mode != 2 && st.reach >= 1 && st.reach <= 2 && !filter3_small(g, st, mode)) {
    const bool sens = mode == 1;
    switch (st.d2max) {
      case 1: return run_filter3<1, 1>(g, st, sens, Hs, in, out, s);
      case 2: return run_filter3<1, 2>(g, st, sens, Hs, in, out, s);
      case 3: return run_filter3<1, 3>(g, st, sens, Hs, in, out, s);
      case 4: return run_filter3<2, 4>(g, st, sens, Hs, in, out, s);
      case 5: return run_filter3<2, 5>(g, st, sens, Hs, in, out, s);
      case 6: return run_filter3<2, 6>(g, st, sens, Hs, in, out, s);
      default: return run_filter3<2, 8>(g, st, sens, Hs, in, out, s);
    }
  }
  else
    k_filter<3><<<nblocks(g.nel, 256), 256, 0, s>>>(g, st, mode, Hs, in, out);
  return cudaGetLastError();
}

bool sensitivity_df_ok(int dim, double penal) {
  return dim == 3 && penal >= 1.0 && penal <= 9.0 && penal == (double)(int)penal;
}

cudaError_t launch_sensitivity_df(const GridP& g, const uint8_t* mask, const double* wht,
                                  const double* u, const double* E, const double* rho,
                                  double penal, double E0, double Emin, double* dc,
                                  double* compliance, double* partials, unsigned* counter,
                                  cudaStream_t s) {
  if (!wht || !sensitivity_df_ok(3, penal)) return cudaErrorInvalidValue;
  WhtDf kb;
  for (int q = 0; q < 72; ++q) {
    const double w = (q % 3 > q / 3 % 3 ? 2.0 : 1.0) * wht[q];
    const float h = (float)w;
    (&kb.h[0][0][0])[q] = h;
    (&kb.l[0][0][0])[q] = (float)(w - (double)h);
  }
  const int zc = sensitivity_chunk(g.nx, g.ny, g.nz);
  if (sensitivity_blocks(g.nx, g.ny, g.nz, zc) > PARTIALS) return cudaErrorInvalidValue;
  const dim3 grid((g.nx + SN_X - 1) / SN_X, (g.ny + SN_Y - 1) / SN_Y, (g.nz + zc - 1) / zc);
  k_sensitivity3_df<<<grid, SN_X * SN_Y, 0, s>>>(g, mask, kb, zc, u, E, rho, -penal * (E0 - Emin),
                                                (int)penal - 1, dc, compliance, partials, counter);
  return cudaGetLastError();
}

cudaError_t launch_filter_norm(int dim, const GridP& g, const StencilP& st, double* Hs,
                               cudaStream_t s) {
  return launch_filter(dim, g, st, 2, nullptr, nullptr, Hs, s);
}

template <int DIM>
static cudaError_t sens_t(const GridP& g, const uint8_t* mask, const double* kev, const double* u,
                          const double* E, const double* rho, double penal, double E0,
                          double Emin, double* dc, double* compliance, double* partials,
                          unsigned* counter, cudaStream_t s, const double* v) {
  constexpr int ND = Geo<DIM>::ND;
  KEP<double, ND> ke;
  for (int q = 0; q < ND * ND; ++q) ke.v[q] = kev[q];
  k_sensitivity<DIM><<<RED_BLOCKS, RED_THREADS, 0, s>>>(g, mask, ke, u, E, rho, penal, E0, Emin,
                                                        dc, compliance, partials, counter, v);
  return cudaGetLastError();
}

cudaError_t launch_sensitivity(int dim, const GridP& g, const uint8_t* mask, const double* ke,
                               const double* wht, const double* u, const double* E,
                               const double* rho, double penal, double E0, double Emin,
                               double* dc, double* compliance, double* partials,
                               unsigned* counter, cudaStream_t s, const double* v) {
  if (dim == 2)
    return sens_t<2>(g, mask, ke, u, E, rho, penal, E0, Emin, dc, compliance, partials, counter, s,
                     v);
  if (wht && !v) {
    WhtBlocks<double> kb;
    for (int q = 0; q < 72; ++q) (&kb.b[0][0][0])[q] = wht[q];
    k_sensitivity3_wht<<<RED_BLOCKS, RED_THREADS, 0, s>>>(g, mask, kb, u, E, rho, penal, E0, Emin,
                                                          dc, compliance, partials, counter);
    return cudaGetLastError();
  }
  return sens_t<3>(g, mask, ke, u, E, rho, penal, E0, Emin, dc, compliance, partials, counter, s,
                   v);
}

cudaError_t launch_oc_prep(long long nel, const double* rho, const double* dc,
                           const double* dv, double* a, double* scal, cudaStream_t s) {
  k_oc_prep<<<nblocks(nel, 256), 256, 0, s>>>(nel, rho, dc, dv, a, scal);
  return cudaGetLastError();
}

cudaError_t launch_oc_step(long long nel, const double* rho, const double* a,
                           const double* dv, double move, double target, double* scal,
                           double* partials, unsigned* counter, cudaStream_t s) {
  k_oc_step<<<RED_BLOCKS, RED_THREADS, 0, s>>>(nel, rho, a, dv, move, target, scal, partials,
                                               counter);
  return cudaGetLastError();
}

static int oc_blocks(long long nel) {
  return (int)std::min<long long>((nel + 2 * OC_T - 1) / (2 * OC_T), OC_BLOCKS);
}

cudaError_t launch_oc_prep_d(long long nel, const double* rho, const double* dc,
                             const double* dv, double move, double target, double* a64, void* a2,
                             void* lo2, void* hi2, void* dv2, double* scal, double* partials,
                             unsigned* counter, cudaStream_t s, double eta) {
  k_oc_prep_d<<<oc_blocks(nel), OC_T, 0, s>>>(nel, rho, dc, dv, move, target, a64, (float2*)a2,
                                              (float2*)lo2, (float2*)hi2, (float2*)dv2, scal, eta,
                                              partials, counter);
  return cudaGetLastError();
}

// resident blocks of a cooperative k_oc_rest, and whether the device takes a
// cluster of OC_CLUSTER (queried at set-up, outside any stream capture)
struct OcShape {
  int slots;
  bool cluster;
};
static OcShape oc_shape() {
  static OcShape cache[64] = {};
  int dev = 0, sms = 0, per_sm = 0, clusters = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (cache[dev].slots > 0) return cache[dev];
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_oc_rest, OC_T, 0) != cudaSuccess ||
      sms <= 0 || per_sm <= 0)
    return {1, false};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(OC_CLUSTER);
  cfg.blockDim = dim3(OC_T);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = OC_CLUSTER;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const bool ok =
      cudaFuncSetAttribute(k_oc_rest, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&clusters, k_oc_rest, &cfg) == cudaSuccess && clusters > 0;
  (void)cudaGetLastError();
  return cache[dev] = {sms * per_sm, ok};
}

void oc_prepare() { oc_shape(); }

cudaError_t launch_oc_search(long long nel, const void* a2, const void* lo2, const void* hi2,
                             const void* dv2, double target, double* scal, double* partials,
                             unsigned* counter, unsigned* turn, int* status, cudaStream_t s,
                             double eta) {
  const OcFields f = {(const float4*)a2, (const float4*)lo2, (const float4*)hi2, (const float4*)dv2};
  const int blocks = oc_blocks(nel);
  cudaError_t e = cudaSuccess;
  for (int q = 0; q < OC_SWEEPS && e == cudaSuccess; ++q)
    e = launch_pdl(k_oc_sweep, dim3(blocks), dim3(OC_T), 0, s, nel, f, target, scal, partials, counter,
                   eta);
  if (e != cudaSuccess) return e;
  // The rest by one cluster up to 128 x 64 x 64 elements, else by the whole grid:
  // cooperative launches in concurrent branches cost a batch of four served grids 20
  // of 390 us.  Update with the target on a plateau of the volume, the rest by one
  // block / so: 765 / 282 us at 48 x 24 x 24, 607 / 508 at 96 x 48 x 48 (430 by the
  // whole grid), 39800 / 660 at 192 x 96 x 96, 217000 / 1910 at 320 x 160 x 160.
  const OcShape sh = oc_shape();
  const bool small = sh.cluster && nel <= 1 << 19;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(small ? OC_CLUSTER : std::min(blocks, sh.slots));
  cfg.blockDim = dim3(OC_T);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  cfg.attrs = at;
  cfg.numAttrs = small ? 2 : 1;
  if (small) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = OC_CLUSTER;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  return cudaLaunchKernelEx(&cfg, k_oc_rest, nel, f, target, (volatile double*)scal, partials, counter,
                            (volatile unsigned*)turn, status, eta);
}

cudaError_t launch_oc_final(long long nel, double* rho, const double* a, double move,
                            double* scal, double* change_dev, double* partials,
                            unsigned* counter, cudaStream_t s, double eta) {
  k_oc_final<<<RED_BLOCKS, RED_THREADS, 0, s>>>(nel, rho, a, move, scal, change_dev, partials,
                                                counter, eta);
  return cudaGetLastError();
}

}  // namespace topo
