// Float64-accurate hex8 stiffness operator in double-float arithmetic.
//
// GB300 runs float64 at 1/128 of the float32 rate, so a float64 transform is
// bound by the FP64 pipe.  Here every value is an unevaluated sum hi + lo of two
// floats (48-bit significand) and all arithmetic runs on the FP32 pipe with
// error-free transformations (TwoSum, FMA-based TwoProduct).  float64 inputs
// are split into (hi, lo) and results widened back with integer bit
// operations, so the FP64 pipe only sees the final additions of the
// epilogue.  The structure (element columns streamed in z, owner-computes
// node sums in shared memory, Walsh blocks) is that of k_apply3_col.
#include <algorithm>
#include <type_traits>

#include "dfmath.cuh"
#include "kernels.h"

namespace topo {

// 4-point Walsh-Hadamard transform in place (self-inverse up to the factor 4)
__device__ __forceinline__ void wht4_df(dfl (&v)[4]) {
  const dfl s0 = df_add(v[0], v[1]), d0 = df_add(v[0], df_neg(v[1]));
  const dfl s1 = df_add(v[2], v[3]), d1 = df_add(v[2], df_neg(v[3]));
  v[0] = df_add(s0, s1);
  v[1] = df_add(d0, d1);
  v[2] = df_add(s0, df_neg(s1));
  v[3] = df_add(d0, df_neg(d1));
}

struct DfBlocks {
  float h[8][3][3], l[8][3][3];
};

constexpr int DX = 16, DY = 8, DOX = DX - 1, DOY = DY - 1;

// S: storage of x, b and y -- float64 (split on load, widened on store) or
// double-float pairs float2 (used as they are)
template <int EPI, typename S>
__global__ void __launch_bounds__(DX * DY)
    k_apply3_df(GridP g, const uint8_t* __restrict__ mask, DfBlocks kb,
                const double* __restrict__ coef, int zc, const S* __restrict__ x,
                S* __restrict__ y, const S* __restrict__ b, double dfix) {
  __shared__ dfl part[2][4][DY][DX][3];
  const int tx = threadIdx.x % DX, ty = threadIdx.x / DX;
  const int x0 = blockIdx.x * DOX, y0 = blockIdx.y * DOY;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, g.nnz);
  const int ex = x0 - 1 + tx, ey = y0 - 1 + ty;
  const bool col_ok = ex >= 0 && ex < g.nx && ey >= 0 && ey < g.ny;
  const long long plane = (long long)g.nnx * g.nny;

  // The transform is separable: a face's xy part is formed once and serves the
  // element below and the one above, and the two elements' contributions to
  // a face are added in the xy-Walsh domain and transformed back once (108
  // double-float additions per element instead of 156): K x of pairs 243 -> 195
  // us at 192 x 96 x 96, three blocks per SM (163 registers).  Staging the
  // faces in shared memory instead of four loads per node measured 203 us, two
  // blocks per SM with more values in flight 248 us.
  dfl Wb[3][4], Wt[3][4], Up[3][4];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int t = 0; t < 4; ++t) Up[c][t] = {0.f, 0.f};

  auto load_face = [&](int kz, dfl (&W)[3][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = ex + (q & 1), j = ey + (q >> 1);
      if (col_ok && kz >= 0 && kz < g.nnz) {
        const long long nd = i + (long long)g.nnx * j + plane * kz;
        const unsigned m = mask[nd];
#pragma unroll
        for (int c = 0; c < 3; ++c)
          W[c][q] = ((m >> c) & 1u) ? dfl{0.f, 0.f} : ld_df(x, 3 * nd + c);
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) W[c][q] = {0.f, 0.f};
      }
    }
  };

  load_face(z0 - 1, Wb);
#pragma unroll
  for (int c = 0; c < 3; ++c) wht4_df(Wb[c]);
  const bool own = tx < DOX && ty < DOY && (x0 + tx) < g.nnx && (y0 + ty) < g.nny;
  int buf = 0;
  for (int ez = z0 - 1; ez < z1; ++ez) {
    load_face(ez + 1, Wt);
#pragma unroll
    for (int c = 0; c < 3; ++c) wht4_df(Wt[c]);
    dfl X[3][8];
    if (col_ok && ez >= 0 && ez < g.nz) {
      const dfl ce = split_d(coef[ex + (long long)g.nx * (ey + (long long)g.ny * ez)]);
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          X[c][t] = df_add(Wb[c][t], Wt[c][t]);
          X[c][t + 4] = df_add(Wb[c][t], df_neg(Wt[c][t]));
        }
      // block tau couples X[c][tau xor e_c], c = 0..2, in place
#pragma unroll
      for (int tau = 0; tau < 8; ++tau) {
        dfl zt[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) zt[c] = df_mul(ce, X[c][tau ^ (1 << c)]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          dfl s = {0.f, 0.f};
          bool first = true;
#pragma unroll
          for (int cp = 0; cp < 3; ++cp) {
            if (wht_zero(tau, c, cp)) continue;
            const dfl t = df_mul(dfl{kb.h[tau][c][cp], kb.l[tau][c][cp]}, zt[cp]);
            s = first ? t : df_add(s, t);
            first = false;
          }
          X[c][tau ^ (1 << c)] = s;
        }
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int t = 0; t < 8; ++t) X[c][t] = {0.f, 0.f};
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      dfl acc[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        acc[t] = df_add(Up[c][t], df_add(X[c][t], X[c][t + 4]));
        Up[c][t] = df_add(X[c][t], df_neg(X[c][t + 4]));
        Wb[c][t] = Wt[c][t];
      }
      wht4_df(acc);
#pragma unroll
      for (int q = 0; q < 4; ++q) part[buf][q][ty][tx][c] = acc[q];
    }
    __syncthreads();
    if (own && ez >= z0) {
      const long long nd = (x0 + tx) + (long long)g.nnx * (y0 + ty) + plane * ez;
      const unsigned m = mask[nd];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const dfl s = df_add(df_add(df_add(part[buf][3][ty][tx][c], part[buf][2][ty][tx + 1][c]),
                                    part[buf][1][ty + 1][tx][c]),
                             part[buf][0][ty + 1][tx + 1][c]);
        const long long d = 3 * nd + c;
        if constexpr (std::is_same<S, double>::value) {
          if ((m >> c) & 1u) {
            const double Ax = dfix * x[d];
            y[d] = EPI == EPI_RESID ? b[d] - Ax : Ax;
          } else if (EPI == EPI_RESID) {
            // b and K x nearly cancel near convergence: subtract the leading
            // part first (exact when close), then the trailing part
            y[d] = (b[d] - f2d(s.h)) - f2d(s.l);
          } else {
            y[d] = f2d(s.h) + f2d(s.l);
          }
        } else {
          // dfix is 0 or 1, so dfix * x is exact in the pair format
          const dfl Ax = ((m >> c) & 1u) ? (dfix != 0.0 ? ld_df(x, d) : dfl{0.f, 0.f}) : s;
          st_df(y, d, EPI == EPI_RESID ? df_add(ld_df(b, d), df_neg(Ax)) : Ax);
        }
      }
    }
    buf ^= 1;
  }
}

// ---------------------------------------------------------------------------
// 2D: q = K p of the mixed CG with p in pairs, in double-float arithmetic,
// rounded to float32 at the end, and p . q of that q.  On a smooth direction
// K p is smaller than K's entries times p by (element size / wave length)^2,
// 2e-6 on a 640-element span, so the float32 product of p rounded to float32
// (6e-8) is off by percents there and the CG takes up to twice the iterations.
// One thread per node gathers its nine nodes (16 bytes each) and forms its two
// rows of the four elements around it, each row a Dot2 sum.  About 950 FP32
// instructions per node; the direction is zero on the fixed DOFs (a fixed row's
// product is 0).  Twelve solves at 640 x 320 to 1e-6: 1001 iterations in 129 ms
// with the float32 product, 730 in 74 ms with this one (float64: 726); at
// 320 x 160 614 in 67 ms and 307 in 24 ms.
// ---------------------------------------------------------------------------
struct DfKe2 {
  float2 v[8][8];
};
constexpr int D2_T = 256, D2_BLOCKS = 8 * 152;

__global__ void __launch_bounds__(D2_T)
    k_cg_q2_df(GridP g, const uint8_t* __restrict__ mask, DfKe2 ke,
               const double* __restrict__ coef, const float2* __restrict__ p,
               float* __restrict__ q, Springs sp, double* partials, unsigned* counter,
               double* pq) {
  __shared__ double sh[1][D2_T / 32], tot[1];
  pdl_wait();
  dfl dot[1] = {{0.f, 0.f}};
  for (long long node = (long long)blockIdx.x * D2_T + threadIdx.x; node < g.nn;
       node += (long long)gridDim.x * D2_T) {
    const int i = (int)(node % g.nnx), j = (int)(node / g.nnx);
    // clamped neighbours: outside the grid their elements' moduli are 0
    float4 x[3][3];
    dfl E[2][2];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int ii = min(max(i + a - 1, 0), g.nnx - 1), jj = min(max(j + b - 1, 0), g.nny - 1);
        x[b][a] = reinterpret_cast<const float4*>(p)[ii + (long long)g.nnx * jj];
      }
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int ei = i - 1 + a, ej = j - 1 + b;
        const bool in = ei >= 0 && ei < g.nx && ej >= 0 && ej < g.ny;
        E[b][a] = in ? split_d(coef[ei + (long long)g.nx * ej]) : dfl{0.f, 0.f};
      }
    dfl acc[2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int corner = (1 - a) + 2 * (1 - b);   // of this node in element (a, b)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          dfl s = {0.f, 0.f};
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const float4 u = x[b + (m >> 1)][a + (m & 1)];
            const float2 k0 = ke.v[2 * corner + c][2 * m], k1 = ke.v[2 * corner + c][2 * m + 1];
            df_dot_acc(s, {k0.x, k0.y}, {u.x, u.y});
            df_dot_acc(s, {k1.x, k1.y}, {u.z, u.w});
          }
          acc[c] = df_fma(E[b][a], df_norm(s), acc[c]);
        }
      }
    const unsigned m = mask[node];
    const dfl own[2] = {{x[1][1].x, x[1][1].y}, {x[1][1].z, x[1][1].w}};
    float out[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      for (int t = 0; t < sp.n; ++t)
        if (sp.dof[t] == 2 * node + c) acc[c] = df_fma(split_d(sp.k[t]), own[c], acc[c]);
      out[c] = ((m >> c) & 1u) ? 0.f : __fadd_rn(acc[c].h, acc[c].l);
      df_dot_acc(dot[0], own[c], {out[c], 0.f});
    }
    reinterpret_cast<float2*>(q)[node] = make_float2(out[0], out[1]);
  }
  pdl_launch_dependents();
  dot[0] = df_norm(dot[0]);
  if (grid_sum_df(dot, sh, tot, partials, counter) && threadIdx.x == 0) *pq = tot[0];
}

cudaError_t launch_cg_q2_df(const GridP& g, const uint8_t* mask, const double* ke64,
                            const double* coef, const void* p, float* q, const Springs& sp,
                            double* partials, unsigned* counter, double* pq, cudaStream_t s) {
  DfKe2 ke;
  for (int e = 0; e < 64; ++e) {
    const float h = (float)ke64[e];
    (&ke.v[0][0])[e] = make_float2(h, (float)(ke64[e] - (double)h));
  }
  const int blocks = std::min(nblocks(g.nn, D2_T), D2_BLOCKS);
  return launch_pdl(k_cg_q2_df, dim3(blocks), dim3(D2_T), 0, s, g, mask, ke, coef, (const float2*)p,
                    q, sp, partials, counter, pq);
}

bool df_blocks_ok(const double* wht64) {
  double mx = 0.0;
  for (int q = 0; q < 72; ++q) mx = fmax(mx, fabs(wht64[q]));
  for (int tau = 0; tau < 8; ++tau)
    for (int c = 0; c < 3; ++c)
      for (int cp = 0; cp < 3; ++cp)
        if (wht_zero(tau, c, cp) && fabs(wht64[(tau * 3 + c) * 3 + cp]) > 1e-14 * mx) return false;
  return true;
}

// resident blocks of the pair-storage double-float kernel (cached per device;
// queried at set-up, outside any stream capture)
template <int EPI>
static long long df_slots() {
  static long long cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (cache[dev] > 0) return cache[dev];
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_apply3_df<EPI, float2>, DX * DY, 0) !=
          cudaSuccess ||
      sms <= 0 || per_sm <= 0)
    return 0;
  cache[dev] = (long long)sms * per_sm;
  return cache[dev];
}

void df_prepare() {
  df_slots<EPI_APPLY>();
  df_slots<EPI_RESID>();
}

template <typename S>
static void run_df(const ApplyArgs& a, const DfBlocks& kb, dim3 grid, int zc, cudaStream_t s) {
  if (a.epi == EPI_RESID)
    k_apply3_df<EPI_RESID, S><<<grid, DX * DY, 0, s>>>(
        a.g, a.mask, kb, static_cast<const double*>(a.coef), zc, static_cast<const S*>(a.x),
        static_cast<S*>(a.y), static_cast<const S*>(a.b), a.dfix);
  else
    k_apply3_df<EPI_APPLY, S><<<grid, DX * DY, 0, s>>>(
        a.g, a.mask, kb, static_cast<const double*>(a.coef), zc, static_cast<const S*>(a.x),
        static_cast<S*>(a.y), static_cast<const S*>(a.b), a.dfix);
}

cudaError_t launch_apply_df(const ApplyArgs& a, cudaStream_t s) {
  if (a.dim != 3 || a.expl || a.gal1 || a.tx != a.ty || (a.tx != T_F64 && a.tx != T_D2) ||
      !a.wht || a.epi == EPI_SMOOTH || (a.tx == T_D2 && a.dfix != 0.0 && a.dfix != 1.0))
    return cudaErrorInvalidValue;
  if (a.g.nn <= 0) return cudaSuccess;
  const double* w = static_cast<const double*>(a.wht);
  DfBlocks kb;
  for (int q = 0; q < 72; ++q) {
    const float h = (float)w[q];
    (&kb.h[0][0][0])[q] = h;
    (&kb.l[0][0][0])[q] = (float)(w[q] - (double)h);
  }
  const int gx = (a.g.nnx + DOX - 1) / DOX, gy = (a.g.nny + DOY - 1) / DOY;
  int zc = 16;
  while (zc > 2 && (long long)gx * gy * ((a.g.nnz + zc - 1) / zc) < 2 * 152) zc /= 2;
  // pair storage (the mixed path's accurate products): the chunk length
  // minimising waves x (layers + 1 recomputed) for the queried occupancy
  const long long slots =
      a.tx == T_D2 ? (a.epi == EPI_RESID ? df_slots<EPI_RESID>() : df_slots<EPI_APPLY>()) : 0;
  if (slots > 0) {
    long long best = -1;
    for (int c = 1; c <= a.g.nnz; ++c) {
      const long long blocks = (long long)gx * gy * ((a.g.nnz + c - 1) / c);
      const long long cost = ((blocks + slots - 1) / slots) * (c + 1);
      if (best < 0 || cost < best) {
        best = cost;
        zc = c;
      }
    }
  }
  if (a.zsplit > 0) zc = min(a.zsplit, (int)a.g.nnz);   // chosen by the autotuner
  dim3 grid(gx, gy, (a.g.nnz + zc - 1) / zc);
  if (a.tx == T_D2)
    run_df<float2>(a, kb, grid, zc, s);
  else
    run_df<double>(a, kb, grid, zc, s);
  return cudaGetLastError();
}

}  // namespace topo
