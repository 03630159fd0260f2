// Finest-grid hex8 operator of the float64 path with the element arithmetic
// in 64-bit fixed point (fxmath.cuh): float64 in, float64 out, the FP64 pipe
// left with the conversions of an element's 24 results, the nodal sums and
// the epilogue (~50 instructions per element instead of ~240).
//
// Same structure as k_apply3_col: a thread owns one element column and
// streams it up in z (a face is converted once and serves the element below
// and the element above), a block covers 16 x 8 columns and owns the 15 x 7
// nodes whose four columns it computes, and the column partials of an owned
// node are summed in shared memory in a fixed order.  An element's result
// depends on its own inputs alone, so tiles and chunks do not change bits.
//
// Bound by instruction issue and the FP64 pipe together (at 96 x 48 x 48, two
// blocks per SM: issue 41 %, FP64 47 %, ALU 38 %); three blocks per SM (168
// registers) gain 8 to 20 %, four nothing more.  K x with float64 arithmetic / in
// fixed point: 53 / 18.0 us at 48 x 24 x 24, 156 / 62 us at 96 x 48 x 48, 1115 /
// 329 us at 192 x 96 x 96.  (Of that 1.3, 5 and 18 us scale the components and the
// strain modes; with one exponent for a whole face a component far smaller than
// another lost its bits.)
#include "fxmath.cuh"
#include "kernels.h"

namespace topo {
namespace {

constexpr int FX_X = 16, FX_Y = 8, FX_OX = FX_X - 1, FX_OY = FX_Y - 1;

template <int EPI>
__global__ void __launch_bounds__(FX_X * FX_Y, 3)
    k_apply3_fx(GridP g, const uint8_t* __restrict__ mask, FxBlocks kb,
                const double* __restrict__ coef, int zc, const double* __restrict__ x,
                double* __restrict__ y, const double* __restrict__ b,
                const double* __restrict__ dinv, double omega, double dfix, bool clean) {
  __shared__ double part[2][4][FX_Y][FX_X][3];
  pdl_wait();
  const int tx = threadIdx.x % FX_X, ty = threadIdx.x / FX_X;
  const int x0 = blockIdx.x * FX_OX, y0 = blockIdx.y * FX_OY;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, g.nnz);
  const int ex = x0 - 1 + tx, ey = y0 - 1 + ty;
  const bool col_ok = ex >= 0 && ex < g.nx && ey >= 0 && ey < g.ny;
  const long long plane = (long long)g.nnx * g.nny;
  // the raw values of the next top face are requested before the current
  // element is computed (clean: x is zero on every fixed DOF already)
  double raw[4][3];
  auto load_face = [&](int kz) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = ex + (q & 1), j = ey + (q >> 1);
      const bool in = col_ok && kz >= 0 && kz < g.nnz;
      const long long nd = i + (long long)g.nnx * j + plane * kz;
      const unsigned m = in ? (clean ? 0u : (unsigned)mask[nd]) : 7u;
#pragma unroll
      for (int c = 0; c < 3; ++c) raw[q][c] = ((m >> c) & 1u) ? 0.0 : x[3 * nd + c];
    }
  };
  FxFace fb, ft;
  load_face(z0 - 1);
  fx_face(raw, fb);
  load_face(z0);
  double acc[4][3];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[q][c] = 0.0;
  const bool own = tx < FX_OX && ty < FX_OY && x0 + tx < g.nnx && y0 + ty < g.nny;
  int buf = 0;
  for (int ez = z0 - 1; ez < z1; ++ez) {
    fx_face(raw, ft);
    if (ez + 2 <= z1) load_face(ez + 2);
    double ye[8][3];
    if (col_ok && ez >= 0 && ez < g.nz) {
      fx_element(kb, coef[ex + (long long)g.nx * (ey + (long long)g.ny * ez)], fb, ft, ye);
    } else {
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) ye[a][c] = 0.0;
    }
    fb = ft;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        part[buf][q][ty][tx][c] = acc[q][c] + ye[q][c];
        acc[q][c] = ye[q + 4][c];
      }
    __syncthreads();
    if (own && ez >= z0) {
      const long long nd = (x0 + tx) + (long long)g.nnx * (y0 + ty) + plane * ez;
      const unsigned m = mask[nd];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double s = ((part[buf][3][ty][tx][c] + part[buf][2][ty][tx + 1][c]) +
                          part[buf][1][ty + 1][tx][c]) + part[buf][0][ty + 1][tx + 1][c];
        const long long d = 3 * nd + c;
        const double Ax = ((m >> c) & 1u) ? dfix * x[d] : s;
        if (EPI == EPI_APPLY)
          y[d] = Ax;
        else if (EPI == EPI_RESID)
          y[d] = b[d] - Ax;
        else
          y[d] = x[d] + omega * dinv[d] * (b[d] - Ax);
      }
    }
    buf ^= 1;
  }
  pdl_launch_dependents();
}

// resident blocks of the device (cached per device; queried at set-up,
// outside any stream capture)
template <int EPI>
long long fx_slots() {
  static long long cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (cache[dev] > 0) return cache[dev];
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_apply3_fx<EPI>, FX_X * FX_Y, 0) !=
          cudaSuccess ||
      sms <= 0 || per_sm <= 0)
    return 2 * 152;
  cache[dev] = (long long)sms * per_sm;
  return cache[dev];
}

template <int EPI>
cudaError_t run_fx(const ApplyArgs& a, cudaStream_t s) {
  const int gx = (a.g.nnx + FX_OX - 1) / FX_OX, gy = (a.g.nny + FX_OY - 1) / FX_OY;
  // z-chunk: each chunk recomputes one element layer, so the length that
  // minimises waves x (layers + 1); the shortest such one
  const long long slots = fx_slots<EPI>();
  int zc = 1;
  long long best = -1;
  for (int c = 1; c <= a.g.nnz; ++c) {
    const long long blocks = (long long)gx * gy * ((a.g.nnz + c - 1) / c);
    const long long cost = ((blocks + slots - 1) / slots) * (c + 1);
    if (best < 0 || cost < best) {
      best = cost;
      zc = c;
    }
  }
  if (a.zsplit > 0) zc = min(a.zsplit, (int)a.g.nnz);   // chosen by the autotuner
  return launch_pdl(k_apply3_fx<EPI>, dim3(gx, gy, (a.g.nnz + zc - 1) / zc), dim3(FX_X * FX_Y), 0,
                    s, a.g, a.mask, *a.fx,
                    static_cast<const double*>(a.coef), zc, static_cast<const double*>(a.x),
                    static_cast<double*>(a.y), static_cast<const double*>(a.b),
                    static_cast<const double*>(a.dinv), a.omega, a.dfix, a.clean_inputs);
}

}  // namespace

void fx_prepare() {
  fx_slots<EPI_APPLY>();
  fx_slots<EPI_RESID>();
  fx_slots<EPI_SMOOTH>();
}

bool make_fx_blocks(const double* wht64, FxBlocks* out) {
  *out = fx_blocks(wht64);
  return fx_blocks_ok(wht64);
}

bool fx_apply_ok(const ApplyArgs& a) {
  return a.dim == 3 && !a.expl && !a.gal1 && a.fx != nullptr && a.tc == T_F64 &&
         a.tx == T_F64 && a.ty == T_F64;
}

cudaError_t launch_apply_fx(const ApplyArgs& a, cudaStream_t s) {
  switch (a.epi) {
    case EPI_APPLY: return run_fx<EPI_APPLY>(a, s);
    case EPI_RESID: return run_fx<EPI_RESID>(a, s);
    default: return run_fx<EPI_SMOOTH>(a, s);
  }
}

}  // namespace topo
