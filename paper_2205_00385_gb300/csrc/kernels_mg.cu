// Multigrid pieces of Algorithm 2: restriction P^T, interpolation P, Jacobi
// smoothing from a zero guess, the Galerkin coarse operators P^T K P as
// per-coarse-element matrices, and the exact coarsest-grid solve.
//
// With 2x coarsening and multilinear P, the fine elements inside one coarse
// element interpolate only from that coarse element's nodes, so P^T K P is
// again element-by-element on the coarse grid with element matrices
//   Kc_E = sum_children P_c^T Ke_child P_c,
// where P_c = W_c (x) I_dim and W_c[a][A] is the product over axes of the
// linear weights of fine corner a of child c at coarse corner A.
#include <math.h>

#include "dfmath.cuh"
#include "kernels.h"
#include "mg_device.cuh"

namespace topo {

// ---------------------------------------------------------------------------
// Restriction and interpolation.  Each value sums its terms in the order of
// restrict_finish / prolong_pair (mg_device.cuh), whose per-node bodies the
// fused coarse V-cycle runs, so the bits are the same.  The restriction
// runs one thread per coarse value: consecutive threads take consecutive
// values of one coarse plane (its rows flattened), so a warp's fine loads
// span few sectors and a thread holds only its 27 terms (more threads in
// flight than one per node, which pays on the small levels).
// ---------------------------------------------------------------------------
constexpr int TVAL = 256;

// r_f is +-0 on every fixed DOF (the cycle's input is cleared there), so the
// fine masks are not loaded: a fixed term then adds w * (+-0) where
// restrict_finish adds +0, and a running sum that starts at +0 is never -0,
// so the bits are the same.
template <int DIM, typename T>
__global__ void __launch_bounds__(TVAL)
    k_restrict(GridP gf, GridP gc, const uint8_t* __restrict__ maskc, const T* __restrict__ rf,
               T* __restrict__ bc, const T* __restrict__ dinvc, T omega, T* __restrict__ zc) {
  constexpr int NZ = DIM == 3 ? 3 : 1;
  const int rowv = DIM * gc.nnx;
  const int pv = blockIdx.x * TVAL + threadIdx.x;
  const int K = DIM == 3 ? (int)blockIdx.y : 0;
  pdl_wait();
  if (pv >= rowv * gc.nny) return;
  const int J = pv / rowv, v = pv - J * rowv;
  const int I = v / DIM, c = v - I * DIM;
  T x[NZ][3][3];
#pragma unroll
  for (int a = 0; a < NZ; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int i = min(max(2 * I + q - 1, 0), gf.nnx - 1);
        const int j = min(max(2 * J + b - 1, 0), gf.nny - 1);
        const int k = DIM == 3 ? min(max(2 * K + a - 1, 0), gf.nnz - 1) : 0;
        x[a][b][q] = rf[DIM * (i + (long long)gf.nnx * (j + (long long)gf.nny * k)) + c];
      }
  T acc = T(0);
#pragma unroll
  for (int a = 0; a < NZ; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int dx = q - 1, dy = b - 1, dz = DIM == 3 ? a - 1 : 0;
        const int i = 2 * I + dx, j = 2 * J + dy, k = 2 * K + dz;
        bool in = i >= 0 && i < gf.nnx && j >= 0 && j < gf.nny;
        if (DIM == 3) in = in && k >= 0 && k < gf.nnz;
        const T w = T((dx ? 0.5 : 1.0) * (dy ? 0.5 : 1.0) * (dz ? 0.5 : 1.0));
        acc = fma(w, in ? x[a][b][q] : T(0), acc);
      }
  const long long node = I + (long long)gc.nnx * (J + (long long)gc.nny * K);
  const long long d = DIM * node + c;
  const T bv = ((maskc[node] >> c) & 1u) ? T(0) : acc;
  bc[d] = bv;
  if (zc) zc[d] = mul_rn(mul_rn(omega, dinvc[d]), bv);
  pdl_launch_dependents();
}

// z_f += Pm z_c: threads on the fine (i, j) grid, each taking the fine nodes
// k = 2q and 2q+1 (3D), which share the coarse plane q (index work shared by
// six values; one thread per value measured 2.5x slower at the finest level).
constexpr int TBX = 32, TBY = 4;

template <typename T>
__host__ __device__ constexpr int transfer_min_blocks() {
  return sizeof(T) == 4 ? 4 : 2;   // registers for all loads in flight
}

template <int DIM, typename T>
__global__ void __launch_bounds__(TBX * TBY, transfer_min_blocks<T>())
    k_prolong_add(GridP gf, const uint8_t* __restrict__ maskf, GridP gc,
                  const T* __restrict__ zc, T* __restrict__ zf) {
  const int i = blockIdx.x * TBX + threadIdx.x, j = blockIdx.y * TBY + threadIdx.y;
  const int q = DIM == 3 ? (int)blockIdx.z : 0;
  pdl_wait();
  if (i >= gf.nnx || j >= gf.nny) return;
  prolong_pair<DIM, T, false>(gf, maskf, gc, zc, zf, i, j, q);
  pdl_launch_dependents();
}

// Element-wise passes: EW_U values per thread, a block's width apart, all
// requested before any is used (one per thread left 24 and 16 us of a V-cycle
// at 192 x 96 x 96 to these two passes).
constexpr int EW_T = 256, EW_U = 4;

// bout = bin and z = omega D^-1 bin (smoothing from a zero guess); with a node
// mask (DIM > 0) the input is taken as zero on the fixed DOFs.
template <int DIM, typename T, typename TIN>
__global__ void __launch_bounds__(EW_T)
    k_presmooth(long long n, const TIN* __restrict__ bin, T* __restrict__ bout,
                const T* __restrict__ dinv, T omega, T* __restrict__ z,
                const uint8_t* __restrict__ mask) {
  const long long q0 = (long long)blockIdx.x * EW_T * EW_U + threadIdx.x;
  pdl_wait();
  TIN bv[EW_U];
  T dv[EW_U];
  bool fx[EW_U];
#pragma unroll
  for (int u = 0; u < EW_U; ++u) {
    const long long q = q0 + u * EW_T;
    if (q >= n) continue;
    bv[u] = bin[q];
    dv[u] = dinv[q];
    fx[u] = DIM > 0 && ((mask[q / (DIM > 0 ? DIM : 1)] >> (int)(q % (DIM > 0 ? DIM : 1))) & 1u);
  }
#pragma unroll
  for (int u = 0; u < EW_U; ++u) {
    const long long q = q0 + u * EW_T;
    if (q >= n) continue;
    const T v = DIM > 0 && fx[u] ? T(0) : cvt<T>(bv[u]);
    bout[q] = v;
    z[q] = omega * dv[u] * v;
  }
  pdl_launch_dependents();
}

// Float64 result of a float32 V-cycle: on a fixed DOF, where the operator is the
// identity, two smoothing steps of the input; elsewhere zin.
template <int DIM>
__global__ void __launch_bounds__(EW_T)
    k_vcycle_out(long long n, const float* __restrict__ zin, const double* __restrict__ r,
                 float omega, const uint8_t* __restrict__ mask, double* __restrict__ out) {
  const long long q0 = (long long)blockIdx.x * EW_T * EW_U + threadIdx.x;
  pdl_wait();
  float zv[EW_U];
  bool fx[EW_U];
#pragma unroll
  for (int u = 0; u < EW_U; ++u) {
    const long long q = q0 + u * EW_T;
    if (q >= n) continue;
    fx[u] = (mask[q / DIM] >> (int)(q % DIM)) & 1u;
    zv[u] = zin[q];
  }
#pragma unroll
  for (int u = 0; u < EW_U; ++u) {
    const long long q = q0 + u * EW_T;
    if (q >= n) continue;
    if (fx[u]) {
      const float b = (float)r[q], z = omega * b;
      zv[u] = z + omega * (b - z);
    }
    out[q] = (double)zv[u];
  }
}

// The same where out already holds the free DOFs (the float64 cycle): four mask
// bytes per thread, and nothing else is read where no DOF is fixed.  Bound by
// launch latency: a V-cycle call at 96x48x48 took 298 us with a thread per DOF
// here, 296 so.
template <int DIM>
__global__ void __launch_bounds__(EW_T)
    k_vcycle_fixed(long long nn, const double* __restrict__ r, double omega,
                   const uint8_t* __restrict__ mask, double* __restrict__ out) {
  const long long b0 = 4 * ((long long)blockIdx.x * EW_T + threadIdx.x);
  uint8_t m[4] = {0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (b0 + k < nn) m[k] = mask[b0 + k];
  pdl_wait();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!m[k]) continue;
    for (int c = 0; c < DIM; ++c) {
      const long long q = (b0 + k) * DIM + c;
      if (!((m[k] >> c) & 1u)) continue;
      const double b = r[q], z = omega * b;
      out[q] = z + omega * (b - z);
    }
  }
}

template <typename TIN, typename TOUT, int U>
__global__ void __launch_bounds__(EW_T)
    k_convert(long long n, const TIN* __restrict__ in, TOUT* __restrict__ out) {
  const long long q0 = (long long)blockIdx.x * EW_T * U + threadIdx.x;
  TIN v[U];
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (q0 + u * EW_T < n) v[u] = in[q0 + u * EW_T];
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (q0 + u * EW_T < n) out[q0 + u * EW_T] = cvt<TOUT>(v[u]);
}

// ---------------------------------------------------------------------------
// Galerkin level 1 from the finest grid: Kc_E = sum_c coef_child(E,c) Q_c,
// Q_c = P_c^T KE P_c (precomputed).  One thread per (entry, coarse element).
// ---------------------------------------------------------------------------
template <int DIM, typename T>
__global__ void __launch_bounds__(256)
    k_galerkin_fine(GridP gc, GridP gf, const T* __restrict__ coef, const T* __restrict__ Qc,
                    T* __restrict__ Kc) {
  constexpr int ND = Geo<DIM>::ND, NPE = Geo<DIM>::NPE, NT = tri_len(ND);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= gc.nel * NT) return;
  const long long E = t / NT;
  const int pk = (int)(t % NT);
  int r, cc;
  tri_rc(pk, ND, r, cc);
  const int entry = r * ND + cc;
  const int EX = (int)(E % gc.nx);
  const long long rest = E / gc.nx;
  const int EY = (int)(rest % gc.ny);
  const int EZ = DIM == 3 ? (int)(rest / gc.ny) : 0;
  T acc = T(0);
#pragma unroll
  for (int c = 0; c < NPE; ++c) {
    const int fx = 2 * EX + (c & 1), fy = 2 * EY + ((c >> 1) & 1), fz = 2 * EZ + ((c >> 2) & 1);
    const long long fe = fx + (long long)gf.nx * (fy + (long long)gf.ny * (DIM == 3 ? fz : 0));
    acc += coef[fe] * Qc[c * ND * ND + entry];
  }
  Kc[(size_t)E * NT + pk] = acc;
}

// Level-1 diagonal without stored matrices (3D): node I of level 1 sums, over
// its coarse elements E and their children ch, E_child * diag(Q_ch) at I's
// corner a.  qd.v[(ch * 8 + a) * 3 + c] = Q_ch[(3a+c),(3a+c)].
template <typename T>
struct QDiagP {
  T v[8 * 8 * 3];
};

template <typename T>
__global__ void __launch_bounds__(256)
    k_diag_l1(GridP g1, GridP gf, const uint8_t* __restrict__ mask, QDiagP<T> qd,
              const T* __restrict__ coef, T* __restrict__ dinv) {
  const long long node = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (node >= g1.nn) return;
  const int i = (int)(node % g1.nnx);
  const long long rest = node / g1.nnx;
  const int j = (int)(rest % g1.nny);
  const int k = (int)(rest / g1.nny);
  T d[3] = {T(0), T(0), T(0)};
  for (int ez = 0; ez < 2; ++ez)
    for (int ey = 0; ey < 2; ++ey)
      for (int ex = 0; ex < 2; ++ex) {
        const int EX = i - 1 + ex, EY = j - 1 + ey, EZ = k - 1 + ez;
        if (EX < 0 || EX >= g1.nx || EY < 0 || EY >= g1.ny || EZ < 0 || EZ >= g1.nz) continue;
        const int a = (1 - ex) + 2 * (1 - ey) + 4 * (1 - ez);
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
          const long long fe = (2 * EX + (ch & 1)) +
                               (long long)gf.nx * ((2 * EY + ((ch >> 1) & 1)) +
                                                   (long long)gf.ny * (2 * EZ + ((ch >> 2) & 1)));
          const T e = coef[fe];
#pragma unroll
          for (int c = 0; c < 3; ++c) d[c] += e * qd.v[(ch * 8 + a) * 3 + c];
        }
      }
  const unsigned m = mask[node];
#pragma unroll
  for (int c = 0; c < 3; ++c) dinv[3 * node + c] = ((m >> c) & 1u) ? T(1) : T(1) / d[c];
}

// Level-2 element matrices straight from the finest moduli (3D): a level-2
// element covers 4x4x4 finest elements f, and
// Kc_E = sum_f E_f R_f with R_f = W_c1^T (W_c0^T KE W_c0) W_c1 for the
// finest element's position c0 inside its level-1 parent and that parent's
// position c1 inside E (64 precomputed tables, R[f * 576 + entry]).
template <typename T>
__global__ void __launch_bounds__(256)
    k_galerkin_l2(GridP g2, GridP gf, const T* __restrict__ coef, const T* __restrict__ R,
                  T* __restrict__ Kc) {
  constexpr int NT = tri_len(24);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= g2.nel * NT) return;
  const long long E = t / NT;
  const int pk = (int)(t % NT);
  int r, cc;
  tri_rc(pk, 24, r, cc);
  const int entry = r * 24 + cc;
  const int EX = (int)(E % g2.nx);
  const long long rest = E / g2.nx;
  const int EY = (int)(rest % g2.ny);
  const int EZ = (int)(rest / g2.ny);
  T acc = T(0);
#pragma unroll 8
  for (int f = 0; f < 64; ++f) {
    const int c1 = f >> 3, c0 = f & 7;
    const int fx = 4 * EX + 2 * (c1 & 1) + (c0 & 1);
    const int fy = 4 * EY + 2 * ((c1 >> 1) & 1) + ((c0 >> 1) & 1);
    const int fz = 4 * EZ + 2 * ((c1 >> 2) & 1) + ((c0 >> 2) & 1);
    acc += coef[fx + (long long)gf.nx * (fy + (long long)gf.ny * fz)] * R[f * 576 + entry];
  }
  Kc[(size_t)E * NT + pk] = acc;
}

// Galerkin level l+1 from stored level-l element matrices.  One block of
// ND*ND threads per coarse element; T = Kchild W in shared memory, then
// Kc += W^T T, summed over the 2^DIM children.  W_c[a][A], the weight of
// coarse corner A at fine corner a of child c, is the product over the axes
// of the linear weights (c + a) / 2 (A's bit set) or (2 - c - a) / 2 (per
// axis bits, positions in half coarse-element units); it is staged in shared
// memory from integer arithmetic, an integer over 2^DIM, exact in any
// floating type.
template <int DIM, typename T>
__global__ void __launch_bounds__(Geo<DIM>::ND * Geo<DIM>::ND)
    k_galerkin_coarse(GridP gc, GridP gf, const T* __restrict__ Kf, T* __restrict__ Kc) {
  constexpr int ND = Geo<DIM>::ND, NPE = Geo<DIM>::NPE, NT = tri_len(ND);
  __shared__ T sK[ND * ND];
  __shared__ T sT[ND * ND];
  __shared__ T sW[NPE * NPE * NPE];   // [child][fine corner][coarse corner]
  const long long E = blockIdx.x;
  const int tid = threadIdx.x;
  for (int q = tid; q < NPE * NPE * NPE; q += ND * ND) {
    const int c = q / (NPE * NPE), a = (q / NPE) % NPE, A = q % NPE;
    int num = 1;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const int p = ((c >> d) & 1) + ((a >> d) & 1);
      num *= ((A >> d) & 1) ? p : 2 - p;
    }
    sW[q] = T(num) / T(1 << DIM);
  }
  __syncthreads();
  const int EX = (int)(E % gc.nx);
  const long long rest = E / gc.nx;
  const int EY = (int)(rest % gc.ny);
  const int EZ = DIM == 3 ? (int)(rest / gc.ny) : 0;
  const int I = tid / ND, J = tid % ND;
  const int AI = I / DIM, ci = I % DIM, AJ = J / DIM, cj = J % DIM;
  T acc = T(0);
  for (int c = 0; c < NPE; ++c) {
    const int fx = 2 * EX + (c & 1), fy = 2 * EY + ((c >> 1) & 1), fz = 2 * EZ + ((c >> 2) & 1);
    const long long fe = fx + (long long)gf.nx * (fy + (long long)gf.ny * (DIM == 3 ? fz : 0));
    sK[tid] = Kf[(size_t)fe * NT + sym_idx(I, J, ND)];
    __syncthreads();
    // T[i][J] = sum_b K[i][(b, cj)] W_c[b][AJ]   (i = I here)
    T tv = T(0);
#pragma unroll
    for (int bcn = 0; bcn < NPE; ++bcn) tv += sK[I * ND + DIM * bcn + cj] * sW[(c * NPE + bcn) * NPE + AJ];
    sT[tid] = tv;
    __syncthreads();
    // acc[I][J] += sum_a W_c[a][AI] T[(a, ci)][J]
#pragma unroll
    for (int acn = 0; acn < NPE; ++acn) acc += sW[(c * NPE + acn) * NPE + AI] * sT[(DIM * acn + ci) * ND + J];
    __syncthreads();
  }
  if (J >= I) Kc[(size_t)E * NT + tri_idx(I, J, ND)] = acc;
}

// ---------------------------------------------------------------------------
// Coarsest grid: dense matrix with identity rows/columns at fixed DOFs.
// One thread per matrix entry, summing over the elements shared by both
// nodes (deterministic).  Row-major n x n.
// ---------------------------------------------------------------------------
template <int DIM, typename T, typename TA>
__global__ void __launch_bounds__(256)
    k_dense_assemble(GridP g, const uint8_t* __restrict__ mask, const T* __restrict__ Kc,
                     TA* __restrict__ A, double shift) {
  constexpr int ND = Geo<DIM>::ND;
  const long long n = DIM * g.nn;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const long long row = t / n, col = t % n;
  const long long nr = row / DIM, nc = col / DIM;
  const int cr = (int)(row % DIM), cc = (int)(col % DIM);
  const bool fr = (mask[nr] >> cr) & 1u, fc = (mask[nc] >> cc) & 1u;
  if (fr || fc) {
    A[t] = (row == col) ? TA(1) : TA(0);
    return;
  }
  const int ir = (int)(nr % g.nnx), jr = (int)((nr / g.nnx) % g.nny), kr = DIM == 3 ? (int)(nr / ((long long)g.nnx * g.nny)) : 0;
  const int ic = (int)(nc % g.nnx), jc = (int)((nc / g.nnx) % g.nny), kc = DIM == 3 ? (int)(nc / ((long long)g.nnx * g.nny)) : 0;
  TA s = TA(0);
  if (abs(ir - ic) <= 1 && abs(jr - jc) <= 1 && abs(kr - kc) <= 1) {
    const int exlo = max(max(ir, ic) - 1, 0), exhi = min(min(ir, ic), g.nx - 1);
    const int eylo = max(max(jr, jc) - 1, 0), eyhi = min(min(jr, jc), g.ny - 1);
    const int ezlo = DIM == 3 ? max(max(kr, kc) - 1, 0) : 0;
    const int ezhi = DIM == 3 ? min(min(kr, kc), g.nz - 1) : 0;
    for (int ez = ezlo; ez <= ezhi; ++ez)
      for (int ey = eylo; ey <= eyhi; ++ey)
        for (int ex = exlo; ex <= exhi; ++ex) {
          const long long e = ex + (long long)g.nx * (ey + (long long)g.ny * ez);
          const int ar = (ir - ex) + 2 * (jr - ey) + (DIM == 3 ? 4 * (kr - ez) : 0);
          const int ac = (ic - ex) + 2 * (jc - ey) + (DIM == 3 ? 4 * (kc - ez) : 0);
          s += (TA)Kc[(size_t)e * tri_len(ND) + sym_idx(DIM * ar + cr, DIM * ac + cc, ND)];
        }
  }
  A[t] = row == col ? (TA)((double)s * (1.0 + shift)) : s;
}

// y = A x with the matrix (and the accumulation) in TA and the vectors in TV
template <typename TA, typename TV>
__global__ void __launch_bounds__(256)
    k_gemv(int n, const TA* __restrict__ A, const TV* __restrict__ x, TV* __restrict__ y) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  pdl_wait();
  if (warp >= n) return;
  TA s = TA(0);
  for (int m = lane; m < n; m += 32) s += A[(size_t)warp * n + m] * (TA)x[m];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) y[warp] = (TV)s;
  pdl_launch_dependents();
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
template <int DIM, typename T>
static cudaError_t restrict_t(const GridP& gf, const GridP& gc, const uint8_t* mc, const void* rf,
                              void* bc, const void* dinvc, double omega, void* zc,
                              cudaStream_t s) {
  if (gc.nn <= 0) return cudaSuccess;
  const long long pv = (long long)DIM * gc.nnx * gc.nny;
  if (pv >= (1LL << 31) - TVAL || gc.nnz > 65535) return cudaErrorInvalidValue;
  dim3 grid((unsigned)((pv + TVAL - 1) / TVAL), DIM == 3 ? gc.nnz : 1);
  return launch_pdl(k_restrict<DIM, T>, grid, dim3(TVAL), 0, s, gf, gc, mc, (const T*)rf, (T*)bc,
                    (const T*)dinvc, T(omega), (T*)zc);
}

cudaError_t launch_restrict(int dim, int t, const GridP& gf, const GridP& gc, const uint8_t* mc,
                            const void* rf, void* bc, const void* dinvc, double omega, void* zc,
                            cudaStream_t s) {
  if (dim == 2) return t == T_F64 ? restrict_t<2, double>(gf, gc, mc, rf, bc, dinvc, omega, zc, s)
                                  : restrict_t<2, float>(gf, gc, mc, rf, bc, dinvc, omega, zc, s);
  return t == T_F64 ? restrict_t<3, double>(gf, gc, mc, rf, bc, dinvc, omega, zc, s)
                    : restrict_t<3, float>(gf, gc, mc, rf, bc, dinvc, omega, zc, s);
}

template <int DIM, typename T>
static cudaError_t prolong_t(const GridP& gf, const uint8_t* mf, const GridP& gc, const void* zc,
                             void* zf, cudaStream_t s) {
  if (gf.nn <= 0) return cudaSuccess;
  dim3 grid((gf.nnx + TBX - 1) / TBX, (gf.nny + TBY - 1) / TBY, DIM == 3 ? (gf.nnz + 1) / 2 : 1);
  return launch_pdl(k_prolong_add<DIM, T>, grid, dim3(TBX, TBY), 0, s, gf, mf, gc, (const T*)zc,
                    (T*)zf);
}

cudaError_t launch_prolong_add(int dim, int t, const GridP& gf, const uint8_t* mf,
                               const GridP& gc, const void* zc, void* zf, cudaStream_t s) {
  if (dim == 2) return t == T_F64 ? prolong_t<2, double>(gf, mf, gc, zc, zf, s)
                                  : prolong_t<2, float>(gf, mf, gc, zc, zf, s);
  return t == T_F64 ? prolong_t<3, double>(gf, mf, gc, zc, zf, s)
                    : prolong_t<3, float>(gf, mf, gc, zc, zf, s);
}

template <typename T, typename TIN>
static cudaError_t presmooth_t(long long n, const void* bin, void* bout, const void* dinv,
                               double omega, void* z, cudaStream_t s, int dim,
                               const uint8_t* mask) {
  auto kern = !mask      ? k_presmooth<0, T, TIN>
              : dim == 2 ? k_presmooth<2, T, TIN>
                         : k_presmooth<3, T, TIN>;
  return launch_pdl(kern, dim3(nblocks(n, EW_T * EW_U)), dim3(EW_T), 0, s, n, (const TIN*)bin,
                    (T*)bout, (const T*)dinv, (T)omega, (T*)z, mask);
}

cudaError_t launch_presmooth(int t, int tin, long long n, const void* bin, void* bout,
                             const void* dinv, double omega, void* z, cudaStream_t s, int dim,
                             const uint8_t* mask) {
  if (t == T_F64 && tin == T_F64)
    return presmooth_t<double, double>(n, bin, bout, dinv, omega, z, s, dim, mask);
  if (t == T_F32 && tin == T_F64)
    return presmooth_t<float, double>(n, bin, bout, dinv, omega, z, s, dim, mask);
  if (t == T_F32 && tin == T_D2)
    return presmooth_t<float, float2>(n, bin, bout, dinv, omega, z, s, dim, mask);
  return cudaErrorInvalidValue;
}

cudaError_t launch_vcycle_out(int dim, long long n, const float* zin, const double* r, double omega,
                              const uint8_t* mask, double* out, cudaStream_t s) {
  if (!zin)
    return launch_pdl(dim == 2 ? k_vcycle_fixed<2> : k_vcycle_fixed<3>,
                      dim3(nblocks(n / dim, EW_T * 4)), dim3(EW_T), 0, s, n / dim, r, omega, mask,
                      out);
  return launch_pdl(dim == 2 ? k_vcycle_out<2> : k_vcycle_out<3>, dim3(nblocks(n, EW_T * EW_U)),
                    dim3(EW_T), 0, s, n, zin, r, (float)omega, mask, out);
}

// (one value per thread on short vectors: a float32 product, which takes two
// conversions, 12.2 us with four and 10.3 to 11.3 with one at 8 x 4 x 4, the same at
// 64 x 32 x 32; with one at 192 x 96 x 96 86 us, with four 78)
template <typename TIN, typename TOUT>
static cudaError_t convert_t(long long n, const void* in, void* out, cudaStream_t s) {
  const int b1 = nblocks(n, EW_T);
  if (b1 <= 8 * 152)
    k_convert<TIN, TOUT, 1><<<b1, EW_T, 0, s>>>(n, (const TIN*)in, (TOUT*)out);
  else
    k_convert<TIN, TOUT, EW_U><<<nblocks(n, EW_T * EW_U), EW_T, 0, s>>>(n, (const TIN*)in, (TOUT*)out);
  return cudaGetLastError();
}

cudaError_t launch_convert(int tin, int tout, long long n, const void* in, void* out,
                           cudaStream_t s) {
  if (tin == T_D2 && tout == T_F32) return convert_t<float2, float>(n, in, out, s);
  if (tin == T_F64 && tout == T_F32) return convert_t<double, float>(n, in, out, s);
  if (tin == T_F32 && tout == T_F64) return convert_t<float, double>(n, in, out, s);
  if (tin == T_F64 && tout == T_F64) return convert_t<double, double>(n, in, out, s);
  return cudaErrorInvalidValue;
}

template <int DIM, typename T>
static cudaError_t gal_fine_t(const GridP& gc, const GridP& gf, const void* coef, const void* Qc,
                              void* Kc, cudaStream_t s) {
  constexpr int ND = Geo<DIM>::ND;
  const long long tot = gc.nel * tri_len(ND);
  k_galerkin_fine<DIM, T><<<nblocks(tot, 256), 256, 0, s>>>(gc, gf, (const T*)coef,
                                                            (const T*)Qc, (T*)Kc);
  return cudaGetLastError();
}

// Springs in the level-1 Galerkin matrices: the spring at fine DOF (node n,
// component c) adds k w_A w_B to entry (DIM A + c, DIM B + c) of one coarse
// element holding n, w the 1D linear weights of n at that element's corners
// (P^T S P; any element holding n gives the same assembled operator, since
// n interpolates only from the corners of each element holding it).  One
// thread per spring, springs applied in order.
template <int DIM, typename T>
__global__ void k_spring_galerkin(GridP gc, GridP gf, Springs sp, T* __restrict__ Kc) {
  constexpr int ND = Geo<DIM>::ND, NPE = Geo<DIM>::NPE, NT = tri_len(ND);
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  for (int q = 0; q < sp.n; ++q) {
    const long long node = sp.dof[q] / DIM;
    const int c = (int)(sp.dof[q] % DIM);
    const int i = (int)(node % gf.nnx);
    const long long rest = node / gf.nnx;
    const int j = (int)(rest % gf.nny);
    const int k = DIM == 3 ? (int)(rest / gf.nny) : 0;
    const int EX = min(i / 2, gc.nx - 1), EY = min(j / 2, gc.ny - 1);
    const int EZ = DIM == 3 ? min(k / 2, gc.nz - 1) : 0;
    const long long E = EX + (long long)gc.nx * (EY + (long long)gc.ny * EZ);
    double w[NPE];
    for (int a = 0; a < NPE; ++a) {
      const double px = 0.5 * (i - 2 * EX), py = 0.5 * (j - 2 * EY), pz = 0.5 * (k - 2 * EZ);
      w[a] = ((a & 1) ? px : 1.0 - px) * (((a >> 1) & 1) ? py : 1.0 - py) *
             (DIM == 3 ? (((a >> 2) & 1) ? pz : 1.0 - pz) : 1.0);
    }
    for (int a = 0; a < NPE; ++a)
      for (int b = a; b < NPE; ++b) {
        const double v = sp.k[q] * w[a] * w[b];
        if (v != 0.0) Kc[(size_t)E * NT + tri_idx(DIM * a + c, DIM * b + c, ND)] += T(v);
      }
  }
}

cudaError_t launch_spring_galerkin(int dim, int t, const GridP& gc, const GridP& gf,
                                   const Springs& sp, void* Kc, cudaStream_t s) {
  if (sp.n <= 0) return cudaSuccess;
  if (dim == 2) {
    if (t == T_F64) k_spring_galerkin<2, double><<<1, 32, 0, s>>>(gc, gf, sp, (double*)Kc);
    else k_spring_galerkin<2, float><<<1, 32, 0, s>>>(gc, gf, sp, (float*)Kc);
  } else {
    if (t == T_F64) k_spring_galerkin<3, double><<<1, 32, 0, s>>>(gc, gf, sp, (double*)Kc);
    else k_spring_galerkin<3, float><<<1, 32, 0, s>>>(gc, gf, sp, (float*)Kc);
  }
  return cudaGetLastError();
}

cudaError_t launch_galerkin_fine(int dim, int t, const GridP& gc, const GridP& gf,
                                 const void* coef, const void* Qc, void* Kc, cudaStream_t s) {
  if (dim == 2) return t == T_F64 ? gal_fine_t<2, double>(gc, gf, coef, Qc, Kc, s)
                                  : gal_fine_t<2, float>(gc, gf, coef, Qc, Kc, s);
  return t == T_F64 ? gal_fine_t<3, double>(gc, gf, coef, Qc, Kc, s)
                    : gal_fine_t<3, float>(gc, gf, coef, Qc, Kc, s);
}

template <typename T>
static cudaError_t diag_l1_t(const GridP& g1, const GridP& gf, const uint8_t* mask,
                             const double* qdiag, const void* coef, void* dinv, cudaStream_t s) {
  QDiagP<T> qd;
  for (int q = 0; q < 192; ++q) qd.v[q] = T(qdiag[q]);
  k_diag_l1<T><<<nblocks(g1.nn, 256), 256, 0, s>>>(g1, gf, mask, qd, (const T*)coef, (T*)dinv);
  return cudaGetLastError();
}

cudaError_t launch_diag_l1(int t, const GridP& g1, const GridP& gf, const uint8_t* mask,
                           const double* qdiag, const void* coef, void* dinv, cudaStream_t s) {
  return t == T_F64 ? diag_l1_t<double>(g1, gf, mask, qdiag, coef, dinv, s)
                    : diag_l1_t<float>(g1, gf, mask, qdiag, coef, dinv, s);
}

cudaError_t launch_galerkin_l2(int t, const GridP& g2, const GridP& gf, const void* coef,
                               const void* R, void* Kc, cudaStream_t s) {
  const long long tot = g2.nel * tri_len(24);
  if (t == T_F64)
    k_galerkin_l2<double><<<nblocks(tot, 256), 256, 0, s>>>(g2, gf, (const double*)coef,
                                                             (const double*)R, (double*)Kc);
  else
    k_galerkin_l2<float><<<nblocks(tot, 256), 256, 0, s>>>(g2, gf, (const float*)coef,
                                                           (const float*)R, (float*)Kc);
  return cudaGetLastError();
}

template <int DIM, typename T>
static cudaError_t gal_coarse_t(const GridP& gc, const GridP& gf, const void* Kf, void* Kc,
                                cudaStream_t s) {
  constexpr int ND = Geo<DIM>::ND;
  if (gc.nel <= 0) return cudaSuccess;
  k_galerkin_coarse<DIM, T><<<(unsigned)gc.nel, ND * ND, 0, s>>>(gc, gf, (const T*)Kf, (T*)Kc);
  return cudaGetLastError();
}

cudaError_t launch_galerkin_coarse(int dim, int t, const GridP& gc, const GridP& gf,
                                   const void* Kf, void* Kc, cudaStream_t s) {
  if (dim == 2) return t == T_F64 ? gal_coarse_t<2, double>(gc, gf, Kf, Kc, s)
                                  : gal_coarse_t<2, float>(gc, gf, Kf, Kc, s);
  return t == T_F64 ? gal_coarse_t<3, double>(gc, gf, Kf, Kc, s)
                    : gal_coarse_t<3, float>(gc, gf, Kf, Kc, s);
}

template <int DIM, typename T, typename TA>
static cudaError_t dense_t(const GridP& g, const uint8_t* mask, const void* Kc, void* A,
                           double shift, cudaStream_t s) {
  const long long n = DIM * g.nn;
  k_dense_assemble<DIM, T, TA><<<nblocks(n * n, 256), 256, 0, s>>>(g, mask, (const T*)Kc,
                                                                   (TA*)A, shift);
  return cudaGetLastError();
}

cudaError_t launch_dense_assemble(int dim, int t, int ta, const GridP& g, const uint8_t* mask,
                                  const void* Kc, void* A, double shift, cudaStream_t s) {
  if (t == T_F64 && ta == T_F64)
    return dim == 2 ? dense_t<2, double, double>(g, mask, Kc, A, shift, s)
                    : dense_t<3, double, double>(g, mask, Kc, A, shift, s);
  if (t == T_F32 && ta == T_F64)
    return dim == 2 ? dense_t<2, float, double>(g, mask, Kc, A, shift, s)
                    : dense_t<3, float, double>(g, mask, Kc, A, shift, s);
  if (t == T_F32 && ta == T_F32)
    return dim == 2 ? dense_t<2, float, float>(g, mask, Kc, A, shift, s)
                    : dense_t<3, float, float>(g, mask, Kc, A, shift, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_dense_gemv(int ta, int t, int n, const void* A, const void* x, void* y,
                              cudaStream_t s) {
  const int nb = nblocks((long long)n * 32, 256);
  if (ta == T_F64 && t == T_F64)
    return launch_pdl(k_gemv<double, double>, dim3(nb), dim3(256), 0, s, n, (const double*)A,
                      (const double*)x, (double*)y);
  if (ta == T_F64)
    return launch_pdl(k_gemv<double, float>, dim3(nb), dim3(256), 0, s, n, (const double*)A,
                      (const float*)x, (float*)y);
  return launch_pdl(k_gemv<float, float>, dim3(nb), dim3(256), 0, s, n, (const float*)A,
                    (const float*)x, (float*)y);
}

}  // namespace topo
