// hex8 element operator E KE u of float64 values in 64-bit fixed point.
//
// GB300 runs one float64 FMA per clock per SM, and integer adds and 32 x 32
// -> 64 bit multiply-adds at tens per clock, so the ~230 additions and
// multiplications of an element (corner Walsh-Hadamard basis, KE = T B T) run
// on integers scaled to the element's own largest nodal value:
//   value    v = u 2^(1075 + FX_S - e), e the largest exponent field among
//            the four nodes of the face, truncated below 2^-57 of that value
//   moduli   60-bit mantissa with its own exponent
//   B        entries scaled by 2^(60 - bs)
// Additions are exact; a product drops its low 64 bits (4 units at most).  A
// unit is 2^-57 of the largest nodal value, below float64's rounding of the
// same sums (2^-53 of partial sums up to 8 times that value): over random,
// smooth and mixed-scale elements at nu = 0.3 the rms error is 0.25 to 0.4 of
// the float64 transform's.  Magnitudes: |v| < 2^58, Walsh sums < 2^61, and bs
// is chosen on the host so that no intermediate of the inverse transform
// reaches 2^62.  Results are
// rounded once to float64.  Zeros are exact; an infinity or NaN among an
// element's inputs makes all its outputs NaN.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "topo_internal.cuh"

namespace topo {

typedef long long fx_t;

// bits kept below a float64 mantissa's last, and bits of the constants
constexpr int FX_S = 5, FX_C = 60;
static_assert(FX_S + FX_C <= 66, "three products of high and low halves fit 63 bits");

struct FxFace {
  fx_t w[3][4];   // xy-Walsh sums of the face's four nodes per component
  int e;          // largest exponent field of the values
  bool bad;       // a value is not finite
};

__host__ __device__ __forceinline__ unsigned long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
__host__ __device__ __forceinline__ double fx_double(unsigned long long u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}

// v 2^-s for s >= 0 (arithmetic shift; more than 62 places leave 0 or -1 unit)
__host__ __device__ __forceinline__ fx_t fx_shr(fx_t v, int s) { return v >> (s < 63 ? s : 63); }

// 4-point Walsh-Hadamard transform in place (self-inverse up to the factor 4)
__host__ __device__ __forceinline__ void fx_wht4(fx_t (&v)[4]) {
  const fx_t s0 = v[0] + v[1], d0 = v[0] - v[1], s1 = v[2] + v[3], d1 = v[2] - v[3];
  v[0] = s0 + s1;
  v[1] = d0 + d1;
  v[2] = s0 - s1;
  v[3] = d0 - d1;
}

__host__ __device__ __forceinline__ void fx_face(const double (&f)[4][3], FxFace& o) {
  unsigned m = 0u;
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const unsigned h = (unsigned)(fx_bits(f[q][c]) >> 32) & 0x7fffffffu;
      m = h > m ? h : m;
    }
  o.bad = m >= 0x7ff00000u;
  o.e = (int)(m >> 20);
  if (o.e < 1) o.e = 1;   // subnormal numbers have exponent field 1 too
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned long long u = fx_bits(f[q][c]);
      const unsigned h = (unsigned)(u >> 32);
      const int ef = (int)((h >> 20) & 0x7ffu);
      unsigned long long t = u & 0xfffffffffffffULL;
      t |= ef ? 1ULL << 52 : 0ULL;
      const int s = o.e - (ef ? ef : 1);
      t = (t << FX_S) >> (s < 63 ? s : 63);
      o.w[c][q] = (h >> 31) ? -(fx_t)t : (fx_t)t;
    }
    fx_wht4(o.w[c]);
  }
}

// signed halves of a 64-bit integer: x = hi 2^32 + lo
__host__ __device__ __forceinline__ void fx_split(fx_t x, int& hi, int& lo) {
  lo = (int)(unsigned)(unsigned long long)x;
  hi = (int)((x + 0x80000000LL) >> 32);
}

// Contributions of one element: Ub, Ut (nodal values of its bottom and top
// face, float64) from the faces' xy-Walsh sums and the modulus.
__host__ __device__ __forceinline__ void fx_element(const FxBlocks& kb, double coef,
                                                    const FxFace& fb, const FxFace& ft,
                                                    double (&ye)[8][3]) {
  const int e = fb.e > ft.e ? fb.e : ft.e;
  const int sb = e - fb.e, st = e - ft.e;
  fx_t X[3][8];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const fx_t a = fx_shr(fb.w[c][t], sb), b = fx_shr(ft.w[c][t], st);
      X[c][t] = a + b;
      X[c][t + 4] = a - b;
    }
  // modulus: 60-bit signed mantissa, exponent field ee
  const unsigned long long cu = fx_bits(coef);
  const int cf = (int)((cu >> 52) & 0x7ff), ee = cf ? cf : 1;
  int ch, cl;
  {
    const unsigned long long t = ((cu & 0xfffffffffffffULL) | (cf ? 1ULL << 52 : 0ULL)) << (FX_C - 53);
    fx_split((cu >> 63) ? -(fx_t)t : (fx_t)t, ch, cl);
  }
#pragma unroll
  for (int tau = 0; tau < 8; ++tau) {
    // block tau couples X[c][tau xor e_c], c = 0..2, in place
    int zh[3], zl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      int xh, xl;
      fx_split(X[c][tau ^ (1 << c)], xh, xl);
      const fx_t H = (fx_t)xh * ch, M = (fx_t)xh * cl + (fx_t)xl * ch;
      fx_split((H << (64 - FX_C)) + (M >> (FX_C - 32)), zh[c], zl[c]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      fx_t H = 0, M = 0;
#pragma unroll
      for (int cp = 0; cp < 3; ++cp) {
        if (wht_zero(tau, c, cp)) continue;
        H += (fx_t)zh[cp] * kb.hi[tau][c][cp];
        M += (fx_t)zh[cp] * kb.lo[tau][c][cp] + (fx_t)zl[cp] * kb.hi[tau][c][cp];
      }
      X[c][tau ^ (1 << c)] = (H << (64 - FX_C)) + (M >> (FX_C - 32));
    }
  }
  // inverse transform, then to float64 with the exponents of u, E and B
  const int k = e + ee + kb.bs - (2097 + FX_S);
  const bool bad = fb.bad || ft.bad || cf == 0x7ff;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    fx_t b[4], t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      b[q] = X[c][q] + X[c][q + 4];
      t[q] = X[c][q] - X[c][q + 4];
    }
    fx_wht4(b);
    fx_wht4(t);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const fx_t v = a < 4 ? b[a & 3] : t[a & 3];
      // v 2^k: one rounding, then the exponent field; below the normal range
      // the result is 0, above it infinite
      unsigned long long d = fx_bits((double)v);
      const int f = (int)((d >> 52) & 0x7ff) + k;
      d += (unsigned long long)(long long)k << 52;
      if (v == 0 || f <= 0) d = 0;
      if (v != 0 && f >= 0x7ff) d = 0x7ff0000000000000ULL | (v < 0 ? 1ULL << 63 : 0ULL);
      if (bad) d = 0x7ff8000000000000ULL;
      ye[a][c] = fx_double(d);
    }
  }
}

// Fixed-point form of the Walsh blocks (host).  bs is the least exponent such
// that every entry is below 2^bs and every intermediate of the inverse
// transform, whose largest possible value over inputs |v| < 2^(53 + FX_S) is its
// coefficients' absolute sum, stays below 2^62.
inline FxBlocks fx_blocks(const double* wht) {
  auto at = [&](int tau, int c, int cp) { return wht[(tau * 3 + c) * 3 + cp]; };
  double mx = 0.0, grow = 0.0;
  for (int q = 0; q < 72; ++q) mx = fmax(mx, fabs(wht[q]));
  double Y[3][8][24];   // Y[c][t] as a combination of the 24 nodal values
  for (int tau = 0; tau < 8; ++tau)
    for (int c = 0; c < 3; ++c)
      for (int a = 0; a < 8; ++a)
        for (int cp = 0; cp < 3; ++cp) {
          const int t = tau ^ (1 << cp);
          Y[c][tau ^ (1 << c)][3 * a + cp] =
              (__builtin_popcount(a & t) & 1 ? -1.0 : 1.0) * at(tau, c, cp);
        }
  auto l1 = [&](const double* r) {
    double s = 0.0;
    for (int q = 0; q < 24; ++q) s += fabs(r[q]);
    grow = fmax(grow, s);
  };
  // the transform's stages in the kernel's order: z, then x, then y
  for (int c = 0; c < 3; ++c)
    for (int t = 0; t < 8; ++t) l1(Y[c][t]);
  const int order[3] = {4, 1, 2};
  for (int s = 0; s < 3; ++s)
    for (int c = 0; c < 3; ++c)
      for (int t = 0; t < 8; ++t)
        if (!(t & order[s])) {
          for (int q = 0; q < 24; ++q) {
            const double u = Y[c][t][q], v = Y[c][t | order[s]][q];
            Y[c][t][q] = u + v;
            Y[c][t | order[s]][q] = u - v;
          }
          l1(Y[c][t]);
          l1(Y[c][t | order[s]]);
        }
  FxBlocks kb;
  kb.bs = -60;
  while (ldexp(1.0, kb.bs) <= mx || ldexp(1.0, 9 - FX_S + kb.bs) <= grow) ++kb.bs;
  for (int tau = 0; tau < 8; ++tau)
    for (int c = 0; c < 3; ++c)
      for (int cp = 0; cp < 3; ++cp)
        fx_split(llrint(ldexp(at(tau, c, cp), FX_C - kb.bs)), kb.hi[tau][c][cp], kb.lo[tau][c][cp]);
  return kb;
}

}  // namespace topo
