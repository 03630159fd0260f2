// hex8 element operator E KE u of float64 values in 64-bit fixed point.
//
// GB300 runs one float64 FMA per clock per SM, and integer adds and 32 x 32
// -> 64 bit multiply-adds at tens per clock, so the ~230 additions and
// multiplications of an element (corner Walsh-Hadamard basis, KE = T B T) run
// on integers:
//   values   each component of a face with the exponent of its own largest
//            nodal value, FX_S bits below that value's mantissa kept
//   modes    the 21 Walsh sums that strain the element (the three translations
//            have no force and are left out), all scaled by one power of two
//            so that the largest has FX_G bits
//   moduli   60-bit mantissa with its own exponent
//   B        entries scaled by 2^(60 - bs)
// Additions are exact; a product drops its low 64 bits (4 units at most).  So an
// element's forces are off by a few units of 2^-FX_G of its largest strain mode
// times the largest entry of B, in norm: a translation, or one component much
// larger than the others, costs no bits.  (A component that the large modes
// do not load, as u_z in a pure xy shear, has that same absolute error, where
// float64 would round it at its own size.)  The float64 transform rounds every
// sum at 2^-53 of the sum, translations included.  Measured against 80-bit
// arithmetic at nu = 0.3, rms over elements, this / float64: random 0.37, linear
// 0.12, quadratic 0.15, rigid rotation 0.05, one component uniform and the others
// 1e-8 of it 0.38, magnitudes over 12 decades 0.37; about the same from nu = -0.95
// to 0.35.  Towards 0.5 the entries of B spread (bulk to shear modulus) and one
// unit no longer suits them all, see
// fx_blocks_ok.  Results are rounded once to float64.  Zeros are exact; an
// infinity or NaN among an element's inputs makes all its outputs NaN.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "topo_internal.cuh"

namespace topo {

typedef long long fx_t;

// Bits kept below a float64 mantissa's last, of the constants, and of the
// largest strain mode.  A face's Walsh sums take 53 + FX_S + 2 bits, an element's
// one more; products of halves: 3 (2^(FX_G - 1) + 2^59) < 2^63.  FX_S may be up to 7;
// the errors above are the same with 5 and with 7 (0.01 of a ratio), and with 5 the
// 48 x 24 x 24 design loop takes the oracle's CG iteration counts, which rounding
// alone moves by a few on its gray designs.
constexpr int FX_S = 5, FX_C = 60, FX_G = 61;
static_assert(53 + FX_S + 3 <= 63 && FX_C <= 60 && FX_G <= 61, "sums and products fit 63 bits");

__host__ __device__ __forceinline__ int fx_clz(unsigned long long m) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)m);
#else
  return m ? __builtin_clzll(m) : 64;
#endif
}

struct FxFace {
  fx_t w[3][4];   // xy-Walsh sums of the face's four nodes per component
  int e[3];       // largest exponent field of the component's values
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
  o.bad = false;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    unsigned m = 1u << 20;   // subnormal numbers have exponent field 1 too
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned h = (unsigned)(fx_bits(f[q][c]) >> 32) & 0x7fffffffu;
      m = h > m ? h : m;
    }
    o.bad = o.bad || m >= 0x7ff00000u;
    o.e[c] = (int)(m >> 20);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned long long u = fx_bits(f[q][c]);
      const unsigned h = (unsigned)(u >> 32);
      const int ef = (int)((h >> 20) & 0x7ffu);
      unsigned long long t = u & 0xfffffffffffffULL;
      t |= ef ? 1ULL << 52 : 0ULL;
      const int s = o.e[c] - (ef ? ef : 1);
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
  // modes, and the least exponent e at which they all stay within FX_G bits
  fx_t X[3][8];
  int ec[3], e = -4096;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ec[c] = fb.e[c] > ft.e[c] ? fb.e[c] : ft.e[c];
    const int sb = ec[c] - fb.e[c], st = ec[c] - ft.e[c];
    unsigned long long m = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const fx_t a = fx_shr(fb.w[c][t], sb), b = fx_shr(ft.w[c][t], st);
      X[c][t] = a + b;
      X[c][t + 4] = a - b;
      if (t) m |= (unsigned long long)(X[c][t] ^ (X[c][t] >> 63));
      m |= (unsigned long long)(X[c][t + 4] ^ (X[c][t + 4] >> 63));
    }
    const int need = ec[c] + (64 - FX_G) - fx_clz(m);
    if (m && need > e) e = need;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // (a component without modes is zero, whatever its shift)
    const int s = ec[c] - e, l = s > 0 ? (s < 63 ? s : 63) : 0, r = s < 0 ? -s : 0;
#pragma unroll
    for (int t = 1; t < 8; ++t) X[c][t] = fx_shr((fx_t)((unsigned long long)X[c][t] << l), r);
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
      if (tau == (1 << c)) continue;   // a translation
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
    for (int q = 0; q < 4; ++q) {
      X[c][q] = b[q];
      X[c][q + 4] = t[q];
    }
  }
  if (k > -1023) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        // v 2^k: one rounding, then the exponent field; above the range infinite
        const fx_t v = X[c][a];
        unsigned long long d = fx_bits((double)v);
        const int f = (int)((d >> 52) & 0x7ff) + k;
        d += (unsigned long long)(long long)k << 52;
        if (v == 0) d = 0;
        if (v != 0 && f >= 0x7ff) d = 0x7ff0000000000000ULL | (v < 0 ? 1ULL << 63 : 0ULL);
        if (bad) d = 0x7ff8000000000000ULL;
        ye[a][c] = fx_double(d);
      }
  } else {
    // results may lie below the normal range: 2^k as two factors (v 2^(k / 2) is
    // normal and exact, so the second product rounds as the number system does)
    const int kk = k > -1200 ? k : -1200, k1 = kk / 2;
    const double f1 = fx_double((unsigned long long)(1023 + k1) << 52);
    const double f2 = fx_double((unsigned long long)(1023 + kk - k1) << 52);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int a = 0; a < 8; ++a)
        ye[a][c] = bad ? fx_double(0x7ff8000000000000ULL) : (double)X[c][a] * f1 * f2;
  }
}

// Whether one unit suits all entries of B: the largest at most FX_SPREAD times
// the least of the diagonal, which holds for nu < 0.37.  The kind of field that
// bounds it is a nearly rigid shear, whose force is small against its modes: at
// nu = 0.35 (spread 6.5) its error is 0.29 to 0.4 of float64's, at 0.4 (9) 0.97, at
// 0.45 (17) 2.4 and at 0.499 (750) 74 times it.
constexpr double FX_SPREAD = 7.0;
inline bool fx_blocks_ok(const double* wht) {
  double mx = 0.0, mn = 1e300;
  for (int tau = 0; tau < 8; ++tau)
    for (int c = 0; c < 3; ++c)
      for (int cp = 0; cp < 3; ++cp) {
        const double v = fabs(wht[(tau * 3 + c) * 3 + cp]);
        mx = fmax(mx, v);
        if (c == cp && !wht_zero(tau, c, c)) mn = fmin(mn, v);
      }
  return mx <= FX_SPREAD * mn;
}

// Fixed-point form of the Walsh blocks (host).  bs is the least exponent such
// that every entry is below 2^bs and every intermediate of the inverse
// transform, at most 2^FX_G times a component's absolute sum of entries, stays
// below 2^62.
inline FxBlocks fx_blocks(const double* wht) {
  auto at = [&](int tau, int c, int cp) { return wht[(tau * 3 + c) * 3 + cp]; };
  double mx = 0.0, grow = 0.0;
  for (int q = 0; q < 72; ++q) mx = fmax(mx, fabs(wht[q]));
  for (int c = 0; c < 3; ++c) {
    double g = 0.0;
    for (int tau = 0; tau < 8; ++tau)
      for (int cp = 0; cp < 3; ++cp) g += fabs(at(tau, c, cp));
    grow = fmax(grow, g);
  }
  FxBlocks kb;
  kb.bs = -60;
  while (ldexp(1.0, kb.bs) <= mx || ldexp(1.0, 62 - FX_G + kb.bs) <= grow) ++kb.bs;
  for (int tau = 0; tau < 8; ++tau)
    for (int c = 0; c < 3; ++c)
      for (int cp = 0; cp < 3; ++cp)
        fx_split(llrint(ldexp(at(tau, c, cp), FX_C - kb.bs)), kb.hi[tau][c][cp], kb.lo[tau][c][cp]);
  return kb;
}

}  // namespace topo
