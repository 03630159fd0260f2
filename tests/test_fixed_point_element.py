"""The fixed-point element product of the float64 operator (fxmath.cuh, compiled
for the host) against 80-bit arithmetic and against the float64 Walsh transform
it stands for: on no kind of field is it further from the exact product than
float64, over the Poisson's ratios it is used at.  The kinds include those
where float64's sums happen to be exact: rigid motions, one component uniform
and the others far smaller, magnitudes of many decades.

Bound: the rms error over the elements of a kind, in the norm of an element's
product, at most float64's (the ratios are 0 to 0.5)."""

import ctypes
import os

import numpy as np
import pytest

from oracle import fe

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_00385_gb300", "csrc")

SRC = r"""
#include "fxmath.cuh"
using namespace topo;
typedef long double ld;
template <typename T> static void had(T (&v)[8]) {
  for (int h = 1; h < 8; h <<= 1)
    for (int a = 0; a < 8; ++a)
      if (!(a & h)) { const T u = v[a], w = v[a + h]; v[a] = u + w; v[a + h] = u - w; }
}
static double mul_add(double a, double b, double c) { return fma(a, b, c); }
static ld mul_add(ld a, ld b, ld c) { return a * b + c; }
template <typename T> static void walsh(const double* W, double E, const double* u, T* y) {
  T X[3][8], Y[3][8];
  for (int c = 0; c < 3; ++c) { for (int a = 0; a < 8; ++a) X[c][a] = u[3 * a + c]; had(X[c]); }
  for (int tau = 0; tau < 8; ++tau) {
    T z[3];
    for (int c = 0; c < 3; ++c) z[c] = (T)E * X[c][tau ^ (1 << c)];
    for (int c = 0; c < 3; ++c) {
      T s = 0;
      for (int cp = 0; cp < 3; ++cp) s = mul_add((T)W[(tau * 3 + c) * 3 + cp], z[cp], s);
      Y[c][tau ^ (1 << c)] = s;
    }
  }
  for (int c = 0; c < 3; ++c) { had(Y[c]); for (int a = 0; a < 8; ++a) y[3 * a + c] = Y[c][a]; }
}
extern "C" int blocks_ok(double* W) {
  for (int q = 0; q < 72; ++q) if (wht_zero(q / 9, q / 3 % 3, q % 3)) W[q] = 0.0;
  return fx_blocks_ok(W);
}
extern "C" void fixed(const double* W, double E, const double* u, double* y) {
  const FxBlocks kb = fx_blocks(W);
  double f[2][4][3], ye[8][3];
  for (int q = 0; q < 24; ++q) f[q / 12][q / 3 % 4][q % 3] = u[q];
  FxFace b, t;
  fx_face(f[0], b);
  fx_face(f[1], t);
  fx_element(kb, E, b, t, ye);
  for (int q = 0; q < 24; ++q) y[q] = ye[q / 3][q % 3];
}
// relative errors of n elements (norm of the product): fixed point, float64
extern "C" void errors(const double* W, int n, const double* E, const double* u, double* e) {
  for (int i = 0; i < n; ++i) {
    double y[24], y64[24];
    ld ex[24], s = 0, d = 0, d64 = 0;
    fixed(W, E[i], u + 24 * i, y);
    walsh(W, E[i], u + 24 * i, y64);
    walsh(W, E[i], u + 24 * i, ex);
    for (int q = 0; q < 24; ++q) {
      s += ex[q] * ex[q];
      d += (y[q] - ex[q]) * (y[q] - ex[q]);
      d64 += (y64[q] - ex[q]) * (y64[q] - ex[q]);
    }
    e[2 * i] = s > 0 ? (double)sqrtl(d / s) : 0.0;
    e[2 * i + 1] = s > 0 ? (double)sqrtl(d64 / s) : 0.0;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import subprocess
    from paper_2205_00385_gb300 import build
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cu").write_text(SRC)
    subprocess.run([nvcc, *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    "-o", str(d / "fx.so"), str(d / "fx.cu")], check=True)
    return ctypes.CDLL(str(d / "fx.so"))


def _ptr(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def _blocks(lib, nu):
    K = fe.element_stiffness(3, nu)
    sgn = np.array([[(-1.0) ** bin(a & t).count("1") for t in range(8)] for a in range(8)])
    W = np.zeros((8, 3, 3))
    for tau in range(8):
        for c in range(3):
            for cp in range(3):
                W[tau, c, cp] = sgn[:, tau ^ (1 << c)] @ K[c::3, cp::3] @ sgn[:, tau ^ (1 << cp)] / 64
    return bool(lib.blocks_ok(_ptr(W))), W


def _fields(rng, n):
    """Nodal values (n, 8, 3) by kind; nodes a = bx + 2 by + 4 bz."""
    v = rng.standard_normal((n, 8, 3))
    a = np.arange(8)
    x = np.stack([a & 1, a >> 1 & 1, a >> 2], 1) + 3.0 * rng.standard_normal((n, 1, 3))
    om, t = rng.standard_normal((n, 1, 3)), rng.standard_normal((n, 1, 3))
    A = rng.standard_normal((n, 3, 3))
    lin = np.einsum("nij,naj->nai", A, x)
    rot = np.cross(np.broadcast_to(om, x.shape), x)
    uni = lambda s: np.where(np.arange(3) == 0, t, s * v)
    plane = np.stack([-x[..., 1], x[..., 0], 0 * x[..., 0]], 2)
    shear = np.stack([A[:, :1, 0] * x[..., 1], A[:, :1, 1] * x[..., 0], 1e-8 * v[..., 2]], 2)
    bend = np.stack([x[..., 0] * x[..., 1], -0.5 * x[..., 0] ** 2 - 0.15 * (x[..., 1] ** 2 - x[..., 2] ** 2),
                     0.3 * x[..., 1] * x[..., 2]], 2)
    hot = np.eye(24)[rng.integers(0, 24, n)].reshape(n, 8, 3)
    return dict(random=v, smooth=t + 1e-4 * v, linear=lin, bending=bend, rotation=rot,
                rotation_translation=rot + 1e3 * t, rotation_strain=plane + 1e-6 * lin,
                uniform_1e3=uni(1e-3), uniform_1e8=uni(1e-8), shear=shear,
                components=v * 10.0 ** np.array([0, -4, -8]),
                decades=v * 10.0 ** -rng.integers(0, 12, v.shape), unit=hot * v,
                zeros=v * (rng.uniform(size=v.shape) < 0.5))


@pytest.mark.parametrize("nu", [-0.95, -0.5, 0.0, 0.2, 0.3, 0.35])
def test_no_further_from_the_exact_product_than_float64(lib, nu):
    ok, W = _blocks(lib, nu)
    assert ok
    rng = np.random.default_rng(17)
    n = 3000
    for kind, u in _fields(rng, n).items():
        E = np.exp(3 * rng.standard_normal(n)) * rng.choice([-1.0, 1.0], n)
        u = np.ascontiguousarray(u * 10.0 ** rng.uniform(-3, 3, (n, 1, 1)))
        e = np.zeros((n, 2))
        lib.errors(_ptr(W), n, _ptr(E), _ptr(u), _ptr(e))
        rms = np.sqrt(np.mean(e ** 2, axis=0))
        print(f"nu {nu} {kind}: fixed {rms[0]:.2e} float64 {rms[1]:.2e} ratio {rms[0] / rms[1]:.2f}")
        assert rms[0] <= rms[1], (kind, rms)


@pytest.mark.parametrize("nu,ok", [(-0.99, True), (0.35, True), (0.4, False), (0.45, False),
                                   (0.49, False), (0.4999, False)])
def test_poisson_ratios(lib, nu, ok):
    """Near 0.5 the entries of the Walsh blocks spread too far for one unit; the
    float64 transform runs there."""
    assert _blocks(lib, nu)[0] == ok


def test_results_below_the_normal_range(lib):
    """Subnormal results are rounded as the number system rounds them (1.5 units
    of 2^-1074 with the product's own rounding), not flushed."""
    ok, W = _blocks(lib, 0.3)
    assert ok
    rng = np.random.default_rng(18)
    for scale in (1e-290, 1e-300, 1e-306, 1e-309, 1e-312, 1e-318, 1e-323):
        for E in (1.0, 1e-9, 3e5, 1e-300):
            u = rng.standard_normal(24) * scale
            y, ref, e = np.zeros(24), np.zeros(24), np.zeros(2)
            lib.fixed(_ptr(W), ctypes.c_double(E), _ptr(u), _ptr(y))
            big = np.ascontiguousarray(u * 2.0 ** 500 * 2.0 ** 500)   # (exact)
            lib.fixed(_ptr(W), ctypes.c_double(E), _ptr(big), _ptr(ref))
            with np.errstate(under="ignore"):
                ref = ref * 2.0 ** -500 * 2.0 ** -500
            assert np.all(np.abs(y - ref) <= 1.5 * 2.0 ** -1074 + 1e-15 * np.max(np.abs(ref)))
            if scale == 1e-309 and E == 1.0:
                assert np.all(y != 0.0) and np.max(np.abs(y)) < 2.0 ** -1022
