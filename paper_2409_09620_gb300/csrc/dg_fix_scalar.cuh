// dg_fix_scalar.cuh -- the P1-P3 basis of the scalar solver (arXiv 2409.09620, eq.
// basisfunc) and its reference derivatives at the vertices in block fixed point
// (dg_fix.cuh; P2 and P3, for P1's sums have two terms); plain C++ where compiled without CUDA (host self-test).
#pragma once
#include "dg_basis.h"
#include "dg_fix.cuh"

namespace dg {
namespace sc {

// --------------------------------------------------------------------------
// Basis of eq. (basisfunc), modes 0..9, and its reference derivatives.  Each
// mode is a sum of terms c xi^p eta^q; d^(r+s)/dxi^r deta^s is taken term by
// term.  constexpr, so evaluations at fixed points fold to constants.
// --------------------------------------------------------------------------
// flat (non-recursive) helpers for exponents and orders up to 3, so that the
// optimiser folds every evaluation at the fixed points into a constant
DG_CONST double ipow(double x, int n) {
  return n <= 0 ? 1.0 : n == 1 ? x : n == 2 ? x * x : x * x * x;
}
DG_CONST double fall(int n, int r) {   // n (n-1) ... (n-r+1)
  return r <= 0 ? 1.0 : r == 1 ? double(n) : r == 2 ? double(n * (n - 1)) : double(n * (n - 1) * (n - 2));
}
DG_CONST double term(double c, int p, int q, int r, int s, double x, double y) {
  return (r > p || s > q) ? 0.0 : c * fall(p, r) * fall(q, s) * ipow(x, p - r) * ipow(y, q - s);
}
DG_CONST double psi_rs(int l, int r, int s, double x, double y) {
#define T(c, p, q) term(c, p, q, r, s, x, y)
  return l == 0 ? T(1, 0, 0)
       : l == 1 ? T(4, 1, 0) + T(2, 0, 1) + T(-2, 0, 0)
       : l == 2 ? T(3, 0, 1) + T(-1, 0, 0)
       : l == 3 ? T(24, 2, 0) + T(24, 1, 1) + T(4, 0, 2) + T(-24, 1, 0) + T(-8, 0, 1) + T(4, 0, 0)
       : l == 4 ? T(20, 1, 1) + T(10, 0, 2) + T(-4, 1, 0) + T(-12, 0, 1) + T(2, 0, 0)
       : l == 5 ? T(10, 0, 2) + T(-8, 0, 1) + T(1, 0, 0)
       : l == 6 ? T(160, 3, 0) + T(240, 2, 1) + T(96, 1, 2) + T(8, 0, 3) + T(-240, 2, 0) + T(-192, 1, 1) +
                      T(-24, 0, 2) + T(96, 1, 0) + T(24, 0, 1) + T(-8, 0, 0)
       : l == 7 ? T(168, 2, 1) + T(168, 1, 2) + T(28, 0, 3) + T(-24, 2, 0) + T(-192, 1, 1) + T(-60, 0, 2) +
                      T(24, 1, 0) + T(36, 0, 1) + T(-4, 0, 0)
       : l == 8 ? T(84, 1, 2) + T(42, 0, 3) + T(-48, 1, 1) + T(-66, 0, 2) + T(4, 1, 0) + T(26, 0, 1) + T(-2, 0, 0)
                : T(35, 0, 3) + T(-45, 0, 2) + T(15, 0, 1) + T(-1, 0, 0);
#undef T
}
// a_K^(l) / |K| (exact rationals: 1, 2/3, 1/2, 16/15, 4/9, 1/3, 16/7, 4/5, 1/3, 1/4)
DG_CONST double sc_inv_mass(int l) {
  return l == 0 ? 1.0 : l == 1 ? 1.5 : l == 2 ? 2.0 : l == 3 ? 0.9375 : l == 4 ? 2.25 : l == 5 ? 3.0
       : l == 6 ? 7.0 / 16.0 : l == 7 ? 1.25 : l == 8 ? 3.0 : 4.0;
}
DG_CONST int sc_degree(int l) { return l == 0 ? 0 : l <= 2 ? 1 : l <= 5 ? 2 : 3; }

// --------------------------------------------------------------------------
// Reference derivatives of order J at the vertices
// --------------------------------------------------------------------------
// Only modes of degree >= J enter, and a smooth flow's modes fall with the degree, so each
// order has a block of its own, in which a mode counts 2^3 times per degree above J (its
// coefficients are that much larger): the sum is then off by about a unit of 2^-58 of its
// own largest terms, less than the FP64 FMA chain (tests/test_fix_scalar_host.py).  With
// one block over all modes and coefficients / 256 a third derivative held 2^-50 of the cell
// average.
template <int K> constexpr int SC_NB = (K + 1) * (K + 2) / 2;
template <int J> constexpr int SC_L0 = J * (J + 1) / 2;   // the first mode of degree J
template <int J>
DG_CONST double sc_coef(int l, int r, int v) {             // of d^J / dxi^r deta^(J-r)
  const int w = 3 * (sc_degree(l) - J);
  return psi_rs(l, r, J - r, vert_xi(v), vert_eta(v)) / double(1 << w);
}
// scale 2^S of the coefficients: each at most 4, the magnitudes of a sum at most 12
template <int K, int J>
DG_CONST int sc_scale() {
  double top = 0.0;
  for (int v = 0; v < 3; ++v)
    for (int r = 0; r <= J; ++r) {
      double sum = 0.0;
      for (int l = SC_L0<J>; l < SC_NB<K>; ++l) {
        const double c = sc_coef<J>(l, r, v), a = c < 0.0 ? -c : c;
        sum += a;
        top = 3.0 * a > top ? 3.0 * a : top;
      }
      top = sum > top ? sum : top;
    }
  int S = 0;
  for (double t = 12.0; t < top; t *= 2.0) ++S;
  return S;
}
constexpr int FX_EBAD = 0x4000;   // exponent of a block with a non-finite mode
template <int K, int J>
FX_HD int sfx_deriv_block(const double c[SC_NB<K>], Fx f[SC_NB<K>]) {
  int mx[4] = {0, 0, 0, 0};   // per degree
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int l = SC_L0<J>; l < SC_NB<K>; ++l) {
    const int a = fx_abs_hi(c[l]);
    mx[sc_degree(l)] = a > mx[sc_degree(l)] ? a : mx[sc_degree(l)];
  }
  int E = FX_EMIN;
  bool bad = false;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int d = J; d <= K; ++d) {
    const int e = (mx[d] >> 20) + 3 * (d - J);
    E = e > E ? e : E;
    bad = bad || mx[d] >= 0x7ff00000;
  }
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int l = SC_L0<J>; l < SC_NB<K>; ++l) f[l] = fx_from(c[l], E - 3 * (sc_degree(l) - J));
  return bad ? FX_EBAD : E;
}
// d^J u / dxi^r deta^(J-r) at vertex v, r = 0 ... J
template <int K, int J>
FX_HD void sfx_derivs(const Fx f[SC_NB<K>], int E, int v, double t[J + 1]) {
  constexpr int S = sc_scale<K, J>();
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int r = 0; r <= J; ++r) {
    FxAcc a{0, 0};
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int l = SC_L0<J>; l < SC_NB<K>; ++l) fx_mac(a, fxc(sc_coef<J>(l, r, v) / double(1 << S)), f[l]);
    t[r] = fx_nan_if(E >= FX_EBAD, fx_to(fx_round(a), E + S));
  }
}

}  // namespace sc
}  // namespace dg
