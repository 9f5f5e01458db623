// dg_fix_vertex.cuh -- first and second physical derivatives of one component at a
// cell's vertices in block fixed point (dg_fix.cuh), for the OE jumps of the FP64 form;
// plain C++ where compiled without CUDA (host self-test).
//
// A derivative does not contain the cell average, and a smooth flow's modes are far
// below it and the second-degree ones far below the first-degree ones.  So the gradients have
// a block of their own over the modes l >= 1, the second-degree ones counted with their
// larger coefficients, and the Hessian one over l >= 3; each row of J^-1 (the derivatives
// of xi and eta by one coordinate) has its exponent, for the cells may be thin.  The
// products are complete and the sums rounded, so that the error stays below that of the FMA
// chain sum_l dPsi_l u_l, J^-T (.) in FP64 (tests/test_fix_vertex_host.py): with
// one block over all modes it was 2^-52 of the average, 10^-10 of a gradient and 10^-8 of a
// Hessian of modes 10^-3 and 10^-6 of the average.
#pragma once
#include "dg_basis.h"
#include "dg_fix.cuh"

namespace dg {

// J^-1 by rows: r[d][0] = dxi/dx_d, r[d][1] = deta/dx_d, |r[d][.]| 2^E[d]
struct FxRows {
  Fx r[2][2];
  int E[2];
};
FX_HD FxRows fx_rows(const double xi[2], const double eta[2]) {
  FxRows J;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int d = 0; d < 2; ++d) {
    const int a = fx_abs_hi(xi[d]), b = fx_abs_hi(eta[d]);
    J.E[d] = fx_exp(a > b ? a : b) - 1022;   // |xi[d]|, |eta[d]| < 2^E: coefficients below 1
    J.r[d][0] = fx_coef(xi[d], -J.E[d]);
    J.r[d][1] = fx_coef(eta[d], -J.E[d]);
  }
  return J;
}
// p dxi/dx_d + q deta/dx_d
FX_HD int64_t fx_turn(const FxRows &J, int d, Fx p, Fx q) {
  FxAccL t{0, 0, 0};
  fx_mac(t, J.r[d][0], p);
  fx_mac(t, J.r[d][1], q);
  return fx_round(t);
}

// sum_l c_l f_l of the modes l0 ... NB - 1, rounded, as a value
template <int NB, typename C>
FX_HD Fx fx_modes(const Fx f[NB], int l0, C coef) {
  FxAcc s{0, 0};
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int l = 1; l < NB; ++l)
    if (l >= l0) fx_mac(s, fxc(coef(l)), f[l]);
  return fx_value(fx_round(s), 0);
}

// Gradients at the three vertices, handed to store(vertex, gx, gy), of exponents EG[d], and
// for P2 the Hessian (xx, xy, yy) of exponents EH, EH + EG[1] - EG[0], EH + 2 (EG[1] - EG[0]).
//   Gradient block: |h_l| 2^(3 (degree - 1)) < 2^(E - 1022), coefficients / 2^FX_GRAD.  The
// |dPsi/dxi| at a vertex sum to at most 7.5 / 16 and the |dPsi/deta| to 9 / 16 in P2, to 4 / 8
// and 5 / 8 in P1: a reference derivative is below 0.63 * 2^58, a gradient below 1.13 * 2^58,
// the difference of two below 2^60 (limbs).
//   Hessian block: the second-degree modes, coefficients / 64, which sum to at most 48 / 64; a
// turn at most doubles: below 3 * 2^58.
//   P2's gradients at vertices 1 and 2 are that at vertex 0 plus the first turn of the Hessian's
// columns (its edges in reference coordinates have length 1): 9 turns in all instead of 13.
template <int NB> constexpr int FX_GRAD = NB == 3 ? 3 : 4;
constexpr int FX_HESS = 6;
template <int NB>
struct FxDerivs {
  int EG[2], EH;
  Fx hess[3];
  template <typename S>
  FX_HD FxDerivs(const double h[NB], const FxRows &J, S store) : EH(0) {
    Fx f[NB];
    int m1 = 0, m2 = 0;   // largest mode of each degree
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int l = 1; l < NB; ++l) {
      const int a = fx_abs_hi(h[l]);
      if (l < 3) m1 = a > m1 ? a : m1;
      else m2 = a > m2 ? a : m2;
    }
    const int E2 = fx_exp(m2), e1 = fx_exp(m1), E = NB > 3 && E2 + 3 > e1 ? E2 + 3 : e1;
    EG[0] = E + FX_GRAD<NB> + J.E[0];
    EG[1] = E + FX_GRAD<NB> + J.E[1];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int l = 1; l < NB; ++l) f[l] = fx_from(h[l], E);
    constexpr double G = 1.0 / (1 << FX_GRAD<NB>);
    const Fx p = fx_modes<NB>(f, 1, [](int l) { return psi_x(l, 0.0, 0.0) * G; });
    const Fx q = fx_modes<NB>(f, 1, [](int l) { return psi_y(l, 0.0, 0.0) * G; });
    const int64_t gx = fx_turn(J, 0, p, q), gy = fx_turn(J, 1, p, q);
    store(0, fx_value(gx, 0), fx_value(gy, 0));
    if constexpr (NB == 3) {
      store(1, fx_value(gx, 0), fx_value(gy, 0));
      store(2, fx_value(gx, 0), fx_value(gy, 0));
    } else {
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
      for (int l = 3; l < NB; ++l) f[l] = fx_from(h[l], E2);
      constexpr double H = 1.0 / (1 << FX_HESS);
      const Fx xx = fx_modes<NB>(f, 3, [](int l) { return psi_2(l, 0) * H; });
      const Fx xe = fx_modes<NB>(f, 3, [](int l) { return psi_2(l, 1) * H; });
      const Fx ee = fx_modes<NB>(f, 3, [](int l) { return psi_2(l, 2) * H; });
      const int64_t ax = fx_turn(J, 0, xx, xe), bx = fx_turn(J, 0, xe, ee);
      const int64_t ay = fx_turn(J, 1, xx, xe), by = fx_turn(J, 1, xe, ee);
      // E >= E2 + 3: from the Hessian's block to the gradient's, rounded
      const int s = E + FX_GRAD<NB> - E2 - FX_HESS < 62 ? E + FX_GRAD<NB> - E2 - FX_HESS : 62;
      const int64_t half = 1LL << (s - 1);
      store(1, fx_value(gx + ((ax + half) >> s), 0), fx_value(gy + ((ay + half) >> s), 0));
      store(2, fx_value(gx + ((bx + half) >> s), 0), fx_value(gy + ((by + half) >> s), 0));
      const Fx cx = fx_value(ax, 0), dx = fx_value(bx, 0);
      EH = E2 + FX_HESS + 2 * J.E[0];
      hess[0] = fx_value(fx_turn(J, 0, cx, dx), 0);
      hess[1] = fx_value(fx_turn(J, 1, cx, dx), 0);
      hess[2] = fx_value(fx_turn(J, 1, fx_value(ay, 0), fx_value(by, 0)), 0);
    }
  }
};

}  // namespace dg
