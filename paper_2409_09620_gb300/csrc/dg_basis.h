// dg_basis.h -- the P1/P2 basis and the quadrature rules (arXiv 2409.09620,
// eq. basisfunc, Appendices A and B) as constexpr functions, shared by the
// kernels and host self-tests (plain C++: no CUDA headers needed).
#pragma once

#ifdef __CUDACC__
#define DG_CONST __host__ __device__ constexpr
#else
#define DG_CONST constexpr
#endif

namespace dg {

// ------------------------------------------------------------------------
// Basis of eq. (basisfunc), modes 0..5, on the reference triangle
// (v1 -> (0,0), v2 -> (1,0), v3 -> (0,1)).  Written as constexpr functions so
// that evaluations at the fixed quadrature points fold to constants.
// ------------------------------------------------------------------------
DG_CONST double psi(int l, double x, double y) {
  return l == 0 ? 1.0
       : l == 1 ? 4.0 * x + 2.0 * y - 2.0
       : l == 2 ? 3.0 * y - 1.0
       : l == 3 ? 24.0 * x * x + 24.0 * x * y + 4.0 * y * y - 24.0 * x - 8.0 * y + 4.0
       : l == 4 ? 20.0 * x * y + 10.0 * y * y - 4.0 * x - 12.0 * y + 2.0
                : 10.0 * y * y - 8.0 * y + 1.0;
}
DG_CONST double psi_x(int l, double x, double y) {   // d/dxi
  return l == 0 ? 0.0 : l == 1 ? 4.0 : l == 2 ? 0.0 : l == 3 ? 48.0 * x + 24.0 * y - 24.0
       : l == 4 ? 20.0 * y - 4.0 : 0.0;
}
DG_CONST double psi_y(int l, double x, double y) {   // d/deta
  return l == 0 ? 0.0 : l == 1 ? 2.0 : l == 2 ? 3.0 : l == 3 ? 24.0 * x + 8.0 * y - 8.0
       : l == 4 ? 20.0 * x + 20.0 * y - 12.0 : 20.0 * y - 8.0;
}
// second reference derivatives: r = 0 (xi xi), 1 (xi eta), 2 (eta eta)
DG_CONST double psi_2(int l, int r) {
  return l == 3 ? (r == 0 ? 48.0 : r == 1 ? 24.0 : 8.0)
       : l == 4 ? (r == 0 ? 0.0 : 20.0)
       : l == 5 ? (r == 2 ? 20.0 : 0.0) : 0.0;
}
// mass a_K^(l) = c_l |K| of the orthogonal basis
DG_CONST double mass_c(int l) {
  return l == 0 ? 1.0 : l == 1 ? 2.0 / 3.0 : l == 2 ? 0.5 : l == 3 ? 16.0 / 15.0 : l == 4 ? 4.0 / 9.0 : 1.0 / 3.0;
}
// 1 / c_l (exact in binary)
DG_CONST double inv_mass_c(int l) {
  return l == 0 ? 1.0 : l == 1 ? 1.5 : l == 2 ? 2.0 : l == 3 ? 0.9375 : l == 4 ? 2.25 : 3.0;
}
DG_CONST int degree_of(int l) { return l == 0 ? 0 : (l <= 2 ? 1 : 2); }

// Gauss-Legendre nodes of Appendix B mapped to s in (0, 1), weights summing to 1.
DG_CONST double gauss_s(int Q, int nu) {
  return Q == 2 ? (nu == 0 ? 0.21132486540518713 : 0.78867513459481287)
                : (nu == 0 ? 0.11270166537925831 : nu == 1 ? 0.5 : 0.88729833462074169);
}
DG_CONST double gauss_w(int Q, int nu) {
  return Q == 2 ? 0.5 : (nu == 1 ? 8.0 / 18.0 : 5.0 / 18.0);
}
// edge i is opposite vertex i, run from vertex i+1 to vertex i+2 (counter-clockwise)
DG_CONST double edge_xi(int i, double s) { return i == 0 ? 1.0 - s : i == 1 ? 0.0 : s; }
DG_CONST double edge_eta(int i, double s) { return i == 0 ? s : i == 1 ? 1.0 - s : 0.0; }
DG_CONST double vert_xi(int v) { return v == 1 ? 1.0 : 0.0; }
DG_CONST double vert_eta(int v) { return v == 2 ? 1.0 : 0.0; }

// Volume rules of Appendix A (tab:2th for N = 3, tab:4th for N = 6); (xi, eta) = (b2, b3).
DG_CONST double vol_xi(int N, int mu) {
  return N == 3 ? (mu == 0 ? 1.0 / 6.0 : mu == 1 ? 2.0 / 3.0 : 1.0 / 6.0)
       : (mu == 0 ? 0.445948490915965 : mu == 1 ? 0.108103018168070 : mu == 2 ? 0.445948490915965
          : mu == 3 ? 0.091576213509771 : mu == 4 ? 0.816847572980458 : 0.091576213509771);
}
DG_CONST double vol_eta(int N, int mu) {
  return N == 3 ? (mu == 0 ? 2.0 / 3.0 : mu == 1 ? 1.0 / 6.0 : 1.0 / 6.0)
       : (mu == 0 ? 0.108103018168070 : mu == 1 ? 0.445948490915965 : mu == 2 ? 0.445948490915965
          : mu == 3 ? 0.816847572980458 : mu == 4 ? 0.091576213509771 : 0.091576213509771);
}
DG_CONST double vol_w(int N, int mu) {
  return N == 3 ? 1.0 / 3.0 : (mu < 3 ? 0.223381589678010 : 0.109951743655322);
}

}  // namespace dg
