// dg_common.cuh -- device data layout, basis, quadrature and physics of the
// GB300 BP RI-OEDG solver (Ding, Cui & Wu, arXiv 2409.09620).
//
// Data layout in HBM (one mesh of nt cells):
//   state     avg[4][nt] (FP64 cell averages, mode 0)  +  hi[4][nb-1][nt] (modes 1..nb-1, Real)
//   geometry  area[nt], jinv[4][nt] (dxi/dx, dxi/dy, deta/dx, deta/dy), nrm[6][nt],
//             len[3][nt], hgeo[6][nt] (h_i, 1/h_i), vxy[6][nt], node[4][nt] (P2 internal
//             nodes, reference coords),
//             limv[2][nt] (P1 limiter vertices), conn[3][nt] (neighbour << 2 | its edge, or -tag)
//   exchange buffers (FP64 form only; the mixed form's passes read the
//   neighbours' modal states instead, see dg_stage_mixed.cuh):
//             tr[nt][3][Q][8]  traces of the stage input at edge Gauss points:
//                              u (4) and F(u).n_i (4), written by the cell that owns them
//             vd[nt][52]       u_h at the three vertices, [3][16]: value (4) and physical
//                              gradient (8) in fixed point, 1/rho, sound speed and momentum
//                              in FP64; then the blocks' exponents per component (4)
//             hs[nt][12]       physical Hessian (xx, xy, yy) of u_h per component (P2), fixed point
//             ej[ne][16]       per edge: the OE jump terms of each component
// The mixed form's kernels are one thread per cell, the FP64 form's four lanes
// per cell; reductions are per-block partials reduced in a fixed order, so
// results are bitwise reproducible.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "dg_basis.h"
#include "dg_math.h"

namespace dg {

constexpr int TPB = 128;                 // threads per block of the stage kernels
// cells per tile (one block's work, one reduction partial): one thread per
// cell in the mixed form, four lanes per cell in the FP64 form
template <typename Real> struct TileCells { static constexpr int value = sizeof(Real) == 4 ? TPB : TPB / 4; };
__host__ __device__ constexpr int tile_cells(int precision) {
  return precision == 0 ? TileCells<double>::value : TileCells<float>::value;
}
constexpr int FIN_THREADS = 1024;        // threads (virtual lanes) of the finalize reductions

template <int K> struct Deg;
template <> struct Deg<1> { static constexpr int NB = 3, NQ = 2, NV = 3; };
template <> struct Deg<2> { static constexpr int NB = 6, NQ = 3, NV = 6; };

struct MeshDev {
  int64_t nt;
  const double *area, *jinv, *nrm, *len, *vxy, *node;
  const double *hgeo;   // [6][nt]: h_i = 2|K| / l_i (i = 0..2), then 1 / h_i
  const int8_t *limv;
  const int32_t *conn;
  // edges, each once, ordered by the owning cell (the lower cell id of an
  // interior edge; the cell of a boundary edge)
  int64_t ne;
  const int32_t *e_cell;   // [ne] owning cell
  const int8_t *e_loc;     // [ne] its local edge
  const int32_t *etile;    // [ntiles + 1] first edge owned by each tile of the FP64 form
  const int32_t *cedge;    // [3][nt] edge index of (cell, local edge)
  // FP32 copies of the geometry the mixed-precision kernels read (the same
  // rounded values, without a conversion per read), and 1/|K| in FP64
  const float *jinv_f, *nrm_f, *len_f, *hgeo_f;
  const double *iarea;
  const float *node_f;     // [4][nt] FP32 copy of node (P2 internal limiter nodes)
  const double *psi_node;  // [2][5][nt] P2 basis psi_1..psi_5 at the two internal nodes
};

// the exchange buffers (traces, vertex records, Hessians, edge records) are
// used by the FP64 form only; the mixed form's passes read the states directly
__host__ __device__ constexpr bool uses_exchange(int precision) { return precision == 0; }
// values per edge Gauss point in the trace buffer tr[nt][3][Q][8]: u and F(u).n
constexpr int TR_STRIDE = 8;
// per-edge OE record ej[ne][4][4]: A^{k,j} beta sqrt(J) of the trapezoidal jump
// sums J, per component and derivative order j = 0..k (one padding value)
constexpr int EJ_STRIDE = 16;
// per-cell vertex record vd[nt][VD_CELL]: per vertex VD_STRIDE values (value and
// gradient of component c at c and 4 + 2 c as limb pairs of dg_fix.cuh; 1/rho,
// sound speed, m1, m2), then per component four 16-bit exponents: of its values, the x
// and the y entries of its gradients, and the xx entry of its Hessian (xy and yy: one and
// two steps from x to y further)
constexpr int VD_STRIDE = 16;
constexpr int VD_EXP = 3 * VD_STRIDE;
constexpr int VD_CELL = VD_EXP + 4;

// 16-byte vector loads and stores of N consecutive values (N a multiple of 16/sizeof(T))
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  using type = float4;
  static constexpr int n = 4;
  static __device__ __forceinline__ void get(const float4 &v, float *o) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
  static __device__ __forceinline__ float4 make(const float *i) { return make_float4(i[0], i[1], i[2], i[3]); }
};
template <> struct Vec16<double> {
  using type = double2;
  static constexpr int n = 2;
  static __device__ __forceinline__ void get(const double2 &v, double *o) { o[0] = v.x; o[1] = v.y; }
  static __device__ __forceinline__ double2 make(const double *i) { return make_double2(i[0], i[1]); }
};
template <int N, typename T>
__device__ __forceinline__ void vload(const T *__restrict__ p, T out[N]) {
  constexpr int L = Vec16<T>::n;
  const typename Vec16<T>::type *q = reinterpret_cast<const typename Vec16<T>::type *>(p);
#pragma unroll
  for (int k = 0; k < N / L; ++k) Vec16<T>::get(q[k], out + k * L);
}
template <int N, typename T>
__device__ __forceinline__ void vstore(T *__restrict__ p, const T in[N]) {
  constexpr int L = Vec16<T>::n;
  typename Vec16<T>::type *q = reinterpret_cast<typename Vec16<T>::type *>(p);
#pragma unroll
  for (int k = 0; k < N / L; ++k) q[k] = Vec16<T>::make(in + k * L);
}

template <typename Real> struct StateDev {
  double *avg;   // [4][nt]
  Real *hi;      // FP64 form: [4][nb-1][nt]; mixed form: [nt][4][nb-1] (one 16-byte aligned record per cell)
};

struct Phys {
  double gamma;
  double bc[4][4];
  double shock_x0, shock_cot, shock_vx;   // x_s(y, t) = x0 + y cot(angle) + t speed / sin(angle)
  int shock_pre, shock_post;
  int oe, bp, k, decomp;   // decomp: 0 optimal convex decomposition, 1 classical (ZXS)
  float gamma_f, gm1_f;    // FP32 roundings of gamma and gamma - 1 (mixed form)
};

// gamma and gamma - 1 in the working precision (no conversion in the kernels)
template <typename Real>
__device__ __forceinline__ Real phys_gamma(const Phys &ph) {
  if constexpr (sizeof(Real) == sizeof(float)) return ph.gamma_f; else return ph.gamma;
}
template <typename Real>
__device__ __forceinline__ Real phys_gm1(const Phys &ph) {
  if constexpr (sizeof(Real) == sizeof(float)) return ph.gm1_f; else return ph.gamma - 1.0;
}

// Device-resident scalars of one solver.
struct Scalars {
  double t, t_end, dt, alpha, cfl, min_ca;
  double mean[4], area_total, dev[5];
  double invD[4];   // 1 / normaliser of the damped quantities (rho, m_n|m1, m_t|m2, E); 0 if constant
  float invDf[4];   // their FP32 roundings (mixed form)
  long long steps, limited, nonphys, breaches;
  int active, pad;
};

// the basis of dg_basis.h evaluated in the arithmetic of T at run-time points
template <typename T>
__device__ __forceinline__ T psi_t(int l, T x, T y) {
  // nested forms with explicit fmas (see fdot2)
  return l == 0 ? T(1)
       : l == 1 ? fma(T(4), x, fma(T(2), y, T(-2)))
       : l == 2 ? fma(T(3), y, T(-1))
       : l == 3 ? fma(x, fma(T(24), x, fma(T(24), y, T(-24))), fma(y, fma(T(4), y, T(-8)), T(4)))
       : l == 4 ? fma(x, fma(T(20), y, T(-4)), fma(y, fma(T(10), y, T(-12)), T(2)))
                : fma(y, fma(T(10), y, T(-8)), T(1));
}
// acc + c * x with a coefficient c known at compile time after unrolling:
// zero terms vanish and unit coefficients become additions.
template <typename T>
__device__ __forceinline__ T cfma(double c, T x, T acc) {
  if (c == 0.0) return acc;
  if (c == 1.0) return acc + x;
  if (c == -1.0) return acc - x;
  return fma(static_cast<T>(c), x, acc);
}

// x != 0 on the integer units (true for NaN, false for +0 and -0, as the
// comparison); on the two words, for a 64-bit test of the bits is compiled to
// an FP64 comparison
__device__ __forceinline__ bool nonzero_bits(double x) {
  return (((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x)) != 0u;
}
__device__ __forceinline__ bool nonzero_bits(float x) { return (__float_as_int(x) << 1) != 0; }
// the first SSP-RK stage, u_h = v + dt L(v), on the integer units (two comparisons per
// warp were 8 of 305 operations of the FP64 pipe per tile of k_rk)
__device__ __forceinline__ bool first_stage(double a, double b) {
  return !nonzero_bits(a) && __double2hiint(b) == 0x3ff00000 && __double2loint(b) == 0;
}

// ------------------------------------------------------------------------
// FP64 operations at the cost of a register-only DFMA
// ------------------------------------------------------------------------
// Measured on GB300 (cycles per warp instruction and scheduler): DFMA with
// three register operands 64; DFMA with an immediate, constant or uniform
// operand 76; DADD and DMUL 76; 1.0 / x 344; sqrt(x) 572.  So sums and products
// are written as a b + c with a 1.0 or -0.0 that the compiler has to keep in a
// register because it comes from memory; x 1.0 + y and x y + (-0.0) are x + y
// and x y bit for bit.
static __device__ const double g_fp_const[3] = {1.0, -0.0, 0.5};
template <int I>
__device__ __forceinline__ double fp_const() {
  double r;
  asm("ld.global.f64 %0, [%1];" : "=d"(r) : "l"(__cvta_generic_to_global(g_fp_const + I)));
  return r;
}
__device__ __forceinline__ double add(double a, double b) { return fma(a, fp_const<0>(), b); }
__device__ __forceinline__ double sub(double a, double b) { return fma(-b, fp_const<0>(), a); }
__device__ __forceinline__ double mul(double a, double b) { return fma(a, b, fp_const<1>()); }
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float mul(float a, float b) { return a * b; }

// 1 / x: the hardware's reciprocal approximation y (relative error e below 2^-20) and one
// step of the fourth-order iteration y (1 + e + e^2 + e^3) (Traub 1964, the reciprocal's
// hyperpower series).  The remainder e^4 is below 2^-80 and e is exact to 2^-73, so the
// result is within 0.50001 ulp (tests/test_gpu_math.py).  4 DFMA (256 cycles) in place of 344.
// Outside the normal range (with two binary orders to spare) it divides.
__device__ __forceinline__ double recip(double x) {
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  if (ex - 2u >= 2042u) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, fp_const<0>());
  return fma(y, fma(fma(e, e, e), e, e), y);
}
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }
// -x / 2
__device__ __forceinline__ double half_neg(double x) { return fma(-x, fp_const<2>(), fp_const<1>()); }
__device__ __forceinline__ float half_neg(float x) { return -0.5f * x; }
// sqrt(x), x >= 0 (or NaN): from the hardware's approximation y of 1 / sqrt(x) (relative error
// d below 2^-20) Goldschmidt's coupled iteration (1964): g -> sqrt(x) and h -> 1 / (2 sqrt(x))
// with r = 1/2 - g h, both then within 1.5 d^2 < 2^-39, and a last Newton step g + (x - g^2) h,
// whose residual is exact in the fma and whose remainder is below 2^-77: within 0.50001 ulp
// (tests/test_gpu_math.py).  6 DFMA (384 cycles) in place of 572.  Zero stays zero; outside
// [2^-895, 2^897) it takes sqrt.
__device__ __forceinline__ double root(double x) {
  const unsigned ex = (unsigned)__double2hiint(x) >> 20;
  const bool zero = !nonzero_bits(x);
  if (ex - 128u >= 1792u && !zero) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double h = __hiloint2double(__double2hiint(y) - 0x100000, __double2loint(y));   // y / 2
  double g = mul(x, y);
  const double r = fma(-g, h, fp_const<2>());
  g = fma(g, r, g);
  h = fma(h, r, h);
  g = fma(fma(-g, g, x), h, g);
  return zero ? x : g;
}
__device__ __forceinline__ float root(float x) { return sqrtf(x); }

// ------------------------------------------------------------------------
// Euler physics (eq. euler, G:Euler)
// ------------------------------------------------------------------------
// a b + c d with the fused product fixed: c d rounds, a b fuses into the
// sum.  Left to the compiler, which product of a two-product sum is fused
// depends on the surrounding code, so the same source inlined into two
// kernels could round differently; every such sum on the shared stage paths
// is written with fdot2 (or an explicit fma) so that all kernels agree bit
// for bit.
template <typename T>
__device__ __forceinline__ T fdot2(T a, T b, T c, T d) { return fma(a, b, mul(c, d)); }

// F(u) . d for any direction d (not necessarily unit); returns pressure.
template <typename T>
__device__ __forceinline__ T flux_dir(const T u[4], T dx, T dy, T gm1, T f[4]) {
  const T ri = recip(u[0]);
  const T p = mul(gm1, fma(half_neg(fdot2(u[1], u[1], u[2], u[2])), ri, u[3]));
  const T md = fdot2(u[1], dx, u[2], dy);
  const T vd = mul(md, ri);
  f[0] = md;
  f[1] = fma(u[1], vd, mul(p, dx));
  f[2] = fma(u[2], vd, mul(p, dy));
  f[3] = mul(add(u[3], p), vd);
  return p;
}

// F(u) . d1 and F(u) . d2 with one reciprocal of the density
template <typename T>
__device__ __forceinline__ void flux_dir2(const T u[4], T d1x, T d1y, T d2x, T d2y, T gm1, T f1[4], T f2[4]) {
  const T ri = recip(u[0]);
  const T p = mul(gm1, fma(half_neg(fdot2(u[1], u[1], u[2], u[2])), ri, u[3]));
  const T ep = add(u[3], p);
  const T m1 = fdot2(u[1], d1x, u[2], d1y), v1 = mul(m1, ri);
  const T m2 = fdot2(u[1], d2x, u[2], d2y), v2 = mul(m2, ri);
  f1[0] = m1; f1[1] = fma(u[1], v1, mul(p, d1x)); f1[2] = fma(u[2], v1, mul(p, d1y)); f1[3] = mul(ep, v1);
  f2[0] = m2; f2[1] = fma(u[1], v2, mul(p, d2x)); f2[2] = fma(u[2], v2, mul(p, d2y)); f2[3] = mul(ep, v2);
}

// x > 0 on the integer units for doubles (differs from the comparison only
// for a NaN with a clear sign bit); a plain comparison for floats
__device__ __forceinline__ bool gt0(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool gt0(float x) { return x > 0.0f; }
// exp(-x), x >= 0 (or NaN): small FP64 arguments, the usual case of the OE
// damping away from discontinuities, take a 7-FMA Taylor polynomial
// (dg_math.h); the rest the library exp; FP32 the fast intrinsic, whose
// error (a few ulp) is far below the mixed form's FP32 arithmetic error
__device__ __forceinline__ double exp_neg(double x) {
  static_assert(EXP_NEG_SMALL_MAX == 0.00390625, "the high word below");
  // x < 2^-8 on the integer units (x >= 0, or NaN, whose high word is above)
  return (unsigned)__double2hiint(x) < 0x3f700000u ? exp_neg_small(x) : exp(-x);
}
__device__ __forceinline__ float exp_neg(float x) { return __expf(-x); }

// F(u) . n and the spectral radius |v.n| + c (+inf for rho <= 0) with one reciprocal
template <typename T>
__device__ __forceinline__ T flux_speed(const T u[4], T nx, T ny, T gm1, T gamma, T f[4]) {
  const T ri = recip(u[0]);
  const T p = mul(gm1, fma(half_neg(fdot2(u[1], u[1], u[2], u[2])), ri, u[3]));
  const T mn = fdot2(u[1], nx, u[2], ny);
  const T vn = mul(mn, ri);
  f[0] = mn;
  f[1] = fma(u[1], vn, mul(p, nx));
  f[2] = fma(u[2], vn, mul(p, ny));
  f[3] = mul(add(u[3], p), vn);
  if (!gt0(u[0])) return T(INFINITY);
  const T pc = gt0(p) ? p : T(0);
  return add(T(fabs(vn)), root(mul(mul(gamma, pc), ri)));
}

// spectral radius |v.n| + c; +inf for rho <= 0, pressure clamped at 0
template <typename T>
__device__ __forceinline__ T wave_speed(const T u[4], T nx, T ny, T gamma) {
  if (!gt0(u[0])) return T(INFINITY);
  const T ri = T(1) / u[0];
  T p = (gamma - T(1)) * fma(T(-0.5) * fdot2(u[1], u[1], u[2], u[2]), ri, u[3]);
  p = gt0(p) ? p : T(0);
  return fma(fabs(fdot2(u[1], nx, u[2], ny)), ri, sqrt(gamma * p * ri));
}

__device__ __forceinline__ double int_energy(const double u[4]) {
  return u[3] - 0.5 * fdot2(u[1], u[1], u[2], u[2]) / u[0];
}

// exterior state of a boundary edge (tag > 0) at physical point (px, py),
// time t, from the interior trace um and the cell average avg
template <typename T>
__device__ __forceinline__ void ghost_state(int tag, const T um[4], const T avg[4], T nx, T ny, double px,
                                            double py, double t, const Phys &ph, T up[4]) {
  if (tag == 1) {                       // reflecting wall: m - 2 (m . n) n, the fused product fixed
    const T mn2 = T(-2) * fdot2(um[1], nx, um[2], ny);
    up[0] = um[0];
    up[1] = fma(mn2, nx, um[1]);
    up[2] = fma(mn2, ny, um[2]);
    up[3] = um[3];
  } else if (tag >= 3 && tag <= 6) {    // constant state
#pragma unroll
    for (int c = 0; c < 4; ++c) up[c] = T(ph.bc[tag - 3][c]);
  } else if (tag == 7) {                // moving shock
    const double xs = fma(py, ph.shock_cot, fma(t, ph.shock_vx, ph.shock_x0));
    const int s = px < xs ? ph.shock_post : ph.shock_pre;
#pragma unroll
    for (int c = 0; c < 4; ++c) up[c] = T(ph.bc[s][c]);
  } else {                              // transmissive: the cell average (a constant state)
#pragma unroll
    for (int c = 0; c < 4; ++c) up[c] = avg[c];
  }
}

// ------------------------------------------------------------------------
// Deterministic block reductions
// ------------------------------------------------------------------------
// Maximum of two non-negative doubles (or +inf, or NaN) on the integer units:
// for x, y >= +0 the IEEE bit patterns order like the numbers, and a NaN of
// either sign compares above every number, so it propagates.  A double
// comparison would occupy GB300's narrow FP64 pipe.
__device__ __forceinline__ double max_nn(double a, double b) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(a);
  const unsigned long long y = (unsigned long long)__double_as_longlong(b);
  return __longlong_as_double((long long)(x > y ? x : y));
}
__device__ __forceinline__ float max_nn(float a, float b) { return (a > b || a != a) ? a : b; }

// x is neither infinite nor NaN, tested on the integer units
__device__ __forceinline__ bool is_finite_bits(double x) {
  return (__double_as_longlong(x) & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool is_finite_bits(float x) {
  return (__float_as_int(x) & 0x7f800000) != 0x7f800000;
}

// FP64 to FP32 and back on the integer units (a conversion instruction takes 64
// cycles of the FP64 pipe, which the mixed form's flux pass keeps half busy).  In that
// pass, 24 conversions per cell, 1,036,800 cells: 0.173 -> 0.157 ms (P2), 0.146 -> 0.135 ms (P1);
// in its OE pass, bound by latency and registers, slower (0.237 -> 0.254 ms), so it converts as is.
//
// To nearest, ties away from zero; results below 2^-126 are zero, those beyond the FP32 range
// infinite, NaN stays NaN.
__device__ __forceinline__ float f32_of(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned long long r = (((unsigned long long)(hi & 0x7fffffffu) << 32) | lo) + 0x10000000ull - 0x3800000000000000ull;
  const int t = (int)(r >> 32);
  unsigned b = __funnelshift_l((unsigned)r, (unsigned)t, 3);
  b = t < 0x00100000 ? 0u : b;
  if (t >= 0x0ff00000) b = r > 0x47f0000010000000ull ? 0x7fffffffu : 0x7f800000u;
  return __uint_as_float(b | (hi & 0x80000000u));
}
// exact; subnormals count as zero, infinities and NaN stay what they are
__device__ __forceinline__ double f64_of(float x) {
  const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
  const unsigned e = a < 0x00800000u ? 0u : (a >> 3) + (a >= 0x7f800000u ? 0x70000000u : 0x38000000u);
  return __hiloint2double((int)(e | (b & 0x80000000u)), a < 0x00800000u ? 0 : (int)(b << 29));
}

// Order-preserving integer key of a double (NaN aside): negative numbers get
// their magnitude bits flipped, so signed integer comparison orders the keys
// like the numbers (-0 sorts just below +0).  The map is its own inverse.
__device__ __forceinline__ long long ord_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double ord_val(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

struct OpSum {
  template <typename T> __device__ T operator()(T a, T b) const { return a + b; }
  template <typename T> __device__ static T ident() { return T(0); }
};
// NaN-propagating maximum of non-negative values
struct OpMaxNN {
  template <typename T> __device__ T operator()(T a, T b) const { return max_nn(a, b); }
  template <typename T> __device__ static T ident() { return T(0); }
};

constexpr int pow2_ceil(int n) { return n <= 1 ? 1 : 2 * pow2_ceil((n + 1) / 2); }

// Warp reduction of N values per lane by transposition: at each of the first
// log2(P) shuffle levels (P = N rounded up to a power of two) a lane keeps half
// of its values and adds the partner's copies of them, so the level costs half
// as many operations as the one before; the remaining levels are a butterfly on
// one value.  Component q ends on lanes q * 32 / P (and their butterfly
// partners).  The tree is fixed, so the result is reproducible.
template <int N, typename T, typename Op>
__device__ __forceinline__ T warp_reduce_transposed(const T v[N], Op op) {
  constexpr int P = pow2_ceil(N);
  static_assert(P <= 32, "too many values for one warp");
  const int lane = threadIdx.x & 31;
  T w[P];
#pragma unroll
  for (int q = 0; q < P; ++q) w[q] = q < N ? v[q] : Op::template ident<T>();
  int o = 16;
#pragma unroll
  for (int cnt = P; cnt > 1; cnt >>= 1, o >>= 1) {
    const int half = cnt >> 1;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const T send = up ? w[j] : w[j + half];
      const T keep = up ? w[j + half] : w[j];
      w[j] = op(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1) w[0] = op(w[0], __shfl_xor_sync(0xffffffffu, w[0], o));
  return w[0];
}

// Block reduction: transposed warp reduction, then the warps in order.  Ends
// with a barrier, so the block may call it again at once.
template <int N, typename T, typename U, typename Op>
__device__ __forceinline__ void block_reduce(const T v[N], U *out, Op op) {
  constexpr int P = pow2_ceil(N);
  __shared__ T red[TPB / 32][N > 0 ? N : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T r = warp_reduce_transposed<N, T, Op>(v, op);
  if (lane % (32 / P) == 0 && lane / (32 / P) < N) red[warp][lane / (32 / P)] = r;
  __syncthreads();
  if (threadIdx.x < N) {
    T s = red[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < TPB / 32; ++w) s = op(s, red[w][threadIdx.x]);
    out[threadIdx.x] = U(s);
  }
  __syncthreads();
}

// Fixed-order reduction of nblk partials of N values by one block: FIN_THREADS
// virtual lanes each reduce a strided subset, then a fixed tree.  The
// arithmetic does not depend on the block size, so a persistent kernel with
// TPB threads reproduces the FIN_THREADS-thread finalize kernels bitwise.  The
// strided loop loads four partials ahead of the operations, in the same order.
// Shared scratch of fin_reduce: one array per kernel, whatever the value type
// and count, so a kernel that reduces several kinds of partials stays within
// the static shared-memory limit.
__device__ __forceinline__ unsigned char *fin_scratch() {
  __shared__ __align__(16) unsigned char buf[FIN_THREADS * 5 * sizeof(double)];
  return buf;
}

template <int N, typename T, typename Op>
__device__ void fin_reduce(const T *part, int nblk, T init, Op op, T out[N]) {
  static_assert(N * sizeof(T) <= 5 * sizeof(double), "fin_scratch too small");
  T (*sh)[N] = reinterpret_cast<T (*)[N]>(fin_scratch());
  for (int vt = threadIdx.x; vt < FIN_THREADS; vt += blockDim.x) {
    T acc[N];
#pragma unroll
    for (int q = 0; q < N; ++q) acc[q] = init;
    int b = vt;
    for (; b + 3 * FIN_THREADS < nblk; b += 4 * FIN_THREADS) {
      T x[4][N];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < N; ++q) x[u][q] = part[(int64_t)(b + u * FIN_THREADS) * N + q];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < N; ++q) acc[q] = op(acc[q], x[u][q]);
    }
    for (; b < nblk; b += FIN_THREADS)
#pragma unroll
      for (int q = 0; q < N; ++q) acc[q] = op(acc[q], part[(int64_t)b * N + q]);
#pragma unroll
    for (int q = 0; q < N; ++q) sh[vt][q] = acc[q];
  }
  __syncthreads();
  for (int st = FIN_THREADS / 2; st > 0; st >>= 1) {
    for (int vt = threadIdx.x; vt < st; vt += blockDim.x)
#pragma unroll
      for (int q = 0; q < N; ++q) sh[vt][q] = op(sh[vt][q], sh[vt + st][q]);
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < N; ++q) out[q] = sh[0][q];
  __syncthreads();
}

// ------------------------------------------------------------------------
// Per-solve finalize steps (one block; thread 0 writes the scalars)
// ------------------------------------------------------------------------
// 1 / D_q of the damped quantities from sc->dev and sc->mean (eqs.
// OEScalar:Coef2, RIOESys:Coef1/Coef2 with the round-off guard of Sec. 2.3:
// a component whose deviation is below 1e-12 max(1, |mean|) is constant)
__device__ __forceinline__ double inv_normaliser(int q, const double dev[5], const double mean[4], int cw) {
  const double eps = 1e-12;
  const bool mom = !cw && (q == 1 || q == 2);
  const double D = q == 0 ? dev[0] : q == 3 ? dev[2] : mom ? dev[1] : q == 1 ? dev[3] : dev[4];
  const double ref = mom ? sqrt(fdot2(mean[1], mean[1], mean[2], mean[2])) : fabs(mean[q]);
  return D <= eps * fmax(1.0, ref) ? 0.0 : 1.0 / D;
}
__device__ __forceinline__ void write_inv_normalisers(Scalars *sc, int cw) {
  for (int q = 0; q < 4; ++q) {
    sc->invD[q] = q == 2 && !cw ? sc->invD[1] : inv_normaliser(q, sc->dev, sc->mean, cw);
    sc->invDf[q] = float(sc->invD[q]);
  }
}

// ------------------------------------------------------------------------
// Finalisation inside the producing kernel, in a fixed order
// ------------------------------------------------------------------------
// The tiles of a reduction (TileCells cells each, one partial per tile) form groups
// of TILE_GROUP consecutive tiles.  After writing the partials of its tiles, a block takes
// their tickets of the group; the block that takes the group's last ticket reduces
// the group's partials with block_reduce and takes a ticket at the top level;
// the block that takes the last top-level ticket reduces the group results in
// chunks of TPB, in order, and writes the scalars.  The arithmetic depends only
// on the number of tiles, not on which block finishes when, so results are
// reproducible and the same in the per-solve kernels and the batch kernel.
// Every ticket counter is reset by the block that takes its last ticket, so it
// is zero again when the next launch (or batch phase) starts.
constexpr int TILE_GROUP = TPB;
__host__ __device__ __forceinline__ int64_t num_groups(int64_t ntiles) {
  return (ntiles + TILE_GROUP - 1) / TILE_GROUP;
}
// ticket counters of one reduction: one per group, then the top level
__host__ __device__ __forceinline__ int64_t ticket_slots(int64_t ntiles) { return num_groups(ntiles) + 1; }

// Called by every thread of the block once the block's results are written:
// takes n tickets of *cnt, true in the block that took the last of `total`.
// The block's writes are ordered before the ticket by the barrier and one
// device-scope fence of thread 0 (cumulative over what the barrier ordered);
// the last block fences again before its threads read the other blocks'
// results.
__device__ __forceinline__ bool take_ticket(unsigned *cnt, unsigned total, unsigned n = 1) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned t = atomicAdd(cnt, n);
    const int last = t + n == total;
    if (last) {
      atomicExch(cnt, 0u);               // every ticket is taken: reset for the next launch
      __threadfence();
    }
    s_last = last;
  }
  __syncthreads();
  const bool last = s_last != 0;
  __syncthreads();                       // s_last may be rewritten by the next call
  return last;
}

// partials of other blocks are read from L2 (L1 is not coherent across SMs)
__device__ __forceinline__ double ld_l2(const double *p) { return __ldcg(p); }
__device__ __forceinline__ long long ld_l2(const long long *p) { return __ldcg(p); }

// group g's partials -> grp[g]
template <int N, typename T, typename Op>
__device__ __forceinline__ void reduce_group(const T *part, int64_t g, int64_t ntiles, T *grp, Op op) {
  const int64_t t0 = g * TILE_GROUP;
  const int64_t n = ntiles - t0 < TILE_GROUP ? ntiles - t0 : TILE_GROUP;
  T v[N];
#pragma unroll
  for (int q = 0; q < N; ++q)
    v[q] = threadIdx.x < n ? ld_l2(part + (t0 + threadIdx.x) * N + q) : Op::template ident<T>();
  block_reduce<N>(v, grp + g * N, op);
}

// all group results, in chunks of TPB -> out[] in every thread
template <int N, typename T, typename Op>
__device__ __forceinline__ void reduce_top(const T *grp, int64_t ng, Op op, T out[N]) {
  __shared__ T res[N];
#pragma unroll
  for (int q = 0; q < N; ++q) out[q] = Op::template ident<T>();
  for (int64_t c0 = 0; c0 < ng; c0 += TPB) {
    T v[N];
#pragma unroll
    for (int q = 0; q < N; ++q)
      v[q] = c0 + threadIdx.x < ng ? ld_l2(grp + (c0 + threadIdx.x) * N + q) : Op::template ident<T>();
    block_reduce<N>(v, res, op);
#pragma unroll
    for (int q = 0; q < N; ++q) out[q] = op(out[q], res[q]);
    __syncthreads();
  }
}

// scratch of the in-kernel finalisation of one solve
struct FinBufs {
  double *grp_sum, *grp_dev, *grp_alpha;   // [ng][4], [ng][5], [ng]
  long long *grp_cnt;                      // [ng][2]
  unsigned *tick;                          // 3 reductions x ticket_slots(ntiles)
};

// Top level of each finalisation: the block that takes the last top-level
// ticket reduces the group results and writes the scalars.  The three kinds
// use consecutive ranges of ticket_slots(ntiles) counters.
__device__ __forceinline__ void finish_means_top(const FinBufs &f, int64_t ntiles, Scalars *sc) {
  const int64_t ng = num_groups(ntiles);
  if (!take_ticket(f.tick + ng, (unsigned)ng)) return;
  double r[4];
  reduce_top<4>(f.grp_sum, ng, OpSum(), r);
  if (threadIdx.x == 0)
    for (int c = 0; c < 4; ++c) sc->mean[c] = r[c] / sc->area_total;
}

__device__ __forceinline__ void finish_deviations_top(const FinBufs &f, int64_t ntiles, Scalars *sc, int cw) {
  const int64_t ng = num_groups(ntiles);
  if (!take_ticket(f.tick + ticket_slots(ntiles) + ng, (unsigned)ng)) return;
  double r[5];
  reduce_top<5>(f.grp_dev, ng, OpMaxNN(), r);
  if (threadIdx.x == 0) {
    for (int q = 0; q < 5; ++q) sc->dev[q] = r[q];
    write_inv_normalisers(sc, cw);
  }
}

// alpha of the next stage input, counters, and after the last stage t += dt
// (stage < 0: outside a step, alpha and counters only)
__device__ __forceinline__ void finish_alpha_top(const FinBufs &f, int64_t ntiles, Scalars *sc, int stage) {
  const int64_t ng = num_groups(ntiles);
  if (!take_ticket(f.tick + 2 * ticket_slots(ntiles) + ng, (unsigned)ng)) return;
  double a[1];
  long long c[2];
  reduce_top<1>(f.grp_alpha, ng, OpMaxNN(), a);
  reduce_top<2>(f.grp_cnt, ng, OpSum(), c);
  if (threadIdx.x == 0) {
    sc->alpha = a[0];
    sc->limited += c[0];
    sc->nonphys += c[1];
    if (stage == 0 || stage == 1) {
      if (a[0] * sc->dt > sc->min_ca * (1.0 + 1e-12)) sc->breaches += 1;
    } else if (stage == 2) {
      sc->t = sc->pad ? sc->t_end : sc->t + sc->dt;
      sc->steps += 1;
    }
  }
}

// Group level.  In the per-solve finalize kernels block g reduces group g
// directly; in the batch kernel the block that finishes a group's last tiles
// does (after the group's tickets), so both produce the same group results.
// A block takes the tickets of a whole chunk of tiles at once: one fence and three barriers
// per chunk, not per tile.  fn(g) for every group that the n tiles from `first` complete.
template <typename F>
__device__ __forceinline__ void complete_groups(const FinBufs &f, int kind, int64_t first, int64_t n, int64_t ntiles,
                                                F fn) {
  for (int64_t g = first / TILE_GROUP; g * TILE_GROUP < first + n; ++g) {
    const int64_t t0 = g * TILE_GROUP, t1 = min(t0 + TILE_GROUP, ntiles);
    const int64_t mine = min(t1, first + n) - max(t0, first);
    if (take_ticket(f.tick + kind * ticket_slots(ntiles) + g, (unsigned)(t1 - t0), (unsigned)mine)) fn(g);
  }
}

// in-kernel finalisation after the n tiles from `first` wrote their partials (batch kernel)
__device__ __forceinline__ void finish_means(const double *part_sum, const FinBufs &f, int64_t first, int64_t n,
                                             int64_t ntiles, Scalars *sc) {
  complete_groups(f, 0, first, n, ntiles, [&](int64_t g) {
    reduce_group<4>(part_sum, g, ntiles, f.grp_sum, OpSum());
    finish_means_top(f, ntiles, sc);
  });
}
__device__ __forceinline__ void finish_deviations(const double *part_dev, const FinBufs &f, int64_t first, int64_t n,
                                                  int64_t ntiles, Scalars *sc, int cw) {
  complete_groups(f, 1, first, n, ntiles, [&](int64_t g) {
    reduce_group<5>(part_dev, g, ntiles, f.grp_dev, OpMaxNN());
    finish_deviations_top(f, ntiles, sc, cw);
  });
}
__device__ __forceinline__ void finish_alpha(const double *part_alpha, const long long *part_cnt, const FinBufs &f,
                                             int64_t first, int64_t n, int64_t ntiles, Scalars *sc, int stage) {
  complete_groups(f, 2, first, n, ntiles, [&](int64_t g) {
    reduce_group<1>(part_alpha, g, ntiles, f.grp_alpha, OpMaxNN());
    reduce_group<2>(part_cnt, g, ntiles, f.grp_cnt, OpSum());
    finish_alpha_top(f, ntiles, sc, stage);
  });
}

// dt of the BP CFL condition (Sec. 5), clamped to t_end; inactive once t >= t_end
__device__ __forceinline__ void step_begin_thread(Scalars *sc) {
  if (sc->t < sc->t_end) {
    double dt = sc->cfl * sc->min_ca / sc->alpha;
    int clamped = 0;
    if (sc->t + dt >= sc->t_end) { dt = sc->t_end - sc->t; clamped = 1; }
    sc->dt = dt;
    sc->pad = clamped;
    sc->active = 1;
  } else {
    sc->dt = 0.0;
    sc->active = 0;
  }
}

// ------------------------------------------------------------------------
// Finalisation inside the consuming kernel (few tiles)
// ------------------------------------------------------------------------
// A finalize kernel of a small mesh is one block and almost all latency
// (launch, partials from L2, a serial chain of FP64 operations, the ticket): about
// 5 us, nine times per step.  With at most FUSE_GROUPS groups of tiles every
// block of the consuming kernel takes the reduction itself, in the order of the
// finalize kernels, into a copy of the scalars in its shared memory, and one block
// more, without a tile, writes them back.  No field that a block of the same launch reads from
// memory for its result is written in that launch.  Vortex, 2,048 P1 cells FP64: 92 us per
// step; Riemann problem, 1,058 P2 cells mixed: 78 us; with finalize launches 127 and 118.
// The limit, separate and fused: P2 FP64, 2 groups (7,688 cells) 178 and 166 us, 4 groups
// 229 and 243 us; mixed, 2 groups (31,250 cells) 125 and 116 us, 4 groups 144 and 161 us.
// The kernels have a variant for it: chosen at run time it cost the mixed form's large
// meshes 1.5 %.
constexpr int FUSE_GROUPS = 2;
struct Fuse {
  int on;                   // which kernel to launch: the one that finishes the reduction itself
  int ntiles;
  const double *part;       // partials of the kernel before (nullptr: none, the step start)
  const long long *cnt;     // counters beside the wave speeds
  Scalars *sc;
};

// Where a tile function gets its scalars: begin() starts the loads, end() returns
// them (every thread of the block calls both).  In between go the tile's own
// loads and whatever work needs no scalar, so that the latency of the
// reduction and that of the state overlap (5 to 6 % of a small mesh's step).
struct PlainScalars {
  static constexpr bool FUSED = false;
  const Scalars *sc;
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ const Scalars *end() { return sc; }
};

// partials of the first group -> v; all partials -> out[] in every thread, the
// arithmetic of reduce_group and reduce_top
template <int N, typename T, typename Op>
__device__ __forceinline__ void fused_load(const T *part, int ntiles, Op op, T v[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q)
    v[q] = (int)threadIdx.x < min(ntiles, TILE_GROUP) ? ld_l2(part + threadIdx.x * N + q) : Op::template ident<T>();
}
template <int N, typename T, typename Op>
__device__ __forceinline__ void fused_reduce(const T *part, int ntiles, Op op, const T first[N], T out[N]) {
  __shared__ T grp[FUSE_GROUPS * N];
  const int ng = (ntiles + TILE_GROUP - 1) / TILE_GROUP;
  block_reduce<N>(first, grp, op);
  for (int g = 1; g < ng; ++g) reduce_group<N>(part, g, ntiles, grp, op);
  if (ng > 1) {
    T v[N];
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = threadIdx.x < ng ? grp[threadIdx.x * N + q] : Op::template ident<T>();
    block_reduce<N>(v, grp, op);
  }
#pragma unroll
  for (int q = 0; q < N; ++q) out[q] = op(Op::template ident<T>(), grp[q]);
}
// The scalars in shared memory, one word per thread.  The block after the last
// tile writes the new ones back.
struct FusedScalars {
  static constexpr bool FUSED = true;
  static_assert(sizeof(Scalars) % 8 == 0 && sizeof(Scalars) / 8 <= TPB, "one word per thread");
  Fuse f;
  Scalars *s;   // shared
  double word;
  __device__ __forceinline__ FusedScalars(const Fuse &f_, Scalars *s_) : f(f_), s(s_), word(0.0) {}
  __device__ __forceinline__ bool writer() const { return (int)blockIdx.x == f.ntiles; }
  __device__ __forceinline__ void load() {
    if (threadIdx.x < sizeof(Scalars) / 8) word = reinterpret_cast<const double *>(f.sc)[threadIdx.x];
  }
  __device__ __forceinline__ void store() {
    if (threadIdx.x < sizeof(Scalars) / 8) reinterpret_cast<double *>(s)[threadIdx.x] = word;
    __syncthreads();
  }
};

// domain means (before K2), normalisers (before K3), alpha of the stage input or
// the step start (before K1)
struct FuseMeans : FusedScalars {
  double v[4];
  using FusedScalars::FusedScalars;
  __device__ __forceinline__ void begin() {
    load();
    fused_load<4>(f.part, f.ntiles, OpSum(), v);
  }
  __device__ __forceinline__ const Scalars *end() {
    double r[4];
    fused_reduce<4>(f.part, f.ntiles, OpSum(), v, r);
    store();
    if (threadIdx.x < 4) {
      const int q = threadIdx.x;
      const double mean = (q == 0 ? r[0] : q == 1 ? r[1] : q == 2 ? r[2] : r[3]) / s->area_total;
      s->mean[q] = mean;
      if (writer() && s->active) f.sc->mean[q] = mean;
    }
    __syncthreads();
    return s;
  }
};
struct FuseDeviations : FusedScalars {
  double v[5];
  int cw;
  __device__ __forceinline__ FuseDeviations(const Fuse &f_, Scalars *s_, int cw_) : FusedScalars(f_, s_), cw(cw_) {}
  __device__ __forceinline__ void begin() {
    load();
    fused_load<5>(f.part, f.ntiles, OpMaxNN(), v);
  }
  __device__ __forceinline__ const Scalars *end() {
    double r[5];
    fused_reduce<5>(f.part, f.ntiles, OpMaxNN(), v, r);
    store();
    if (threadIdx.x < 4) {   // one component per thread
      const int q = threadIdx.x;
      const double iD = inv_normaliser(q, r, s->mean, cw);
      s->invD[q] = iD;
      s->invDf[q] = float(iD);
      if (writer() && s->active) {
        f.sc->invD[q] = iD;
        f.sc->invDf[q] = float(iD);
      }
    }
    if (threadIdx.x == 0 && writer() && s->active)
      for (int q = 0; q < 5; ++q) f.sc->dev[q] = r[q];
    __syncthreads();
    return s;
  }
};
struct FuseAlpha : FusedScalars {
  double v[1];
  using FusedScalars::FusedScalars;
  __device__ __forceinline__ void begin() {
    load();
    if (f.part) fused_load<1>(f.part, f.ntiles, OpMaxNN(), v);
  }
  __device__ __forceinline__ const Scalars *end() {
    if (f.part) {
      double a[1];
      fused_reduce<1>(f.part, f.ntiles, OpMaxNN(), v, a);
      store();
      if (!s->active) return s;   // an idle step leaves the counters alone
      long long n[2] = {0, 0};
      if (writer()) {
        long long c[2];
        fused_load<2>(f.cnt, f.ntiles, OpSum(), c);
        fused_reduce<2>(f.cnt, f.ntiles, OpSum(), c, n);
      }
      if (threadIdx.x == 0) {
        s->alpha = a[0];
        if (writer()) {   // as finish_alpha_top after stage 0 or 1
          f.sc->alpha = a[0];
          f.sc->limited += n[0];
          f.sc->nonphys += n[1];
          if (a[0] * s->dt > s->min_ca * (1.0 + 1e-12)) f.sc->breaches += 1;
        }
      }
    } else {
      store();
      if (threadIdx.x == 0) {
        step_begin_thread(s);
        if (writer()) {
          f.sc->dt = s->dt;
          f.sc->pad = s->pad;
          f.sc->active = s->active;
        }
      }
    }
    __syncthreads();
    return s;
  }
};

}  // namespace dg
