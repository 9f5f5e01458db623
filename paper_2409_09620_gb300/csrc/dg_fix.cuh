// dg_fix.cuh -- block fixed-point arithmetic for the FP64 form's contractions
// with constant tables (basis values at points, quadrature sums), plain C++
// where compiled without CUDA (host self-test).
//
// GB300 runs an FP64 warp instruction in 64 cycles per scheduler when all
// operands are registers and in 76 when one is an immediate or a constant
// (a compile-time basis value always is; DADD and DMUL always take 76), while
// a 32 x 32 + 64 bit integer multiply-add takes about 2.  A sum
// sum_j c_j x_j with constants c_j therefore runs on the integer units, about
// 9 cycles per term, beside the FP64 pipe:
//
//   * the values x_j of a block (a cell's modes of one component, its fluxes
//     at the volume points, ...) share the exponent E of the largest:
//     x_j = (h 2^29 + l) 2^(E - 1080), |h 2^29 + l| < 2^58, truncated at 2^-58
//     of the block's largest magnitude (FP64 rounds at 2^-53 of each term);
//   * a constant |c| <= 4 is (h 2^29 + l) 2^-56 with |l| <= 2^28;
//   * the products h h and h l + l h accumulate exactly in two 64-bit
//     integers (l l, below 2^-57 of the block, is dropped), so the order of
//     the terms does not matter;
//   * the result converts to FP64 with one rounding.
//
// The error of a sum is a few 2^-57 of the block's largest magnitude
// (tests/test_fix_host.py).  Where that value is a term of the sum (point values,
// quadrature sums), an FMA chain rounds at 2^-53 of it.  Where it would not be,
// the terms have a block of their own: derivatives, which do not contain the
// cell average (dg_fix_vertex.cuh, dg_fix_scalar.cuh; tests/test_fix_vertex_host.py and
// tests/test_fix_scalar_host.py compare them with the chain).  Zeros stay zero,
// subnormals count as zero and blocks below 2^-959 keep an absolute 2^-1016;
// a result beyond FP64's range is infinite; a block that holds an infinity or a
// NaN has E = 0x7ff, and the callers turn its results into NaN.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#define FX_CONST __host__ __device__ constexpr
#else
#define FX_HD inline
#define FX_CONST constexpr
#endif

namespace dg {

constexpr int FX_LIMB = 29;          // bits of the low limb
constexpr int FX_ONE = 56;           // a constant c is stored as round(c 2^56)
constexpr int FX_EMIN = 64, FX_ENAN = 0x7ff;   // smallest block exponent used; exponent of a non-finite block

FX_HD int fx_hiword(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
FX_HD unsigned fx_loword(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return (unsigned)b;
#endif
}
FX_HD double fx_make(int hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, (int)lo);
#else
  const int64_t b = (int64_t)(((uint64_t)(unsigned)hi << 32) | lo);
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
// 127 + floor(log2 a), 0 for a = 0, from the exponent field of the leading 32
// bits rounded toward zero to FP32 (a 64-bit conversion would run on the FP64
// pipe, 64 cycles)
FX_HD int fx_log2_127(uint64_t a) {
  const unsigned hi = (unsigned)(a >> 32), t = hi ? hi : (unsigned)a;
#ifdef __CUDA_ARCH__
  const int e = __float_as_int(__uint2float_rz(t)) >> 23;
#else
  const int e = t == 0 ? 0 : 158 - __builtin_clz(t);
#endif
  return hi ? e + 32 : e;
}

// constant: c = (h 2^29 + l) 2^-56, |l| <= 2^28
struct FxC {
  int h, l;
};
FX_CONST FxC fxc(double c) {
  const double s = c * double(1LL << FX_ONE);
  const int64_t v = (int64_t)(s < 0.0 ? s - 0.5 : s + 0.5);
  const int64_t h = (v + (1LL << (FX_LIMB - 1))) >> FX_LIMB;
  return FxC{(int)h, (int)(v - h * (1LL << FX_LIMB))};
}

// the constant c f with one rounding, f of a few bits (a product in FP64 would round by up to
// 2^-53 of it first, the same in every cell and step): c split into halves of 26 bits (Dekker 1971)
FX_CONST FxC fxc(double c, double f) {
  const double t = c * 134217729.0, ch = t - (t - c), cl = c - ch, one = double(1LL << FX_ONE);
  const double s1 = ch * f * one, s2 = cl * f * one;   // exact
  const int64_t i = (int64_t)s1;
  const double r = (s1 - double(i)) + s2;
  const int64_t v = i + (int64_t)(r < 0.0 ? r - 0.5 : r + 0.5);
  const int64_t h = (v + (1LL << (FX_LIMB - 1))) >> FX_LIMB;
  return FxC{(int)h, (int)(v - h * (1LL << FX_LIMB))};
}

// exponent of a block from the bitwise-positive high words of its values
FX_HD int fx_abs_hi(double x) { return fx_hiword(x) & 0x7fffffff; }
FX_HD int fx_exp(int max_abs_hi) {
  const int e = max_abs_hi >> 20;
  return e < FX_EMIN ? FX_EMIN : e;
}

// a value of a block with exponent E (|x| < 2^(E - 1022))
struct Fx {
  int h, l;
};
FX_HD Fx fx_from(double x, int E) {
  const int hi = fx_hiword(x);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const uint64_t m = (((uint64_t)mh << 32) | fx_loword(x)) << 5;
  // E >= 64, so a zero or subnormal x (exponent field 0) shifts out
  int s = E - ((hi >> 20) & 0x7ff);
  s = s > 63 ? 63 : s;
  const uint64_t v = m >> s;
  const int g = (hi >> 31) | 1;        // sign
  return Fx{(int)(v >> FX_LIMB) * g, ((int)v & ((1 << FX_LIMB) - 1)) * g};
}

// s + a b as one 32 x 32 + 64 bit multiply-add (left to itself the compiler
// multiplies sign-extended 64-bit values, several instructions each)
FX_HD void fx_mad(int64_t &s, int a, int b) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
#else
  s += (int64_t)a * b;
#endif
}
// sum of products, exact but for the dropped l l
struct FxAcc {
  int64_t a, b;
};
FX_HD void fx_mac(FxAcc &s, FxC c, Fx x) {
  if (c.h != 0) {
    fx_mad(s.a, c.h, x.h);
    fx_mad(s.b, c.h, x.l);
  }
  if (c.l != 0) fx_mad(s.b, c.l, x.h);
}
// run-time coefficient c = x 2^k (|c| < 4) in the format of a constant, as fx_mac takes it
FX_HD Fx fx_coef(double x, int k) {
  return (fx_hiword(x) & 0x7ff00000) == 0 ? Fx{0, 0} : fx_from(x, 1024 - k);
}
FX_HD void fx_mac(FxAcc &s, Fx c, Fx x) {
  fx_mad(s.a, c.h, x.h);
  fx_mad(s.b, c.h, x.l);
  fx_mad(s.b, c.l, x.h);
}
// difference of two values of a block, one bit longer than a value
FX_HD Fx operator-(Fx p, Fx q) { return Fx{p.h - q.h, p.l - q.l}; }
// a sum back as a value, shifted right by s (its block's exponent grows by s); |r| < 2^(58 + s)
FX_HD Fx fx_value(int64_t r, int s) {
  const int64_t v = r >> s;
  return Fx{(int)(v >> FX_LIMB), (int)v & ((1 << FX_LIMB) - 1)};
}
// a value as one integer
FX_HD int64_t fx_join(Fx x) { return (int64_t)x.h * (1LL << FX_LIMB) + x.l; }
// a - b of blocks with exponents Ea, Eb, in that of E >= Ea, Eb; below 2^61
FX_HD int64_t fx_diff(Fx a, int Ea, Fx b, int Eb, int E) {
  return (fx_join(a) >> (E - Ea < 63 ? E - Ea : 63)) - (fx_join(b) >> (E - Eb < 63 ? E - Eb : 63));
}
// the same as limbs of exponent E + S; |a - b| < 2^(60 + S), for the high limb has 32 bits
template <int S>
FX_HD Fx fx_jump(Fx a, int Ea, Fx b, int Eb, int E) {
  return fx_value(fx_diff(a, Ea, b, Eb, E), S);
}
// r 2^-s to nearest, |r| < 2^62, s >= 0
FX_HD int64_t fx_shift(int64_t r, int s) {
  s = s < 63 ? s : 63;
  return (r + (int64_t)((1ULL << s) >> 1)) >> s;
}
// the sum's last unit is rounded down, from FxAcc{0, FX_HALF} on to nearest
constexpr int64_t FX_HALF = 1LL << (FX_ONE - FX_LIMB - 1);
FX_HD int64_t fx_sum(const FxAcc &s) {
  return s.a * (1LL << (2 * FX_LIMB - FX_ONE)) + (s.b >> (FX_ONE - FX_LIMB));
}
// the same rounded to nearest
FX_HD int64_t fx_round(const FxAcc &s) { return fx_sum(FxAcc{s.a, s.b + FX_HALF}); }
// sum of products with run-time coefficients, l l included (their low limbs reach
// 2^29, so that dropping it costs up to 4 units of the result per term), and rounded
struct FxAccL {
  int64_t a, b, l;
};
FX_HD void fx_mac(FxAccL &s, Fx c, Fx x) {
  fx_mad(s.a, c.h, x.h);
  fx_mad(s.b, c.h, x.l);
  fx_mad(s.b, c.l, x.h);
  fx_mad(s.l, c.l, x.l);
}
FX_HD int64_t fx_round(const FxAccL &s) { return fx_round(FxAcc{s.a, s.b + (s.l >> FX_LIMB)}); }
// r 2^(E - 1080) rounded to nearest, |r| < 2^63 and E >= FX_NEAR_MIN, so that it is not below
// FP64's normal numbers: fx_near for E <= FX_NEAR_MAX, fx_to infinite beyond FP64's range
constexpr int FX_NEAR_MIN = 58, FX_NEAR_MAX = 2040;
template <bool WIDE>
FX_HD double fx_convert(int64_t r, int E) {
  const int64_t g = r >> 63;
  const uint64_t a = (uint64_t)(r ^ g) - (uint64_t)g;   // |r|
  const int e8 = fx_log2_127(a);
  const uint64_t m = a << (189 - e8 < 63 ? 189 - e8 : 63);   // leading bit at 62
  const uint64_t q = (m + 512u) >> 10;
  const int f = e8 == 0 ? 0 : E + e8 - 185;   // exponent field, less the one that q carries
  const bool over = WIDE && f >= 2046;
  const int hi = over ? 0x7ff00000 : (int)(q >> 32) + (int)((unsigned)f << 20);
  return fx_make(hi | ((int)(g >> 32) & (int)0x80000000), over ? 0u : (unsigned)q);
}
FX_HD double fx_near(int64_t r, int E) { return fx_convert<false>(r, E); }
FX_HD double fx_to(int64_t r, int E) { return fx_convert<true>(r, E); }
// r1 2^(E1 - 1080) + r2 2^(E2 - 1080) as r 2^(E - 1080), each rounded to nearest
FX_HD int64_t fx_add(int64_t r1, int E1, int64_t r2, int E2, int &E) {
  E = (E1 > E2 ? E1 : E2) + 1;
  return fx_shift(r1, E - E1) + fx_shift(r2, E - E2);
}

// |r| as an integer; the top 62 bits of values whose largest is top (left shift, if negative right)
FX_HD uint64_t fx_mag(int64_t r) { return (uint64_t)(r < 0 ? -r : r); }
FX_HD int fx_norm_shift(uint64_t top) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)top) - 2;
#else
  return top == 0 ? 62 : __builtin_clzll(top) - 2;
#endif
}
// bits by which |r| < 2^61 may grow as a value of limbs (-1: it has to shrink by one), at most 40
FX_HD int fx_room(int64_t r) {
  const int z = fx_norm_shift(fx_mag(r)) - 2;
  return z < 40 ? z : 40;
}
// r 2^z as a value; its block's exponent falls by z >= -1
FX_HD Fx fx_value_up(int64_t r, int z) { return fx_value(z >= 0 ? r * (1LL << z) : r, z >= 0 ? 0 : 1); }
// the top 64 bits of (a 2^s)^2, a 2^s < 2^62: squares compare to 2^-58 of the largest
FX_HD uint64_t fx_square(uint64_t a, int s) {
  a = s >= 0 ? a << s : a >> (s < -63 ? 63 : -s);
#ifdef __CUDA_ARCH__
  return __umul64hi(a, a);
#else
  return (uint64_t)(((unsigned __int128)a * a) >> 64);
#endif
}

// block fixed point of N values; returns the block's exponent
template <int N>
FX_HD int fx_block(const double x[N], Fx f[N]) {
  int mx = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int j = 0; j < N; ++j) mx = fx_abs_hi(x[j]) > mx ? fx_abs_hi(x[j]) : mx;
  const int E = fx_exp(mx);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int j = 0; j < N; ++j) f[j] = fx_from(x[j], E);
  return E;
}
// x, or NaN (a selection: as the arms of a conditional the compiler would branch around the
// whole conversion)
FX_HD double fx_nan_if(bool bad, double x) { return bad ? NAN : x; }
// fx_to for a block's own exponent, NaN for a block that holds a non-finite value
FX_HD double fx_out(int64_t r, int E) { return fx_nan_if(E >= FX_ENAN, fx_to(r, E)); }

}  // namespace dg
