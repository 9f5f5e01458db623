// dg_stage_fp64.cuh -- stage kernels of the FP64 form (Ding, Cui & Wu, arXiv
// 2409.09620, Sec. 4.5).
//
// What bounds them: GB300's FP64 pipe takes 64 cycles per warp instruction and
// scheduler (76 with an immediate or constant operand), whatever the number
// of active lanes, and a dependent instruction waits as long.  So
//
//   * four lanes share a cell, one per conserved component: a tile of 32 cells
//     is a block of 128 threads.  A quarter of the serial chain per thread,
//     four times the warps of one thread per cell on a small mesh, and few
//     enough registers for several blocks per SM;
//   * sums with compile-time coefficients (values at points, quadrature sums,
//     vertex derivatives) run in block fixed point on the integer units
//     beside the FP64 pipe (dg_fix.cuh);
//   * work that needs all four components (fluxes, wave speeds) is dealt out
//     one (cell, point) per lane through shared memory.  The warp that starts
//     depends on the tile: warp w sits on scheduler w mod 4, and 6 or 9 points
//     are no multiple of 4.
//
// Threads beyond the last cell repeat the last cell and store nothing.
//
// 1,036,800 P2 cells (double Mach reflection), ms per launch, against one thread per cell
// with every sum on the FP64 pipe: k_rk 2.37 -> 0.91, k_stats 0.96 -> 0.59, k_oe_bp 1.39 ->
// 0.71, step 14.2 -> 6.67; 460,800 P1 cells: 0.468 -> 0.200, 0.273 -> 0.200,
// 0.370 -> 0.210.  The errors against 64 bits are those of the FMA chains (vortex 1.54e-15, DMR 3.6e-16, forward facing step 7.6e-16).
#pragma once

namespace dg {

constexpr int FT = TileCells<double>::value;   // cells per tile
static_assert(4 * FT == TPB, "four lanes per cell");

// a cell's four components of one point, in shared memory
struct __align__(16) Vec4d {
  double c[4];
};

// Shared memory of the tile functions.  A kernel that holds several of them (both degrees,
// or both phases, in the batch kernels) gives all the same BYTES and so one buffer, which
// every function leaves free with a barrier.
template <int K>
struct RkShared {
  Vec4d u[Deg<K>::NV][FT], g[Deg<K>::NV][FT];
  int64_t y[3 * Deg<K>::NQ][TPB];
  double cell[4][FT], jac[4][FT], m[TPB];
};
template <int K>
struct OeShared {
  Vec4d u[3 * Deg<K>::NQ + 2][FT], a[FT];
};
constexpr int FP64_TILE_BYTES = sizeof(RkShared<2>);   // the largest of them
static_assert(sizeof(OeShared<2>) <= FP64_TILE_BYTES && sizeof(RkShared<1>) <= FP64_TILE_BYTES, "one buffer");
template <int BYTES>
__device__ __forceinline__ unsigned char *tile_shared() {
  __shared__ __align__(16) unsigned char buf[BYTES];
  return buf;
}

// one component's average and modes
template <int NB>
__device__ __forceinline__ void load_comp(const StateDev<double> &s, int64_t nt, int64_t K, int c, double x[NB]) {
  x[0] = s.avg[c * nt + K];
#pragma unroll
  for (int l = 1; l < NB; ++l) x[l] = s.hi[(c * (NB - 1) + (l - 1)) * nt + K];
}
// value of the component's polynomial at a fixed reference point: sum_l psi_l(x) f_l
template <int NB>
__device__ __forceinline__ int64_t fx_point(const Fx f[NB], double xi, double eta) {
  FxAcc s{0, 0};
#pragma unroll
  for (int l = 0; l < NB; ++l) fx_mac(s, fxc(psi(l, xi, eta)), f[l]);
  return fx_sum(s);
}
// component c of four values held by every lane
__device__ __forceinline__ double pick4(const double v[4], int c) {
  const double a = c & 1 ? v[1] : v[0], b = c & 1 ? v[3] : v[2];
  return c & 2 ? b : a;
}

// ==========================================================================
// K1: u_h = a u_n + b (v + dt L(v))
// ==========================================================================
// one tile; block partial -> part_sum[4 * tile]
template <int K, int BYTES, typename Sc>
__device__ __forceinline__ void rk_tile_fp64(const MeshDev &m, const Phys &ph, StateDev<double> v, StateDev<double> un,
                                             StateDev<double> uh, const double *__restrict__ tr,
                                             double *__restrict__ vdo, double *__restrict__ hso, double *part_sum,
                                             Sc get, double a, double b, double c_in, int64_t tile) {
  constexpr int NB = Deg<K>::NB, NQ = Deg<K>::NQ, NV = Deg<K>::NV;
  RkShared<K> &sh = *reinterpret_cast<RkShared<K> *>(tile_shared<BYTES>());
  auto &s_u = sh.u, &s_g = sh.g;
  auto &s_cell = sh.cell;   // dt / |K|, then alpha l_i
  auto &s_jac = sh.jac;     // |K| times the inverse Jacobian
  const int c = threadIdx.x & 3, lc = threadIdx.x >> 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warp0 = (warp + (int)tile) & 3;
  const int64_t nt = m.nt, K0 = tile * FT;
  const bool live = K0 + lc < nt;
  const int64_t Kc = live ? K0 + lc : nt - 1;
  const double gm1 = phys_gm1<double>(ph);
  get.begin();

  // ---- values at the volume points -----------------------------------------
  {
    double x[NB];
    Fx f[NB];
    load_comp<NB>(v, nt, Kc, c, x);
    const int E = fx_block<NB>(x, f);
#pragma unroll
    for (int mu = 0; mu < NV; ++mu)
      s_u[mu][lc].c[c] = fx_out(fx_point<NB>(f, vol_xi(NV, mu), vol_eta(NV, mu)), E);
  }
  const Scalars *sc = get.end();
  if (Sc::FUSED && !sc->active) return;
  const double dt = sc->dt, alpha = sc->alpha;
  // products that belong to a cell or an edge, once per cell instead of in every lane
  {
    const int64_t Kl = K0 + lane < nt ? K0 + lane : nt - 1;
    s_cell[warp][lane] = mul(warp == 0 ? dt : alpha, warp == 0 ? m.iarea[Kl] : m.len[(warp - 1) * nt + Kl]);
    s_jac[warp][lane] = mul(m.area[Kl], m.jinv[warp * nt + Kl]);
  }
  __syncthreads();
  // ---- volume fluxes, one (cell, point) per lane -----------------------------
  // F . grad Psi = (F . grad xi) dPsi/dxi + (F . grad eta) dPsi/deta; |K| rides on the gradients
  {
    const double jx = s_jac[0][lane], jy = s_jac[1][lane], ex = s_jac[2][lane], ey = s_jac[3][lane];
#pragma unroll 1
    for (int p = warp0; p < NV; p += 4) {
      Vec4d u = s_u[p][lane], g1, g2;
      flux_dir2(u.c, jx, jy, ex, ey, gm1, g1.c, g2.c);
      s_u[p][lane] = g1;
      s_g[p][lane] = g2;
    }
  }
  // ---- edge fluxes of this component -------------------------------------------
  // y = l_i ((F(u-) + F(u+)) . n - alpha (u+ - u-)) in fixed point: the traces of
  // an edge share one block, its fluxes another, and l_i and alpha l_i scaled to
  // the larger of the two products are run-time coefficients.  Beside a
  // conversion per trace value this takes 6 integer multiply-adds per point
  // where the FP64 pipe took 4 operations (64 cycles each).  The two cells of
  // an edge form opposite values to 2^-58 of the larger product.
  // One edge after another in a loop, its values in shared memory: unrolled, the
  // kernel was 67 KB of straight-line code that waited for instructions more than
  // for anything else (28 % of the stalls, P2), and held 9 sums in registers.
  // A loop gave 4 % of k_rk in P2 and 11 % in P1.
  auto &s_y = sh.y;   // this thread's, in its own column
  int ei[3] = {0, 0, 0};
  bool bad = false;
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    const int32_t cn = m.conn[i * nt + Kc];
    const double li = m.len[i * nt + Kc];
    double um[NQ], fm[NQ], up[NQ], fn[NQ];   // fn = - F(u+).n (a negated double would be an FP64 operation)
    int mu = 0, mf = 0;
#pragma unroll
    for (int nu = 0; nu < NQ; ++nu) {
      const double *po = tr + ((Kc * 3 + i) * NQ + nu) * 8;
      um[nu] = po[c];
      fm[nu] = po[4 + c];
      if (cn >= 0) {
        const double *pn = tr + (((int64_t)(cn >> 2) * 3 + (cn & 3)) * NQ + (NQ - 1 - nu)) * 8;
        up[nu] = pn[c];
        fn[nu] = pn[4 + c];   // the neighbour's normal is the negative
      } else {
        const double nx = m.nrm[(2 * i) * nt + Kc], ny = m.nrm[(2 * i + 1) * nt + Kc];
        double px = 0.0, py = 0.0, ow[4], av[4], gh[4], gf[4];
        const double t_in = fma(c_in, sc->dt, sc->t);
        if (cn == -7) {
          const double s = gauss_s(NQ, nu);
          const int ia = i == 2 ? 0 : i + 1, ib = i == 0 ? 2 : i - 1;
          const double xa = m.vxy[(2 * ia) * nt + Kc], ya = m.vxy[(2 * ia + 1) * nt + Kc];
          const double xb = m.vxy[(2 * ib) * nt + Kc], yb = m.vxy[(2 * ib + 1) * nt + Kc];
          px = fma(xb - xa, s, xa);
          py = fma(yb - ya, s, ya);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          ow[q] = po[q];
          av[q] = v.avg[q * nt + Kc];
        }
        ghost_state(-cn, ow, av, nx, ny, px, py, t_in, ph, gh);
        flux_dir(gh, nx, ny, gm1, gf);
        up[nu] = pick4(gh, c);
        fn[nu] = -pick4(gf, c);
      }
      mu = max(mu, max(fx_abs_hi(um[nu]), fx_abs_hi(up[nu])));
      mf = max(mf, max(fx_abs_hi(fm[nu]), fx_abs_hi(fn[nu])));
    }
    const double al = s_cell[1 + i][lc];
    const int Eu = fx_exp(mu), Ef = fx_exp(mf);
    // both coefficients are below 1: x < 2^(exponent field - 1022)
    const int e = max(Ef + (fx_abs_hi(li) >> 20), Eu + (fx_abs_hi(al) >> 20)) - 1022;
#pragma unroll
    for (int j = 0; j < 3; ++j) ei[j] = j == i ? e : ei[j];
    const Fx cf = fx_coef(li, Ef - e), cu = fx_coef(al, Eu - e);
    bad = bad || max(Eu, Ef) >= FX_ENAN || (fx_abs_hi(al) >> 20) >= FX_ENAN;
#pragma unroll
    for (int nu = 0; nu < NQ; ++nu) {
      FxAcc y{0, FX_HALF};
      fx_mac(y, cf, fx_from(fm[nu], Ef) - fx_from(fn[nu], Ef));
      fx_mac(y, cu, fx_from(um[nu], Eu) - fx_from(up[nu], Eu));
      s_y[i * NQ + nu][threadIdx.x] = fx_sum(y);   // below 2^60
    }
  }
  __syncthreads();
  // ---- quadrature sums, mass inverse, SSP-RK combination ---------------------------
  // volume |K| sum_mu w_mu F . grad Psi_l, edges - sum_i l_i sum_nu w_nu Fhat Psi_l, both with
  // the mass inverse (and the 1/2 of the LF flux) on their coefficients.  Every sum and shift to
  // nearest: rounded down, each stage had the same bias of about 2^-56 in every cell, and the
  // error against 64 bits grew (forward facing step, 48 stages: 8.6e-16, now 7.6e-16).
  double h[NB];
  {
    int64_t rv[NB];
    int Ev;
    {
      double g1[NV], g2[NV];
      int mx = 0;
#pragma unroll
      for (int mu = 0; mu < NV; ++mu) {
        g1[mu] = s_u[mu][lc].c[c];
        g2[mu] = s_g[mu][lc].c[c];
        mx = max(mx, max(fx_abs_hi(g1[mu]), fx_abs_hi(g2[mu])));
      }
      Ev = fx_exp(mx);
      FxAcc s[NB];
#pragma unroll
      for (int l = 1; l < NB; ++l) s[l] = FxAcc{0, FX_HALF};
#pragma unroll
      for (int mu = 0; mu < NV; ++mu) {
        const double xi = vol_xi(NV, mu), eta = vol_eta(NV, mu), w = vol_w(NV, mu);
        const Fx f1 = fx_from(g1[mu], Ev), f2 = fx_from(g2[mu], Ev);
#pragma unroll
        for (int l = 1; l < NB; ++l) {
          fx_mac(s[l], fxc(w * psi_x(l, xi, eta), inv_mass_c(l)), f1);
          fx_mac(s[l], fxc(w * psi_y(l, xi, eta), inv_mass_c(l)), f2);
        }
      }
#pragma unroll
      for (int l = 1; l < NB; ++l) rv[l] = fx_sum(s[l]);
    }
    const int Ee = max(max(max(ei[0], ei[1]), ei[2]) + 2, FX_NEAR_MIN);
    FxAcc s[NB];
#pragma unroll
    for (int l = 0; l < NB; ++l) s[l] = FxAcc{0, FX_HALF};
#pragma unroll
    for (int p = 0; p < 3 * NQ; ++p) {
      const double sg = gauss_s(NQ, p % NQ), w = 0.5 * gauss_w(NQ, p % NQ);
      const Fx f = fx_value(fx_shift(s_y[p][threadIdx.x], Ee - ei[p / NQ]), 0);
#pragma unroll
      for (int l = 0; l < NB; ++l)
        fx_mac(s[l], fxc(-psi(l, edge_xi(p / NQ, sg), edge_eta(p / NQ, sg)) * w, inv_mass_c(l)), f);
    }
    const double dta = s_cell[0][lc];
    const bool first = first_stage(a, b);   // the first stage skips the zero term and the load of u_n
    bad = bad || Ev >= FX_ENAN;
    double x[NB], xn[NB];
    load_comp<NB>(v, nt, Kc, c, x);
    if (!first) load_comp<NB>(un, nt, Kc, c, xn);
#pragma unroll
    for (int l = 0; l < NB; ++l) {
      int E = Ee;
      int64_t r = fx_sum(s[l]);
      if (l > 0) r = fx_add(rv[l], Ev, r, Ee, E);
      const double d = fx_nan_if(bad, fx_to(r, E));
      const double L = fma(dta, d, x[l]);
      h[l] = first ? L : fdot2(a, xn[l], b, L);
    }
  }
  if (live) {
    uh.avg[c * nt + Kc] = h[0];
#pragma unroll
    for (int l = 1; l < NB; ++l) uh.hi[(c * (NB - 1) + (l - 1)) * nt + Kc] = h[l];
  }
  auto &s_m = sh.m;
  s_m[threadIdx.x] = live ? mul(m.area[Kc], h[0]) : 0.0;   // summed after the barrier below

  // ---- vertex values and derivatives of u_h for the OE jumps --------------------
  // stored as limb pairs (FP64 would be rounded here and taken apart again in K2)
  {
    double *vo = vdo + Kc * VD_CELL;
    short4 ex = make_short4(0, 0, 0, 0);
    {
      Fx f[NB];
      const int E = fx_block<NB>(h, f);
      bad = bad || E >= FX_ENAN;
      ex.x = (short)(E + 2);
#pragma unroll
      for (int vv = 0; vv < 3; ++vv) {
        const int64_t val = fx_point<NB>(f, vert_xi(vv), vert_eta(vv));   // below 11 * 2^58
        s_u[vv][lc].c[c] = fx_out(val, E);   // this thread's slot; read after the barrier below
        const Fx v2 = fx_value(val, 2);      // below 2^59.5
        if (live) *reinterpret_cast<int2 *>(vo + vv * VD_STRIDE + c) = make_int2(v2.h, v2.l);
      }
    }
    const double jxi[2] = {m.jinv[Kc], m.jinv[nt + Kc]}, jeta[2] = {m.jinv[2 * nt + Kc], m.jinv[3 * nt + Kc]};
    const FxRows J = fx_rows(jxi, jeta);
    auto gradient = [&](int vv, Fx gx, Fx gy) {
      if (live) *reinterpret_cast<int4 *>(vo + vv * VD_STRIDE + 4 + 2 * c) = make_int4(gx.h, gx.l, gy.h, gy.l);
    };
    FxDerivs<NB> d(h, J, gradient);
    ex.y = (short)d.EG[0];
    ex.z = (short)d.EG[1];
    if constexpr (K == 2) {
      ex.w = (short)d.EH;
#pragma unroll
      for (int r = 0; r < 3; ++r)
        if (live) *reinterpret_cast<int2 *>(hso + Kc * 12 + 3 * c + r) = make_int2(d.hess[r].h, d.hess[r].l);
    }
    if (bad) ex = make_short4(FX_ENAN, FX_ENAN, FX_ENAN, FX_ENAN);
    if (live) *reinterpret_cast<short4 *>(vo + VD_EXP + c) = ex;
  }
  __syncthreads();
  // 1/rho and sound speed at the vertices, for the wave speeds beta of the OE (+inf for rho <= 0)
  if (warp0 < 3 && K0 + lane < nt) {
    const double gamma = phys_gamma<double>(ph);
    const Vec4d u = s_u[warp0][lane];
    double ri = 0.0, cs = INFINITY;
    if (gt0(u.c[0])) {
      ri = recip(u.c[0]);
      double p = mul(gm1, fma(half_neg(fdot2(u.c[1], u.c[1], u.c[2], u.c[2])), ri, u.c[3]));
      p = gt0(p) ? p : 0.0;
      cs = root(mul(mul(gamma, p), ri));
    }
    double *rec = vdo + (K0 + lane) * VD_CELL + warp0 * VD_STRIDE;
    *reinterpret_cast<double2 *>(rec + 12) = make_double2(ri, cs);
    *reinterpret_cast<double2 *>(rec + 14) = make_double2(u.c[1], u.c[2]);
  }
  // block sums of |K| u^(0) by one warp: four cells per lane, then the lanes of a component
  if (warp == 0) {
    double t = add(add(s_m[lane], s_m[32 + lane]), add(s_m[64 + lane], s_m[96 + lane]));
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) t = add(t, __shfl_xor_sync(0xffffffffu, t, o));
    if (lane < 4) part_sum[4 * tile + lane] = t;
  }
  __syncthreads();
}

// ==========================================================================
// K2: sup deviations from the domain mean at the volume points
// ==========================================================================
template <int K, typename Sc>
__device__ __forceinline__ void stats_tile_fp64(const MeshDev &m, StateDev<double> uh, double *part_dev, Sc get,
                                                int64_t tile) {
  constexpr int NB = Deg<K>::NB, NV = Deg<K>::NV;
  const int c = threadIdx.x & 3, lc = threadIdx.x >> 2;
  const int64_t nt = m.nt, K0 = tile * FT;
  const int64_t Kc = K0 + lc < nt ? K0 + lc : nt - 1;   // a repeated cell changes no maximum
  double x[NB];
  get.begin();
  load_comp<NB>(uh, nt, Kc, c, x);
  const Scalars *sc = get.end();
  if (Sc::FUSED && !sc->active) return;
  x[0] = sub(x[0], sc->mean[c]);
  int mx = 0;
#pragma unroll
  for (int l = 0; l < NB; ++l) mx = max(mx, fx_abs_hi(x[l]));
  const int E = fx_exp(mx);
  // the squares of the two momentum components compare in the larger of their blocks
  const bool mom = c == 1 || c == 2;
  const int Ep = __shfl_xor_sync(0xffffffffu, E, 3);
  const int down = mom && Ep > E ? min(Ep - E, 63) : 0;
  Fx f[NB];
#pragma unroll
  for (int l = 0; l < NB; ++l) f[l] = fx_from(x[l], E);
  // maxima in fixed point; the point of the largest |m|^2 is found from the top 64 bits
  // of the squares (of the values scaled to 62 bits: to 2^-58 of the largest), its norm
  // taken in FP64
  int64_t r[NV];
  uint64_t top = 0;
#pragma unroll
  for (int mu = 0; mu < NV; ++mu) {
    r[mu] = fx_point<NB>(f, vol_xi(NV, mu), vol_eta(NV, mu));
    top = max(top, fx_mag(r[mu]));
  }
  const uint64_t ta = top >> down, tb = __shfl_xor_sync(0xffffffffu, (unsigned long long)ta, 3);
  const int sh = fx_norm_shift(max(ta, tb)) - down;
  uint64_t best = 0;
  int64_t b1 = 0;
#pragma unroll
  for (int mu = 0; mu < NV; ++mu) {
    const uint64_t sq = fx_square(fx_mag(r[mu]), sh);
    const uint64_t s = sq + (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)sq, 3);
    if (mu == 0 || s > best) { best = s; b1 = r[mu]; }
  }
  const double d = fx_out((int64_t)top, E), m1 = fx_out(b1, E), m2 = __shfl_xor_sync(0xffffffffu, m1, 3);
  // rho, |m|, E, |m1|, |m2|; the lanes of the other components hold 0
  double dr[5] = {c == 0 ? d : 0.0, c == 1 ? root(fdot2(m1, m1, m2, m2)) : 0.0, c == 3 ? d : 0.0, c == 1 ? d : 0.0,
                  c == 2 ? d : 0.0};
  block_reduce<5>(dr, part_dev + 5 * tile, OpMaxNN());
}

// --------------------------------------------------------------------------
// OE jump data of one edge, computed once for both cells that share it: per
// component and derivative order j, A^{k,j} beta sqrt(J) of the trapezoidal
// sums J = 1/2 sum_{|alpha| = j} C_j^alpha1 [d^alpha q]^2 over the two
// endpoints (eqs. OEScalar:Coef2 with the trapezoidal rule, RIOESys:Coef1/
// Coef2), seen from the owning cell; beta is the largest spectral radius of
// both sides at both endpoints.  Jump sums are even in the sign of the jump
// and of the normal, so both cells share them.  With RIOE both momentum rows
// hold the larger of the normal and tangential sums.
// Edges [etile[tile], etile[tile + 1]), four lanes per edge, one per component;
// for beta the lanes take the four (endpoint, side) pairs.  The jumps and their
// rotation are taken in fixed point from K1's records (27 FP64 operations per
// lane otherwise), the squares and square roots in FP64.
// --------------------------------------------------------------------------
__device__ __forceinline__ Fx ld_fx(const double *p) {
  const int2 v = *reinterpret_cast<const int2 *>(p);
  return Fx{v.x, v.y};
}
// beta and 2 J of component c at a boundary edge, from the exterior polynomial
// of all components of this side
template <int K>
__device__ __noinline__ void boundary_jumps(const MeshDev &m, const Phys &ph, const double *__restrict__ avg,
                                            const double *__restrict__ vme, const double *__restrict__ hsi,
                                            int64_t Kc, int i, int32_t cn, double nx, double ny, double t_out,
                                            int c, int cw, double gamma, double &beta, double *J) {
  const int64_t nt = m.nt;
  double ab[4], hme[12];
  short4 xo[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    ab[q] = avg[q * nt + Kc];   // the exterior state of a transmissive edge
    xo[q] = *reinterpret_cast<const short4 *>(vme + VD_EXP + q);
  }
  // only squared jumps are taken of these: beyond 2^+-900 infinite or zero either way
  auto get = [&](const double *p, int q, int E) {
    return fx_nan_if(xo[q].x >= FX_ENAN, fx_near(fx_join(ld_fx(p)), min(max(E, FX_NEAR_MIN), FX_NEAR_MAX)));
  };
#pragma unroll
  for (int q = 0; q < 12; ++q)   // xx, xy, yy: the exponents step as those of the gradient's x and y
    hme[q] = K == 2 ? get(hsi + Kc * 12 + q, q / 3, xo[q / 3].w + q % 3 * (xo[q / 3].z - xo[q / 3].y)) : 0.0;
  beta = 0.0;
  // row c of a jump per component, the momentum in (m_n, m_t) for RIOE
  auto row = [&](const double d[4]) {
    const double n = fdot2(d[1], nx, d[2], ny), t = fdot2(d[2], nx, -d[1], ny);
    const double e[4] = {d[0], cw ? d[1] : n, cw ? d[2] : t, d[3]};
    return pick4(e, c);
  };
#pragma unroll 1
  for (int ev = 0; ev < 2; ++ev) {
    int ov = i + 1 + ev;
    ov = ov >= 3 ? ov - 3 : ov;
    const double *ro = vme + ov * VD_STRIDE;
    double val[4], grd[8], xv[4], xg[8], xh[12];
#pragma unroll
    for (int q = 0; q < 4; ++q) val[q] = get(ro + q, q, xo[q].x);
#pragma unroll
    for (int q = 0; q < 8; ++q) grd[q] = get(ro + 4 + q, q / 2, q & 1 ? xo[q / 2].z : xo[q / 2].y);
    double px = 0.0, py = 0.0;
    if (cn == -7) { px = m.vxy[(2 * ov) * nt + Kc]; py = m.vxy[(2 * ov + 1) * nt + Kc]; }
    ghost_vertex(-cn, val, grd, hme, ab, nx, ny, px, py, t_out, ph, xv, xg, xh);
    const double r_own = fma(fabs(fdot2(ro[14], nx, ro[15], ny)), ro[12], ro[13]);
    // a mirror state has the same spectral radius
    beta = max_nn(beta, max_nn(r_own, cn == -1 ? r_own : wave_speed(xv, nx, ny, gamma)));
    double dv[4], d0[4], d1[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      dv[q] = val[q] - xv[q];
      d0[q] = grd[2 * q] - xg[2 * q];
      d1[q] = grd[2 * q + 1] - xg[2 * q + 1];
    }
    const double q = row(dv), g0 = row(d0), g1 = row(d1);
    J[0] = ev == 0 ? q * q : fma(q, q, J[0]);
    J[1] = ev == 0 ? fdot2(g0, g0, g1, g1) : fma(g0, g0, fma(g1, g1, J[1]));
    if (K == 2 && ev == 0) {   // the exterior Hessian is constant: taken at v_c, for both endpoints
      double h[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const double dh[4] = {hme[r] - xh[r], hme[3 + r] - xh[3 + r], hme[6 + r] - xh[6 + r], hme[9 + r] - xh[9 + r]};
        h[r] = row(dh);
      }
      const double f = fma(h[0], h[0], fma(h[1] + h[1], h[1], h[2] * h[2]));
      J[K] = f + f;
    }
  }
}

template <int K>
__device__ __forceinline__ void edge_tile_fp64(const MeshDev &m, const Phys &ph, const double *__restrict__ avg,
                                               const double *__restrict__ vdi, const double *__restrict__ hsi,
                                               double *__restrict__ ej, const Scalars *sc, double c_out,
                                               int64_t tile) {
  const int64_t nt = m.nt;
  const int64_t e0 = m.etile[tile], e1 = m.etile[tile + 1];
  const double gamma = phys_gamma<double>(ph);
  const int cw = ph.oe == 2;
  const int c = threadIdx.x & 3;
  const int slot = ((threadIdx.x >> 2) + 8 * (int)(tile & 3)) & 31;   // an uneven last round moves over the schedulers
  const bool mom = !cw && (c == 1 || c == 2);
  for (int64_t eb = e0; eb < e1; eb += FT) {
    if (eb + (slot & ~7) >= e1) continue;   // no edge left for this warp
    const bool live = eb + slot < e1;
    const int64_t e = live ? eb + slot : e1 - 1;
    const int64_t Kc = m.e_cell[e];
    const int i = m.e_loc[e];
    const int32_t cn = m.conn[i * nt + Kc];
    const double nx = m.nrm[(2 * i) * nt + Kc], ny = m.nrm[(2 * i + 1) * nt + Kc];
    const double *vme = vdi + Kc * VD_CELL;
    const short4 xo = *reinterpret_cast<const short4 *>(vme + VD_EXP + c);
    // jumps of this component: values and gradients at v_c then v_d, the Hessian once; with
    // the exponent of each kind (the momentum components share it, for their rotation)
    Fx jv[2], jg[2][2], jh[3];
    int E0, Ev[2], E1[2], E2[3] = {0, 0, 0};
    // the larger exponents of two components, two kinds at a time
    auto shared_exp = [&](int Ea, int Eb, int &a, int &b) {
      const int p = __shfl_xor_sync(0xffffffffu, (Ea << 16) | (Eb & 0xffff), 3);
      a = mom ? max(Ea, p >> 16) : Ea;
      b = mom ? max(Eb, (int)(short)p) : Eb;
    };
    double r;
    bool bad = xo.x >= FX_ENAN;
    const int64_t nb = cn >= 0 ? cn >> 2 : Kc;
    const int jn = cn >= 0 ? cn & 3 : i;
    const double *vnb = vdi + nb * VD_CELL;
    const short4 xx = *reinterpret_cast<const short4 *>(vnb + VD_EXP + c);
    bad = bad || xx.x >= FX_ENAN;
    int ho[3] = {xo.w, xo.w + xo.z - xo.y, xo.w + 2 * (xo.z - xo.y)};   // Hessian: xx, xy, yy
    int hx[3] = {xx.w, xx.w + xx.z - xx.y, xx.w + 2 * (xx.z - xx.y)};
    shared_exp(max(xo.x, xx.x), max(xo.y, xx.y), E0, E1[0]);
    shared_exp(max(xo.z, xx.z), max(ho[0], hx[0]), E1[1], E2[0]);
    if (K == 2) shared_exp(max(ho[1], hx[1]), max(ho[2], hx[2]), E2[1], E2[2]);
#pragma unroll
    for (int ev = 0; ev < 2; ++ev) {   // v_c then v_d, and the neighbour's copy of it
      int ov = i + 1 + ev, xv = jn + 2 - ev;
      ov = ov >= 3 ? ov - 3 : ov;
      xv = xv >= 3 ? xv - 3 : xv;
      const double *ro = vme + ov * VD_STRIDE, *rx = vnb + xv * VD_STRIDE;
      const int4 go = *reinterpret_cast<const int4 *>(ro + 4 + 2 * c),
                 gx = *reinterpret_cast<const int4 *>(rx + 4 + 2 * c);
      // the values' difference is far below their block: scaled up, so that it keeps its
      // bits in the rotation (gradients and Hessians contain no average)
      const int64_t d = fx_diff(ld_fx(ro + c), xo.x, ld_fx(rx + c), xx.x, E0);
      int z = fx_room(d);
      const int zp = __shfl_xor_sync(0xffffffffu, z, 3);
      z = mom ? min(z, zp) : z;
      jv[ev] = fx_value_up(d, z);
      Ev[ev] = E0 - z;
      jg[ev][0] = fx_jump<0>(Fx{go.x, go.y}, xo.y, Fx{gx.x, gx.y}, xx.y, E1[0]);
      jg[ev][1] = fx_jump<0>(Fx{go.z, go.w}, xo.z, Fx{gx.z, gx.w}, xx.z, E1[1]);
    }
    if (K == 2) {
#pragma unroll
      for (int q = 0; q < 3; ++q)
        jh[q] = fx_jump<1>(ld_fx(hsi + Kc * 12 + 3 * c + q), ho[q], ld_fx(hsi + nb * 12 + 3 * c + q), hx[q], E2[q]);
    }
    {
      int vv = c & 1 ? (c & 2 ? jn + 1 : i + 2) : (c & 2 ? jn + 2 : i + 1);
      vv = vv >= 3 ? vv - 3 : vv;
      const double *rr = (c & 2 ? vnb : vme) + vv * VD_STRIDE;
      r = fma(fabs(fdot2(rr[14], nx, rr[15], ny)), rr[12], rr[13]);
    }
    r = max_nn(r, __shfl_xor_sync(0xffffffffu, r, 1));
    double beta = max_nn(r, __shfl_xor_sync(0xffffffffu, r, 2));
    // RIOE: rotate the momentum jumps to (m_n, m_t) with the owner's normal
    const Fx rs = fx_coef(mom ? nx : 1.0, 0), ry = fx_coef(mom ? ny : 0.0, 0);
    const Fx rp = c == 2 ? Fx{-ry.h, -ry.l} : ry;
    auto rot = [&](Fx q, int E) {
      const Fx p{__shfl_xor_sync(0xffffffffu, q.h, 3), __shfl_xor_sync(0xffffffffu, q.l, 3)};
      FxAcc t{0, 0};
      fx_mac(t, rs, q);
      fx_mac(t, rp, p);
      // only squared, beyond 2^+-900 to an infinity or zero either way
      return fx_nan_if(bad, fx_near(fx_sum(t), min(max(E, FX_NEAR_MIN), FX_NEAR_MAX)));
    };
    double J[K + 1];
#pragma unroll
    for (int ev = 0; ev < 2; ++ev) {
      const double q = rot(jv[ev], Ev[ev]), g0 = rot(jg[ev][0], E1[0]), g1 = rot(jg[ev][1], E1[1]);
      // 2 J: the 1/2 of the trapezoidal rule moves into A (sqrt(1/2))
      J[0] = ev == 0 ? mul(q, q) : fma(q, q, J[0]);
      J[1] = ev == 0 ? fdot2(g0, g0, g1, g1) : fma(g0, g0, fma(g1, g1, J[1]));
    }
    if (K == 2) {   // the Hessian jump counts at both endpoints
      const double h0 = rot(jh[0], E2[0] + 1), h1 = rot(jh[1], E2[1] + 1), h2 = rot(jh[2], E2[2] + 1);
      const double f = fma(h0, h0, fma(add(h1, h1), h1, mul(h2, h2)));
      J[K] = add(f, f);
    }
    if (cn < 0) boundary_jumps<K>(m, ph, avg, vme, hsi, Kc, i, cn, nx, ny, fma(c_out, sc->dt, sc->t), c, cw, gamma, beta, J);
    const bool finite = is_finite_bits(beta);
    double er[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j <= K; ++j) {
      const double Jp = __shfl_xor_sync(0xffffffffu, J[j], 3);
      if (mom) J[j] = max_nn(J[j], Jp);   // delta_m = max(delta_mn, delta_mt)
      const double s = root(J[j]);
      // A^{k,j} = (2j + 1) / ((2k - 1) j!); a zero jump adds nothing, also where beta is
      // +inf (a vertex with rho <= 0) and 0 * inf would be NaN
      constexpr double r2 = 0.70710678118654752440;
      const double A = (2.0 * j + 1.0) / ((2.0 * K - 1.0) * (j == 2 ? 2.0 : 1.0)) * r2;
      er[j] = finite || nonzero_bits(s) ? mul(A * beta, s) : 0.0;
    }
    if (live) vstore<4>(ej + e * EJ_STRIDE + 4 * c, er);
  }
}

// ==========================================================================
// K3: RIOE + BP limiter + traces / alpha of the limited state
// ==========================================================================
// |x| truncated to FP32 from its high word: in [t, t (1 + 2^-20)] up to
// 2^-126; +inf above the FP32 range or if not finite
__device__ __forceinline__ float abs_f32_down(double x) {
  const int t = (fx_hiword(x) & 0x7fffffff) - 0x38000000;
  return __int_as_float(min(max(t, 0), 0x0ff00000) << 3);
}

template <int K, int BYTES, typename Sc>
__device__ __forceinline__ void oe_bp_tile_fp64(const MeshDev &m, const Phys &ph, StateDev<double> uh,
                                                StateDev<double> out, const double *__restrict__ ej,
                                                double *__restrict__ tr, double *part_alpha, long long *part_cnt,
                                                Sc get, int do_oe, int do_bp, double c_out, int end_of_step,
                                                int64_t tile) {
  constexpr int NB = Deg<K>::NB, NQ = Deg<K>::NQ;
  constexpr int NE = 3 * NQ;          // edge Gauss points
  OeShared<K> &sh = *reinterpret_cast<OeShared<K> *>(tile_shared<BYTES>());
  auto &s_u = sh.u;
  auto &s_a = sh.a;
  const unsigned FULL = 0xffffffffu;
  const int c = threadIdx.x & 3, lc = threadIdx.x >> 2;
  const int lane = threadIdx.x & 31, warp0 = ((threadIdx.x >> 5) + (int)tile) & 3, q0 = lane & ~3;
  const int64_t nt = m.nt, K0 = tile * FT;
  const bool live = K0 + lc < nt;
  const int64_t Kc = live ? K0 + lc : nt - 1;
  long long cnt[2] = {0, 0};
  double x[NB];
  get.begin();
  load_comp<NB>(uh, nt, Kc, c, x);
  s_a[lc].c[c] = x[0];

  // ---------------------------- RIOE ---------------------------------------
  double sig[K + 1];
  if (do_oe) {
    // sigma^j = sum_i (beta_i / h_i) delta_i^j with delta = A^{k,j} h^j sqrt(J) / D: the
    // edge records hold A beta sqrt(J), the edge sum is scaled by 1 / D once (a constant
    // component, 1 / D = 0, gets sigma = 0)
#pragma unroll
    for (int j = 0; j <= K; ++j) sig[j] = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double *er = ej + (int64_t)m.cedge[i * nt + Kc] * EJ_STRIDE + 4 * c;
      const double2 e01 = *reinterpret_cast<const double2 *>(er);
      sig[0] = fma(m.hgeo[(3 + i) * nt + Kc], e01.x, sig[0]);
      sig[1] = add(sig[1], e01.y);
      if (K == 2) sig[K] = fma(m.hgeo[i * nt + Kc], er[2], sig[K]);
    }
  }
  const Scalars *sc = get.end();
  if (Sc::FUSED && !sc->active) return;
  const double dt = sc->dt;
  if (do_oe) {
    const double iD = sc->invD[c];
    // exact solution of the damping ODE: mode of degree d times exp(-dt sum_{j<=d} sigma^j)
    const double s = nonzero_bits(iD) ? mul(iD, dt) : 0.0;
    double sacc = sig[0];
#pragma unroll
    for (int d = 1; d <= K; ++d) {
      sacc = add(sacc, sig[d]);
      const double fac = exp_neg(nonzero_bits(iD) ? mul(s, sacc) : 0.0);
#pragma unroll
      for (int l = 1; l < NB; ++l)
        if (degree_of(l) == d) x[l] = mul(x[l], fac);
    }
  }

  // ---------------------------- BP limiter ----------------------------------
  // A bound over the whole cell settles the usual (smooth) cell without its
  // limiter points: with |Psi_l| <= 4 on K, every point's density is at least
  // rho_bar - 4 sum |rho_l|, its energy at least E_bar - 4 sum |E_l| and the L1
  // norm of its momentum at most |m1_bar| + |m2_bar| + 4 sum (|m1_l| + |m2_l|).
  // If these keep rho and the internal energy above the thresholds with a
  // margin (1e-5 relative) far above the rounding of this FP32 bound and of
  // the point evaluations, every point passes the paper's tests and theta = 1,
  // as the points themselves would give.
  bool todo = false;
  if (do_bp) {
    float S = 0.0f;
#pragma unroll
    for (int l = 1; l < NB; ++l) S += abs_f32_down(x[l]);
    const float D = fmaf(4.00002f, S, 1e-37f), A = abs_f32_down(x[0]);
    const float B = fmaf(1.000002f, A, D);              // upper bound of |component|
    const float lo = gt0(x[0]) ? A - D : -1.0f;         // lower bound of rho, E
    const float r_lo = __shfl_sync(FULL, lo, q0), r_hi = __shfl_sync(FULL, B, q0);
    const float M_hi = __shfl_sync(FULL, B, q0 + 1) + __shfl_sync(FULL, B, q0 + 2);
    const float E_lo = __shfl_sync(FULL, lo, q0 + 3), E_hi = __shfl_sync(FULL, B, q0 + 3);
    const float M2 = M_hi * M_hi, S2 = fmaf(E_hi, r_lo, M2);
    // a NaN or an infinity (also above the FP32 range) leaves S2 infinite or NaN: such a cell
    // is looked at point by point, and its average counted if it is not in G
    const bool settled = r_lo >= fmaf(1e-5f, r_hi, 2e-13f) && S2 < INFINITY &&
                         r_lo * E_lo - 0.5f * M2 >= fmaf(1e-5f, S2, 2e-13f * r_lo);
    todo = !settled;
  }

  // values at the edge Gauss points (the traces, if the cell is not limited)
  auto traces = [&]() {
    Fx f[NB];
    const int E = fx_block<NB>(x, f);
#pragma unroll
    for (int p = 0; p < NE; ++p) {
      const double sg = gauss_s(NQ, p % NQ);
      s_u[p][lc].c[c] = fx_out(fx_point<NB>(f, edge_xi(p / NQ, sg), edge_eta(p / NQ, sg)), E);
    }
  };
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    traces();
    if (pass == 1 || !__any_sync(FULL, todo)) break;
    // the limiter's points: the edge Gauss points and two extra points
    double ext[2];
    if (ph.decomp) {
      // classical decomposition: P1 repeats edge point 0 (its edge weights sum to one), P2 takes
      // the weighted internal state of Sec. 4.1: u_* - ubar = -1/6 sum w_nu dev
      double acc = 0.0;
#pragma unroll
      for (int p = 0; p < NE; ++p) acc = fma(gauss_w(NQ, p % NQ), s_u[p][lc].c[c] - x[0], acc);
      ext[0] = ext[1] = K == 1 ? s_u[0][lc].c[c] : fma(-1.0 / 6.0, acc, x[0]);
    } else {
      // P1: the vertices v1, v2; P2: the internal nodes, whose basis values the mesh holds
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        double s = 0.0;
        if (K == 1) {
          const int vp = m.limv[p * nt + Kc];
#pragma unroll
          for (int l = 1; l < NB; ++l) s = fma(psi(l, vert_xi(vp), vert_eta(vp)), x[l], s);
        } else {
#pragma unroll
          for (int l = 1; l < NB; ++l) s = fma(m.psi_node[(5 * p + l - 1) * nt + Kc], x[l], s);
        }
        ext[p] = x[0] + s;
      }
    }
    s_u[NE][lc].c[c] = ext[0];
    s_u[NE + 1][lc].c[c] = ext[1];
    __syncwarp();
    const Vec4d av = s_a[lc];
    const double Ebar = int_energy(av.c);
    const bool adm = av.c[0] > 0.0 && Ebar > 0.0;
    // Step 1: density.  Minimum on the integer units through order-preserving keys
    long long kmin = ord_key(INFINITY);
#pragma unroll
    for (int p = c; p < NE + 2; p += 4) kmin = min(kmin, ord_key(s_u[p][lc].c[0]));
    kmin = min(kmin, __shfl_xor_sync(FULL, kmin, 1));
    kmin = min(kmin, __shfl_xor_sync(FULL, kmin, 2));
    const double rmin = ord_val(kmin);
    const double eps1 = fmin(av.c[0], 1e-13);
    const double th1 = rmin < eps1 ? (av.c[0] - eps1) / (av.c[0] - rmin) : 1.0;
    // Step 2: internal energy of the density-limited polynomial
    // E - |m|^2 / (2 rho) < eps2 is tested as rho E - |m|^2 / 2 < eps2 rho (rho > 0):
    // the division is only needed at points that violate the bound
    const double eps2 = fmin(Ebar, 1e-13);
    long long kem = ord_key(INFINITY);
#pragma unroll 1
    for (int p = c; p < NE + 2; p += 4) {
      const Vec4d u = s_u[p][lc];
      const double w0 = th1 < 1.0 ? fma(th1, u.c[0] - av.c[0], av.c[0]) : u.c[0];
      const double q = 0.5 * fdot2(u.c[1], u.c[1], u.c[2], u.c[2]);
      if (!(w0 > 0.0) || fma(u.c[3], w0, -q) < eps2 * w0) kem = min(kem, ord_key(u.c[3] - q / w0));
    }
    kem = min(kem, __shfl_xor_sync(FULL, kem, 1));
    kem = min(kem, __shfl_xor_sync(FULL, kem, 2));
    const double emin = ord_val(kem);
    const double th2 = emin < eps2 ? (Ebar - eps2) / (Ebar - emin) : 1.0;
    const bool lim = todo && adm && (th1 < 1.0 || th2 < 1.0);
    if (todo && live && c == 0) {
      if (!adm) cnt[1] = 1;
      if (lim) cnt[0] = 1;
    }
    if (!__any_sync(FULL, lim)) break;
    // scale the modes; the traces are taken again from the scaled (stored)
    // modes, so that a run resumed from the stored state sees the same traces
    // bit for bit
    const double th = c == 0 ? th1 * th2 : th2;
#pragma unroll
    for (int l = 1; l < NB; ++l) x[l] = lim && th < 1.0 ? th * x[l] : x[l];
    __syncwarp();   // every lane has read the points
  }
  if (live) {
    out.avg[c * nt + Kc] = x[0];
#pragma unroll
    for (int l = 1; l < NB; ++l) out.hi[(c * (NB - 1) + (l - 1)) * nt + Kc] = x[l];
  }
  __syncthreads();

  // ---------------------------- output ----------------------------------------
  // traces, F.n and wave speed of the limited state, one (cell, edge point) per lane
  double amax = 0.0;
  if (K0 + lane < nt) {
    const int64_t Kl = K0 + lane;
    const double gamma = phys_gamma<double>(ph), gm1 = phys_gm1<double>(ph);
#pragma unroll 1
    for (int p = warp0; p < NE; p += 4) {
      const int i = p / NQ;
      const int32_t cn = m.conn[i * nt + Kl];
      const double nx = m.nrm[(2 * i) * nt + Kl], ny = m.nrm[(2 * i + 1) * nt + Kl];
      const Vec4d u = s_u[p][lane];
      double o8[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) o8[q] = u.c[q];
      amax = max_nn(amax, flux_speed(u.c, nx, ny, gm1, gamma, o8 + 4));
      vstore<8>(tr + (Kl * NE + p) * 8, o8);
      if (cn <= -2) {   // constant exterior states (walls mirror the trace: same speed)
        // exterior states for the next stage's alpha at the time of the stage
        // result: t + c_out dt, and after the last stage of a step clamped to
        // the end time, the end time itself (the next step starts there)
        const double t_out = end_of_step && sc->pad ? sc->t_end : fma(c_out, sc->dt, sc->t);
        double px = 0.0, py = 0.0;
        if (cn == -7) {
          const int ia = i == 2 ? 0 : i + 1, ib = i == 0 ? 2 : i - 1, nu = p - i * NQ;
          const double s = nu == 0 ? gauss_s(NQ, 0) : nu == 1 ? gauss_s(NQ, 1) : gauss_s(NQ, NQ - 1);
          const double xa = m.vxy[(2 * ia) * nt + Kl], ya = m.vxy[(2 * ia + 1) * nt + Kl];
          const double xb = m.vxy[(2 * ib) * nt + Kl], yb = m.vxy[(2 * ib + 1) * nt + Kl];
          px = fma(xb - xa, s, xa);
          py = fma(yb - ya, s, ya);
        }
        double up[4];
        ghost_state(-cn, u.c, s_a[lane].c, nx, ny, px, py, t_out, ph, up);
        amax = max_nn(amax, wave_speed(up, nx, ny, gamma));
      }
    }
  }
  double am[1] = {amax};
  block_reduce<1>(am, part_alpha + tile, OpMaxNN());
  block_reduce<2>(cnt, part_cnt + 2 * tile, OpSum());
}

}  // namespace dg
