// dg_stage.cuh -- the per-stage kernels of the SSP-RK3 BP RI-OEDG scheme
// (Ding, Cui & Wu, arXiv 2409.09620, Sec. 4.5).  The work of a tile of cells is
// in dg_stage_fp64.cuh and dg_stage_mixed.cuh.
//
//   k_rk      volume quadrature + edge LF fluxes + mass inverse + RK combine
//             (eqs. DGSystem:Dis, fluxLF, RKTime); publishes the vertex
//             derivatives of u_h and block sums of |K| u_h^(0)
//   k_stats   sup deviations from the domain mean at the volume points
//             (eqs. normOmg, RIOESys:Coef1)
//   k_oe_bp   RIOE damping (eqs. oe:sys, OEScalar:Coef1/Coef2, oe:sysdelta2,
//             RIOESys:CoefM) + BP limiter (Sec. 4.4) + traces, F.n and the
//             maximum wave speed of the limited state at the edge Gauss points
//             (eq. 1250) for the next stage
#pragma once
#include <type_traits>

#include "dg_common.cuh"
#include "dg_fix.cuh"
#include "dg_fix_vertex.cuh"

namespace dg {

// Resident blocks per SM requested from the register allocator.  Higher
// occupancy hides the latency of the neighbour gathers and of the FP64 pipe
// until the spills cost more, which for the fewer modes of P1 happens later.
// 1,036,800 cells, ms per launch:
//   FP64  k_rk     P2 0.911 with 7 blocks, 0.916 with 8, 0.955 with 9; P1 the same from 9 to 12
//         k_stats  P2 0.601 with 8, 0.592 with 10, 0.610 with 12; P1 0.406 with 10, 0.401 with
//                  12, 0.434 with 14
//         k_oe_bp  P2 0.711 with 6, 0.714 with 8, 0.720 with 10; P1 0.465, 0.450 and 0.454
//   mixed k_rk     P2 0.181 with 3 blocks, 0.157 with 4, 0.166 with 5;
//                  P1 0.136 with 4, 0.112 with 6, 0.105 with 7, 0.103 with 8, 0.106 with 9;
//                  259,200 cells 0.0380 with 4, 0.0330 with 6, 0.0337 with 7, 0.0347 with 8
//         k_oe_bp  P2 0.229 with 3 and 4 blocks, 0.265 with 5;
//                  P1 0.149 with 4, 0.136 with 5, 0.135 with 6, 0.141 with 7;
//                  259,200 cells 0.0468 with 4, 0.0453 with 5, 0.0496 with 6
//         k_stats  the same from 5 to 8 (bound by memory)
// A small mesh (FUSED) has at most FUSE_GROUPS * TILE_GROUP blocks, not two per SM: its
// kernels get all the registers they want.  us per step with 2 / 4 / 6 blocks: 1,058 P2
// cells, mixed, 85 / 90 / 100; 20,000 P2 cells, mixed, 104 / 108 / 130; 2,048 P1 cells, FP64,
// 100 / 100 / 102.
// The batch kernels hold both degrees and take the values of P2.
template <int K, typename Real, bool FUSED = false>
struct MinBlocks {
  static constexpr bool F = sizeof(Real) == 4;
  static constexpr int rk = FUSED ? 2 : F ? (K == 1 ? 7 : 4) : (K == 1 ? 10 : 7);
  static constexpr int stats = FUSED ? 2 : F ? 6 : (K == 1 ? 12 : 10);
  static constexpr int oe_bp = FUSED ? 2 : F ? (K == 1 ? 5 : 4) : 8;
};

// A cell's state.  The FP64 form keeps the modes component- and mode-major
// ([4][NB-1][nt]); the mixed form keeps each cell's 4 (NB - 1) FP32 modes
// together (80 bytes for P2, 32 for P1, both multiples of 16), so that a cell
// -- its own or a neighbour's -- comes in (NB - 1) 16-byte loads from one
// address instead of 4 (NB - 1) scattered ones.
template <int NB>
__device__ __forceinline__ void load_state(const StateDev<float> &s, int64_t nt, int64_t K, double avg[4],
                                           float hi[4][NB]) {
  constexpr int NM = 4 * (NB - 1);
#pragma unroll
  for (int c = 0; c < 4; ++c) avg[c] = s.avg[c * nt + K];
  const float4 *p = reinterpret_cast<const float4 *>(s.hi + K * NM);
  float v[NM];
#pragma unroll
  for (int j = 0; j < NM / 4; ++j) {
    const float4 q = p[j];
    v[4 * j] = q.x; v[4 * j + 1] = q.y; v[4 * j + 2] = q.z; v[4 * j + 3] = q.w;
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    hi[c][0] = 0.0f;
#pragma unroll
    for (int l = 1; l < NB; ++l) hi[c][l] = v[c * (NB - 1) + l - 1];
  }
}
// store the modes of cell K in the mixed form's per-cell record
template <int NB>
__device__ __forceinline__ void store_modes_mixed(const StateDev<float> &s, int64_t K, const float hi[4][NB]) {
  constexpr int NM = 4 * (NB - 1);
  float4 *p = reinterpret_cast<float4 *>(s.hi + K * NM);
#pragma unroll
  for (int j = 0; j < NM / 4; ++j) {
    float q[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) q[r] = hi[(4 * j + r) / (NB - 1)][(4 * j + r) % (NB - 1) + 1];
    p[j] = make_float4(q[0], q[1], q[2], q[3]);
  }
}

// value of the cell polynomial at a fixed reference point (compile-time after unrolling)
template <typename Real, int NB, typename A>
__device__ __forceinline__ void eval_fixed(const A avg[4], const Real hi[4][NB], double xi, double eta,
                                           Real out[4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    Real s = Real(avg[c]);
#pragma unroll
    for (int l = 1; l < NB; ++l) s = cfma(psi(l, xi, eta), hi[c][l], s);
    out[c] = s;
  }
}

// exterior vertex data of a boundary edge: value, gradient (x, y) and Hessian (xx, xy, yy)
template <typename Real>
__device__ __forceinline__ void ghost_vertex(int tag, const Real val[4], const Real grd[8], const Real hes[12],
                                             const Real avg[4], Real nx, Real ny, double px, double py, double t,
                                             const Phys &ph, Real ov[4], Real og[8], Real oh[12]) {
  if (tag == 1) {
    // mirror polynomial: q(Rx) for rho, E and R m(Rx) for the momentum, R = I - 2 n n^T
    // with the fused products fixed (left to the compiler, the fusion could
    // differ between the kernels that inline this, and a batch would not
    // reproduce its solves bit for bit)
    const Real R00 = fma(Real(-2) * nx, nx, Real(1)), R01 = Real(-2) * nx * ny, R11 = fma(Real(-2) * ny, ny, Real(1));
    Real RHR[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const Real hxx = hes[3 * c], hxy = hes[3 * c + 1], hyy = hes[3 * c + 2];
      // (R H R)_ab with R symmetric
      const Real a0 = fdot2(R00, hxx, R01, hxy), a1 = fdot2(R00, hxy, R01, hyy);   // row 0 of R H
      const Real b0 = fdot2(R01, hxx, R11, hxy), b1 = fdot2(R01, hxy, R11, hyy);   // row 1 of R H
      RHR[c][0] = fdot2(a0, R00, a1, R01);
      RHR[c][1] = fdot2(a0, R01, a1, R11);
      RHR[c][2] = fdot2(b0, R01, b1, R11);
    }
#pragma unroll
    for (int c = 0; c < 4; c += 3) {
      ov[c] = val[c];
      og[2 * c] = fdot2(R00, grd[2 * c], R01, grd[2 * c + 1]);
      og[2 * c + 1] = fdot2(R01, grd[2 * c], R11, grd[2 * c + 1]);
      oh[3 * c] = RHR[c][0]; oh[3 * c + 1] = RHR[c][1]; oh[3 * c + 2] = RHR[c][2];
    }
    ov[1] = fdot2(R00, val[1], R01, val[2]);
    ov[2] = fdot2(R01, val[1], R11, val[2]);
    // gradient matrix G[a][b] = d m_a / d x_b -> R G R
    const Real G00 = grd[2], G01 = grd[3], G10 = grd[4], G11 = grd[5];
    const Real A00 = fdot2(R00, G00, R01, G10), A01 = fdot2(R00, G01, R01, G11);
    const Real A10 = fdot2(R01, G00, R11, G10), A11 = fdot2(R01, G01, R11, G11);
    og[2] = fdot2(A00, R00, A01, R01); og[3] = fdot2(A00, R01, A01, R11);
    og[4] = fdot2(A10, R00, A11, R01); og[5] = fdot2(A10, R01, A11, R11);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      oh[3 + r] = fdot2(R00, RHR[1][r], R01, RHR[2][r]);
      oh[6 + r] = fdot2(R01, RHR[1][r], R11, RHR[2][r]);
    }
  } else {   // constant exterior states (Dirichlet, moving shock, the transmissive cell average): no derivatives
    Real st[4];
    ghost_state(tag, val, avg, nx, ny, px, py, t, ph, st);
#pragma unroll
    for (int c = 0; c < 4; ++c) ov[c] = st[c];
#pragma unroll
    for (int q = 0; q < 8; ++q) og[q] = Real(0);
#pragma unroll
    for (int q = 0; q < 12; ++q) oh[q] = Real(0);
  }
}

}  // namespace dg

#include "dg_stage_fp64.cuh"
#include "dg_stage_mixed.cuh"

namespace dg {

// ==========================================================================
// The tile functions of both precisions, and the kernels of one solve
// ==========================================================================
// BYTES: the FP64 form's shared memory (dg_stage_fp64.cuh)
template <int K, typename Real, int BYTES = sizeof(RkShared<K>), typename Sc>
__device__ __forceinline__ void rk_tile(const MeshDev &m, const Phys &ph, StateDev<Real> v, StateDev<Real> un,
                                        StateDev<Real> uh, const Real *__restrict__ tr, Real *__restrict__ vdo,
                                        Real *__restrict__ hso, double *part_sum, Sc get, double a,
                                        double b, double c_in, int64_t tile) {
  if constexpr (sizeof(Real) == sizeof(float)) rk_tile_mixed<K>(m, ph, v, un, uh, part_sum, get, a, b, c_in, tile);
  else rk_tile_fp64<K, BYTES>(m, ph, v, un, uh, tr, vdo, hso, part_sum, get, a, b, c_in, tile);
}
template <int K, typename Real, typename Sc>
__device__ __forceinline__ void stats_tile(const MeshDev &m, StateDev<Real> uh, double *part_dev, Sc get,
                                           int64_t tile) {
  if constexpr (sizeof(Real) == sizeof(float)) stats_tile_mixed<K>(m, uh, part_dev, get, tile);
  else stats_tile_fp64<K>(m, uh, part_dev, get, tile);
}
// the mixed form takes its jumps in K3
template <int K, typename Real>
__device__ __forceinline__ void edge_tile(const MeshDev &m, const Phys &ph, const double *__restrict__ avg,
                                          const Real *__restrict__ vdi, const Real *__restrict__ hsi,
                                          Real *__restrict__ ej, const Scalars *sc, double c_out, int64_t tile) {
  if constexpr (sizeof(Real) == sizeof(double)) edge_tile_fp64<K>(m, ph, avg, vdi, hsi, ej, sc, c_out, tile);
}
template <int K, typename Real, int BYTES = sizeof(OeShared<K>), typename Sc>
__device__ __forceinline__ void oe_bp_tile(const MeshDev &m, const Phys &ph, StateDev<Real> uh, StateDev<Real> out,
                                           const Real *__restrict__ ej, Real *__restrict__ tr, double *part_alpha,
                                           long long *part_cnt, Sc get, int do_oe, int do_bp,
                                           double c_out, int end_of_step, int64_t tile) {
  if constexpr (sizeof(Real) == sizeof(float))
    oe_bp_tile_mixed<K>(m, ph, uh, out, part_alpha, part_cnt, get, do_oe, do_bp, c_out, end_of_step, tile);
  else
    oe_bp_tile_fp64<K, BYTES>(m, ph, uh, out, ej, tr, part_alpha, part_cnt, get, do_oe, do_bp, c_out, end_of_step, tile);
}

template <int K, typename Real, bool FUSED>
__global__ void __launch_bounds__(TPB, MinBlocks<K, Real, FUSED>::rk)
    k_rk(MeshDev m, Phys ph, StateDev<Real> v, StateDev<Real> un, StateDev<Real> uh, const Real *__restrict__ tr,
         Real *__restrict__ vdo, Real *__restrict__ hso, double *part_sum, const Scalars *sc, double a, double b,
         double c_in, Fuse f) {
  if constexpr (FUSED) {
    __shared__ Scalars s_sc;
    FuseAlpha g(f, &s_sc);
    if (g.writer()) {
      g.begin();
      g.end();
      return;
    }
    rk_tile<K, Real>(m, ph, v, un, uh, tr, vdo, hso, part_sum, g, a, b, c_in, blockIdx.x);
  } else {
    if (!sc->active) return;
    rk_tile<K, Real>(m, ph, v, un, uh, tr, vdo, hso, part_sum, PlainScalars{sc}, a, b, c_in, blockIdx.x);
  }
}

// OE statistics of the tile's cells and the jump data of the edges it owns
template <int K, typename Real, bool FUSED>
__global__ void __launch_bounds__(TPB, MinBlocks<K, Real, FUSED>::stats)
    k_stats(const __grid_constant__ MeshDev m, const __grid_constant__ Phys ph, StateDev<Real> uh, double *part_dev, const Real *__restrict__ vdi,
            const Real *__restrict__ hsi, Real *__restrict__ ej, const Scalars *sc, double c_out, Fuse f) {
  if constexpr (FUSED) {
    __shared__ Scalars s_sc;
    FuseMeans g(f, &s_sc);
    if (g.writer()) {
      g.begin();
      g.end();
      return;
    }
    stats_tile<K, Real>(m, uh, part_dev, g, blockIdx.x);
    sc = &s_sc;
    if (!sc->active) return;
  } else {
    if (!sc->active) return;
    stats_tile<K, Real>(m, uh, part_dev, PlainScalars{sc}, blockIdx.x);
  }
  edge_tile<K, Real>(m, ph, uh.avg, vdi, hsi, ej, sc, c_out, blockIdx.x);
}

// RIOE damping, BP limiter, traces and wave speeds of the stage result
template <int K, typename Real, bool FUSED>
__global__ void __launch_bounds__(TPB, MinBlocks<K, Real, FUSED>::oe_bp)
    k_oe_bp(MeshDev m, Phys ph, StateDev<Real> uh, StateDev<Real> out, const Real *__restrict__ ej,
            Real *__restrict__ tr, double *part_alpha, long long *part_cnt, const Scalars *sc, int do_oe,
            int do_bp, double c_out, int end_of_step, Fuse f) {
  if constexpr (FUSED) {
    __shared__ Scalars s_sc;
    FuseDeviations g(f, &s_sc, ph.oe == 2);
    if (g.writer()) {
      g.begin();
      g.end();
      return;
    }
    oe_bp_tile<K, Real>(m, ph, uh, out, ej, tr, part_alpha, part_cnt, g, do_oe, do_bp, c_out, end_of_step, blockIdx.x);
  } else {
    if (!sc->active) return;
    oe_bp_tile<K, Real>(m, ph, uh, out, ej, tr, part_alpha, part_cnt, PlainScalars{sc}, do_oe, do_bp, c_out,
                        end_of_step, blockIdx.x);
  }
}

}  // namespace dg

