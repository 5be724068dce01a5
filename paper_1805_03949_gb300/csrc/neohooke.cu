// neohooke.cu -- Jacobian and internal force of the finite-strain solid
// (total Lagrangian, first Piola-Kirchhoff stress): the Newton step of the
// paper's structure solver, Sec. 2.2, whose costly part is the constitutive
// evaluation at every Gauss point (Sec. 5.2).
//
// The paper names no material; the engine reads it as the compressible
// neo-Hookean solid (Bonet and Wood 2008, Sec. 6.4.3):
//   Psi = mu/2 (F:F - 3) - mu ln J + lam/2 (ln J)^2,
//   P   = mu (F - F^-T) + lam ln J F^-T,
//   dP_iJ/dF_kL = mu d_ik d_JL + lam F^-1_Ji F^-1_Lk + (mu - lam ln J) F^-1_Jk F^-1_Li.
// Contracted with the reference gradients g_a = grad0 N_a, and with
// h_a = F^-T g_a (the spatial gradients), the element blocks are
//   A^e_ab = sum_q W_q [mu (g_a . g_b) I + lam h_a h_b^T + (mu - lam ln J) h_b h_a^T + m N_a N_b I],
//   f^e_a  = sum_q W_q P g_a,         W_q = w_q det J0_q,
// m N_a N_b I being the inertia term of the Newmark Jacobian.  Per Gauss
// point, FP64: the reference geometry, F = I + sum_a u_a (x) g_a, det F,
// F^-T, ln J and P.  The gradient products (h_a and the blocks) run in the
// tile precision (FP32 for FEA_FP32_INTEGRATE) and are added into A and b in
// FP64, by atomics (ATOMIC) or plain read-modify-writes (COLOR).
//
// Both precisions are bound by the number of FP64 instructions (pairs.cuh).
// F - I = Ju C^T / det of every type from the displacement field's reference
// Jacobian Ju (RefMap, or the modal transform), reciprocals by rcp64, and FP64
// tiles form the node pairs of the symmetric element matrix: with
// g^_a = sqrt(W) g_a and h^_a = sqrt(W) h_a,
//   A^e_ab = lam M + N^T + (mu D + m sum_q W N_a N_b) I,
//   M = sum_q h^_a (x) h^_b,  N = sum_q (mu - lam ln J) h^_a (x) h^_b,
//   D = sum_q g^_a . g^_b,
// 24 products per pair and point where a row block took 28 per ordered pair.
// 65,559 hex8, FP64, one GB300: 2.81 -> 1.29 ms.
#include <cmath>
#include <cstddef>
#include <cstring>
#include <type_traits>

#include "coop_scatter.cuh"
#include "element.cuh"
#include "fea_internal.cuh"
#include "pairs.cuh"

namespace fea {

struct NHParams : ElemParams {
  const double* u;
  double lam, mu, mass;
};

// FP32 tiles: lane a of an element's NN lanes holds its row block.
template <int TYPE, int SLOT>
struct NHCfg {
  static constexpr int NN = nodes_of(TYPE);
  static constexpr int NQ = rule_nq(SLOT);
  static constexpr int LPE = NN;
  static constexpr int EPW = 32 / LPE;
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int EPC = EPW * WARPS;
  static constexpr bool kHex = TYPE == FEA_HEX8;
  static_assert(!kHex || (EPC * 8 % 32 == 0 && EPC * 8 <= THREADS), "modal hex geometry needs whole warps");
  struct Smem {
    double X[EPC][NN][3];
    double U[EPC][NN][3];
    float G[EPC][NQ][grad_stride(NN)];  // g_a = grad0 N_a [point][node][component]
    float H[EPC][NQ][grad_stride(NN)];  // h_a = F^-T g_a
    float C[EPC][NQ][4];      // W mu, W lam, W (mu - lam ln J), W m
    float S[EPC][NQ][9];      // W P, row-major
  };
  // with the cooperative scatter's rows, where its staging fits the place of the
  // coordinates and displacements (every type but pyramids; a plain
  // read-modify-write scatter has the L1 cache that they would take)
  using CS = CoopScatter<NN, FEA_SCATTER_ATOMIC>;
  static constexpr bool kCoop = WARPS * CS::kVals * sizeof(float) <= 2 * sizeof(double[EPC][NN][3]);
  struct CoopSmem : Smem {
    typename CS::Rows rows[WARPS];
  };
};

// The kinematics of one point (FP64), from the Jacobian J' = s J0 (s a power
// of two) and Ju' = s Ju of the displacement field: C' and det' of J', F^-T,
// ln J and W P.  False (and latched) if the element is inverted in the
// reference configuration or by the deformation.
struct NHPoint {
  double C[3][3], Fit[3][3], WP[3][3];
  double rdet, W, lnJ;
};

__device__ __forceinline__ bool nh_kinematics(const NHParams& P, int64_t id, double w, const double (&J)[3][3],
                                              const double (&Ju)[3][3], double s, NHPoint& r) {
  cofactors(J, r.C);
  const double det = J[0][0] * r.C[0][0] + J[0][1] * r.C[0][1] + J[0][2] * r.C[0][2];
  double F[3][3], Fc[3][3], detF = 0.0;
  if (det > 0.0) {
    r.rdet = rcp64(det);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double h = fma(Ju[i][2], r.C[j][2], fma(Ju[i][1], r.C[j][1], Ju[i][0] * r.C[j][0]));
        F[i][j] = i == j ? fma(h, r.rdet, 1.0) : h * r.rdet;
      }
    cofactors(F, Fc);  // cof F = det F * F^-T
    detF = F[0][0] * Fc[0][0] + F[0][1] * Fc[0][1] + F[0][2] * Fc[0][2];
  }
  if (!(det > 0.0) || !(detF > 0.0)) {
    latch_error(P.st, FEA_ERR_INVERTED_ELEMENT, (unsigned long long)id);
    return false;
  }
  const double rJ = rcp64(detF);
  r.lnJ = log(detF);
  r.W = w * det * (1.0 / (s * s * s));
  // P = mu (F - F^-T) + lam ln J F^-T
  const double a = r.W * P.mu, b = fma(r.W * P.lam, r.lnJ, -a);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      r.Fit[i][j] = Fc[i][j] * rJ;
      r.WP[i][j] = fma(b, r.Fit[i][j], a * F[i][j]);
    }
  return true;
}

// Phase 1 of point q of element le of an FP32 tile.  Hex gradients are formed
// in FP32 from C' and det' rounded once, the other types' in FP64 and rounded.
template <class Cfg>
__device__ __forceinline__ void nh_point(typename Cfg::Smem& sm, const RefRule& rr, const NHParams& P, int le, int q,
                                         int64_t et, const double (&J)[3][3], const double (&Ju)[3][3], double s) {
  constexpr int NN = Cfg::NN;
  NHPoint r;
  if (!nh_kinematics(P, original_id(P, et), rr.w[q], J, Ju, s, r)) {
#pragma unroll
    for (int k = 0; k < 4; ++k) sm.C[le][q][k] = 0.0f;
#pragma unroll
    for (int k = 0; k < 9; ++k) sm.S[le][q][k] = 0.0f;
#pragma unroll
    for (int a = 0; a < NN; ++a)
#pragma unroll
      for (int i = 0; i < 3; ++i) sm.G[le][q][3 * a + i] = sm.H[le][q][3 * a + i] = 0.0f;
    return;
  }
  sm.C[le][q][0] = f64_to_f32_rn(r.W * P.mu);
  sm.C[le][q][1] = f64_to_f32_rn(r.W * P.lam);
  sm.C[le][q][2] = f64_to_f32_rn(r.W * (P.mu - P.lam * r.lnJ));
  sm.C[le][q][3] = f64_to_f32_rn(r.W * P.mass);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) sm.S[le][q][3 * i + j] = f64_to_f32_rn(r.WP[i][j]);
  float gt[NN][3];  // g_a
  if constexpr (Cfg::kHex) {
    const double det = J[0][0] * r.C[0][0] + J[0][1] * r.C[0][1] + J[0][2] * r.C[0][2];
    float Cf[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) Cf[i][j] = f64_to_f32_rn(r.C[i][j]);
    const float invf = (float)s / f64_to_f32_rn(det);
#pragma unroll
    for (int a = 0; a < NN; ++a)
#pragma unroll
      for (int i = 0; i < 3; ++i)
        gt[a][i] = (rr.dNf[q][a][0] * Cf[i][0] + rr.dNf[q][a][1] * Cf[i][1] + rr.dNf[q][a][2] * Cf[i][2]) * invf;
  } else {
    const double inv = s * r.rdet;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double c0 = r.C[i][0] * inv, c1 = r.C[i][1] * inv, c2 = r.C[i][2] * inv;
#pragma unroll
      for (int a = 0; a < NN; ++a)
        gt[a][i] = f64_to_f32_rn(fma(rr.dN[q][a][2], c2, fma(rr.dN[q][a][1], c1, rr.dN[q][a][0] * c0)));
    }
  }
  // h_a = F^-T g_a in FP32, like the other gradient products
  float Ft[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Ft[i][j] = f64_to_f32_rn(r.Fit[i][j]);
#pragma unroll
  for (int a = 0; a < NN; ++a) {
    const float g0 = gt[a][0], g1 = gt[a][1], g2 = gt[a][2];
    float *g = sm.G[le][q] + 3 * a, *h = sm.H[le][q] + 3 * a;
    g[0] = g0;
    g[1] = g1;
    g[2] = g2;
#pragma unroll
    for (int i = 0; i < 3; ++i) h[i] = Ft[i][0] * g0 + Ft[i][1] * g1 + Ft[i][2] * g2;
  }
}

// One FP32 tile of EPC elements from launch index e0 (elements at or past
// n_end are skipped).  Every thread of the CTA calls it; it ends with a barrier.
template <int TYPE, int SLOT, int SC, class Smem>
__device__ __forceinline__ void nh_tile_body(Smem& sm, const RefRule& rr, const NHParams& P, int64_t e0,
                                             int64_t n_end) {
  using Cfg = NHCfg<TYPE, SLOT>;
  constexpr int NN = Cfg::NN, NQ = Cfg::NQ, EPC = Cfg::EPC, LPE = Cfg::LPE, EPW = Cfg::EPW;
  constexpr int NB = column_group(NN, 3, SC);  // columns a lane accumulates at a time
  // phase 0: coordinates and displacements of the tile's nodes
  for (int t = threadIdx.x; t < EPC * NN; t += Cfg::THREADS) {
    const int le = t / NN, a = t % NN;
    const int64_t et = e0 + le;
    if (et < n_end) {
      const int64_t node = P.tconn[group_index(P, et) * NN + a];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        sm.X[le][a][i] = P.coords[3 * node + i];
        sm.U[le][a][i] = P.u[3 * node + i];
      }
    }
  }
  __syncthreads();
  // phase 1: one thread per (element, point)
  field_points<TYPE, NQ, EPC, Cfg::THREADS>(
      sm, rr, e0, n_end, [](int p) { return hex8_corner_node(p); },
      [&](int le, int q, int64_t et, const double(&J)[3][3], const double(&Ju)[3][3], double s) {
        nh_point<Cfg>(sm, rr, P, le, q, et, J, Ju, s);
      });
  __syncthreads();
  if constexpr (SC == FEA_SCATTER_ATOMIC) wait_for_previous();

  // phase 2: lane a accumulates its row block
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lw = lane / LPE;
  const int le = warp * EPW + lw;
  const int64_t et = e0 + le;
  const bool active = lw < EPW && et < n_end;
  const int a = lane % LPE;
  const int64_t g = active ? group_index(P, et) : 0;
  const int64_t node = active ? (int64_t)P.tconn[g * NN + a] : 0;
  using CS = CoopScatter<NN, SC>;
  // the cooperative scatter stages its values where the coordinates and
  // displacements were
  float* vals = reinterpret_cast<float*>(&sm) + warp * CS::kVals;
  constexpr bool kCoop = CS::kOn && Cfg::kCoop;
  if constexpr (kCoop) {
    CS::begin(sm.rows[warp], P, active, g, a);
  }
  float rhs[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 1
  for (int b0 = 0; b0 < NN; b0 += NB) {
    float K[NB][3][3];
#pragma unroll
    for (int bb = 0; bb < NB; ++bb)
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) K[bb][c][cc] = 0.0f;
    if (active) {
#pragma unroll 1
      for (int q = 0; q < NQ; ++q) {
        const float wm = sm.C[le][q][0], wl = sm.C[le][q][1], wp = sm.C[le][q][2], wn = sm.C[le][q][3];
        const float *pg = sm.G[le][q], *ph = sm.H[le][q];
        const float ga[3] = {pg[3 * a], pg[3 * a + 1], pg[3 * a + 2]};
        const float gm[3] = {wm * ga[0], wm * ga[1], wm * ga[2]};
        const float hl[3] = {wl * ph[3 * a], wl * ph[3 * a + 1], wl * ph[3 * a + 2]};
        const float hp[3] = {wp * ph[3 * a], wp * ph[3 * a + 1], wp * ph[3 * a + 2]};
        const float mn = wn * rr.Nf[q][a];
#pragma unroll
        for (int bb = 0; bb < NB; ++bb) {
          const float gb[3] = {pg[3 * (b0 + bb)], pg[3 * (b0 + bb) + 1], pg[3 * (b0 + bb) + 2]};
          const float hb[3] = {ph[3 * (b0 + bb)], ph[3 * (b0 + bb) + 1], ph[3 * (b0 + bb) + 2]};
          const float diag = gm[0] * gb[0] + gm[1] * gb[1] + gm[2] * gb[2] + mn * rr.Nf[q][b0 + bb];
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) K[bb][c][cc] += hl[c] * hb[cc] + hb[c] * hp[cc];
#pragma unroll
          for (int c = 0; c < 3; ++c) K[bb][c][c] += diag;
        }
        if (b0 == 0) {
          const float* S = sm.S[le][q];
#pragma unroll
          for (int c = 0; c < 3; ++c) rhs[c] += S[3 * c] * ga[0] + S[3 * c + 1] * ga[1] + S[3 * c + 2] * ga[2];
        }
      }
    }
    if constexpr (kCoop) {
      CS::add(sm.rows[warp], vals, b0, K);
    } else if (active) {
      const int64_t id = P.ids ? (int64_t)P.ids[g] : g;
      const int32_t* mp = P.node_map + (P.mapoff ? P.mapoff[g] : id * NN * NN) + a * NN + b0;
      int64_t rb[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) rb[c] = P.row_ptr[3 * node + c];
#pragma unroll
      for (int bb = 0; bb < NB; ++bb) {
        const int64_t k = mp[bb];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          double* row = P.A + rb[c] + 3 * k;
#pragma unroll
          for (int cc = 0; cc < 3; ++cc) scatter_add<SC>(row + cc, widen(K[bb][c][cc]));
        }
      }
    }
  }
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) scatter_add<SC>(P.b + 3 * node + c, widen(rhs[c]));
  __syncthreads();
}

// ---------------------------------------------------------------------------
// FP64 tiles, by node pairs
// ---------------------------------------------------------------------------
template <int TYPE, int SLOT>
struct NHPairCfg : PairShape<TYPE, SLOT, 3, pair_epc(rule_nq(SLOT))> {
  using Base = PairShape<TYPE, SLOT, 3, pair_epc(rule_nq(SLOT))>;
  struct Smem : Base::Nodes {
    double U[Base::EPC][Base::NN][3];
    double G[Base::EPC][Base::NQ][Base::GS];  // g^
    double H[Base::EPC][Base::NQ][Base::GS];  // h^
    double C[Base::EPC][Base::NQ][2];         // mu - lam ln J, W m
    double S[Base::EPC][Base::NQ][9];         // sqrt(W) P, row-major
  };
};

template <class Cfg>
__device__ __forceinline__ void nh_pair_point(typename Cfg::Smem& sm, const RefRule& rr, const NHParams& P, int le,
                                              int q, int64_t et, const double (&J)[3][3], const double (&Ju)[3][3],
                                              double s) {
  constexpr int NN = Cfg::NN;
  NHPoint r;
  double *g = sm.G[le][q], *h = sm.H[le][q];
  if (!nh_kinematics(P, original_id(P, et), rr.w[q], J, Ju, s, r)) {
#pragma unroll
    for (int k = 0; k < 3 * NN; ++k) g[k] = h[k] = 0.0;
    sm.C[le][q][0] = sm.C[le][q][1] = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) sm.S[le][q][k] = 0.0;
    return;
  }
  const double rroot = rsqrt(r.W), inv = r.W * rroot * (s * r.rdet);
  sm.C[le][q][0] = fma(-P.lam, r.lnJ, P.mu);
  sm.C[le][q][1] = r.W * P.mass;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      sm.S[le][q][3 * i + j] = r.WP[i][j] * rroot;
      r.C[i][j] *= inv;
    }
#pragma unroll
  for (int u = 0; u < NN; ++u) {
    const double* d = rr.dN[q][Cfg::node_of(u)];
    double v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) g[3 * u + i] = v[i] = fma(d[2], r.C[i][2], fma(d[1], r.C[i][1], d[0] * r.C[i][0]));
#pragma unroll
    for (int i = 0; i < 3; ++i) h[3 * u + i] = fma(r.Fit[i][2], v[2], fma(r.Fit[i][1], v[1], r.Fit[i][0] * v[0]));
  }
}

template <class Cfg, int SC, bool DIAG>
__device__ __forceinline__ void nh_pair_task(const typename Cfg::Smem& sm, const RefRule& rr, const NHParams& P,
                                             int le, int u, int v) {
  const typename Cfg::Node nu = sm.nd[le][u], nv = sm.nd[le][v];
  int64_t kuv, kvu;
  pair_ranks<Cfg>(sm, P, le, u, v, &kuv, &kvu);
  const int au = Cfg::node_of(u), av = Cfg::node_of(v);
  double M[3][3], N[3][3], dot = 0.0, mass = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < 3; ++k) M[c][k] = N[c][k] = 0.0;
  double f[1][3] = {{0.0, 0.0, 0.0}};
#pragma unroll 1
  for (int q = 0; q < Cfg::NQ; ++q) {
    const double *a = sm.G[le][q] + 3 * u, *b = sm.G[le][q] + 3 * v;
    const double *ha = sm.H[le][q] + 3 * u, *hb = sm.H[le][q] + 3 * v;
    const double p = sm.C[le][q][0];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double y = p * ha[c];
      dot = fma(a[c], b[c], dot);
#pragma unroll
      for (int k = DIAG ? c : 0; k < 3; ++k) {
        M[c][k] = fma(ha[c], hb[k], M[c][k]);
        N[c][k] = fma(y, hb[k], N[c][k]);
      }
    }
    if (P.mass != 0.0) mass = fma(sm.C[le][q][1] * rr.N[q][au], rr.N[q][av], mass);
    if constexpr (DIAG) {
      const double* S = sm.S[le][q];
#pragma unroll
      for (int c = 0; c < 3; ++c) f[0][c] = fma(S[3 * c + 2], a[2], fma(S[3 * c + 1], a[1], fma(S[3 * c], a[0], f[0][c])));
    }
  }
  const double d = fma(P.mu, dot, mass);
  double K[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const bool low = DIAG && k < c;  // M and N are symmetric on the diagonal
      const double nt = DIAG ? (low ? N[k][c] : N[c][k]) : N[k][c];
      K[c][k] = low ? K[k][c] : fma(P.lam, M[c][k], c == k ? nt + d : nt);
    }
  pair_block<SC, DIAG>(P, nu, nv, kuv, kvu, K);
  if constexpr (DIAG) pair_add<SC>(P.b + 3 * (int64_t)nu.id, 0, f);
}

template <int TYPE, int SLOT, int SC>
__device__ __forceinline__ void nh_pair_body(typename NHPairCfg<TYPE, SLOT>::Smem& sm, const RefRule& rr,
                                             const NHParams& P, int64_t e0, int64_t n_end) {
  using Cfg = NHPairCfg<TYPE, SLOT>;
  pair_nodes<Cfg>(sm, P, e0, n_end, P.u, sm.U);
  __syncthreads();
  field_points<TYPE, Cfg::NQ, Cfg::EPC, Cfg::THREADS>(
      sm, rr, e0, n_end, [](int p) { return p; },
      [&](int le, int q, int64_t et, const double(&J)[3][3], const double(&Ju)[3][3], double s) {
        nh_pair_point<Cfg>(sm, rr, P, le, q, et, J, Ju, s);
      });
  __syncthreads();
  if constexpr (SC == FEA_SCATTER_ATOMIC) wait_for_previous();
  pair_rounds<Cfg>(
      sm, e0, n_end, [&](int le, int u, int v) { nh_pair_task<Cfg, SC, false>(sm, rr, P, le, u, v); },
      [&](int le, int u) { nh_pair_task<Cfg, SC, true>(sm, rr, P, le, u, u); });
  __syncthreads();
}

// the tile of an element type in a precision
template <int TYPE, int SLOT, int PREC>
struct NHTile {
  using Cfg = NHCfg<TYPE, SLOT>;
  template <int SC>
  using Smem = std::conditional_t<SC == FEA_SCATTER_ATOMIC && Cfg::kCoop, typename Cfg::CoopSmem, typename Cfg::Smem>;
  template <int SC>
  __device__ static __forceinline__ void run(Smem<SC>& sm, const RefRule& rr, const NHParams& P, int64_t e0) {
    nh_tile_body<TYPE, SLOT, SC>(sm, rr, P, e0, P.n);
  }
};
template <int TYPE, int SLOT>
struct NHTile<TYPE, SLOT, FEA_FP64> {
  using Cfg = NHPairCfg<TYPE, SLOT>;
  template <int SC>
  using Smem = typename Cfg::Smem;
  template <int SC>
  __device__ static __forceinline__ void run(Smem<SC>& sm, const RefRule& rr, const NHParams& P, int64_t e0) {
    nh_pair_body<TYPE, SLOT, SC>(sm, rr, P, e0, P.n);
  }
};

template <int TYPE, int SLOT, int PREC, int SC>
__global__ void __launch_bounds__(128, PREC == FEA_FP64 || SC != FEA_SCATTER_ATOMIC ? 0 : 5)
    k_nh_tile(const __grid_constant__ RefRule rr, const __grid_constant__ NHParams P) {
  using T = NHTile<TYPE, SLOT, PREC>;
  extern __shared__ __align__(16) unsigned char nh_smem_raw[];
  let_next_start();
  T::template run<SC>(*reinterpret_cast<typename T::template Smem<SC>*>(nh_smem_raw), rr, P,
                      (int64_t)blockIdx.x * T::Cfg::EPC);
}

template <int TYPE, int SLOT, int PREC, int SC>
static int launch_nh(const NHParams& P, cudaStream_t s) {
  using Cfg = typename NHTile<TYPE, SLOT, PREC>::Cfg;
  constexpr size_t smem = sizeof(typename NHTile<TYPE, SLOT, PREC>::template Smem<SC>);
  static_assert(smem <= 227 * 1024, "finite-strain tile exceeds shared memory");
  auto kern = k_nh_tile<TYPE, SLOT, PREC, SC>;
  if (smem > 48 * 1024) FEA_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const unsigned grid = grid_for(P.n, Cfg::EPC);
  const bool early = P.early && starts_early(grid, P.early == 1, false);
  FEA_CUDA(launch_tiles(kern, grid, Cfg::THREADS, smem, s, early, host_rule(SLOT), P));
  return FEA_OK;
}

template <int PREC, int SC>
static int launch_nh_type(int type, const NHParams& P, cudaStream_t s) {
  switch (type) {
    case FEA_TET4: return launch_nh<FEA_TET4, kRuleTet4, PREC, SC>(P, s);
    case FEA_PYR5: return launch_nh<FEA_PYR5, kRulePyr8, PREC, SC>(P, s);
    case FEA_PRISM6: return launch_nh<FEA_PRISM6, kRulePrism6, PREC, SC>(P, s);
    default: return launch_nh<FEA_HEX8, kRuleHex8, PREC, SC>(P, s);
  }
}

int assemble_nh(const fea_operator* op, fea_mesh* m, const int64_t* row_ptr, const int32_t* node_map, double* A,
                double* b, cudaStream_t s) {
  if (op->scatter != FEA_SCATTER_ATOMIC && op->scatter != FEA_SCATTER_COLOR)
    return fail(FEA_ERR_UNSUPPORTED, "fea_assemble: the finite-strain solid supports the ATOMIC and COLOR scatters");
  if (op->schedule != FEA_SCHED_PER_TYPE)
    return fail(FEA_ERR_UNSUPPORTED, "fea_assemble: the finite-strain solid runs per element type");
  if (!op->u_d) return fail(FEA_ERR_ARG, "fea_assemble: the finite-strain solid needs the displacements u_d");
  if (!(op->poisson > -1.0 && op->poisson < 0.5)) return fail(FEA_ERR_ARG, "fea_assemble: poisson must be in (-1, 0.5)");
  if (!(op->mass >= 0.0)) return fail(FEA_ERR_ARG, "fea_assemble: mass must be >= 0");
  if (op->scatter == FEA_SCATTER_COLOR && !m->color) {
    int rc = build_color_plan(m, s);  // host-synchronous, first call only
    if (rc) return rc;
  }
  cudaEvent_t* ev = (cudaEvent_t*)op->events;
  const int nev = ev ? op->n_events : 0;
  if (nev > 0) FEA_CUDA(cudaEventRecord(ev[0], s));
  const int zrc = zero_system(A, 9 * m->nnz_node, b, m->n_nodes * 3, s);
  if (zrc) return zrc;
  if (nev > 1) FEA_CUDA(cudaEventRecord(ev[1], s));

  NHParams P;
  std::memset(&P, 0, sizeof(P));
  P.coords = m->coords;
  P.row_ptr = row_ptr;
  P.node_map = node_map;
  P.A = A;
  P.b = b;
  P.st = m->status;
  P.u = op->u_d;
  const double E = op->young, nu = op->poisson;
  P.lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu));
  P.mu = E / (2.0 * (1.0 + nu));
  P.mass = op->mass;
  const bool color = op->scatter == FEA_SCATTER_COLOR;
  P.early = !color && small_system(9 * m->nnz_node);
  int launched = 0;
  auto run = [&](int t) -> int {
    int rc;
    if (op->precision == FEA_FP64)
      rc = color ? launch_nh_type<FEA_FP64, FEA_SCATTER_COLOR>(t, P, s)
                 : launch_nh_type<FEA_FP64, FEA_SCATTER_ATOMIC>(t, P, s);
    else
      rc = color ? launch_nh_type<FEA_FP32_INTEGRATE, FEA_SCATTER_COLOR>(t, P, s)
                 : launch_nh_type<FEA_FP32_INTEGRATE, FEA_SCATTER_ATOMIC>(t, P, s);
    if (rc) return rc;
    if (2 + launched < nev) FEA_CUDA(cudaEventRecord(ev[2 + launched], s));
    ++launched;
    if (P.early) P.early = 2;
    return FEA_OK;
  };
  if (color) {
    const ColorPlan& Cp = *m->color;
    for (int c = 0; c < Cp.n_colors; ++c)
      for (int t = 0; t < kNumTypes; ++t) {
        const size_t k = (size_t)c * kNumTypes + t;
        const int64_t n = Cp.seg_off[k + 1] - Cp.seg_off[k];
        if (!n) continue;
        const TypeGroup& g = m->group[t];
        P.tconn = g.conn;
        P.ids = g.ids;
        P.mapoff = g.mapoff;
        P.list = Cp.lists + Cp.seg_off[k];
        P.n = n;
        int rc = run(t);
        if (rc) return rc;
      }
    return FEA_OK;
  }
  for (int t = 0; t < kNumTypes; ++t) {
    const TypeGroup& g = m->group[t];
    if (!g.n) continue;
    P.tconn = g.conn;
    P.ids = g.ids;
    P.mapoff = g.mapoff;
    P.list = nullptr;
    P.n = g.n;
    int rc = run(t);
    if (rc) return rc;
  }
  for (int k = 2 + launched; k < nev; ++k) FEA_CUDA(cudaEventRecord(ev[k], s));
  return FEA_OK;
}

}  // namespace fea
