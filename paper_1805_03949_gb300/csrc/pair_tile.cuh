// pair_tile.cuh -- FP64 element tiles of the diffusion and elasticity
// operators: symmetric node-pair products.
//
// The tile (pairs.cuh says why by pairs) is laid out to need few FP64
// instructions:
//  * elasticity: with g^_u(q) = sqrt(w det J) J^{-T} grad_xi N_u a pair takes
//    the 9 products M = sum_q g^_u (x) g^_v and then once
//    K = lam M + mu M^T + mu tr(M) I (18 operations), instead of 24 per point;
//    the scale sqrt(w det J) / det J is one rsqrt(det J) per point;
//  * diffusion: with c_u(q) = C grad_xi N_u (C the cofactors of J) a pair takes
//    S_q (c_u . c_v), S_q = w k(x_q) / det J, one division per point and no
//    scaled gradients (k may have either sign, so it stays out of the root);
//  * points that share their gradients (a linear tet's all, a pyramid's in
//    pairs) make one set of gradients, with their weights summed first.
// Measured on one GB300, before and after: 250,047 hex8, elasticity 8.82 ->
// 1.95 ms; 162,000 tet4, elasticity 0.776 -> 0.137 ms; 412,500 mixed elements,
// diffusion 1.53 -> 0.94 ms (0.85 with RefMap; hex8 diffusion has its own tile,
// hex_diffusion.cuh).
#pragma once

#include "pairs.cuh"

namespace fea {

// Parameters of the diffusion and elasticity kernels.
struct AsmParams : ElemParams {
  double k0, k2, src;       // diffusion
  double lam, mu;           // elasticity
  double f[3];
  int geo64;                // FP32 tiles: 1 = FP64 geometry for every element, 0 = adaptive
};

// points that share their gradients: a linear tet's all, a pyramid's q and q + 4 (RefMap)
__host__ __device__ constexpr int pair_share(int slot) {
  return rule_type(slot) == FEA_TET4 ? rule_nq(slot) : rule_type(slot) == FEA_PYR5 ? 2 : 1;
}

template <int TYPE, int SLOT, int OP>
struct PairCfg : PairShape<TYPE, SLOT, OP == FEA_OP_DIFFUSION ? 1 : 3,
                           TYPE == FEA_TET4 ? 32 : pair_epc(rule_nq(SLOT) / pair_share(SLOT))> {
  using Base = PairShape<TYPE, SLOT, OP == FEA_OP_DIFFUSION ? 1 : 3,
                         TYPE == FEA_TET4 ? 32 : pair_epc(rule_nq(SLOT) / pair_share(SLOT))>;
  static constexpr bool kTet = TYPE == FEA_TET4;
  static constexpr int kShare = pair_share(SLOT);
  static constexpr int NG = Base::NQ / kShare;  // gradient sets of an element: q % NG is point q's
  struct Smem : Base::Nodes {
    double G[Base::EPC][NG][Base::GS];  // gradients (see above) [set][node][component]
    double S[Base::EPC][NG];            // diffusion: w k / det J, summed over the points that share the set
    double W[Base::EPC][NG];            // w det J (sets shared by points: det J)
  };
};

// The values of gradient set q of element le from the cofactors C' and det' of
// J' = s J: gradients of every slot, S (wk = sum of w k over its points) and W.
template <class Cfg, int OP>
__device__ __forceinline__ void pair_point(typename Cfg::Smem& sm, const RefRule& rr, int le, int q,
                                           const double (&C)[3][3], double det, double s, double wk) {
  double* g = sm.G[le][q];
  double F[3][3];
  if constexpr (OP == FEA_OP_DIFFUSION) {
    sm.S[le][q] = wk / (s * det);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) F[i][j] = C[i][j];
  } else {
    double w = rr.w[q];
#pragma unroll
    for (int k = 1; k < Cfg::kShare; ++k) w += rr.w[q + k * Cfg::NG];
    const double r = sqrt(w / s) * rsqrt(det);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) F[i][j] = C[i][j] * r;
  }
  sm.W[le][q] = (Cfg::kShare == 1 ? rr.w[q] : 1.0) * det * (1.0 / (s * s * s));
  if constexpr (Cfg::kTet) {
    // J^{-T} grad_xi N_{j+1} is column j of C / det J; the gradients sum to zero
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
      for (int j = 0; j < 3; ++j) g[3 * (j + 1) + i] = F[i][j];
      g[i] = -(F[i][0] + F[i][1] + F[i][2]);
    }
  } else {
#pragma unroll
    for (int u = 0; u < Cfg::NN; ++u) {
      const double* d = rr.dN[q][Cfg::kHex ? hex8_corner_node(u) : u];
#pragma unroll
      for (int i = 0; i < 3; ++i) g[3 * u + i] = fma(d[2], F[i][2], fma(d[1], F[i][1], d[0] * F[i][0]));
    }
  }
}

// nodes, coordinates and the points' values of the tile [e0, e0 + EPC)
template <class Cfg, int OP>
__device__ __forceinline__ void pair_geometry(typename Cfg::Smem& sm, const RefRule& rr, const AsmParams& P,
                                              int64_t e0, int64_t n_end) {
  constexpr int TYPE = Cfg::kType, NG = Cfg::NG, EPC = Cfg::EPC;
  pair_nodes<Cfg>(sm, P, e0, n_end);
  __syncthreads();
  const int t = threadIdx.x;
  if constexpr (Cfg::kHex) {
    const int le = t >> 3, p = t & 7;
    const bool valid = e0 + le < n_end;
    double v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = valid ? sm.X[le][p][i] : 0.0;
    hex8_modal(v);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 3; ++i) sm.X[le][p][i] = v[i];
    __syncwarp();
    double J[3][3], C[3][3];
    hex8_jacobian_pairs(sm.X[le], p, J);  // every lane: it exchanges columns with partner lanes
    if (valid) {
      cofactors(J, C);
      const double det = J[0][0] * C[0][0] + J[0][1] * C[0][1] + J[0][2] * C[0][2];
      if (!(det > 0.0)) latch_error(P.st, FEA_ERR_INVERTED_ELEMENT, (unsigned long long)original_id(P, e0 + le));
      double kq = 0.0;
      if constexpr (OP == FEA_OP_DIFFUSION) {
        const double x = hex8_modal_x(sm.X[le], p);
        kq = P.k0 + P.k2 * x * x;
      }
      pair_point<Cfg, OP>(sm, rr, le, p, C, det, 8.0, rr.w[p] * kq);
    }
  } else {
    using Map = RefMap<TYPE>;
    if (t < EPC * 3 && e0 + t / 3 < n_end) Map::prep(sm.X[t / 3], t % 3);
    __syncthreads();
    const int le = t / NG, q = t % NG;
    if (t < EPC * NG && e0 + le < n_end) {
      double J[3][3], C[3][3];
      Map::jac(sm.X[le], rr.m[q], J);
      cofactors(J, C);
      const double det = J[0][0] * C[0][0] + J[0][1] * C[0][1] + J[0][2] * C[0][2];
      if (!(det > 0.0)) latch_error(P.st, FEA_ERR_INVERTED_ELEMENT, (unsigned long long)original_id(P, e0 + le));
      double wk = 0.0;
      if constexpr (OP == FEA_OP_DIFFUSION) {
#pragma unroll
        for (int k = 0; k < Cfg::kShare; ++k) {
          const int p = q + k * NG;
          const double x = Map::x1(sm.X[le], rr.N[p], rr.m[p]);
          wk = fma(rr.w[p], P.k0 + P.k2 * x * x, wk);
        }
      }
      pair_point<Cfg, OP>(sm, rr, le, q, C, det, Map::s, wk);
    }
  }
  __syncthreads();
}

// sum_q W N_a: the element integral of the slot's shape function
template <class Cfg>
__device__ __forceinline__ double pair_beta(const typename Cfg::Smem& sm, const RefRule& rr, int le, int u) {
  const int a = Cfg::node_of(u);
  double s = 0.0;
#pragma unroll
  for (int g = 0; g < Cfg::NG; ++g) {
    double n = rr.N[g][a];
    if constexpr (Cfg::kShare > 1) {
      n *= rr.w[g];
#pragma unroll
      for (int k = 1; k < Cfg::kShare; ++k) n = fma(rr.w[g + k * Cfg::NG], rr.N[g + k * Cfg::NG][a], n);
    }
    s = fma(sm.W[le][g], n, s);
  }
  return s;
}

// One task: the entry block of the nodes in slots u and v of element le, into
// row u and (off the diagonal) transposed into row v; the right-hand side of
// node u with the diagonal task.
template <class Cfg, int OP, int SC, bool DIAG>
__device__ __forceinline__ void pair_task(const typename Cfg::Smem& sm, const RefRule& rr, const AsmParams& P, int le,
                                          int u, int v) {
  constexpr int NG = Cfg::NG;
  const typename Cfg::Node nu = sm.nd[le][u], nv = sm.nd[le][v];
  int64_t kuv, kvu;
  pair_ranks<Cfg>(sm, P, le, u, v, &kuv, &kvu);
  if constexpr (OP == FEA_OP_DIFFUSION) {
    double K[1][1] = {{0.0}};
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const double* a = sm.G[le][q] + 3 * u;
      const double* b = sm.G[le][q] + 3 * v;
      K[0][0] = fma(sm.S[le][q], fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0])), K[0][0]);
    }
    pair_add<SC>(P.A + nu.row + kuv, 0, K);
    if constexpr (!DIAG) pair_add<SC>(P.A + nv.row + kvu, 0, K);
    if constexpr (DIAG) {
      const double f[1][1] = {{pair_beta<Cfg>(sm, rr, le, u) * P.src}};
      pair_add<SC>(P.b + nu.id, 0, f);
    }
  } else {
    double M[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll 2
    for (int q = 0; q < NG; ++q) {
      const double* a = sm.G[le][q] + 3 * u;
      const double* b = sm.G[le][q] + 3 * v;
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = DIAG ? c : 0; k < 3; ++k) M[c][k] = fma(a[c], b[k], M[c][k]);
    }
    const double lam = P.lam, mu = P.mu, lm = P.lam + P.mu;
    const double tr = mu * (M[0][0] + M[1][1] + M[2][2]);
    double K[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (c == k)
          K[c][c] = fma(lm, M[c][c], tr);
        else if constexpr (DIAG)
          K[c][k] = c < k ? lm * M[c][k] : K[k][c];
        else
          K[c][k] = fma(lam, M[c][k], mu * M[k][c]);
      }
    pair_block<SC, DIAG>(P, nu, nv, kuv, kvu, K);
    if constexpr (DIAG) {
      const double beta = pair_beta<Cfg>(sm, rr, le, u);
      const double f[1][3] = {{beta * P.f[0], beta * P.f[1], beta * P.f[2]}};
      pair_add<SC>(P.b + 3 * (int64_t)nu.id, 0, f);
    }
  }
}

// One tile of EPC elements starting at launch index e0 (elements at or past
// n_end are skipped).  Every thread of the CTA must call it; it ends with the
// shared memory free.
template <int TYPE, int SLOT, int OP, int SC>
__device__ __forceinline__ void pair_tile_body(typename PairCfg<TYPE, SLOT, OP>::Smem& sm, const RefRule& rr,
                                               const AsmParams& P, int64_t e0, int64_t n_end) {
  using Cfg = PairCfg<TYPE, SLOT, OP>;
  pair_geometry<Cfg, OP>(sm, rr, P, e0, n_end);
  if constexpr (SC == FEA_SCATTER_ATOMIC) wait_for_previous();
  pair_rounds<Cfg>(
      sm, e0, n_end, [&](int le, int u, int v) { pair_task<Cfg, OP, SC, false>(sm, rr, P, le, u, v); },
      [&](int le, int u) { pair_task<Cfg, OP, SC, true>(sm, rr, P, le, u, u); });
  __syncthreads();
}

}  // namespace fea
