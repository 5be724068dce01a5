// hex_diffusion.cuh -- FP64 diffusion tile of hex8.
//
// With T(q) = w k / det J C^T C (C the cofactors of J; symmetric, 6 values),
//   A^e_ab = sum_q grad_xi N_a . T(q) grad_xi N_b,
// and only T depends on the element: the reference gradients are products of
// one factor per axis, d_j N_a = a_j/8 prod_{s != j} (1 + a_s xi_s) with the
// corner's signs a_s, and the 2x2x2 points are xi_s = +-g, g^2 = 1/3.  So the
// sum over the points factorises axis by axis, starting from the
// Walsh-Hadamard transform T^[m] = sum_q prod_{s in m} sigma_s(q) T(q) (the
// butterflies of hex8_modal), into 63 values per element:
//   U_j(c_s, c_t) for d_j N_a d_j N_b: along the other axes s, t the product
//     (1 + a xi)(1 + b xi) has three forms c: a = b = +, a = b = -, a != b;
//   V_ji(x_i, x_j, c_t) for d_j N_a d_i N_b, j != i: one factor along i and j;
// and every entry is a signed sum of nine of them:
//   A^e_ab = sum_j a_j b_j U_j + sum_{j<i} [a_j b_i V_ji(a_i, b_j) + a_i b_j V_ji(b_i, a_j)].
// About 1,440 FP64 instructions per element where the gradients at the points
// and their products take 2,340 (pair_tile.cuh); FP64 instructions are what
// bounds the tile (pairs.cuh).  One GB300: 412,500 mixed elements (30 % hex8)
// 0.846 -> 0.669 ms, their hex8 tiles 0.517 -> 0.339 ms.
#pragma once

#include "pair_tile.cuh"

namespace fea {

struct HexDiffusionCfg : PairShape<FEA_HEX8, kRuleHex8, 1, 16> {
  using Base = PairShape<FEA_HEX8, kRuleHex8, 1, 16>;
  struct Smem : Base::Nodes {
    double T[EPC][8][7];        // T^[m] / 64: 00, 11, 22, 01, 12, 02 (and a pad against bank conflicts)
    double U[EPC][3][3][3];     // [j][c of axis j + 1][c of axis j + 2]
    double V[EPC][3][2][2][3];  // [pair (0,1), (1,2), (0,2)][x of the second axis][x of the first][c of the third]
    double W[EPC][8];           // w det J
  };
};

// the three forms (1 + a xi)(1 + b xi) = alpha + beta sigma along one axis,
// applied to the sums without (f0) and with (f1) the axis' sign
__device__ __forceinline__ void hex_axis_forms(double f0, double f1, double* out) {
  constexpr double g2 = 2.0 * 0.57735026918962576451;
  const double e = (4.0 / 3.0) * f0;
  out[0] = fma(g2, f1, e);
  out[1] = fma(-g2, f1, e);
  out[2] = (2.0 / 3.0) * f0;
}

__device__ __forceinline__ double hex_signed(double v, int minus) {
  return __hiloint2double(__double2hiint(v) ^ (minus << 31), __double2loint(v));
}

template <int SC>
__device__ __forceinline__ void hex_diffusion_body(HexDiffusionCfg::Smem& sm, const RefRule& rr, const AsmParams& P,
                                                   int64_t e0, int64_t n_end) {
  using Cfg = HexDiffusionCfg;
  constexpr int EPC = Cfg::EPC;
  constexpr double g = 0.57735026918962576451;
  pair_nodes<Cfg>(sm, P, e0, n_end);
  __syncthreads();
  {
    // T^ / 64 and w det J of the lane's point
    const int le = threadIdx.x >> 3, p = threadIdx.x & 7;
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
    double d[3] = {0.0, 0.0, 0.0}, o[3] = {0.0, 0.0, 0.0};
    if (valid) {
      cofactors(J, C);
      const double det = J[0][0] * C[0][0] + J[0][1] * C[0][1] + J[0][2] * C[0][2];
      if (!(det > 0.0)) latch_error(P.st, FEA_ERR_INVERTED_ELEMENT, (unsigned long long)original_id(P, e0 + le));
      const double x = hex8_modal_x(sm.X[le], p);
      // J' = 8 J: w k / det J C^T C = w k / (8 det') C'^T C'
      const double s = rr.w[p] * (P.k0 + P.k2 * x * x) / (512.0 * det);
      sm.W[le][p] = rr.w[p] * det * (1.0 / 512.0);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int k = (j + 1) % 3;  // d: 00, 11, 22; o: 01, 12, 20
        d[j] = s * fma(C[2][j], C[2][j], fma(C[1][j], C[1][j], C[0][j] * C[0][j]));
        o[j] = s * fma(C[2][j], C[2][k], fma(C[1][j], C[1][k], C[0][j] * C[0][k]));
      }
    }
    hex8_modal(d);
    hex8_modal(o);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      sm.T[le][p][j] = d[j];
      sm.T[le][p][3 + j] = o[j];
    }
  }
  __syncthreads();
  // the tables: (element, j, c) and (element, pair, x) per thread
  for (int t = threadIdx.x; t < EPC * 9; t += Cfg::THREADS) {
    const int le = t / 9, j = (t % 9) / 3, c = t % 3;
    const int ms = 1 << ((j + 1) % 3), mt = 1 << ((j + 2) % 3);
    const double(*T)[7] = sm.T[le];
    const double alpha = c == 2 ? 2.0 / 3.0 : 4.0 / 3.0, beta = c == 2 ? 0.0 : c == 0 ? 2.0 * g : -2.0 * g;
    hex_axis_forms(fma(beta, T[ms][j], alpha * T[0][j]), fma(beta, T[ms | mt][j], alpha * T[mt][j]), sm.U[le][j][c]);
  }
  for (int t = threadIdx.x; t < EPC * 6; t += Cfg::THREADS) {
    const int le = t / 6, pr = (t % 6) >> 1, xi = t & 1;  // xi: 1 for +
    const int j = pr == 1 ? 1 : 0, i = pr == 0 ? 1 : 2, mj = 1 << j, mi = 1 << i, mt = 7 ^ mj ^ mi, k = 3 + pr;
    const double(*T)[7] = sm.T[le];
    const double gi = xi ? g : -g;
    const double b00 = fma(gi, T[mi][k], T[0][k]), bj0 = fma(gi, T[mi | mj][k], T[mj][k]);
    const double b0t = fma(gi, T[mi | mt][k], T[mt][k]), bjt = fma(gi, T[7][k], T[mj | mt][k]);
    hex_axis_forms(fma(-g, bj0, b00), fma(-g, bjt, b0t), sm.V[le][pr][xi][0]);
    hex_axis_forms(fma(g, bj0, b00), fma(g, bjt, b0t), sm.V[le][pr][xi][1]);
  }
  __syncthreads();
  if constexpr (SC == FEA_SCATTER_ATOMIC) wait_for_previous();
  // entry of corners u and v (binary order: bit s set for sign + along axis s)
  auto entry = [&](int le, int u, int v) {
    const int differ = u ^ v;
    int form[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) form[s] = (differ >> s) & 1 ? 2 : 1 - ((u >> s) & 1);
    double K = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j)
      K += hex_signed(sm.U[le][j][form[(j + 1) % 3]][form[(j + 2) % 3]], (differ >> j) & 1);
#pragma unroll
    for (int pr = 0; pr < 3; ++pr) {
      const int j = pr == 1 ? 1 : 0, i = pr == 0 ? 1 : 2, t = 3 - i - j;
      const int uj = (u >> j) & 1, ui = (u >> i) & 1, vj = (v >> j) & 1, vi = (v >> i) & 1;
      K += hex_signed(sm.V[le][pr][ui][vj][form[t]], uj ^ vi);
      K += hex_signed(sm.V[le][pr][vi][uj][form[t]], ui ^ vj);
    }
    return K;
  };
  pair_rounds<Cfg>(
      sm, e0, n_end,
      [&](int le, int u, int v) {
        int64_t kuv, kvu;
        pair_ranks<Cfg>(sm, P, le, u, v, &kuv, &kvu);
        const double K[1][1] = {{entry(le, u, v)}};
        pair_add<SC>(P.A + sm.nd[le][u].row + kuv, 0, K);
        pair_add<SC>(P.A + sm.nd[le][v].row + kvu, 0, K);
      },
      [&](int le, int u) {
        int64_t kuu, same;
        pair_ranks<Cfg>(sm, P, le, u, u, &kuu, &same);
        const double K[1][1] = {{entry(le, u, u)}};
        pair_add<SC>(P.A + sm.nd[le][u].row + kuu, 0, K);
        double beta = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) beta = fma(sm.W[le][q], rr.N[q][Cfg::node_of(u)], beta);
        const double f[1][1] = {{beta * P.src}};
        pair_add<SC>(P.b + sm.nd[le][u].id, 0, f);
      });
  __syncthreads();
}

}  // namespace fea
