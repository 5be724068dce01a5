// pair_tile.cuh -- FP64 element tiles of the diffusion and elasticity
// operators: symmetric node-pair products.
//
// On GB300 an FP64 instruction of a warp holds the SM's FP64 unit for 16
// cycles (2 lanes per clock), so an FP64 tile is bound by the number of FP64
// instructions and by nothing else: ncu of the tile that gave each lane a row
// block (all columns of one node) read the FP64 unit 87 % busy with the issue
// slots 7 % used.  This tile is laid out to need few of them:
//  * the element matrices are symmetric, so only the node pairs (u, v), u < v,
//    and the diagonal ones are formed, one per thread ("task"), and each is
//    added to row u and, transposed, to row v;
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
// diffusion 1.53 -> 0.94 ms.
// A tile holds as many elements as give each of its 128 threads one
// quadrature point; its tasks are numbered element by element, the
// off-diagonal ones first, and go to the warps in rounds of 32.
#pragma once

#include "element.cuh"

namespace fea {

// Parameters of the diffusion and elasticity kernels.
struct AsmParams {
  const double* coords;
  const int32_t* tconn;     // [n][NN] packed connectivity of the group
  const int32_t* ids;       // [n] original element ids (nullptr: identity)
  const int64_t* mapoff;    // [n] node_map offsets (nullptr: id * NN^2)
  const int32_t* list;      // launch index -> index in the group (nullptr: identity; coloring)
  int64_t n;                // elements of this launch
  const int64_t* row_ptr;
  const int32_t* node_map;
  double* A;
  double* b;
  DevStatus* st;
  double k0, k2, src;       // diffusion
  double lam, mu;           // elasticity
  double f[3];
  int geo64;                // FP32 tiles: 1 = FP64 geometry for every element, 0 = adaptive
};

__device__ __forceinline__ int64_t group_index(const AsmParams& P, int64_t et) {
  return P.list ? (int64_t)P.list[et] : et;
}
__device__ __forceinline__ int64_t original_id(const AsmParams& P, int64_t et) {
  const int64_t g = group_index(P, et);
  return P.ids ? (int64_t)P.ids[g] : g;
}

template <int TYPE, int SLOT, int OP>
struct PairCfg {
  static constexpr int kType = TYPE;
  static constexpr int NN = nodes_of(TYPE);
  static constexpr int NQ = rule_nq(SLOT);
  static constexpr int D = OP == FEA_OP_DIFFUSION ? 1 : 3;
  static constexpr bool kHex = TYPE == FEA_HEX8;
  static constexpr bool kTet = TYPE == FEA_TET4;
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int EPC = kTet ? 32 : TYPE == FEA_PYR5 ? 32 : (THREADS / NQ) & ~3;  // elements per tile
  // points that share their gradients: a linear tet's all, a pyramid's q and q + 4 (RefMap)
  static constexpr int kShare = kTet ? NQ : TYPE == FEA_PYR5 ? 2 : 1;
  static constexpr int NG = NQ / kShare;                       // gradient sets of an element: q % NG is point q's
  static constexpr int GS = 3 * NN + 1;                        // odd stride: points spread over the banks
  static constexpr int kOff = NN * (NN - 1) / 2;               // off-diagonal pairs
  static_assert(!kHex || EPC * 8 == THREADS, "the modal transform needs whole warps");
  // a node of an element: start of its first row, length of its rows, id
  struct Node {
    int64_t row;
    int32_t len, id;
  };
  struct Smem {
    double X[EPC][NN][3];   // node coordinates (hex8: corners in binary order)
    double G[EPC][NG][GS];  // gradients (see above) [point][node][component]
    double S[EPC][NG];      // diffusion: w k / det J, summed over the points that share the set
    double W[EPC][NG];      // w det J (sets shared by points: det J)
    Node nd[EPC][NN];
    int64_t moff[EPC];      // node_map offset of the element
    uint8_t pair[kOff][2];
  };
  // local node of slot u
  __device__ static __forceinline__ int node_of(int u) { return kHex ? hex8_corner_node(u) : u; }
};

// v[c][k] into p[c stride + k] (A or b) under the race treatment SC: this
// thread is the only one of the launch that touches the entries unless SC is
// ATOMIC.  MULTIDEP: CTAs on other SMs wrote them before the locks changed
// hands, so they are read from and written to L2.  All loads come before the
// stores: the compiler may not move a load over a store into A.
template <int SC, int R, int K>
__device__ __forceinline__ void pair_add(double* p, int64_t stride, const double (&v)[R][K]) {
  if constexpr (SC == FEA_SCATTER_ATOMIC) {
#pragma unroll
    for (int c = 0; c < R; ++c)
#pragma unroll
      for (int k = 0; k < K; ++k) red_add(p + c * stride + k, v[c][k]);
  } else {
    double old[R][K];
#pragma unroll
    for (int c = 0; c < R; ++c)
#pragma unroll
      for (int k = 0; k < K; ++k)
        old[c][k] = SC == FEA_SCATTER_MULTIDEP ? __ldcg(p + c * stride + k) : p[c * stride + k];
#pragma unroll
    for (int c = 0; c < R; ++c)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if constexpr (SC == FEA_SCATTER_MULTIDEP)
          __stcg(p + c * stride + k, old[c][k] + v[c][k]);
        else
          p[c * stride + k] = old[c][k] + v[c][k];
      }
  }
}

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
template <class Cfg, int OP, class Params>
__device__ __forceinline__ void pair_geometry(typename Cfg::Smem& sm, const RefRule& rr, const Params& P, int64_t e0,
                                              int64_t n_end) {
  constexpr int TYPE = Cfg::kType, NN = Cfg::NN, NG = Cfg::NG, EPC = Cfg::EPC, D = Cfg::D;
  static_assert(EPC * 3 <= Cfg::THREADS, "a thread per element and component");
  for (int p = threadIdx.x; p < Cfg::kOff; p += Cfg::THREADS) {
    int u = 0, r = p;
    while (r >= NN - 1 - u) r -= NN - 1 - u++;
    sm.pair[p][0] = (uint8_t)u;
    sm.pair[p][1] = (uint8_t)(u + 1 + r);
  }
  for (int t = threadIdx.x; t < EPC * NN; t += Cfg::THREADS) {
    const int le = t / NN, u = t % NN;
    const int64_t et = e0 + le;
    if (et >= n_end) continue;
    const int64_t g = group_index(P, et);
    const int64_t node = P.tconn[g * NN + Cfg::node_of(u)];
    if (u == 0) sm.moff[le] = P.mapoff ? P.mapoff[g] : (P.ids ? (int64_t)P.ids[g] : g) * NN * NN;
    const int64_t r0 = P.row_ptr[D * node];
    sm.nd[le][u] = {r0, D == 1 ? 0 : (int32_t)(P.row_ptr[D * node + 1] - r0), (int32_t)node};
#pragma unroll
    for (int i = 0; i < 3; ++i) sm.X[le][u][i] = P.coords[3 * node + i];
  }
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
template <class Cfg, int OP, int SC, bool DIAG, class Params>
__device__ __forceinline__ void pair_task(const typename Cfg::Smem& sm, const RefRule& rr, const Params& P, int le,
                                          int u, int v) {
  constexpr int NN = Cfg::NN, NG = Cfg::NG;
  const typename Cfg::Node nu = sm.nd[le][u], nv = sm.nd[le][v];
  const int au = Cfg::node_of(u), av = Cfg::node_of(v);
  const int32_t* mp = P.node_map + sm.moff[le];
  const int64_t kuv = mp[au * NN + av], kvu = DIAG ? kuv : (int64_t)mp[av * NN + au];
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
    pair_add<SC>(P.A + nu.row + 3 * kuv, nu.len, K);
    if constexpr (!DIAG) {
      double T[3][3];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < 3; ++k) T[k][c] = K[c][k];
      pair_add<SC>(P.A + nv.row + 3 * kvu, nv.len, T);
    }
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
template <int TYPE, int SLOT, int OP, int SC, class Params>
__device__ __forceinline__ void pair_tile_body(typename PairCfg<TYPE, SLOT, OP>::Smem& sm, const RefRule& rr,
                                               const Params& P, int64_t e0, int64_t n_end) {
  using Cfg = PairCfg<TYPE, SLOT, OP>;
  constexpr int NN = Cfg::NN, EPC = Cfg::EPC, kOff = Cfg::kOff;
  pair_geometry<Cfg, OP>(sm, rr, P, e0, n_end);
  // rounds of 32 tasks: the off-diagonal ones, then the diagonal ones
  constexpr int kOffRounds = (EPC * kOff + 31) / 32, kRounds = kOffRounds + (EPC * NN + 31) / 32;
  const int lane = threadIdx.x & 31;
  int r = threadIdx.x >> 5;
  for (; r < kOffRounds; r += Cfg::WARPS) {
    const int t = 32 * r + lane, le = t / kOff, p = t % kOff;
    if (le < EPC && e0 + le < n_end) pair_task<Cfg, OP, SC, false>(sm, rr, P, le, sm.pair[p][0], sm.pair[p][1]);
  }
  for (; r < kRounds; r += Cfg::WARPS) {
    const int t = 32 * (r - kOffRounds) + lane, le = t / NN, u = t % NN;
    if (le < EPC && e0 + le < n_end) pair_task<Cfg, OP, SC, true>(sm, rr, P, le, u, u);
  }
  __syncthreads();
}

}  // namespace fea
