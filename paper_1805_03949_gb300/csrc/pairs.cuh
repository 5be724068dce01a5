// pairs.cuh -- what the FP64 element tiles of every operator share: node pairs
// as tasks, and their scatter.
//
// On GB300 an FP64 instruction of a warp holds the SM's FP64 unit for 16
// cycles (2 lanes per clock), so an FP64 tile is bound by the number of FP64
// instructions and by nothing else: ncu of the tiles that gave each lane a row
// block (all columns of one node) read the FP64 unit 87 % busy with the issue
// slots 7 % used.  The element matrices are symmetric, so the tiles form only
// the node pairs (u, v), u < v, and the diagonal ones, one per thread
// ("task"), and add each to row u and, transposed, to row v.  A tile's tasks
// are numbered element by element, the off-diagonal ones first, and go to its
// warps in rounds of 32.
#pragma once

#include "element.cuh"
#include "zero.cuh"

namespace fea {

// What the kernels of every operator know of one launch's elements.
struct ElemParams {
  const double* coords;
  const int32_t* tconn;     // [n][NN] packed connectivity of the type group
  const int32_t* ids;       // [n] original element ids (nullptr: identity)
  const int64_t* mapoff;    // [n] node_map offsets (nullptr: id * NN^2)
  const int32_t* list;      // launch index -> index in the group (nullptr: identity; coloring)
  int64_t n;                // elements of this launch
  const int64_t* row_ptr;
  const int32_t* node_map;
  double* A;
  double* b;
  DevStatus* st;
  int early;                // host: tile kernels may start early (zero.cuh): 1 after the clearing, 2 after a type
};

// (Params: const ElemParams or a derived struct, volatile where its fields are
// to be read from shared memory at each use instead of kept in registers)
template <class Params>
__device__ __forceinline__ int64_t group_index(Params& P, int64_t et) {
  return P.list ? (int64_t)P.list[et] : et;
}
template <class Params>
__device__ __forceinline__ int64_t original_id(Params& P, int64_t et) {
  const int64_t g = group_index(P, et);
  return P.ids ? (int64_t)P.ids[g] : g;
}

// EPC_ elements per tile, DOF values per node
template <int TYPE, int SLOT, int DOF, int EPC_>
struct PairShape {
  static constexpr int kType = TYPE;
  static constexpr int NN = nodes_of(TYPE);
  static constexpr int NQ = rule_nq(SLOT);
  static constexpr int D = DOF;
  static constexpr bool kHex = TYPE == FEA_HEX8;
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int EPC = EPC_;
  static constexpr int GS = 3 * NN + 1;           // gradients of a point: an odd stride spreads points over the banks
  static constexpr int kOff = NN * (NN - 1) / 2;  // off-diagonal pairs
  static_assert(!kHex || EPC * 8 == THREADS, "the modal transform needs whole warps");
  static_assert(EPC * 3 <= THREADS, "a thread per element and component");
  // a node of an element: start of its first row, length of its rows, id
  struct Node {
    int64_t row;
    int32_t len, id;
  };
  struct Nodes {
    double X[EPC][NN][3];  // node coordinates (hex8: corners in binary order)
    Node nd[EPC][NN];
    int64_t moff[EPC];     // node_map offset of the element
    uint8_t pair[kOff][2];
  };
  // local node of slot u
  __device__ static __forceinline__ int node_of(int u) { return kHex ? hex8_corner_node(u) : u; }
};

// elements per tile that give each of a tile's 128 threads a quadrature point
// (whole groups of 4 elements)
__host__ __device__ constexpr int pair_epc(int points) { return (128 / points) & ~3; }

// The pair list and the nodes of the tile [e0, e0 + EPC); field (may be
// nullptr): a nodal vector field to gather into U beside the coordinates.  No
// barrier at the end.
template <class Cfg, class Smem>
__device__ __forceinline__ void pair_nodes(Smem& sm, const ElemParams& P, int64_t e0, int64_t n_end,
                                           const double* field = nullptr, double (*U)[Cfg::NN][3] = nullptr) {
  constexpr int NN = Cfg::NN, D = Cfg::D;
  for (int p = threadIdx.x; p < Cfg::kOff; p += Cfg::THREADS) {
    int u = 0, r = p;
    while (r >= NN - 1 - u) r -= NN - 1 - u++;
    sm.pair[p][0] = (uint8_t)u;
    sm.pair[p][1] = (uint8_t)(u + 1 + r);
  }
  for (int t = threadIdx.x; t < Cfg::EPC * NN; t += Cfg::THREADS) {
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
    if (field)
#pragma unroll
      for (int i = 0; i < 3; ++i) U[le][u][i] = field[3 * node + i];
  }
}

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

// places of node v's columns in row u of element le, and of u's in row v
template <class Cfg, class Smem>
__device__ __forceinline__ void pair_ranks(const Smem& sm, const ElemParams& P, int le, int u, int v, int64_t* kuv,
                                           int64_t* kvu) {
  const int32_t* mp = P.node_map + sm.moff[le];
  const int au = Cfg::node_of(u), av = Cfg::node_of(v);
  *kuv = mp[au * Cfg::NN + av];
  *kvu = u == v ? *kuv : (int64_t)mp[av * Cfg::NN + au];
}

// the entry block K of nodes u and v into row u, and transposed into row v
// unless u is v (DIAG)
template <int SC, bool DIAG, class Node>
__device__ __forceinline__ void pair_block(const ElemParams& P, const Node& nu, const Node& nv, int64_t kuv,
                                           int64_t kvu, const double (&K)[3][3]) {
  pair_add<SC>(P.A + nu.row + 3 * kuv, nu.len, K);
  if constexpr (!DIAG) {
    double T[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < 3; ++k) T[k][c] = K[c][k];
    pair_add<SC>(P.A + nv.row + 3 * kvu, nv.len, T);
  }
}

// J' and Ju' of every point of the tile to point(le, q, et, J, Ju, s), which
// the valid points' threads call.  sm.X and sm.U hold the nodes' coordinates
// and displacements (hex8: node_of(corner) gives the slot of a corner in
// binary order) and are used up.  Every thread of the CTA calls it.
template <int TYPE, int NQ, int EPC, int THREADS, class Smem, class NodeOf, class Point>
__device__ __forceinline__ void field_points(Smem& sm, const RefRule& rr, int64_t e0, int64_t n_end, NodeOf node_of,
                                          Point point) {
  const int t = threadIdx.x;
  if constexpr (TYPE == FEA_HEX8) {
    if (t < EPC * 8) {
      const int le = t >> 3, p = t & 7;
      const bool valid = e0 + le < n_end;
      const int a = node_of(p);
      double v[3], vu[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        v[i] = valid ? sm.X[le][a][i] : 0.0;
        vu[i] = valid ? sm.U[le][a][i] : 0.0;
      }
      hex8_modal(v);
      hex8_modal(vu);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        sm.X[le][p][i] = v[i];
        sm.U[le][p][i] = vu[i];
      }
      __syncwarp();
      // every lane forms its Jacobians (the lanes of an element exchange
      // columns); the valid ones use them
      double J[3][3], Ju[3][3];
      hex8_jacobian_pairs(sm.X[le], p, J);
      hex8_jacobian_pairs(sm.U[le], p, Ju);
      if (valid) point(le, p, e0 + le, J, Ju, 8.0);
    }
  } else {
    using Map = RefMap<TYPE>;
    for (int k = t; k < EPC * 6; k += THREADS) {
      const int le = k / 6, i = k % 6;
      if (e0 + le < n_end) Map::prep(i < 3 ? sm.X[le] : sm.U[le], i % 3);
    }
    __syncthreads();
    for (int k = t; k < EPC * NQ; k += THREADS) {
      const int le = k / NQ, q = k % NQ;
      if (e0 + le >= n_end) continue;
      double J[3][3], Ju[3][3];
      Map::jac(sm.X[le], rr.m[q], J);
      Map::jac(sm.U[le], rr.m[q], Ju);
      point(le, q, e0 + le, J, Ju, Map::s);
    }
  }
}

// off(le, u, v) and diag(le, u) of every pair of the tile's elements
template <class Cfg, class Smem, class Off, class Diag>
__device__ __forceinline__ void pair_rounds(const Smem& sm, int64_t e0, int64_t n_end, Off off, Diag diag) {
  constexpr int NN = Cfg::NN, EPC = Cfg::EPC, kOff = Cfg::kOff;
  constexpr int kOffRounds = (EPC * kOff + 31) / 32, kRounds = kOffRounds + (EPC * NN + 31) / 32;
  const int lane = threadIdx.x & 31;
  int r = threadIdx.x >> 5;
  for (; r < kOffRounds; r += Cfg::WARPS) {
    const int t = 32 * r + lane, le = t / kOff, p = t % kOff;
    if (le < EPC && e0 + le < n_end) off(le, (int)sm.pair[p][0], (int)sm.pair[p][1]);
  }
  for (; r < kRounds; r += Cfg::WARPS) {
    const int t = 32 * (r - kOffRounds) + lane, le = t / NN;
    if (le < EPC && e0 + le < n_end) diag(le, t % NN);
  }
}

}  // namespace fea
