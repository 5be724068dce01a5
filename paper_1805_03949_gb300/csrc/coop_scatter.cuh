// coop_scatter.cuh -- shared-memory layout and warp-cooperative FP64
// reductions of the FP32 element tiles with three dofs per node.
#pragma once

#include "pairs.cuh"

namespace fea {

// Floats of one point's gradients in the FP32 tiles: 3 per node, odd, so that
// neither the points' stores (32 points of 4 hexes in a warp) nor the row
// blocks' loads (the same node's gradient of each of the warp's elements) meet
// in a bank.  With 24 floats per hex point the elements of a warp were 192
// floats apart, the same bank: four wavefronts per load; 373,248
// hex8 J2 1.96 -> 1.89 ms with the odd stride and the scatter below.
__host__ __device__ constexpr int grad_stride(int nn) { return (3 * nn) | 1; }

// Columns a lane accumulates at a time: a row block of 3 x 3 entries per column
// node takes 9 registers per column, and 72 of them held a hex8 tile at 128
// registers and four CTAs per SM, with its FP64 phase and its FP32 phase
// taking turns.  In groups of four (prisms three) the tiles fit six CTAs
// (elasticity: 682 us per step of 258,048 hex8 at 4, 614 at 5, 564 at 6, 590 at
// 7) or five (J2, finite strain: more would not fit the shared memory), at the
// cost of reading the row's own gradient once per group.  Only with
// reductions: a coloring or multidependence launch waits for the
// read-modify-writes of each group (hex8, FP32, grouped: elasticity 1.29
// against 1.20 ms, finite strain 0.93 against 0.62).
__host__ __device__ constexpr int column_group(int nn, int dofs, int sc) {
  return dofs == 1 || sc != FEA_SCATTER_ATOMIC ? nn : nn == 8 ? 4 : nn == 6 ? 3 : nn;
}

// Warp-cooperative reduction of FP32 row blocks.  A lane's row block holds, for
// each row c and column node, three consecutive entries of A (24 bytes).  One
// lane per entry scatters each warp-wide reduction over 32 rows; here the
// lanes hand one row of a column group at a time to the warp through shared
// memory, and three lanes of each group of four reduce one 24-byte run, so
// that a reduction touches eight or a few more sectors (measured on GB300 with
// A in L2: 192 G reductions/s scattered, 443 G/s in runs of three).  A group of
// four serves the rows of the same lanes throughout, and takes a row's start
// and places once per column group; its four rows one after the other (unrolled
// they cost the registers of two CTAs per SM: 1.94 against 1.78 ms in J2).
// With the column groups, one GB300: 258,048 hex8 elasticity 0.695 -> 0.546 ms
// per step, 374,400 tet4 0.264 -> 0.183 ms, 373,248 hex8 J2 1.89 -> 1.78 ms.
template <int NN, int SC>
struct CoopScatter {
  static constexpr bool kOn = SC == FEA_SCATTER_ATOMIC;
  static constexpr int NB = column_group(NN, 3, FEA_SCATTER_ATOMIC);
  static constexpr int kVals = 32 * 3 * NB;  // floats a warp stages (16-byte aligned)
  // what a warp knows of its lanes' rows
  struct Rows {
    double* row[32];     // the node's first row in A
    int32_t len[32];     // length of its rows
    int16_t k3[32][NN];  // 3 times the place of every column node (-1: idle lane; a row has at most 1,024 nodes)
  };

  // Every lane of the warp; g: the element's index in the group, a: the lane's node.
  template <class Params>
  static __device__ __forceinline__ void begin(Rows& R, Params& P, bool active, int64_t g, int a) {
    const int lane = threadIdx.x & 31;
    if (active) {
      const int64_t node = P.tconn[g * NN + a];
      const int64_t id = P.ids ? (int64_t)P.ids[g] : g;
      const int32_t* mp = P.node_map + (P.mapoff ? P.mapoff[g] : id * NN * NN) + a * NN;
      const int64_t r0 = P.row_ptr[3 * node];
      R.row[lane] = P.A + r0;
      R.len[lane] = (int32_t)(P.row_ptr[3 * node + 1] - r0);
#pragma unroll
      for (int b = 0; b < NN; ++b) R.k3[lane][b] = (int16_t)(3 * mp[b]);
    } else {
#pragma unroll
      for (int b = 0; b < NN; ++b) R.k3[lane][b] = -1;
    }
  }

  // Columns b0 .. b0 + NB of every lane's row block, K [column node][row][column
  // component].  Every lane of the warp; vals is the warp's own.
  static __device__ __forceinline__ void add(const Rows& R, float* vals, int b0, const float (&K)[NB][3][3]) {
    const int lane = threadIdx.x & 31, run = lane >> 2, m = lane & 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      __syncwarp();
      if constexpr (NB % 4 == 0) {
        float4* v4 = reinterpret_cast<float4*>(vals + 3 * NB * lane);
#pragma unroll
        for (int i = 0; i < 3 * NB / 4; ++i) {
          float t[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) t[u] = K[(4 * i + u) / 3][c][(4 * i + u) % 3];
          v4[i] = make_float4(t[0], t[1], t[2], t[3]);
        }
      } else {
#pragma unroll
        for (int f = 0; f < 3 * NB; ++f) vals[3 * NB * lane + f] = K[f / 3][c][f % 3];
      }
      __syncwarp();
      if (m < 3) {
#pragma unroll 1
        for (int r = 0; r < 4; ++r) {
          const int s = 8 * r + run;
          const int16_t* k = &R.k3[s][b0];
          if (k[0] >= 0) {
            double* p = R.row[s] + (c * R.len[s] + m);
#pragma unroll
            for (int j = 0; j < NB; ++j) red_add(p + k[j], widen(vals[3 * NB * s + 3 * j + m]));
          }
        }
      }
    }
  }
};

}  // namespace fea
