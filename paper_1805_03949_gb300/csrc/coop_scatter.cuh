// coop_scatter.cuh -- shared-memory layout and warp-cooperative FP64
// reductions of the FP32 element tiles with three dofs per node.
#pragma once

#include "pairs.cuh"

namespace fea {

// Floats of one point's gradients in the FP32 tiles: 3 per node, odd, so that
// neither the points' stores (32 points of 4 hexes in a warp) nor the row
// blocks' loads (the same node's gradient of each of the warp's elements) meet
// in a bank.  With 24 floats per hex point the elements of a warp were 192
// floats apart, the same bank: four wavefronts per load.  @@LAYOUT@@
__host__ __device__ constexpr int grad_stride(int nn) { return (3 * nn) | 1; }

// Warp-cooperative reduction of FP32 row blocks.  A lane's row block holds,
// for each row c and column node b, three consecutive entries of A (24 bytes);
// one lane per entry scatters each warp-wide reduction over 32 rows, while
// three neighbouring lanes on one 24-byte run and ten runs from one or two
// rows make each reduction touch about a third of the sectors (measured on
// GB300 with A in L2: 192 G reductions/s scattered, 443 G/s in runs of three).
// The lanes hand their entries to the warp through `region`, kBytes of
// 16-byte aligned shared memory of the warp's own: row starts (rbs), column
// positions (ks, -1 for an idle lane) and PB columns' entries at a time
// (vals).  The tiles give it the gradients of the warp's own elements, which
// their row blocks no longer need.  128^3 hex8 elasticity 6.20 -> 5.69 ms per
// step; 72^3 J2 @@J2@@.
template <int NN, int SC, size_t kBytes>
struct CoopScatter {
  static constexpr size_t kValsOff = 256 + 4 * 32 * NN;  // after rbs[32] and ks[32][NN]
  static constexpr int pb() {
    for (int p = NN; p > 0; --p)
      if (NN % p == 0 && kValsOff + 4 * 32 * 3 * p <= kBytes) return p;
    return 0;
  }
  static constexpr int PB = pb();
  // hex8 (PB = 4, 16-byte staging stores) is the tile it serves; staged in
  // pairs of columns, the tet4 items of a 256-mesh batch made it slower (17.97
  // against 17.09 ms)
  static constexpr bool kOn = SC == FEA_SCATTER_ATOMIC && NN == 8 && PB > 0 && kBytes % 16 == 0 && (3 * PB) % 4 == 0;

  // K [column node][row][column component]; every lane of the warp calls it,
  // after the warp's last use of the region's earlier content.  g: the
  // element's index in the group, a: the lane's node.
  static __device__ __forceinline__ void run(unsigned char* region, const ElemParams& P, bool active, int64_t g, int a,
                                             const float (&K)[NN][3][3], const float (&rhs)[3]) {
    const int lane = threadIdx.x & 31;
    int64_t rb[3] = {}, node = 0;
    const int32_t* mp = nullptr;
    if (active) {
      node = P.tconn[g * NN + a];
      const int64_t id = P.ids ? (int64_t)P.ids[g] : g;
      mp = P.node_map + (P.mapoff ? P.mapoff[g] : id * NN * NN) + a * NN;
#pragma unroll
      for (int c = 0; c < 3; ++c) rb[c] = P.row_ptr[3 * node + c];
    }
    __syncwarp();
    int64_t* rbs = reinterpret_cast<int64_t*>(region);
    int32_t* ks = reinterpret_cast<int32_t*>(region + 256);
    float* vals = reinterpret_cast<float*>(region + kValsOff);
#pragma unroll
    for (int bb = 0; bb < NN; ++bb) ks[lane * NN + bb] = active ? mp[bb] : -1;
    // run j of a round: lanes 3j .. 3j+2 (lanes 30 and 31 rest)
    const int run = lane / 3, m = lane - 3 * run;
    constexpr int kRuns = 32 * PB, kRounds = (kRuns + 9) / 10;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      __syncwarp();
      rbs[lane] = rb[c];
#pragma unroll
      for (int part = 0; part < NN / PB; ++part) {
        __syncwarp();
        float4* v4 = reinterpret_cast<float4*>(vals + lane * PB * 3);
#pragma unroll
        for (int i = 0; i < 3 * PB / 4; ++i) {
          float t[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int f = 4 * i + u;
            t[u] = K[part * PB + f / 3][c][f % 3];
          }
          v4[i] = make_float4(t[0], t[1], t[2], t[3]);
        }
        __syncwarp();
#pragma unroll 2
        for (int r = 0; r < kRounds; ++r) {
          const int ch = 10 * r + run;  // run ch: lane ch / PB, column part * PB + ch % PB
          if (run < 10 && ch < kRuns) {
            const int s = ch / PB, j = ch - PB * s;
            const int32_t k = ks[s * NN + part * PB + j];
            if (k >= 0) red_add(P.A + rbs[s] + 3 * (int64_t)k + m, widen(vals[3 * ch + m]));
          }
        }
      }
    }
    if (active)
#pragma unroll
      for (int c = 0; c < 3; ++c) red_add(P.b + 3 * node + c, widen(rhs[c]));
  }
};

}  // namespace fea
