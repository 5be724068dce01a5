// j2.cu -- tangent matrix and internal force of small-strain J2 plasticity
// with isotropic Voce hardening: the element loop of a nonlinear solid, whose
// Gauss-point constitutive update is the costly, data-dependent part (the
// paper's solid mechanics case, Sec. 2.2 and 5.2).
//
// Per Gauss point, in FP64: the strain eps = sym(grad u) of the nodal
// displacements, the radial return from the committed state (eps_p_n,
// alpha_n) with a scalar Newton iteration on the consistency condition
//   g(dg) = |s_tr| - 2 mu dg - sqrt(2/3) sigma_y(alpha_n + sqrt(2/3) dg) = 0,
//   sigma_y(a) = sigma0 + H a + (sigma_inf - sigma0)(1 - exp(-delta a)),
// and the consistent tangent
//   D_ep = kappa 1(x)1 + 2 mu theta I_dev - 2 mu theta_bar n(x)n
//        = lam' 1(x)1 + 2 mu' I_sym - beta n(x)n,
//   lam' = kappa - 2 mu theta / 3,  mu' = mu theta,  beta = 2 mu theta_bar,
//   theta = 1 - 2 mu dg / |s_tr|,  theta_bar = 1/(1 + sigma_y'/(3 mu)) - (1 - theta).
// The element blocks are then
//   A^e_ab = sum_q W_q [lam' g_a g_b^T + mu' g_b g_a^T + mu' (g_a . g_b) I - beta h_a h_b^T],
//   f^e_a  = sum_q W_q sigma g_a,       h_a = n g_a,  W_q = w_q det J_q,
// in the tile precision (FP32 for FEA_FP32_INTEGRATE: the return map and D_ep
// stay FP64, the D_ep B products are FP32; FP64 otherwise), accumulated into
// A and b in FP64 by atomics (ATOMIC) or plain read-modify-writes (COLOR).
//
// The Gauss-point update is bound by the number of its FP64 instructions (a
// warp instruction holds the SM's FP64 unit for 16 cycles; ncu of the element
// loop: unit 87 % busy, issue slots 12 %), so:
//  * the displacement gradient of every type is Ju C^T / det from the
//    displacement field's reference Jacobian Ju (RefMap, or the modal
//    transform), only its symmetric part is formed, and the committed plastic
//    strain is subtracted in the same FMAs;
//  * a point clearly inside the yield surface is told by the squared norm: no
//    square root (a point near the surface takes the root and the same test
//    as a yielding one, so ties fall as before);
//  * reciprocals of det J, of the Newton slope and of the norm are rcp64, and
//    constant divisors are the host's factors;
//  * the element loop forms no tile factors (they go nowhere there).
// 499,200 hex8, element loop, one GB300: 2.18 -> 1.58 ms; 373,248 hex8, FP32
// assembly: 2.24 -> 1.75 ms with the scatter of coop_scatter.cuh.
#include <cmath>
#include <cstring>
#include <type_traits>

#include "coop_scatter.cuh"
#include "element.cuh"
#include "fea_internal.cuh"
#include "pairs.cuh"
#include "sched.cuh"

namespace fea {

struct J2Params : ElemParams {
  const double* u;
  const double* state_in;
  double* state_out;
  uint8_t* yield_out;
  uint8_t* iters_out;
  double* stress_out;     // element loop: [E][8][6] Cauchy stress per point slot (may be nullptr)
  double lam, mu, kappa;
  double s0, sinf, delta, hard, tol_g, tol_step;
  double mu2, mu2_3;      // 2 mu, 2 mu / 3
  double gp0, gp1;        // dg/d(dgamma) = gp0 + gp1 exp(-delta a)
  double inv3mu;          // 1 / (3 mu)
  int max_iter;
};

// FP32 tiles: lane a of an element's NN lanes holds its row block.
template <int TYPE, int SLOT>
struct J2Cfg {
  static constexpr int kType = TYPE;
  static constexpr int NN = nodes_of(TYPE);
  static constexpr int NQ = rule_nq(SLOT);
  static constexpr int LPE = NN;
  static constexpr int EPW = 32 / LPE;
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int EPC = EPW * WARPS;
  static constexpr bool kHex = TYPE == FEA_HEX8;
  static_assert(!kHex || (EPC * 8 % 32 == 0 && EPC * 8 <= THREADS), "modal hex geometry needs whole warps");
  // what the Gauss-point update of the element loop needs
  struct Fields {
    double X[EPC][NN][3];
    double U[EPC][NN][3];
  };
  struct Smem : Fields {
    float G[EPC][NQ][grad_stride(NN)];  // grad N_a [point][node][component]
    float H[EPC][NQ][grad_stride(NN)];  // h_a = n grad N_a
    float C[EPC][NQ][4];      // W, W lam', W mu', W beta
    float S[EPC][NQ][6];      // W sigma (xx, yy, zz, xy, yz, xz)
  };
  // with the cooperative scatter's rows, where its staging fits the place of the
  // coordinates and displacements (every type but pyramids)
  using CS = CoopScatter<NN, FEA_SCATTER_ATOMIC>;
  static constexpr bool kCoop = WARPS * CS::kVals * sizeof(float) <= sizeof(Fields);
  struct CoopSmem : Smem {
    typename CS::Rows rows[WARPS];
  };
};

// Radial return at one point (all FP64): trial strain e = eps - eps_p_n.
struct J2Point {
  double sig[6], n[6], ep[6];
  double theta, theta_bar, alpha;
  int iters, yielded, ok;
};

__device__ __forceinline__ void j2_return(const J2Params& P, const double e[6], const double epn[6], double an,
                                          J2Point& r) {
  const double r23 = 0.81649658092772603273;  // sqrt(2/3)
  const double tr = e[0] + e[1] + e[2];
  const double m = -P.mu2_3 * tr;  // the volumetric part of 2 mu e
  double s[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) s[i] = i < 3 ? fma(P.mu2, e[i], m) : P.mu2 * e[i];
  const double n2 = fma(2.0, fma(s[5], s[5], fma(s[4], s[4], s[3] * s[3])), fma(s[2], s[2], fma(s[1], s[1], s[0] * s[0])));
  const double dsy = P.sinf - P.s0;
  // sigma_y(alpha_n); at alpha_n = 0 (a point that never yielded) it is s0
  // exactly, and the exp is not taken
  double sy_n = P.s0;
  if (an != 0.0) sy_n = P.s0 + P.hard * an + dsy * (1.0 - exp(-P.delta * an));
  r.theta = 1.0;
  r.theta_bar = 0.0;
  r.iters = 0;
  r.ok = 1;
  r.yielded = 0;
  r.alpha = an;
#pragma unroll
  for (int i = 0; i < 6; ++i) r.n[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) r.ep[i] = epn[i];
  const double thr = r23 * sy_n;
  double norm = 0.0;
  // clearly elastic (thr > 0 and the norm below it by more than rounding): no root
  bool plastic = !(thr > 0.0 && n2 < 0.999999 * (thr * thr));
  if (plastic) {
    norm = sqrt(n2);
    plastic = !(norm - thr <= 0.0);
  }
  if (plastic) {
    double dg = 0.0, ex = 1.0;
    int it = 0, ok = 0;
    bool ex_final = false;  // ex belongs to the final dg (no step after it)
    for (;;) {
      const double a = fma(r23, dg, an);
      ex = exp(-P.delta * a);
      const double g = norm - P.mu2 * dg - r23 * (P.s0 + P.hard * a + dsy * (1.0 - ex));
      if (fabs(g) <= P.tol_g * sy_n) {
        ok = 1;
        ex_final = true;
        break;
      }
      if (it == P.max_iter) {
        ex_final = true;
        break;
      }
      const double step = -g * rcp64(fma(P.gp1, ex, P.gp0));
      dg += step;
      ++it;
      if (fabs(step) <= P.tol_step) {
        ok = 1;
        break;
      }
    }
    r.iters = it;
    r.ok = ok;
    const double a = fma(r23, dg, an);
    // exp(-delta a) at the final dg: the loop's last value when it stopped at
    // the residual test or the iteration limit (the same a), else a new one
    const double slope = P.hard + dsy * P.delta * (ex_final ? ex : exp(-P.delta * a));
    const double inv = rcp64(norm);
#pragma unroll
    for (int i = 0; i < 6; ++i) r.n[i] = s[i] * inv;
    r.theta = fma(-P.mu2 * dg, inv, 1.0);
    r.theta_bar = rcp64(fma(slope, P.inv3mu, 1.0)) - (1.0 - r.theta);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      s[i] *= r.theta;
      r.ep[i] = fma(dg, r.n[i], epn[i]);
    }
    r.alpha = a;
    r.yielded = 1;
  }
  const double p = P.kappa * tr;
#pragma unroll
  for (int i = 0; i < 6; ++i) r.sig[i] = i < 3 ? s[i] + p : s[i];
}

// The Gauss-point update of point q of the element with original id `id`:
// strain from the displacement field's reference Jacobian Ju' = s Ju and the
// cofactors C' and determinant of J' = s J, return map from the committed
// state, and its results to the state, flag and stress arrays.
__device__ __forceinline__ void j2_update(const J2Params& P, int64_t id, int q, const double (&C)[3][3], double rdet,
                                          const double (&Ju)[3][3], J2Point& r) {
  double epn[6] = {0, 0, 0, 0, 0, 0}, an = 0.0;
  const int64_t slot = id * 8 + q;
  if (P.state_in) {
    const double* sp = P.state_in + slot * 7;
#pragma unroll
    for (int i = 0; i < 6; ++i) epn[i] = sp[i];
    an = sp[6];
  }
  // e = sym(Ju' C'^T) / det' - eps_p_n: the displacement gradient is Ju J^-1
  double e[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int i = k < 3 ? k : k == 4 ? 1 : 0, j = k < 3 ? k : k == 3 ? 1 : 2;
    double h = fma(Ju[i][2], C[j][2], fma(Ju[i][1], C[j][1], Ju[i][0] * C[j][0]));
    if (k >= 3) h = fma(Ju[j][2], C[i][2], fma(Ju[j][1], C[i][1], fma(Ju[j][0], C[i][0], h)));
    e[k] = fma(h, k < 3 ? rdet : 0.5 * rdet, -epn[k]);
  }
  j2_return(P, e, epn, an, r);
  if (!r.ok) latch_error(P.st, FEA_ERR_NO_CONVERGENCE, (unsigned long long)id);
  if (P.state_out) {
    double* sp = P.state_out + slot * 7;
#pragma unroll
    for (int i = 0; i < 6; ++i) sp[i] = r.ep[i];
    sp[6] = r.alpha;
  }
  if (P.yield_out) P.yield_out[slot] = (uint8_t)r.yielded;
  if (P.iters_out) P.iters_out[slot] = (uint8_t)r.iters;
  if (P.stress_out) {
#pragma unroll
    for (int i = 0; i < 6; ++i) P.stress_out[slot * 6 + i] = r.sig[i];
  }
}

// Cofactors and determinant of J' at point q; det' <= 0 latches the element.
__device__ __forceinline__ bool j2_jacobian(const J2Params& P, int64_t id, const double (&J)[3][3], double (&C)[3][3],
                                            double* det) {
  cofactors(J, C);
  *det = J[0][0] * C[0][0] + J[0][1] * C[0][1] + J[0][2] * C[0][2];
  if (*det > 0.0) return true;
  latch_error(P.st, FEA_ERR_INVERTED_ELEMENT, (unsigned long long)id);
  return false;
}

// Phase 1 of point q of element le of an FP32 tile: the update, then
// (SCATTER) the point's factors in FP32 into shared memory.  Hex gradients are
// formed in FP32 from C' and det' rounded once each, as the elasticity tile
// forms them; the other types' in FP64 and rounded.
template <class Cfg, bool SCATTER, class Smem>
__device__ __forceinline__ void j2_point(Smem& sm, const RefRule& rr, const J2Params& P, int le, int q, int64_t et,
                                         const double (&J)[3][3], const double (&Ju)[3][3], double s) {
  constexpr int NN = Cfg::NN;
  const int64_t id = original_id(P, et);
  double C[3][3], det;
  const bool ok = j2_jacobian(P, id, J, C, &det);
  if (!ok) {
    if constexpr (SCATTER) {
#pragma unroll
      for (int k = 0; k < 4; ++k) sm.C[le][q][k] = 0.0f;
#pragma unroll
      for (int k = 0; k < 6; ++k) sm.S[le][q][k] = 0.0f;
#pragma unroll
      for (int a = 0; a < NN; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) sm.G[le][q][3 * a + i] = sm.H[le][q][3 * a + i] = 0.0f;
    }
    return;
  }
  J2Point r;
  const double rdet = rcp64(det);
  j2_update(P, id, q, C, rdet, Ju, r);
  if constexpr (SCATTER) {
    const double W = rr.w[q] * det * (1.0 / (s * s * s));
    sm.C[le][q][0] = f64_to_f32_rn(W);
    sm.C[le][q][1] = f64_to_f32_rn(W * (P.kappa - (r.yielded ? P.mu2_3 * r.theta : P.mu2_3)));
    sm.C[le][q][2] = f64_to_f32_rn(W * P.mu * r.theta);
    sm.C[le][q][3] = r.yielded ? f64_to_f32_rn(W * P.mu2 * r.theta_bar) : 0.0f;
#pragma unroll
    for (int k = 0; k < 6; ++k) sm.S[le][q][k] = f64_to_f32_rn(W * r.sig[k]);
    float gt[NN][3];
    if constexpr (Cfg::kHex) {
      float Cf[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) Cf[i][j] = f64_to_f32_rn(C[i][j]);
      const float invf = (float)s / f64_to_f32_rn(det);
#pragma unroll
      for (int a = 0; a < NN; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i)
          gt[a][i] = (rr.dNf[q][a][0] * Cf[i][0] + rr.dNf[q][a][1] * Cf[i][1] + rr.dNf[q][a][2] * Cf[i][2]) * invf;
    } else {
      const double inv = s * rdet;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double c0 = C[i][0] * inv, c1 = C[i][1] * inv, c2 = C[i][2] * inv;
#pragma unroll
        for (int a = 0; a < NN; ++a)
          gt[a][i] = f64_to_f32_rn(fma(rr.dN[q][a][2], c2, fma(rr.dN[q][a][1], c1, rr.dN[q][a][0] * c0)));
      }
    }
    // h_a = n g_a (n = 0 at elastic points)
    float n[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) n[k] = r.yielded ? f64_to_f32_rn(r.n[k]) : 0.0f;
#pragma unroll
    for (int a = 0; a < NN; ++a) {
      const float g0 = gt[a][0], g1 = gt[a][1], g2 = gt[a][2];
      float *g = sm.G[le][q] + 3 * a, *h = sm.H[le][q] + 3 * a;
      g[0] = g0;
      g[1] = g1;
      g[2] = g2;
      h[0] = n[0] * g0 + n[3] * g1 + n[5] * g2;
      h[1] = n[3] * g0 + n[1] * g1 + n[4] * g2;
      h[2] = n[5] * g0 + n[4] * g1 + n[2] * g2;
    }
  }
}

// One FP32 tile of EPC elements from launch index e0 (elements at or past
// n_end are skipped).  Every thread of the CTA calls it; it ends with a
// barrier.  SCATTER = false is the element-wise loop: the Gauss-point update
// only.
template <int TYPE, int SLOT, int SC, bool SCATTER, class Smem>
__device__ __forceinline__ void j2_tile_body(Smem& sm, const RefRule& rr, const J2Params& P, int64_t e0,
                                             int64_t n_end) {
  using Cfg = J2Cfg<TYPE, SLOT>;
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
        j2_point<Cfg, SCATTER>(sm, rr, P, le, q, et, J, Ju, s);
      });
  __syncthreads();
  if constexpr (!SCATTER) return;
  if constexpr (SC == FEA_SCATTER_ATOMIC) wait_for_previous();

  // phase 2: lane a accumulates its row block
  if constexpr (SCATTER) {
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
          const float wl = sm.C[le][q][1], wm = sm.C[le][q][2], wb = sm.C[le][q][3];
          const float *pg = sm.G[le][q], *ph = sm.H[le][q];
          const float ga[3] = {pg[3 * a], pg[3 * a + 1], pg[3 * a + 2]};
          const float gl[3] = {wl * ga[0], wl * ga[1], wl * ga[2]};
          const float gm[3] = {wm * ga[0], wm * ga[1], wm * ga[2]};
          const float hb[3] = {wb * ph[3 * a], wb * ph[3 * a + 1], wb * ph[3 * a + 2]};
#pragma unroll
          for (int bb = 0; bb < NB; ++bb) {
            const float gb[3] = {pg[3 * (b0 + bb)], pg[3 * (b0 + bb) + 1], pg[3 * (b0 + bb) + 2]};
            const float hh[3] = {ph[3 * (b0 + bb)], ph[3 * (b0 + bb) + 1], ph[3 * (b0 + bb) + 2]};
            const float dot = gm[0] * gb[0] + gm[1] * gb[1] + gm[2] * gb[2];
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
              for (int cc = 0; cc < 3; ++cc) K[bb][c][cc] += gl[c] * gb[cc] + gm[cc] * gb[c] - hb[c] * hh[cc];
#pragma unroll
            for (int c = 0; c < 3; ++c) K[bb][c][c] += dot;
          }
          if (b0 == 0) {
            const float* S = sm.S[le][q];
            rhs[0] += S[0] * ga[0] + S[3] * ga[1] + S[5] * ga[2];
            rhs[1] += S[3] * ga[0] + S[1] * ga[1] + S[4] * ga[2];
            rhs[2] += S[5] * ga[0] + S[4] * ga[1] + S[2] * ga[2];
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
}

// ---------------------------------------------------------------------------
// FP64 tiles, by node pairs (pairs.cuh).  With g^_a = sqrt(W) g_a, h^_a = n g^_a
// and eta = 1 - theta (0 at an elastic point), mu' = mu (1 - eta) and
// lam' = lam + 2 mu eta / 3, so
//   A^e_ab = lam M + mu M^T + mu tr(M) I + 2/3 mu N - mu N^T - mu tr(N) I - B,
//   M = sum_q g^_a (x) g^_b,  N = sum_q eta g^_a (x) g^_b,  B = sum_q beta h^_a (x) h^_b:
// an elastic point takes the 9 products of M, a plastic one 24 more, where a
// row block took 36 per ordered pair and point.
// ---------------------------------------------------------------------------
template <int TYPE, int SLOT>
struct J2PairCfg : PairShape<TYPE, SLOT, 3, pair_epc(rule_nq(SLOT))> {
  using Base = PairShape<TYPE, SLOT, 3, pair_epc(rule_nq(SLOT))>;
  struct Smem : Base::Nodes {
    double U[Base::EPC][Base::NN][3];
    double G[Base::EPC][Base::NQ][Base::GS];  // g^
    double H[Base::EPC][Base::NQ][Base::GS];  // h^ (plastic points)
    double C[Base::EPC][Base::NQ][2];         // eta, beta (0, 0 at an elastic point)
    double S[Base::EPC][Base::NQ][6];         // sqrt(W) sigma
  };
};

template <class Cfg>
__device__ __forceinline__ void j2_pair_point(typename Cfg::Smem& sm, const RefRule& rr, const J2Params& P, int le,
                                              int q, int64_t et, const double (&J)[3][3], const double (&Ju)[3][3],
                                              double s) {
  constexpr int NN = Cfg::NN;
  const int64_t id = original_id(P, et);
  double C[3][3], det;
  double *g = sm.G[le][q], *h = sm.H[le][q];
  if (!j2_jacobian(P, id, J, C, &det)) {
#pragma unroll
    for (int k = 0; k < 3 * NN; ++k) g[k] = h[k] = 0.0;
    sm.C[le][q][0] = sm.C[le][q][1] = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) sm.S[le][q][k] = 0.0;
    return;
  }
  J2Point r;
  const double rdet = rcp64(det);
  j2_update(P, id, q, C, rdet, Ju, r);
  const double root = sqrt(rr.w[q] * det * (1.0 / (s * s * s))), inv = root * (s * rdet);
  sm.C[le][q][0] = 1.0 - r.theta;
  sm.C[le][q][1] = P.mu2 * r.theta_bar;
#pragma unroll
  for (int k = 0; k < 6; ++k) sm.S[le][q][k] = root * r.sig[k];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i][j] *= inv;
#pragma unroll
  for (int u = 0; u < NN; ++u) {
    const double* d = rr.dN[q][Cfg::node_of(u)];
    double v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) g[3 * u + i] = v[i] = fma(d[2], C[i][2], fma(d[1], C[i][1], d[0] * C[i][0]));
    if (r.yielded) {
      h[3 * u] = fma(r.n[5], v[2], fma(r.n[3], v[1], r.n[0] * v[0]));
      h[3 * u + 1] = fma(r.n[4], v[2], fma(r.n[1], v[1], r.n[3] * v[0]));
      h[3 * u + 2] = fma(r.n[2], v[2], fma(r.n[4], v[1], r.n[5] * v[0]));
    }
  }
}

template <class Cfg, int SC, bool DIAG>
__device__ __forceinline__ void j2_pair_task(const typename Cfg::Smem& sm, const J2Params& P, int le, int u, int v) {
  const typename Cfg::Node nu = sm.nd[le][u], nv = sm.nd[le][v];
  int64_t kuv, kvu;
  pair_ranks<Cfg>(sm, P, le, u, v, &kuv, &kvu);
  double M[3][3], N[3][3], B[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < 3; ++k) M[c][k] = N[c][k] = B[c][k] = 0.0;
  double f[1][3] = {{0.0, 0.0, 0.0}};
#pragma unroll 1
  for (int q = 0; q < Cfg::NQ; ++q) {
    const double *a = sm.G[le][q] + 3 * u, *b = sm.G[le][q] + 3 * v;
    const double eta = sm.C[le][q][0], beta = sm.C[le][q][1];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = DIAG ? c : 0; k < 3; ++k) M[c][k] = fma(a[c], b[k], M[c][k]);
    if (eta != 0.0 || beta != 0.0) {
      const double *ha = sm.H[le][q] + 3 * u, *hb = sm.H[le][q] + 3 * v;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double x = eta * a[c], y = beta * ha[c];
#pragma unroll
        for (int k = DIAG ? c : 0; k < 3; ++k) {
          N[c][k] = fma(x, b[k], N[c][k]);
          B[c][k] = fma(y, hb[k], B[c][k]);
        }
      }
    }
    if constexpr (DIAG) {
      const double* S = sm.S[le][q];
      f[0][0] = fma(S[5], a[2], fma(S[3], a[1], fma(S[0], a[0], f[0][0])));
      f[0][1] = fma(S[4], a[2], fma(S[1], a[1], fma(S[3], a[0], f[0][1])));
      f[0][2] = fma(S[2], a[2], fma(S[4], a[1], fma(S[5], a[0], f[0][2])));
    }
  }
  const double tr = P.mu * ((M[0][0] + M[1][1] + M[2][2]) - (N[0][0] + N[1][1] + N[2][2]));
  double K[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const bool low = DIAG && k < c;  // M, N and B are symmetric on the diagonal
      const double mt = DIAG ? (low ? M[k][c] : M[c][k]) : M[k][c], nt = DIAG ? (low ? N[k][c] : N[c][k]) : N[k][c];
      K[c][k] = low ? K[k][c]
                    : fma(P.lam, M[c][k], fma(P.mu, mt - nt, fma(P.mu2_3, N[c][k], c == k ? tr - B[c][k] : -B[c][k])));
    }
  pair_block<SC, DIAG>(P, nu, nv, kuv, kvu, K);
  if constexpr (DIAG) pair_add<SC>(P.b + 3 * (int64_t)nu.id, 0, f);
}

template <int TYPE, int SLOT, int SC>
__device__ __forceinline__ void j2_pair_body(typename J2PairCfg<TYPE, SLOT>::Smem& sm, const RefRule& rr,
                                             const J2Params& P, int64_t e0, int64_t n_end) {
  using Cfg = J2PairCfg<TYPE, SLOT>;
  pair_nodes<Cfg>(sm, P, e0, n_end, P.u, sm.U);
  __syncthreads();
  field_points<TYPE, Cfg::NQ, Cfg::EPC, Cfg::THREADS>(
      sm, rr, e0, n_end, [](int p) { return p; },
      [&](int le, int q, int64_t et, const double(&J)[3][3], const double(&Ju)[3][3], double s) {
        j2_pair_point<Cfg>(sm, rr, P, le, q, et, J, Ju, s);
      });
  __syncthreads();
  if constexpr (SC == FEA_SCATTER_ATOMIC) wait_for_previous();
  pair_rounds<Cfg>(
      sm, e0, n_end, [&](int le, int u, int v) { j2_pair_task<Cfg, SC, false>(sm, P, le, u, v); },
      [&](int le, int u) { j2_pair_task<Cfg, SC, true>(sm, P, le, u, u); });
  __syncthreads();
}

// The tile of an element type in a precision; POINTS: the element loop's.
template <int TYPE, int SLOT, int PREC, bool POINTS = false>
struct J2Tile {
  using Cfg = J2Cfg<TYPE, SLOT>;
  template <int SC>
  using Smem = std::conditional_t<POINTS, typename Cfg::Fields,
                                  std::conditional_t<SC == FEA_SCATTER_ATOMIC && Cfg::kCoop, typename Cfg::CoopSmem,
                                                     typename Cfg::Smem>>;
  template <int SC>
  __device__ static __forceinline__ void run(unsigned char* raw, const RefRule& rr, const J2Params& P, int64_t e0,
                                             int64_t n_end) {
    j2_tile_body<TYPE, SLOT, SC, !POINTS>(*reinterpret_cast<Smem<SC>*>(raw), rr, P, e0, n_end);
  }
};
template <int TYPE, int SLOT>
struct J2Tile<TYPE, SLOT, FEA_FP64, false> {
  using Cfg = J2PairCfg<TYPE, SLOT>;
  template <int SC>
  using Smem = typename Cfg::Smem;
  template <int SC>
  __device__ static __forceinline__ void run(unsigned char* raw, const RefRule& rr, const J2Params& P, int64_t e0,
                                             int64_t n_end) {
    j2_pair_body<TYPE, SLOT, SC>(*reinterpret_cast<Smem<SC>*>(raw), rr, P, e0, n_end);
  }
};

// one tile per CTA
template <int TYPE, int SLOT, int PREC, int SC, bool POINTS>
__global__ void __launch_bounds__(128, POINTS || PREC == FEA_FP64 || SC != FEA_SCATTER_ATOMIC ? 0 : 5)
    k_j2_tile(const __grid_constant__ RefRule rr, const __grid_constant__ J2Params P) {
  using T = J2Tile<TYPE, SLOT, PREC, POINTS>;
  extern __shared__ __align__(16) unsigned char j2_smem_raw[];
  if constexpr (!POINTS) let_next_start();
  T::template run<SC>(j2_smem_raw, rr, P, (int64_t)blockIdx.x * T::Cfg::EPC, P.n);
}

template <int TYPE, int SLOT, int PREC, int SC, bool POINTS = false>
static int launch_j2(const J2Params& P, cudaStream_t s) {
  using T = J2Tile<TYPE, SLOT, PREC, POINTS>;
  constexpr size_t smem = sizeof(typename T::template Smem<SC>);
  static_assert(smem <= 227 * 1024, "J2 tile exceeds shared memory");
  auto kern = k_j2_tile<TYPE, SLOT, PREC, SC, POINTS>;
  if (smem > 48 * 1024) FEA_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const unsigned grid = grid_for(P.n, T::Cfg::EPC);
  const bool early = P.early && starts_early(grid, P.early == 1, false);
  FEA_CUDA(launch_tiles(kern, grid, T::Cfg::THREADS, smem, s, early, host_rule(SLOT), P));
  return FEA_OK;
}

template <int PREC, int SC, bool POINTS = false>
static int launch_j2_type(int type, const J2Params& P, cudaStream_t s) {
  switch (type) {
    case FEA_TET4: return launch_j2<FEA_TET4, kRuleTet4, PREC, SC, POINTS>(P, s);
    case FEA_PYR5: return launch_j2<FEA_PYR5, kRulePyr8, PREC, SC, POINTS>(P, s);
    case FEA_PRISM6: return launch_j2<FEA_PRISM6, kRulePrism6, PREC, SC, POINTS>(P, s);
    default: return launch_j2<FEA_HEX8, kRuleHex8, PREC, SC, POINTS>(P, s);
  }
}

static int launch_j2_any(int type, int precision, bool color, const J2Params& P, cudaStream_t s) {
  if (precision == FEA_FP64)
    return color ? launch_j2_type<FEA_FP64, FEA_SCATTER_COLOR>(type, P, s)
                 : launch_j2_type<FEA_FP64, FEA_SCATTER_ATOMIC>(type, P, s);
  return color ? launch_j2_type<FEA_FP32_INTEGRATE, FEA_SCATTER_COLOR>(type, P, s)
               : launch_j2_type<FEA_FP32_INTEGRATE, FEA_SCATTER_ATOMIC>(type, P, s);
}

// ---------------------------------------------------------------------------
// persistent schedule (sched.cuh): every element type in one launch
// ---------------------------------------------------------------------------
__constant__ RefRule c_rules_j2[kNumRules];

struct PersistJ2Args {
  J2Params table[kNumTypes];
  int32_t slot[kNumTypes];
  SchedArgs S;
};

template <int PREC, bool POINTS>
struct PersistJ2Cfg {
  template <int TYPE, int SLOT>
  static constexpr size_t bytes() { return sizeof(typename J2Tile<TYPE, SLOT, PREC, POINTS>::template Smem<FEA_SCATTER_ATOMIC>); }
  static constexpr size_t mx(size_t a, size_t b) { return a > b ? a : b; }
  static constexpr size_t smem = mx(mx(bytes<FEA_TET4, kRuleTet4>(), bytes<FEA_PYR5, kRulePyr8>()),
                                    mx(bytes<FEA_PRISM6, kRulePrism6>(), bytes<FEA_HEX8, kRuleHex8>()));
};

template <int TYPE, int SLOT, int PREC, bool POINTS>
__device__ __forceinline__ void persist_j2_item(unsigned char* raw, const J2Params& P, int64_t first, int64_t end) {
  using T = J2Tile<TYPE, SLOT, PREC, POINTS>;
  for (int64_t e0 = first; e0 < end; e0 += T::Cfg::EPC)
    T::template run<FEA_SCATTER_ATOMIC>(raw, c_rules_j2[SLOT + opaque_zero()], P, e0, end);
}

// One item of the any-type kernel, not inlined: four inlined tile bodies take
// 213 registers in FP32 where the largest needs 126.
template <int TYPE, int SLOT, int PREC, bool POINTS>
__device__ __noinline__ void persist_j2_call(unsigned char* raw, const J2Params& P, int64_t first, int64_t end) {
  persist_j2_item<TYPE, SLOT, PREC, POINTS>(raw, P, first, end);
}

// ONLY == kRuleHex8: a mesh of hexes only (one tile body); -1: any type.
// CTAs per SM: what the shared memory (FP64) or the registers without large
// spills allow.  The element loop could run 8, but is no faster (512,000 hex8,
// stealing: 2.39 ms at four, 2.42 at eight), and with that many CTAs on an SM an
// item's time says little about its cost (the network of the cost model
// explained 2 % of it, 55 % at four).
template <int PREC, int ONLY, bool POINTS>
__global__ void __launch_bounds__(128, PREC == FEA_FP64 ? 3 : POINTS || ONLY < 0 ? 4 : 5)
    k_persistent_j2(const __grid_constant__ PersistJ2Args A) {
  extern __shared__ __align__(16) unsigned char persist_j2_smem[];
  __shared__ int s_item;
  sched_start(A.S);
  int k = 0;
  for (;;) {
    const int item = sched_next(A.S, k, &s_item);
    if (item < 0) break;
    const uint64_t t0 = global_ns();
    const WorkItem it = A.S.items[item];
    const int64_t first = it.first, end = (int64_t)it.first + it.count;
    // entry t is type t: the parameters are read at constant offsets
    if constexpr (ONLY == kRuleHex8) {
      persist_j2_item<FEA_HEX8, kRuleHex8, PREC, POINTS>(persist_j2_smem, A.table[FEA_HEX8], first, end);
    } else {
      switch (A.slot[it.entry]) {
        case kRulePyr8: persist_j2_call<FEA_PYR5, kRulePyr8, PREC, POINTS>(persist_j2_smem, A.table[FEA_PYR5], first, end); break;
        case kRulePrism6:
          persist_j2_call<FEA_PRISM6, kRulePrism6, PREC, POINTS>(persist_j2_smem, A.table[FEA_PRISM6], first, end);
          break;
        case kRuleHex8: persist_j2_call<FEA_HEX8, kRuleHex8, PREC, POINTS>(persist_j2_smem, A.table[FEA_HEX8], first, end); break;
        default: persist_j2_call<FEA_TET4, kRuleTet4, PREC, POINTS>(persist_j2_smem, A.table[FEA_TET4], first, end); break;
      }
    }
    sched_record(A.S, item, it.entry, t0);
  }
}

int init_rule_constants_j2() {
  RefRule all[kNumRules];
  for (int r = 0; r < kNumRules; ++r) all[r] = host_rule(r);
  FEA_CUDA(cudaMemcpyToSymbol(c_rules_j2, all, sizeof(all)));
  return FEA_OK;
}

static int j2_validate(const fea_operator* op) {
  if (!op->u_d) return fail(FEA_ERR_ARG, "fea_assemble: J2 needs the displacements u_d");
  if (op->max_iter < 1 || op->max_iter > 255) return fail(FEA_ERR_ARG, "fea_assemble: J2 max_iter must be in [1, 255]");
  if (!(op->poisson > -1.0 && op->poisson < 0.5)) return fail(FEA_ERR_ARG, "fea_assemble: poisson must be in (-1, 0.5)");
  if (op->state_out_d && op->state_out_d == op->state_in_d)
    return fail(FEA_ERR_ARG, "fea_assemble: J2 state_out must not alias state_in");
  return FEA_OK;
}

static J2Params j2_base_params(const fea_operator* op, fea_mesh* m, const int64_t* row_ptr, const int32_t* node_map,
                               double* A, double* b) {
  J2Params P;
  std::memset(&P, 0, sizeof(P));
  P.coords = m->coords;
  P.row_ptr = row_ptr;
  P.node_map = node_map;
  P.A = A;
  P.b = b;
  P.st = m->status;
  P.u = op->u_d;
  P.state_in = op->state_in_d;
  P.state_out = op->state_out_d;
  P.yield_out = op->yield_out_d;
  P.iters_out = op->iters_out_d;
  const double E = op->young, nu = op->poisson;
  P.lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu));
  P.mu = E / (2.0 * (1.0 + nu));
  P.kappa = P.lam + 2.0 * P.mu / 3.0;
  P.mu2 = 2.0 * P.mu;
  P.mu2_3 = 2.0 * P.mu / 3.0;
  P.inv3mu = 1.0 / (3.0 * P.mu);
  P.s0 = op->sigma0;
  P.sinf = op->sigma_inf;
  P.delta = op->delta;
  P.hard = op->hardening;
  P.tol_g = op->tol_g;
  P.tol_step = op->tol_step;
  P.gp0 = -2.0 * P.mu - (2.0 / 3.0) * P.hard;
  P.gp1 = -(2.0 / 3.0) * (P.sinf - P.s0) * P.delta;
  P.max_iter = op->max_iter;
  return P;
}

template <int PREC, int ONLY, bool POINTS = false>
static int launch_persistent_j2_t(const PersistJ2Args& args, int n_ctas, bool dry, cudaStream_t s, int* grid_out) {
  constexpr size_t smem = ONLY == kRuleHex8
                              ? sizeof(typename J2Tile<FEA_HEX8, kRuleHex8, PREC, POINTS>::template Smem<FEA_SCATTER_ATOMIC>)
                              : PersistJ2Cfg<PREC, POINTS>::smem;
  auto kern = k_persistent_j2<PREC, ONLY, POINTS>;
  if (smem > 48 * 1024) FEA_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int grid = n_ctas;
  if (grid <= 0) {
    int dev = 0, sms = 0, per_sm = 0;
    FEA_CUDA(cudaGetDevice(&dev));
    FEA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    FEA_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128, smem));
    grid = sms * (per_sm > 0 ? per_sm : 1);
  }
  if (grid_out) *grid_out = grid;
  if (!dry) {
    kern<<<sched_ctas(args.S, grid), 128, smem, s>>>(args);
    FEA_CUDA(cudaGetLastError());
  }
  return FEA_OK;
}

int launch_persistent_j2(const fea_operator* op, fea_mesh* m, const int64_t* row_ptr, const int32_t* node_map,
                         double* A, double* b, const SchedArgs& S, int n_ctas, bool dry, cudaStream_t s,
                         int* grid_out, double* stress, bool points_only) {
  if (!dry) {
    int rc = j2_validate(op);
    if (rc) return rc;
  }
  PersistJ2Args args;
  std::memset(&args, 0, sizeof(args));
  J2Params base = j2_base_params(op, m, row_ptr, node_map, A, b);
  base.stress_out = stress;
  const int slots[kNumTypes] = {kRuleTet4, kRulePyr8, kRulePrism6, kRuleHex8};
  for (int t = 0; t < kNumTypes; ++t) {
    args.table[t] = base;
    const TypeGroup& g = m->group[t];
    args.table[t].tconn = g.conn;
    args.table[t].ids = g.ids;
    args.table[t].mapoff = g.mapoff;
    args.table[t].n = g.n;
    args.slot[t] = slots[t];
  }
  args.S = S;
  bool hex_only = m->group[FEA_HEX8].n > 0;
  for (int t = 0; t < kNumTypes; ++t)
    if (t != FEA_HEX8 && m->group[t].n) hex_only = false;
  if (points_only)  // the element-wise loop: Gauss-point updates only
    return hex_only ? launch_persistent_j2_t<FEA_FP32_INTEGRATE, kRuleHex8, true>(args, n_ctas, dry, s, grid_out)
                    : launch_persistent_j2_t<FEA_FP32_INTEGRATE, -1, true>(args, n_ctas, dry, s, grid_out);
  if (op->precision == FEA_FP64)
    return hex_only ? launch_persistent_j2_t<FEA_FP64, kRuleHex8>(args, n_ctas, dry, s, grid_out)
                    : launch_persistent_j2_t<FEA_FP64, -1>(args, n_ctas, dry, s, grid_out);
  return hex_only ? launch_persistent_j2_t<FEA_FP32_INTEGRATE, kRuleHex8>(args, n_ctas, dry, s, grid_out)
                  : launch_persistent_j2_t<FEA_FP32_INTEGRATE, -1>(args, n_ctas, dry, s, grid_out);
}

int assemble_j2(const fea_operator* op, fea_mesh* m, const int64_t* row_ptr, const int32_t* node_map, double* A,
                double* b, cudaStream_t s) {
  if (op->scatter != FEA_SCATTER_ATOMIC && op->scatter != FEA_SCATTER_COLOR)
    return fail(FEA_ERR_UNSUPPORTED, "fea_assemble: J2 supports the ATOMIC and COLOR scatters");
  int vrc = j2_validate(op);
  if (vrc) return vrc;
  if (op->scatter == FEA_SCATTER_COLOR && !m->color) {
    int rc = build_color_plan(m, s);
    if (rc) return rc;
  }
  cudaEvent_t* ev = (cudaEvent_t*)op->events;
  const int nev = ev ? op->n_events : 0;
  const int64_t nnz = 9 * m->nnz_node;
  if (nev > 0) FEA_CUDA(cudaEventRecord(ev[0], s));
  int zrc = zero_system(A, nnz, b, m->n_nodes * 3, s);
  if (zrc) return zrc;
  if (nev > 1) FEA_CUDA(cudaEventRecord(ev[1], s));

  J2Params P = j2_base_params(op, m, row_ptr, node_map, A, b);
  P.early = op->scatter == FEA_SCATTER_ATOMIC && small_system(nnz);
  int launched = 0;
  auto run = [&](int t) -> int {
    int rc = launch_j2_any(t, op->precision, op->scatter == FEA_SCATTER_COLOR, P, s);
    if (rc) return rc;
    if (2 + launched < nev) FEA_CUDA(cudaEventRecord(ev[2 + launched], s));
    ++launched;
    if (P.early) P.early = 2;
    return FEA_OK;
  };
  if (op->scatter == FEA_SCATTER_COLOR) {
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

// The element-wise loop (no scatter): the J2 update at every Gauss point,
// per type or by a persistent schedule (sched.cuh), writing the new state,
// the stress, the yield flags and the Newton iteration counts.
int element_loop_j2(const fea_operator* op, fea_mesh* m, double* stress, cudaStream_t s) {
  int rc = j2_validate(op);
  if (rc) return rc;
  if (op->schedule != FEA_SCHED_PER_TYPE) return element_loop_persistent(op, m, stress, s);
  cudaEvent_t* ev = (cudaEvent_t*)op->events;
  const int nev = ev ? op->n_events : 0;
  if (nev > 0) FEA_CUDA(cudaEventRecord(ev[0], s));
  if (nev > 1) FEA_CUDA(cudaEventRecord(ev[1], s));
  J2Params P = j2_base_params(op, m, nullptr, nullptr, nullptr, nullptr);
  P.stress_out = stress;
  int launched = 0;
  for (int t = 0; t < kNumTypes; ++t) {
    const TypeGroup& g = m->group[t];
    if (!g.n) continue;
    P.tconn = g.conn;
    P.ids = g.ids;
    P.mapoff = g.mapoff;
    P.list = nullptr;
    P.n = g.n;
    rc = launch_j2_type<FEA_FP32_INTEGRATE, FEA_SCATTER_ATOMIC, true>(t, P, s);
    if (rc) return rc;
    if (2 + launched < nev) FEA_CUDA(cudaEventRecord(ev[2 + launched], s));
    ++launched;
  }
  return FEA_OK;
}

}  // namespace fea

extern "C" int fea_element_loop(const fea_operator* op, fea_mesh* mesh, double* stress_d, void* stream) {
  using namespace fea;
  if (!op || !mesh) return fail(FEA_ERR_ARG, "fea_element_loop: null argument");
  if (op->kind != FEA_OP_J2) return fail(FEA_ERR_UNSUPPORTED, "fea_element_loop: the loop runs the J2 operator");
  if (op->schedule < FEA_SCHED_PER_TYPE || op->schedule > FEA_SCHED_QUEUES_STEAL)
    return fail(FEA_ERR_ARG, "fea_element_loop: unknown schedule");
  return element_loop_j2(op, mesh, stress_d, (cudaStream_t)stream);
}
