// element.cuh -- reference elements, quadrature rules and the per-quadrature
// point geometry shared by every assembly kernel of the engine.
//
// Element formulations (the paper states the PDEs, Sec. 2.1.1 and 2.2.1, but
// no element formulation; these are the textbook Galerkin ones):
//   diffusion  A^e_ab = sum_q w_q detJ_q k(x_q) grad N_a . grad N_b,
//              b^e_a  = sum_q w_q detJ_q f N_a,            k(x) = k0 + k2 x^2
//   elasticity A^e_(a,c)(b,c') = sum_q w_q detJ_q [lam g_a,c g_b,c' +
//              mu g_a,c' g_b,c + mu delta_cc' g_a . g_b]  (= B_a^T D B_b for
//              isotropic D), b^e_(a,c) = sum_q w_q detJ_q f_c N_a
// with g_a = grad N_a = J^{-T} grad_xi N_a and J_ij = dx_i / dxi_j.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fea_internal.cuh"

namespace fea {

// quadrature rule slots
enum RuleSlot { kRuleTet1 = 0, kRuleTet4 = 1, kRulePyr8 = 2, kRulePrism6 = 3, kRuleHex8 = 4, kNumRules = 5 };

__host__ __device__ constexpr int rule_nq(int slot) {
  return slot == kRuleTet1 ? 1 : slot == kRuleTet4 ? 4 : slot == kRulePrism6 ? 6 : 8;
}
__host__ __device__ constexpr int rule_type(int slot) {
  return slot <= kRuleTet4 ? FEA_TET4 : slot == kRulePyr8 ? FEA_PYR5 : slot == kRulePrism6 ? FEA_PRISM6 : FEA_HEX8;
}

// Reference values at the quadrature points of one rule.
struct RefRule {
  double w[8];
  double N[8][8];       // [q][a]
  double dN[8][8][3];   // [q][a][j] = dN_a / dxi_j
  double m[8][4];       // [q] parameters of the point for RefMap
  float wf[8];
  float Nf[8][8];
  float dNf[8][8][3];
};

// Host-built tables (computed once per process from the closed forms); passed
// to kernels by value as __grid_constant__ parameters.
const RefRule& host_rule(int slot);

// ---------------------------------------------------------------------------
// FP32 -> FP64 without the FP64 pipe.  On GB300 a cvt.f64.f32 issues on the
// FP64 unit (about 0.6 T/s per GPU, the same as DADD), which would make the
// conversion of every accumulated entry cost as much as the assembly itself;
// the widening below is exact and uses integer instructions only.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double f32_to_f64_exact(float x) {
  const uint32_t u = __float_as_uint(x);
  const uint32_t mag = u & 0x7fffffffu;
  if (mag - 0x00800000u < 0x7f000000u || mag == 0u) {
    // a normal number (or a zero, which entries of axis-aligned elements often
    // are: a select, not a branch of the warp): the exponent field moves 3 bits down and its bias
    // grows by 1023 - 127 = 896; the 23 fraction bits split 20 | 3 across
    // the two words
    const uint32_t hi = mag == 0u ? 0u : (mag >> 3) + (896u << 20);
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
  }
  const uint32_t sign = u & 0x80000000u;
  int e = (int)((u >> 23) & 0xffu);
  uint32_t m = u & 0x7fffffu;
  if (e == 0) {
    const int lz = __clz((int)m) - 8;  // normalise a subnormal: bring the leading bit to position 23
    m = (m << lz) & 0x7fffffu;
    e = 1 - lz;
  } else if (e == 255) {
    return (double)x;  // inf / nan: keep the IEEE semantics
  }
  const uint32_t hi = sign | ((uint32_t)(e + 896) << 20) | (m >> 3);
  return __hiloint2double((int)hi, (int)(m << 29));
}

// 1 / d for a normal d away from the ends of the range: the hardware's
// approximate reciprocal (PTX rcp.approx.ftz.f64, not on the FP64 unit) and
// one step of the third-order Newton (Householder) iteration r (1 + e + e^2),
// e = 1 - d r, whose error is e^3: three FP64 instructions, where the IEEE
// division takes about three times as many.  Not correctly rounded: within
// one unit in the last place of the quotient for exponents in [-1000, 1000]
// (the test compares 2^28 arguments).  Beyond, and for zeros, infinities and
// subnormals, the result can be a NaN: its callers pass determinants of
// Jacobians (edge lengths of 1e-100 to 1e100), the slope of the consistency
// condition and the norm of a yielding point's stress; a branch to the division
// for the others cost 2 % of an FP32 J2 assembly.
__device__ __forceinline__ double rcp64(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// cofactor matrix C of J (J^{-1} = C^T / det J, det J = J_0j C_0j)
__device__ __forceinline__ void cofactors(const double J[3][3], double C[3][3]) {
  C[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
  C[0][1] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
  C[0][2] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
  C[1][0] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
  C[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
  C[1][2] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
  C[2][0] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
  C[2][1] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
  C[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
}

// ---------------------------------------------------------------------------
// Trilinear hex at the 2x2x2 Gauss points in modal form.  With corners in
// binary order p = bx + 2 by + 4 bz (hex8_corner_node maps p to the local node
// order), the map is x(xi) = (1/8) sum_k c_k prod_{s in k} xi_s, where bit s of
// k selects the coordinate xi_s and c_k = sum_p x_p prod_{s in k} sigma_s(p),
// sigma_s(p) = +1 if bit s of p is set, else -1 (a Walsh-Hadamard transform of
// the corner coordinates).  The Jacobian columns are bilinear in the other two
// coordinates, so all eight Jacobians cost 27 FMAs each instead of 63.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int hex8_corner_node(int p) {
  return 4 * (p >> 2) + ((p & 2) ? ((p & 1) ? 2 : 3) : (p & 1));
}

// Lane p of an aligned group of 8 lanes holds the coordinates of corner p on
// entry and c_p on exit (one FP64 add per stage and component: the partner's
// value enters with the sign of the stage).  Every lane of the warp must call it.
// The sign is applied to the partner's value by flipping its sign bit with an
// integer XOR: a per-lane select between v + o and v - o compiles to both FP64
// adds, which doubles the transform's cost on the FP64 pipe.  v + (-o) equals
// v - o exactly (IEEE 754), so the result is unchanged.
__device__ __forceinline__ void hex8_modal(double v[3]) {
  const int p = threadIdx.x & 7;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int bit = 1 << s;
    const int flip = (p & bit) ? (int)0x80000000 : 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double o = __shfl_xor_sync(0xffffffffu, v[i], bit);
      v[i] += __hiloint2double(__double2hiint(o) ^ flip, __double2loint(o));
    }
  }
}

// J' = 8 J at Gauss point q (xi_s = +-1/sqrt(3) by bit s of q) from the modal
// coefficients c[k][i] of hex8_modal, for the lane's own point, with the work
// shared by the 8 lanes of an element (lane p of an aligned group of 8 holds
// point p; every lane of the warp must call it).  Column j of J' is
// sum_k c_k d(prod_{s in k} xi_s)/d xi_j, four terms; the coordinate products
// are +-1/3 (the rounded square of the point), chosen by sign so that they
// cost no FP64 multiply.  Column 0 depends only on (y, z) and column 1 only
// on (x, z), so each takes 4 distinct values over the 8 points: lanes whose
// bits 0 and 1 agree form column 0, the others column 1, and each lane takes
// the column it lacks from the partner with the same coordinates (lane p ^ 2
// for column 1, p ^ 1 for column 0).  Column 2 depends only on (x, y), shared
// by lanes p and p ^ 4: the lane with bit 2 clear forms its components 0 and
// 1, the other component 2 (twice: the warp issues two slots either way),
// and they exchange: 15 FMAs per lane instead of 27, each entry the same FMA
// chain as a lane forming all of J would evaluate.  SHARE_Z = false forms
// column 2 on every lane (18 FMAs, no selects or shuffles): the block-task
// producers, which are bound by issue rather than by the FP64 unit, measured
// 3.82 against 3.80 ms per 128^3 step with the shared column.
template <bool SHARE_Z = true>
__device__ __forceinline__ void hex8_jacobian_pairs(const double (*c)[3], int q, double J[3][3]) {
  constexpr double g = 0.57735026918962576451;
  constexpr double g2 = g * g;
  const double x = (q & 1) ? g : -g, y = (q & 2) ? g : -g, z = (q & 4) ? g : -g;
  const double xy = ((q ^ (q >> 1)) & 1) ? -g2 : g2;
  const double xz = ((q ^ (q >> 2)) & 1) ? -g2 : g2;
  const double yz = (((q >> 1) ^ (q >> 2)) & 1) ? -g2 : g2;
  const bool first = ((q ^ (q >> 1)) & 1) == 0;  // this lane forms column 0
  const double s = first ? y : x, st = first ? yz : xz;
  const int partner = (int)(threadIdx.x & 31) ^ (first ? 2 : 1);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double ca = first ? c[1][i] : c[2][i], cc = first ? c[5][i] : c[6][i];
    const double own = fma(c[7][i], st, fma(cc, z, fma(c[3][i], s, ca)));
    const double other = __shfl_sync(0xffffffffu, own, partner);
    J[i][0] = first ? own : other;
    J[i][1] = first ? other : own;
    if constexpr (!SHARE_Z) J[i][2] = fma(c[7][i], xy, fma(c[6][i], y, fma(c[5][i], x, c[4][i])));
  }
  if constexpr (!SHARE_Z) return;
  const bool low = (q & 4) == 0;
  const int zpartner = (int)(threadIdx.x & 31) ^ 4;
  double m[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    // slot u: component u on the low lane, component 2 on the high one
    const double a4 = low ? c[4][u] : c[4][2], a5 = low ? c[5][u] : c[5][2];
    const double a6 = low ? c[6][u] : c[6][2], a7 = low ? c[7][u] : c[7][2];
    m[u] = fma(a7, xy, fma(a6, y, fma(a5, x, a4)));
  }
  const double o0 = __shfl_sync(0xffffffffu, m[0], zpartner), o1 = __shfl_sync(0xffffffffu, m[1], zpartner);
  J[0][2] = low ? m[0] : o0;
  J[1][2] = low ? m[1] : o1;
  J[2][2] = low ? o0 : m[0];
}

// x coordinate at Gauss point q of the 2x2x2 rule from the modal
// coefficients c_k of hex8_modal: (1/8) sum_k c_k prod_{s in k} xi_s, with
// xi_s = +-1/sqrt(3) by bit s of q.  Each weight is (1/8) g^|k| with the sign
// of the product (negative when an odd number of the bits of k are clear in
// q), set by flipping the constant's sign bit with an integer XOR, so the sum
// costs 8 FMAs and no FP64 multiply.  Equal to (1/8) times the sum with the
// weights formed as products of +-g: the powers of g round the same way, and
// the factor 1/8 is exact.
__device__ __forceinline__ double hex8_modal_x(const double (*c)[3], int q) {
  constexpr double g = 0.57735026918962576451;
  constexpr double g2 = g * g, g3 = g2 * g;
  constexpr double mag[8] = {0.125, 0.125 * g, 0.125 * g, 0.125 * g2, 0.125 * g, 0.125 * g2, 0.125 * g2, 0.125 * g3};
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int flip = (__popc(k & ~q) & 1) ? (int)0x80000000 : 0;
    acc = fma(c[k][0], __hiloint2double(__double2hiint(mag[k]) ^ flip, __double2loint(mag[k])), acc);
  }
  return acc;
}

// ---------------------------------------------------------------------------
// The maps of the other types from a few combinations of the node values,
// taken once per element and component, instead of a sum over the nodes with
// tabulated derivatives at every point.  prep(X, i) replaces component i of an
// element's node values X [NN][3] (coordinates or any nodal field) by its
// combinations; jac gives J' = s dx/dxi at a point from them, s a power of
// two; x1 gives component 0 of the field itself (coordinates: before prep the
// node values were absolute, the combinations are differences).  FP64
// instructions per element for J and x at every point: prism 330 -> 117,
// pyramid 348 -> 142 (one J serves two points), both with 8 or 6 points.
//  tet4    J's columns are the edges x_{j+1} - x_0
//  prism6  x = [(1 - z) B + (1 + z) T] / 2 with B, T the bottom and top
//          triangles: columns 0, 1 are linear in z, column 2 in (r, s)
//  pyr5    with (x, y, z) = (t xi, t eta, 1 - t) the shape functions are t
//          times the bilinear ones of the base and z: the columns depend on
//          (xi, eta) only, so the points q and q + 4 share J
// ---------------------------------------------------------------------------
template <int TYPE>
struct RefMap;
template <>
struct RefMap<FEA_TET4> {
  static constexpr double s = 1.0;
  static __device__ __forceinline__ void prep(double (*X)[3], int i) {
#pragma unroll
    for (int a = 1; a < 4; ++a) X[a][i] -= X[0][i];
  }
  static __device__ __forceinline__ void jac(const double (*X)[3], const double*, double (&J)[3][3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) J[i][j] = X[j + 1][i];
  }
  static __device__ __forceinline__ double x1(const double (*X)[3], const double* N, const double*) {
    return fma(N[3], X[3][0], fma(N[2], X[2][0], fma(N[1], X[1][0], X[0][0])));
  }
};
template <>
struct RefMap<FEA_PRISM6> {  // m: r, s, z
  static constexpr double s = 2.0;
  static __device__ __forceinline__ void prep(double (*X)[3], int i) {
    const double x0 = X[0][i], x3 = X[3][i];
    const double e1 = X[1][i] - x0, e2 = X[2][i] - x0, f1 = X[4][i] - x3, f2 = X[5][i] - x3;
    X[0][i] = e1 + f1;
    X[1][i] = e2 + f2;
    X[2][i] = f1 - e1;
    X[3][i] = f2 - e2;
    X[4][i] = x3 - x0;
    X[5][i] = x0 + x3;
  }
  static __device__ __forceinline__ void jac(const double (*X)[3], const double* m, double (&J)[3][3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      J[i][0] = fma(m[2], X[2][i], X[0][i]);
      J[i][1] = fma(m[2], X[3][i], X[1][i]);
      J[i][2] = fma(m[1], X[3][i], fma(m[0], X[2][i], X[4][i]));
    }
  }
  static __device__ __forceinline__ double x1(const double (*X)[3], const double*, const double* m) {
    const double c = fma(m[1], X[3][0], fma(m[0], X[2][0], X[4][0]));
    return 0.5 * fma(m[2], c, fma(m[1], X[1][0], fma(m[0], X[0][0], X[5][0])));
  }
};
template <>
struct RefMap<FEA_PYR5> {  // m: xi, eta, xi eta, z
  static constexpr double s = 4.0;
  static __device__ __forceinline__ void prep(double (*X)[3], int i) {
    const double x0 = X[0][i], x1 = X[1][i], x2 = X[2][i], x3 = X[3][i];
    const double p = x1 - x0, q = x2 - x3, r = x3 - x0;
    const double b = p + q, w = fma(2.0, r, b);  // w: the other base nodes' distances to node 0
    X[0][i] = b;
    X[1][i] = (x2 - x1) + r;
    X[2][i] = q - p;
    X[3][i] = fma(4.0, X[4][i] - x0, -w);
    X[4][i] = fma(4.0, x0, w);
  }
  static __device__ __forceinline__ void jac(const double (*X)[3], const double* m, double (&J)[3][3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      J[i][0] = fma(m[1], X[2][i], X[0][i]);
      J[i][1] = fma(m[0], X[2][i], X[1][i]);
      J[i][2] = fma(m[2], X[2][i], X[3][i]);
    }
  }
  static __device__ __forceinline__ double x1(const double (*X)[3], const double*, const double* m) {
    const double base = fma(m[2], X[2][0], fma(m[1], X[1][0], m[0] * X[0][0]));
    return 0.25 * fma(1.0 - m[3], base, fma(m[3], X[3][0], X[4][0]));
  }
};

// FP64 -> FP32, rounded to nearest even, with integer instructions only
// (IEEE 754 binary64 to binary32).  On GB300 the hardware conversion issues
// on the FP64 unit, and a fallback to it for rare inputs was still issued by
// every warp once the compiler predicated it (ncu: one FP64-pipe instruction
// per conversion beyond the FP64 arithmetic), so no case uses it:
// - a normal result (inline): the 52-bit significand keeps its top 23 bits
//   and rounds up when the 29 dropped bits exceed half an ulp, or equal it
//   with an odd kept part; a carry out of the significand moves into the
//   exponent, which also gives the correct overflow to infinity;
// - a zero or an FP64 subnormal (inline): a zero of the same sign;
// - the rest, in a function of its own so that the common path stays a
//   branch and not predicated code: a subnormal or zero binary32 result (the
//   significand with its leading 1, shifted down to units of 2^-149 and
//   rounded the same way; a carry into bit 23 is the smallest normal number's
//   encoding), overflow to infinity, infinities, and NaNs (quiet, with the top
//   bits of the payload).
static __device__ __noinline__ float f64_to_f32_rare(uint32_t hi, uint32_t lo) {
  const uint32_t sign = hi & 0x80000000u;
  const int Ed = (int)((hi >> 20) & 0x7ffu);
  if (Ed == 0x7ff) {
    const uint32_t payload = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const bool nan = ((hi & 0xfffffu) | lo) != 0u;
    return __uint_as_float(sign | 0x7f800000u | (nan ? (0x00400000u | payload) : 0u));
  }
  const int E = Ed - 896;
  if (E >= 255) return __uint_as_float(sign | 0x7f800000u);
  // value = M 2^(Ed - 1075) with M = 2^52 + fraction; in units of 2^-149 it
  // is M 2^-(30 - E), a shift of at least 30; from 54 on the value is below
  // half a unit and rounds to zero
  const int sh = 30 - E;
  if (sh >= 54) return __uint_as_float(sign);
  const unsigned long long M = (((unsigned long long)(hi & 0xfffffu) | 0x100000ull) << 32) | lo;
  const unsigned long long kept = M >> sh;
  const unsigned long long rest = M & ((1ull << sh) - 1ull);
  const unsigned long long half = 1ull << (sh - 1);
  const uint32_t up = (rest > half) || (rest == half && (kept & 1ull));
  return __uint_as_float(sign | ((uint32_t)kept + up));
}

__device__ __forceinline__ float f64_to_f32_rn(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int Ed = (int)((hi >> 20) & 0x7ffu);
  const int E = Ed - 896;  // binary32 biased exponent
  if (E > 0 && E < 255) {
    const uint32_t kept = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const uint32_t rest = lo & 0x1fffffffu;
    const uint32_t up = (rest > 0x10000000u) || (rest == 0x10000000u && (kept & 1u));
    return __uint_as_float(((hi & 0x80000000u) | ((uint32_t)E << 23) | kept) + up);
  }
  if (Ed == 0) return __uint_as_float(hi & 0x80000000u);
  return f64_to_f32_rare(hi, lo);
}

// an FP64 value in the tile precision: exact for FP64 tiles, rounded to
// nearest even by integer instructions for FP32 tiles (keeps the FP64 pipe,
// which also runs the hardware conversion, free for the arithmetic)
template <typename R>
__device__ __forceinline__ R to_tile(double x);
template <>
__device__ __forceinline__ double to_tile<double>(double x) {
  return x;
}
template <>
__device__ __forceinline__ float to_tile<float>(double x) {
  return f64_to_f32_rn(x);
}

__device__ __forceinline__ void cofactors(const float J[3][3], float C[3][3]) {
  C[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
  C[0][1] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
  C[0][2] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
  C[1][0] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
  C[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
  C[1][2] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
  C[2][0] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
  C[2][1] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
  C[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
}


// FP64 value of a contribution: exact integer widening of FP32 (keeps the
// FP64 pipe free), identity for FP64
__device__ __forceinline__ double widen(float x) { return f32_to_f64_exact(x); }
__device__ __forceinline__ double widen(double x) { return x; }

// FP64 add into global memory that returns nothing: a reduction carried out
// in L2 on a global-space address (red.global.add.f64), so the warp never
// waits for it.  atomicAdd compiles to that only where the compiler can tell
// the pointer is global; in the persistent kernels, whose pointers come from
// a parameter table indexed at run time, it became a generic-address atomic
// whose result every warp waited for (ncu: no reduction sectors in L2,
// long-scoreboard stalls 4.8 per issue against 1.1 in the per-type kernel).
// A generic-address red behaves the same, hence the explicit conversion.
__device__ __forceinline__ void red_add(double* p, double v) {
  const size_t g = __cvta_generic_to_global(p);
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(g), "d"(v) : "memory");
}


// 32 zero bytes at a 32-byte aligned address
__device__ __forceinline__ void zero32(double* p) {
  asm volatile("st.global.v4.f64 [%0], {%1, %1, %1, %1};" ::"l"(__cvta_generic_to_global(p)), "d"(0.0) : "memory");
}

// add into A or b: FP64 atomic (ATOMIC, Alg. "no coloring"), or a plain
// read-modify-write when no other element of the launch touches the entry
// (COLOR: the launch holds one color class, Alg. "coloring")
template <int SC>
__device__ __forceinline__ void scatter_add(double* p, double v) {
  if constexpr (SC == FEA_SCATTER_ATOMIC)
    red_add(p, v);
  else
    *p += v;
}

}  // namespace fea
