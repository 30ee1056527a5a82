// D3Q27 lattice and moment transforms used by the kernels.
//
// Velocities are held in tensor order t = (cx+1) + 3(cy+1) + 9(cz+1), so the
// rest velocity is t = 13 and the opposite of t is 26 - t.  The D3Q27 weights
// of Sec. II are the products of the D1Q3 weights (1/6, 2/3, 1/6) of the three
// components.  The paper's own direction order (Eq. velSet, fixed by rows 2-4
// of the printed M in App. A) is used only at the C ABI.
//
// Moments.  The raw moments R_abc = sum_i cx^a cy^b cz^c f_i (a,b,c in 0..2)
// follow from three one-dimensional 3-point transforms (one per axis,
// raw_forward; raw_inverse undoes them).  The moments m_1..m_27 of
// Eq. (momentSet) are sparse integer combinations of the R_abc
// (moment_forward, M = T V3: the moment matrix the library exports and checks itself against), and
// T^-1 K T falls into small blocks (relax_moments), so the kernels hold neither T nor a dense
// 27x27 matrix.
#pragma once
#include <stdint.h>

#include <type_traits>

#include "lbm_f2.cuh"

namespace lbmk {

constexpr int Q = 27;
constexpr int REST = 13;

__host__ __device__ constexpr int cx_of(int t) { return t % 3 - 1; }
__host__ __device__ constexpr int cy_of(int t) { return (t / 3) % 3 - 1; }
__host__ __device__ constexpr int cz_of(int t) { return t / 9 - 1; }
__host__ __device__ constexpr int opp_of(int t) { return 26 - t; }
__host__ __device__ constexpr int tensor_index(int cx, int cy, int cz) { return (cx + 1) + 3 * (cy + 1) + 9 * (cz + 1); }
__host__ __device__ constexpr int speed2_of(int t) {
  return cx_of(t) * cx_of(t) + cy_of(t) * cy_of(t) + cz_of(t) * cz_of(t);
}
__host__ __device__ constexpr double w1d(int c) { return c == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
// D3Q27 weight w_i (Sec. II): 8/27, 2/27, 1/54, 1/216 by |c|^2 = 0, 1, 2, 3.
__host__ __device__ constexpr double weight_of(int t) { return w1d(cx_of(t)) * w1d(cy_of(t)) * w1d(cz_of(t)); }

// Paper direction i (0-based, i.e. the paper's i-1) -> tensor index.
// Eq. (velSet) gives the groups; the order inside each group is the one of
// rows 2-4 (c_x, c_y, c_z) of the transformation matrix printed in App. A.
__host__ __device__ inline int paper_to_tensor(int i) {
  switch (i) {
    case 0: return tensor_index(0, 0, 0);
    case 1: return tensor_index(1, 0, 0);
    case 2: return tensor_index(-1, 0, 0);
    case 3: return tensor_index(0, 1, 0);
    case 4: return tensor_index(0, -1, 0);
    case 5: return tensor_index(0, 0, 1);
    case 6: return tensor_index(0, 0, -1);
    case 7: return tensor_index(1, 1, 0);
    case 8: return tensor_index(-1, -1, 0);
    case 9: return tensor_index(1, -1, 0);
    case 10: return tensor_index(-1, 1, 0);
    case 11: return tensor_index(0, 1, 1);
    case 12: return tensor_index(0, -1, -1);
    case 13: return tensor_index(0, 1, -1);
    case 14: return tensor_index(0, -1, 1);
    case 15: return tensor_index(1, 0, 1);
    case 16: return tensor_index(-1, 0, -1);
    case 17: return tensor_index(-1, 0, 1);
    case 18: return tensor_index(1, 0, -1);
    case 19: return tensor_index(1, 1, 1);
    case 20: return tensor_index(-1, -1, -1);
    case 21: return tensor_index(1, 1, -1);
    case 22: return tensor_index(-1, -1, 1);
    case 23: return tensor_index(-1, 1, 1);
    case 24: return tensor_index(1, -1, -1);
    case 25: return tensor_index(1, -1, 1);
    default: return tensor_index(-1, 1, -1);
  }
}

// Relaxation slot of moment j (0-based) in K = diag[s1 x4, s5, s6 x2, s8 x3,
// s11 x3, s14 x3, s17, s18, s19 x2, s21 x3, s24 x3, s27] (Sec. II).
__host__ __device__ inline int kslot_of(int j) {
  if (j < 4) return 1;
  if (j == 4) return 5;
  if (j < 7) return 6;
  if (j < 10) return 8;
  if (j < 13) return 11;
  if (j < 16) return 14;
  if (j == 16) return 17;
  if (j == 17) return 18;
  if (j < 20) return 19;
  if (j < 23) return 21;
  if (j < 26) return 24;
  return 27;
}

// c_T . (a0, a1, a2) with the zero components of c_T left out (IEEE arithmetic
// cannot drop a product with zero on its own).
template <int C, typename R>
__host__ __device__ __forceinline__ R signed_(R a) {
  if constexpr (C > 0) return a;
  else return -a;
}
template <int T, typename R>
__host__ __device__ __forceinline__ R cdot(R a0, R a1, R a2) {
  constexpr int c0 = cx_of(T), c1 = cy_of(T), c2 = cz_of(T);
  if constexpr (c0 != 0 && c1 != 0 && c2 != 0) return signed_<c0>(a0) + signed_<c1>(a1) + signed_<c2>(a2);
  else if constexpr (c0 != 0 && c1 != 0) return signed_<c0>(a0) + signed_<c1>(a1);
  else if constexpr (c0 != 0 && c2 != 0) return signed_<c0>(a0) + signed_<c2>(a2);
  else if constexpr (c1 != 0 && c2 != 0) return signed_<c1>(a1) + signed_<c2>(a2);
  else if constexpr (c0 != 0) return signed_<c0>(a0);
  else if constexpr (c1 != 0) return signed_<c1>(a1);
  else if constexpr (c2 != 0) return signed_<c2>(a2);
  else return R(0);
}

// ---------------------------------------------------------------------------
// raw moments: in-place 1D 3-point transforms along x, y and z.
// (f_-, f_0, f_+) -> (f_- + f_0 + f_+, f_+ - f_-, f_+ + f_-): orders 0, 1, 2.
template <typename R>
__host__ __device__ __forceinline__ void tri_forward(R& a, R& b, R& c) {
  R s = c + a, d = c - a;
  a = s + b;
  b = d;
  c = s;
}
#if defined(__CUDA_ARCH__)
// FP32 on the device: the y and z transforms treat the lines at x-index 0 and 2 alike, so
// those two lines go through one packed FP32x2 transform (a - b as fma(b, -1, a): the
// same rounding as the subtraction); the values and their rounding are the scalar ones.
__device__ __forceinline__ void tri_forward2(float& a0, float& a2, float& b0, float& b2, float& c0, float& c2) {
  const float2 a = make_float2(a0, a2), b = make_float2(b0, b2), c = make_float2(c0, c2);
  const float2 sum = __fadd2_rn(c, a), d = __ffma2_rn(a, make_float2(-1.f, -1.f), c);
  const float2 o = __fadd2_rn(sum, b);
  a0 = o.x;
  a2 = o.y;
  b0 = d.x;
  b2 = d.y;
  c0 = sum.x;
  c2 = sum.y;
}
__device__ __forceinline__ void tri_inverse2(float& a0, float& a2, float& b0, float& b2, float& c0, float& c2) {
  const float2 k0 = make_float2(a0, a2), k1 = make_float2(b0, b2), k2 = make_float2(c0, c2);
  const float2 a = __ffma2_rn(k1, make_float2(-1.f, -1.f), k2);
  const float2 b = __ffma2_rn(k2, make_float2(-2.f, -2.f), k0);
  const float2 c = __fadd2_rn(k2, k1);
  a0 = a.x;
  a2 = a.y;
  b0 = b.x;
  b2 = b.y;
  c0 = c.x;
  c2 = c.y;
}
#endif

template <typename R>
__host__ __device__ __forceinline__ void raw_forward(R v[27]) {
#pragma unroll
  for (int l = 0; l < 9; ++l) tri_forward(v[3 * l + 0], v[3 * l + 1], v[3 * l + 2]);  // x
#if defined(__CUDA_ARCH__)
  if constexpr (std::is_same<R, float>::value) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // y: lines (x, z) = (0|2, k), then (1, k)
      tri_forward2(v[9 * k], v[9 * k + 2], v[9 * k + 3], v[9 * k + 5], v[9 * k + 6], v[9 * k + 8]);
      tri_forward(v[9 * k + 1], v[9 * k + 4], v[9 * k + 7]);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {  // z: lines (x, y) = (0|2, j), then (1, j)
      tri_forward2(v[3 * j], v[3 * j + 2], v[3 * j + 9], v[3 * j + 11], v[3 * j + 18], v[3 * j + 20]);
      tri_forward(v[3 * j + 1], v[3 * j + 10], v[3 * j + 19]);
    }
    return;
  }
#endif
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    int base = (l % 3) + 9 * (l / 3);
    tri_forward(v[base], v[base + 3], v[base + 6]);  // y
  }
#pragma unroll
  for (int l = 0; l < 9; ++l) tri_forward(v[l], v[l + 9], v[l + 18]);  // z
}

// inverse of tri_forward on moments whose orders 1 and 2 come halved (exactly, by a power of two):
// (k0, k1/2, k2/2) -> ((k2 - k1)/2, k0 - k2, (k2 + k1)/2).
template <typename R>
__host__ __device__ __forceinline__ void tri_inverse(R& a, R& b, R& c) {
  const R k0 = a, k1 = b, k2 = c;
  a = k2 - k1;
  b = fma_(R(-2), k2, k0);
  c = k2 + k1;
}

// populations from raw moments scaled by 1/2 per axis of non-zero order: the inverse of
// raw_forward (z, then y, then x).
template <typename R>
__host__ __device__ __forceinline__ void raw_inverse(R v[27]) {
#if defined(__CUDA_ARCH__)
  if constexpr (std::is_same<R, float>::value) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {  // z
      tri_inverse2(v[3 * j], v[3 * j + 2], v[3 * j + 9], v[3 * j + 11], v[3 * j + 18], v[3 * j + 20]);
      tri_inverse(v[3 * j + 1], v[3 * j + 10], v[3 * j + 19]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // y
      tri_inverse2(v[9 * k], v[9 * k + 2], v[9 * k + 3], v[9 * k + 5], v[9 * k + 6], v[9 * k + 8]);
      tri_inverse(v[9 * k + 1], v[9 * k + 4], v[9 * k + 7]);
    }
#pragma unroll
    for (int l = 0; l < 9; ++l) tri_inverse(v[3 * l + 0], v[3 * l + 1], v[3 * l + 2]);  // x
    return;
  }
#endif
#pragma unroll
  for (int l = 0; l < 9; ++l) tri_inverse(v[l], v[l + 9], v[l + 18]);
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    int base = (l % 3) + 9 * (l / 3);
    tri_inverse(v[base], v[base + 3], v[base + 6]);
  }
#pragma unroll
  for (int l = 0; l < 9; ++l) tri_inverse(v[3 * l + 0], v[3 * l + 1], v[3 * l + 2]);
}

#define LBMK_R(a, b, c) r[(a) + 3 * (b) + 9 * (c)]

// Moments 5..27 of Eq. (momentSet) (0-based m[4..26]) from the raw moments.
// Moments 1..4 (density and momentum) are conserved and not needed here.
template <typename R>
__host__ __device__ __forceinline__ void moment_forward(const R r[27], R m[27]) {
  const R S2 = LBMK_R(2, 0, 0) + LBMK_R(0, 2, 0) + LBMK_R(0, 0, 2);
  const R S4 = LBMK_R(2, 2, 0) + LBMK_R(0, 2, 2) + LBMK_R(2, 0, 2);
  m[0] = LBMK_R(0, 0, 0);
  m[1] = LBMK_R(1, 0, 0);
  m[2] = LBMK_R(0, 1, 0);
  m[3] = LBMK_R(0, 0, 1);
  m[4] = fma_(R(-2), LBMK_R(0, 0, 0), S2);                                   // -2<1> + <|c|^2>
  m[5] = fma_(R(3), LBMK_R(2, 0, 0), -S2);                                   // 2<cx^2> - <cy^2+cz^2>
  m[6] = LBMK_R(0, 2, 0) - LBMK_R(0, 0, 2);                                  // <cy^2 - cz^2>
  m[7] = LBMK_R(1, 1, 0);                                                    // <cx cy>
  m[8] = LBMK_R(0, 1, 1);                                                    // <cy cz>
  m[9] = LBMK_R(1, 0, 1);                                                    // <cz cx>
  const R Ax = LBMK_R(1, 2, 0) + LBMK_R(1, 0, 2), Ay = LBMK_R(0, 1, 2) + LBMK_R(2, 1, 0);
  const R Az = LBMK_R(2, 0, 1) + LBMK_R(0, 2, 1);
  m[10] = fma_(R(3), Ax, R(-4) * LBMK_R(1, 0, 0));
  m[11] = fma_(R(3), Ay, R(-4) * LBMK_R(0, 1, 0));
  m[12] = fma_(R(3), Az, R(-4) * LBMK_R(0, 0, 1));
  m[13] = fma_(R(9), LBMK_R(1, 2, 2), fma_(R(-6), Ax, R(4) * LBMK_R(1, 0, 0)));
  m[14] = fma_(R(9), LBMK_R(2, 1, 2), fma_(R(-6), Ay, R(4) * LBMK_R(0, 1, 0)));
  m[15] = fma_(R(9), LBMK_R(2, 2, 1), fma_(R(-6), Az, R(4) * LBMK_R(0, 0, 1)));
  m[16] = fma_(R(3), S4, R(4) * (LBMK_R(0, 0, 0) - S2));                                     // 4<1-|c|^2> + 3<..>
  m[17] = fma_(R(27), LBMK_R(2, 2, 2), fma_(R(-18), S4, fma_(R(12), S2, R(-8) * LBMK_R(0, 0, 0))));
  m[18] = fma_(R(2), LBMK_R(0, 0, 2) + LBMK_R(0, 2, 0),
               fma_(R(3), LBMK_R(2, 2, 0) + LBMK_R(2, 0, 2), fma_(R(-4), LBMK_R(2, 0, 0), R(-6) * LBMK_R(0, 2, 2))));
  m[19] = fma_(R(2), LBMK_R(0, 0, 2) - LBMK_R(0, 2, 0), R(3) * (LBMK_R(2, 2, 0) - LBMK_R(2, 0, 2)));
  m[20] = fma_(R(3), LBMK_R(1, 1, 2), R(-2) * LBMK_R(1, 1, 0));
  m[21] = fma_(R(3), LBMK_R(2, 1, 1), R(-2) * LBMK_R(0, 1, 1));
  m[22] = fma_(R(3), LBMK_R(1, 2, 1), R(-2) * LBMK_R(1, 0, 1));
  m[23] = LBMK_R(1, 2, 0) - LBMK_R(1, 0, 2);
  m[24] = LBMK_R(0, 1, 2) - LBMK_R(2, 1, 0);
  m[25] = LBMK_R(2, 0, 1) - LBMK_R(0, 2, 1);
  m[26] = LBMK_R(1, 1, 1);
}

// ---------------------------------------------------------------------------
// The MRT relaxation in raw moments.  The relaxation matrix K couples only raw moments of one
// parity class (even / odd order in c_x, c_y, c_z), and Eq. (momentSet) is symmetric in the axes, so
// T^-1 K T splits into small blocks with closed forms (S2, S4: sums of the three second-order and
// of the three c_a^2 c_b^2 moments of h = f - f^(e) + F'/2; s: the shear rate of the node):
//   d<a^2>       = -s h<a^2> + (s - s5)/3 S2
//   d<b^2 c^2>   = -s19 h<b^2 c^2> + 2/3 (s - s19) h<a^2> + (s19 - s17)/3 S4
//                  + (4/9 (s17 - s5) - 2/9 (s - s19)) S2                      (a, b, c distinct)
//   d<222>       = -s18 h<222> + 2/3 (s18 - s17) S4 + (8/9 (s17 - s5) - 4/9 (s18 - s5)) S2
//   d<a b>       = -s h<ab>,   d<a b c^2> = -s21 h<abc^2> + 2/3 (s21 - s) h<ab>
//   d<a b^2>     = -(s11 + s24)/2 h<ab^2> - (s11 - s24)/2 h<ac^2>
//   d<a b^2 c^2> = -s14 h<ab^2c^2> + 2/3 (s14 - s11) (h<ab^2> + h<ac^2>),   d<111> = -s27 h<111>
// (S11 and S24 relax the sum and the difference of <ab^2> and <ac^2>).  The collided moments leave
// scaled by 1/2 per axis of non-zero order, which raw_inverse expects: powers of two, folded into
// the coefficients below, so the inverse transform needs no multiplications by 1/2.
template <typename R>
struct RelaxConst {
  R s5h;               // s5 / 6
  R q1, q4, q2s;       // <b^2 c^2>: -s19/4, (s19 - s17)/12, (s17 - s5)/9
  R s19_6;             // s19 / 6
  R t1, t2, t4;        // <222>: -s18/8, S2 and S4 coefficients / 8
  R v1, v2;            // <a b^2>: -(s11 + s24)/8, -(s11 - s24)/8
  R z1, z2;            // <a b^2 c^2>: -s14/8, (s14 - s11)/12
  R p1, pk;            // <a b c^2>: -s21/8, s21/12
  R d1;                // <111>: (1 - s27)/8
  // the folded form: (1 - s19)/4, s19/12, (1 - s18)/8, s18/72, (1 - (s11 + s24)/2)/4, s11/12,
  // (1 - s14)/8, coefficient of j / 8, (1 - s21)/8, s21/48
  R q1f, q2f, t1f, tbf, v1f, vjf, z1f, zjf, p1f, ptf;
};

// rate[j]: relaxation rate of moment j + 1 (the shear slots are not read)
template <typename R>
inline RelaxConst<R> make_relax(const double rate[27]) {
  const double s5 = rate[4], s11 = rate[10], s14 = rate[13], s17 = rate[16], s18 = rate[17], s19 = rate[18],
               s21 = rate[20], s24 = rate[23], s27 = rate[26];
  RelaxConst<R> K;
  K.s5h = (R)(s5 / 6.0);
  K.q1 = (R)(-s19 / 4.0);
  K.q4 = (R)((s19 - s17) / 12.0);
  K.q2s = (R)((s17 - s5) / 9.0);
  K.s19_6 = (R)(s19 / 6.0);
  K.t1 = (R)(-s18 / 8.0);
  K.t2 = (R)(((s17 - s5) * 8.0 / 9.0 - (s18 - s5) * 4.0 / 9.0) / 8.0);
  K.t4 = (R)((s18 - s17) / 12.0);
  K.v1 = (R)(-(s11 + s24) / 8.0);
  K.v2 = (R)(-(s11 - s24) / 8.0);
  K.z1 = (R)(-s14 / 8.0);
  K.z2 = (R)((s14 - s11) / 12.0);
  K.p1 = (R)(-s21 / 8.0);
  K.pk = (R)(s21 / 12.0);
  K.d1 = (R)((1.0 - s27) / 8.0);
  K.q1f = (R)((1.0 - s19) / 4.0);
  K.q2f = (R)(s19 / 12.0);
  K.t1f = (R)((1.0 - s18) / 8.0);
  K.tbf = (R)(s18 / 72.0);
  K.v1f = (R)((1.0 - 0.5 * (s11 + s24)) / 4.0);
  K.vjf = (R)(s11 / 12.0);
  K.z1f = (R)((1.0 - s14) / 8.0);
  K.zjf = (R)((s14 / 9.0 - (s14 - s11) * 4.0 / 9.0) / 8.0);
  K.p1f = (R)((1.0 - s21) / 8.0);
  K.ptf = (R)(s21 / 48.0);
  return K;
}

// Raw moments r of the total populations -> raw moments of f* = f - M^-1 K M h + F' + Omega^(2),
// scaled as raw_inverse expects.  Every term but f has the form w_i Q(c_i) (+ a rest-direction
// term, which only touches the conserved mass moment) with Q quadratic in c, so its raw moments are
// products of the D1Q3 weight moments 1, 1/3.  With w = rho u - F/2 + 2 nu_bar grad(rho) - F/2 and
// B = (P + 3 nu_bar u.grad(rho))/3 (P: sum_k rho_k crest_k; Eqs. EES, varphi_ik, Phi), the
// equilibrium minus half the forcing has the moments
//   <a^2> = B + u_a w_a,  <b^2c^2> = (B + u_b w_b + u_c w_c)/3,  <222> = (B + u.w)/9,
//   <ab> = (u_a w_b + u_b w_a)/2 = 3 <abc^2>,  <ab^2> = <ac^2> = 3 <ab^2c^2> = j_a/3
// (j_a = <a>: the F/2 terms cancel), and F' + Omega^(2) (Eq. ketFd; Eq. perturb, B_i) with
// pi_a = 2 u_a F_a + m_a n_a, m = (2/9) A |grad phi| n
//   <a> = F_a,  <a^2> = pi_a - |m|,  <b^2c^2> = (sum pi - |m| - pi_a)/3,  <222> = (sum pi - |m|)/9,
//   <ab> = u_a F_b + u_b F_a + m_a n_b = 3 <abc^2>,  <ab^2> = <ac^2> = 3 <ab^2c^2> = F_a/3.
// FOLD: each moment as a scaled moment plus a scaled equilibrium (about 170 operations); otherwise as
// itself plus its change (about 190), which rounds it once at its own size.  Error against FP64 relative to
// relaxing the 23 moments one by one (below), folded / rounded once, geometric means over droplets, jets and
// Rayleigh-Taylor boxes of several seeds:
//   FP64 storage, u 1.00 / 0.90, red density 0.98 / 0.97, blue 1.04 / 0.98;
//   FP32 storage, u 1.03 / 0.85, red density 1.05 / 0.98, blue 1.13 / 0.98;
//   compact half, red density 1.007 / 1.003, blue 1.004 / 1.000 (70 runs);
//   packed half, u 1.000 / 1.000, densities 0.999 / 1.000 (70 runs).
// So only the packed 16-bit storages fold (the rounding of the stored populations is all that counts
// there), which takes 488 instead of 515 us a step on the 128x128x512 jet; rounding once costs FP64
// storage 3 % of a step (32^3 55.5 -> 57.2 us) and compact storage 1.5 % (128x128x512 536 -> 545 us).
// Relaxing the 23 moments of Eq. (momentSet) one by one between T and T^-1, with the closed forms
// added per raw moment, took about 330 operations.  Measured folded, with the gradients by
// opposite pairs: collide-stream pass in FP64 on a 32^3 box (bound by the FP64 pipe) 69 -> 56 us;
// packed half, interior tiles of a 128^3 jet 78 -> 72 us on even and 88 -> 85 us on odd steps.
template <bool FOLD, typename R>
__host__ __device__ __forceinline__ void relax_moments(const RelaxConst<R>& K, R r[27], R s_sh, R B, const R u[3],
                                                       const R w[3], const R F[3], R m_abs, const R m[3],
                                                       const R n[3]) {
  // second-order and even moments
  const R sg0 = u[0] * w[0], sg1 = u[1] * w[1], sg2 = u[2] * w[2];
  const R tr = sg0 + sg1 + sg2, Btr = B + tr;
  const R pi0 = fma_(u[0], F[0], fma_(u[0], F[0], m[0] * n[0]));
  const R pi1 = fma_(u[1], F[1], fma_(u[1], F[1], m[1] * n[1]));
  const R pi2 = fma_(u[2], F[2], fma_(u[2], F[2], m[2] * n[2]));
  const R Z = pi0 + pi1 + pi2 - m_abs;
  const R h0 = LBMK_R(2, 0, 0) - B - sg0, h1 = LBMK_R(0, 2, 0) - B - sg1, h2 = LBMK_R(0, 0, 2) - B - sg2;
  const R S2 = h0 + h1 + h2;
  const R S4 = LBMK_R(2, 2, 0) + LBMK_R(0, 2, 2) + LBMK_R(2, 0, 2) - fma_(R(2.0 / 3.0), tr, B);
  const R b = fma_(R(1.0 / 6.0), s_sh, -K.s19_6);                        // (s - s19)/6
  const R a2 = fma_(R(-1.0 / 3.0), b, K.q2s);
  if constexpr (FOLD) {
    const R c = fma_(R(-0.5), s_sh, R(0.5));                              // (1 - s)/2
    const R L = fma_(fma_(R(1.0 / 6.0), s_sh, -K.s5h), S2, R(0.5) * (B - m_abs));
    LBMK_R(2, 0, 0) = fma_(c, h0, fma_(R(0.5), sg0 + pi0, L));
    LBMK_R(0, 2, 0) = fma_(c, h1, fma_(R(0.5), sg1 + pi1, L));
    LBMK_R(0, 0, 2) = fma_(c, h2, fma_(R(0.5), sg2 + pi2, L));
    const R CQ = fma_(a2, S2, fma_(K.q4, S4, fma_(R(1.0 / 12.0), Z, K.q2f * Btr)));
    LBMK_R(0, 2, 2) = fma_(K.q1f, LBMK_R(0, 2, 2), fma_(b, h0, fma_(-K.q2f, sg0, fma_(R(-1.0 / 12.0), pi0, CQ))));
    LBMK_R(2, 0, 2) = fma_(K.q1f, LBMK_R(2, 0, 2), fma_(b, h1, fma_(-K.q2f, sg1, fma_(R(-1.0 / 12.0), pi1, CQ))));
    LBMK_R(2, 2, 0) = fma_(K.q1f, LBMK_R(2, 2, 0), fma_(b, h2, fma_(-K.q2f, sg2, fma_(R(-1.0 / 12.0), pi2, CQ))));
    LBMK_R(2, 2, 2) =
        fma_(K.t1f, LBMK_R(2, 2, 2), fma_(K.t4, S4, fma_(K.t2, S2, fma_(K.tbf, Btr, R(1.0 / 72.0) * Z))));
    // pairs <ab>, <abc^2>
    const R c4 = R(0.5) * c, k = fma_(R(-1.0 / 12.0), s_sh, K.pk);         // (1 - s)/4, (s21 - s)/12
#define LBMK_PAIR(P, Q, x, y)                                                                       \
    {                                                                                               \
      const R t = fma_(u[x], w[y], u[y] * w[x]);                                                    \
      const R g = fma_(m[x], n[y], fma_(u[x], F[y], u[y] * F[x]));                                  \
      const R h = fma_(R(-0.5), t, P);                                                              \
      P = fma_(c4, h, fma_(R(0.125), t, R(0.25) * g));                                              \
      Q = fma_(K.p1f, Q, fma_(K.ptf, t, fma_(k, h, R(1.0 / 24.0) * g)));                            \
    }
    LBMK_PAIR(LBMK_R(1, 1, 0), LBMK_R(1, 1, 2), 0, 1)
    LBMK_PAIR(LBMK_R(0, 1, 1), LBMK_R(2, 1, 1), 1, 2)
    LBMK_PAIR(LBMK_R(1, 0, 1), LBMK_R(1, 2, 1), 0, 2)
#undef LBMK_PAIR
    // vectors <a>, <ab^2>, <ac^2>, <ab^2c^2>
#define LBMK_VEC(J, P, Q, T, x)                                                                     \
    {                                                                                               \
      const R j = J, e = fma_(K.vjf, j, R(1.0 / 12.0) * F[x]), p = P, q = Q;                         \
      J = R(0.5) * (j + F[x]);                                                                      \
      P = fma_(K.v1f, p, fma_(K.v2, q, e));                                                         \
      Q = fma_(K.v1f, q, fma_(K.v2, p, e));                                                         \
      T = fma_(K.z1f, T, fma_(K.z2, p + q, fma_(K.zjf, j, R(1.0 / 72.0) * F[x])));                   \
    }
    LBMK_VEC(LBMK_R(1, 0, 0), LBMK_R(1, 2, 0), LBMK_R(1, 0, 2), LBMK_R(1, 2, 2), 0)
    LBMK_VEC(LBMK_R(0, 1, 0), LBMK_R(0, 1, 2), LBMK_R(2, 1, 0), LBMK_R(2, 1, 2), 1)
    LBMK_VEC(LBMK_R(0, 0, 1), LBMK_R(2, 0, 1), LBMK_R(0, 2, 1), LBMK_R(2, 2, 1), 2)
#undef LBMK_VEC
  } else {
    const R hs = R(-0.5) * s_sh;
    const R L = fma_(fma_(R(1.0 / 6.0), s_sh, -K.s5h), S2, R(-0.5) * m_abs);
    LBMK_R(2, 0, 0) = fma_(R(0.5), LBMK_R(2, 0, 0), fma_(hs, h0, fma_(R(0.5), pi0, L)));
    LBMK_R(0, 2, 0) = fma_(R(0.5), LBMK_R(0, 2, 0), fma_(hs, h1, fma_(R(0.5), pi1, L)));
    LBMK_R(0, 0, 2) = fma_(R(0.5), LBMK_R(0, 0, 2), fma_(hs, h2, fma_(R(0.5), pi2, L)));
    const R CQ = fma_(a2, S2, fma_(K.q4, S4, R(1.0 / 12.0) * Z));
    const R E3 = R(1.0 / 3.0) * Btr;                                       // equilibrium of <b^2c^2>: E3 - sg_a/3
#define LBMK_EVEN(Q, h2a, sg, pi)                                                                   \
    {                                                                                                 \
      const R hq = Q - fma_(R(-1.0 / 3.0), sg, E3);                                                   \
      Q = fma_(R(0.25), Q, fma_(K.q1, hq, fma_(b, h2a, fma_(R(-1.0 / 12.0), pi, CQ))));               \
    }
    LBMK_EVEN(LBMK_R(0, 2, 2), h0, sg0, pi0)
    LBMK_EVEN(LBMK_R(2, 0, 2), h1, sg1, pi1)
    LBMK_EVEN(LBMK_R(2, 2, 0), h2, sg2, pi2)
#undef LBMK_EVEN
    {
      const R ht = fma_(R(-1.0 / 3.0), E3, LBMK_R(2, 2, 2));
      LBMK_R(2, 2, 2) = fma_(R(0.125), LBMK_R(2, 2, 2),
                             fma_(K.t1, ht, fma_(K.t4, S4, fma_(K.t2, S2, R(1.0 / 72.0) * Z))));
    }
    // pairs <ab>, <abc^2>
    const R c4 = R(0.5) * hs, k = fma_(R(-1.0 / 12.0), s_sh, K.pk);        // -s/4, (s21 - s)/12
#define LBMK_PAIR(P, Q, x, y)                                                                       \
    {                                                                                                 \
      const R t = fma_(u[x], w[y], u[y] * w[x]);                                                      \
      const R g = fma_(m[x], n[y], fma_(u[x], F[y], u[y] * F[x]));                                    \
      const R h = fma_(R(-0.5), t, P);                                                                \
      P = fma_(R(0.25), P, fma_(c4, h, R(0.25) * g));                                                 \
      const R hq = fma_(R(-1.0 / 6.0), t, Q);                                                         \
      Q = fma_(R(0.125), Q, fma_(K.p1, hq, fma_(k, h, R(1.0 / 24.0) * g)));                           \
    }
    LBMK_PAIR(LBMK_R(1, 1, 0), LBMK_R(1, 1, 2), 0, 1)
    LBMK_PAIR(LBMK_R(0, 1, 1), LBMK_R(2, 1, 1), 1, 2)
    LBMK_PAIR(LBMK_R(1, 0, 1), LBMK_R(1, 2, 1), 0, 2)
#undef LBMK_PAIR
    // vectors <a>, <ab^2>, <ac^2>, <ab^2c^2>
#define LBMK_VEC(J, P, Q, T, x)                                                                     \
    {                                                                                                 \
      const R j3 = R(1.0 / 3.0) * J, F12 = R(1.0 / 12.0) * F[x], hp = P - j3, hq = Q - j3;            \
      P = fma_(R(0.25), P, fma_(K.v1, hp, fma_(K.v2, hq, F12)));                                      \
      Q = fma_(R(0.25), Q, fma_(K.v1, hq, fma_(K.v2, hp, F12)));                                      \
      const R ht = fma_(R(-1.0 / 3.0), j3, T);                                                        \
      T = fma_(R(0.125), T, fma_(K.z1, ht, fma_(K.z2, hp + hq, R(1.0 / 72.0) * F[x])));               \
      J = R(0.5) * (J + F[x]);                                                                        \
    }
    LBMK_VEC(LBMK_R(1, 0, 0), LBMK_R(1, 2, 0), LBMK_R(1, 0, 2), LBMK_R(1, 2, 2), 0)
    LBMK_VEC(LBMK_R(0, 1, 0), LBMK_R(0, 1, 2), LBMK_R(2, 1, 0), LBMK_R(2, 1, 2), 1)
    LBMK_VEC(LBMK_R(0, 0, 1), LBMK_R(2, 0, 1), LBMK_R(0, 2, 1), LBMK_R(2, 2, 1), 2)
#undef LBMK_VEC
  }
  LBMK_R(1, 1, 1) = K.d1 * LBMK_R(1, 1, 1);
}

#undef LBMK_R

// Full 27x27 transformation matrix as the kernels apply it, column t = tensor
// index (host helper for the self-check; the kernels never form it).
inline void moment_matrix_tensor(double M[27][27]) {
  for (int t = 0; t < Q; ++t) {
    double v[27] = {0};
    v[t] = 1.0;
    raw_forward(v);
    double m[27];
    moment_forward(v, m);
    for (int j = 0; j < Q; ++j) M[j][t] = m[j];
  }
}

// SplitMix64 finaliser (Steele, Lea & Flood, OOPSLA 2014) and the inlet-noise
// variate xi in [-1, 1) keyed by (seed, step, node, component).
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ double inlet_noise(uint64_t seed, int64_t step, int64_t node, int comp) {
  uint64_t h = splitmix64(seed);
  h = splitmix64(h ^ (uint64_t)step);
  h = splitmix64(h ^ (uint64_t)node);
  h = splitmix64(h ^ (uint64_t)comp);
  return (double)(h >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
}

}  // namespace lbmk
