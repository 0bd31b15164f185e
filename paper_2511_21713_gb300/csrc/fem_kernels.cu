// Element kernels of the FEM block on the solvent shell Omega_i.
//
// Quantities (weak form of Sec. 2.2, operator split of Eqs. general_nonlinear /
// Vector_c, Jacobian of Eq. NR_main, second derivative of Appendix A):
//   N(u)_i       = eps_s kappa^2 int F(u_h) v_i
//   J(u)_ij      = eps_s kappa^2 int F'(u_h) v_i v_j
//   N''[d,d]_i   = eps_s kappa^2 int F''(u_h) d_h^2 v_i
// with F = u (linear), u + u^3/6 (T3) or sinh u (HS), 14-point rule per tet.
//
// Assembly is deterministic and atomic-free: one thread per tetrahedron writes
// its local values to tet-local storage (structure of arrays, coalesced), and
// a gather kernel sums, for every CSR slot or vertex, a fixed list of those
// entries in a fixed order.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>
#include <vector>

#include "fp64_math.cuh"
#include "pbfb_internal.cuh"
#include "quad_tables.cuh"
#include "warp_sum.cuh"

namespace pbfb {

namespace {

__device__ __forceinline__ void scheme_F(int scheme, double u, double& F, double& Fp, double& Fpp) {
  if (scheme == PBFB_LINEAR) {
    F = u;
    Fp = 1.0;
    Fpp = 0.0;
  } else if (scheme == PBFB_T3 || scheme == PBFB_T5 || scheme == PBFB_T7) {
    // Taylor polynomials of sinh: F = sum u^(2j+1)/(2j+1)!, F' = sum u^(2j)/(2j)!, F'' = F of one degree less
    const double u2 = u * u;
    const int deg = scheme == PBFB_T3 ? 3 : (scheme == PBFB_T5 ? 5 : 7);
    double term_odd = u, term_even = 1.0;  // u^(2j+1)/(2j+1)!, u^(2j)/(2j)!
    F = u;
    Fp = 1.0;
    Fpp = 0.0;
    for (int k = 3; k <= deg; k += 2) {
      Fpp += term_odd;                            // F'' gets the odd terms up to degree deg-2
      term_even *= u2 / ((k - 2) * (k - 1));      // u^(k-1)/(k-1)!
      term_odd *= u2 / ((k - 1) * k);             // u^k/k!
      F += term_odd;
      Fp += term_even;
    }
  } else {
    double e = exp(u);
    double ei = 1.0 / e;
    F = 0.5 * (e - ei);
    Fp = 0.5 * (e + ei);
    Fpp = F;
  }
}

// ------------------------------------------------------------ float-float sinh scheme
// The mixed precision evaluates the sinh scheme's element integrals on the float32 pipes
// (GB300's float64 rate is 1/64 of its float32 rate) in float-float arithmetic: a value is a
// pair hi + lo of float32 numbers with |lo| <= ulp(hi) / 2, sums by Knuth's two-sum and products
// by the FMA two-product (Dekker 1971; Ogita, Rump & Oishi 2005), about 2^-47 relative per
// operation.  Only the scaling by eps_s kappa^2 |T| and the conversion of the final sums to
// float64 (in the gather kernels) use the float64 pipes.
struct f2 { float h, l; };
__device__ __forceinline__ f2 f2_fast(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ f2 f2_two(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  const f2 s = f2_two(a.h, b.h);
  return f2_fast(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
  return f2_fast(p, e);
}
// product without the last normalisation: p + e, |e| a few ulps of p
__device__ __forceinline__ f2 f2_mul_raw(f2 a, f2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
  return {p, e};
}
// a += x with the low parts added plainly; f2_norm after the last term of a sum
__device__ __forceinline__ void f2_acc(f2& a, f2 x) {
  const f2 s = f2_two(a.h, x.h);
  a = {s.h, __fadd_rn(a.l, __fadd_rn(s.l, x.l))};
}
__device__ __forceinline__ f2 f2_norm(f2 a) { return f2_fast(a.h, a.l); }
__device__ __forceinline__ f2 f2_sum(f2 a, f2 b) {  // one f2_acc of two values
  f2_acc(a, b);
  return a;
}
// x rounded to float32 and the rest, by integer operations (four conversions and a subtraction of the float64 pipe
// otherwise: a third of an element kernel's time): 2^28 added to the low word rounds the 52-bit fraction to 23
// bits, the low 29 bits less 2^28 are the remainder in units of 2^(e - 52).  Outside [2^-73, 2^126) (0 among it)
// the conversions.
__device__ __forceinline__ f2 f2_split(double x) {
  const unsigned hi = __double2hiint(x), lo = __double2loint(x), sign = hi & 0x80000000u;
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - 950u >= 1149u - 950u) {
    const float h = __double2float_rn(x);
    return {h, __double2float_rn(x - (double)h)};
  }
  const unsigned lo2 = lo + 0x10000000u;
  const unsigned mag = (hi & 0x7fffffffu) + (lo2 < lo ? 1u : 0u);
  const float h = __uint_as_float((__funnelshift_l(lo2, mag, 3) - 0xC0000000u) | sign);
  const float r = (float)((int)(lo2 & 0x1fffffffu) - 0x10000000);
  return {h, __fmul_rn(r, __uint_as_float(((e - 948u) << 23) | sign))};
}
__device__ __forceinline__ double f2_val(f2 a) { return (double)a.h + (double)a.l; }

// Constants as float-float pairs, split at compile time from their float64 values.
#define PBFB_FF(name, x)                                 \
  constexpr float name##_h = (float)(x);                 \
  constexpr float name##_l = (float)((x) - (double)(float)(x))
#define PBFB_FFV(name) (f2{name##_h, name##_l})

// |u| = k ln2 / FX_N + f: the step in three parts, the first with 8 bits so that k FX_L1 is exact for k < 2^16
constexpr int FX_N = 512;
constexpr double FX_STEP = 0.69314718055994530942 / FX_N;
constexpr float FX_L1 = 0.00135040283203125f;
constexpr float FX_L2 = (float)(FX_STEP - (double)FX_L1);
constexpr float FX_L3 = (float)(FX_STEP - (double)FX_L1 - (double)FX_L2);

// Quadrature orbits of the 14-point tet rule: S31 orbits k = 1, 2 (three barycentrics alpha_k,
// one beta_k, delta_k = beta_k - alpha_k) and the S22 orbit (two c, two d, e = d - c), with
// u_q = alpha_k sum(u) + delta_k u_i and u_P = c sum(u) + e (u_p + u_q) for the pair P = {p, q}.
// The element sums reduce to orbit sums (l_{q,a} l_{q,b} expanded): the products of the weights
// with the orbit parameters below.
PBFB_FF(OR_A1, PBFB_T_A1);
PBFB_FF(OR_D1, PBFB_T_B1 - PBFB_T_A1);
PBFB_FF(OR_A2, PBFB_T_A2);
PBFB_FF(OR_D2, PBFB_T_B2 - PBFB_T_A2);
PBFB_FF(OR_C3, PBFB_T_C3);
PBFB_FF(OR_E3, PBFB_T_D3 - PBFB_T_C3);
PBFB_FF(OR_WA1, PBFB_T_W1 * PBFB_T_A1);
PBFB_FF(OR_WD1, PBFB_T_W1 * (PBFB_T_B1 - PBFB_T_A1));
PBFB_FF(OR_WAA1, PBFB_T_W1 * PBFB_T_A1 * PBFB_T_A1);
PBFB_FF(OR_WAD1, PBFB_T_W1 * PBFB_T_A1 * (PBFB_T_B1 - PBFB_T_A1));
PBFB_FF(OR_WDD1, PBFB_T_W1 * (PBFB_T_B1 - PBFB_T_A1) * (PBFB_T_B1 - PBFB_T_A1));
PBFB_FF(OR_WA2, PBFB_T_W2 * PBFB_T_A2);
PBFB_FF(OR_WD2, PBFB_T_W2 * (PBFB_T_B2 - PBFB_T_A2));
PBFB_FF(OR_WAA2, PBFB_T_W2 * PBFB_T_A2 * PBFB_T_A2);
PBFB_FF(OR_WAD2, PBFB_T_W2 * PBFB_T_A2 * (PBFB_T_B2 - PBFB_T_A2));
PBFB_FF(OR_WDD2, PBFB_T_W2 * (PBFB_T_B2 - PBFB_T_A2) * (PBFB_T_B2 - PBFB_T_A2));
PBFB_FF(OR_WC3, PBFB_T_W3 * PBFB_T_C3);
PBFB_FF(OR_WE3, PBFB_T_W3 * (PBFB_T_D3 - PBFB_T_C3));
PBFB_FF(OR_WCC3, PBFB_T_W3 * PBFB_T_C3 * PBFB_T_C3);
PBFB_FF(OR_WCE3, PBFB_T_W3 * PBFB_T_C3 * (PBFB_T_D3 - PBFB_T_C3));
PBFB_FF(OR_WEE3, PBFB_T_W3 * (PBFB_T_D3 - PBFB_T_C3) * (PBFB_T_D3 - PBFB_T_C3));

// float-float path for |u| < 60 (e^60 ~ 1.1e26): the upper word of 60.0, compared as integers (a NaN is above)
constexpr int FX_UMAX_HI = 0x404E0000;

// sinh u and cosh u for |u| <= 60, by |u| = v + f, v = k ln2 / 512, |f| <= 6.8e-4.  With c = cosh f - 1 and
// B = sinh f (c = f^2/2 + f^4/24 and B = f + f^3/6 + f^5/120: c is below 2^-22, so that f^4 and f^3 need float32
// only): sinh = sinh v + (B cosh v + c sinh v), cosh = cosh v + (B sinh v + c cosh v), where the bracket's terms
// come in falling order, so the fast two-sum does.  sinh v and cosh v: from the table for k < 512 (sinh keeps its
// relative accuracy near 0), else (2^m T[j] -+ 2^-m / T[j]) / 2, k = 512 m + j (no cancellation).
// tab[j] = (sinh, cosh)(j ln2 / 512), tab[512 + j] = (2^(j/512), 2^(-j/512)), j = 0..511: 16 KB, cached.
// 102 float32 operations; 172 with a table of step 1/32 and the series in float-float.  The error against 64 bits
// is no larger: rms 1.9e-15 (sinh and cosh, |u| <= 8) against 2.6e-15 and 2.7e-15, largest 1.6e-14 against 2.3e-14.
__device__ __forceinline__ f2 fx_bracket(f2 x, f2 y, f2 B, f2 c) {  // x + (B y + c x)
  const f2 p = f2_mul_raw(B, y), q = f2_mul_raw(c, x);
  const f2 t = f2_fast(p.h, q.h);
  const f2 s = f2_fast(x.h, t.h);
  return f2_fast(s.h, __fadd_rn(s.l, __fadd_rn(x.l, __fadd_rn(t.l, __fadd_rn(p.l, q.l)))));
}

__device__ __forceinline__ void ff_sinh_cosh(f2 u, const float4* __restrict__ tab, f2& S, f2& C) {
  const unsigned sign = __float_as_uint(u.h) & 0x80000000u;
  const float ah = fabsf(u.h), al = __uint_as_float(__float_as_uint(u.l) ^ sign);
  const float mg = __fmaf_rn(ah, (float)(1.0 / FX_STEP), 12582912.f);
  const int k = __float_as_int(mg) - 0x4B400000;
  const float kf = __fsub_rn(mg, 12582912.f);
  const float p2 = __fmul_rn(kf, FX_L2);
  const f2 r = f2_two(__fmaf_rn(-kf, FX_L1, ah), -p2);
  f2 f = f2_two(r.h, al);
  f = f2_fast(f.h, __fmaf_rn(-kf, FX_L3, __fadd_rn(__fsub_rn(r.l, __fmaf_rn(kf, FX_L2, -p2)), f.l)));
  const float s = __fmul_rn(f.h, f.h);
  const float sl = __fmaf_rn(2.f * f.h, f.l, __fmaf_rn(f.h, f.h, -s));
  const f2 c{0.5f * s, __fmaf_rn(__fmul_rn(s, s), 1.f / 24.f, 0.5f * sl)};
  const f2 B{f.h, __fmaf_rn(__fmul_rn(f.h, s), __fmaf_rn(s, 1.f / 120.f, 1.f / 6.f), f.l)};
  const float4 t = __ldg(&tab[k < FX_N ? k : FX_N + (k & (FX_N - 1))]);
  const int m = k / FX_N;
  const float sp = __int_as_float((126 + m) << 23), sm = __int_as_float((126 - m) << 23);  // 2^(m-1), 2^(-m-1)
  const f2 P{__fmul_rn(t.x, sp), __fmul_rn(t.y, sp)}, Q{__fmul_rn(t.z, sm), __fmul_rn(t.w, sm)};
  f2 sv = f2_fast(P.h, -Q.h), cv = f2_fast(P.h, Q.h);
  sv.l = __fadd_rn(sv.l, __fsub_rn(P.l, Q.l));
  cv.l = __fadd_rn(cv.l, __fadd_rn(P.l, Q.l));
  if (m == 0) {
    sv = {t.x, t.y};
    cv = {t.z, t.w};
  }
  S = fx_bracket(sv, cv, B, c);
  C = fx_bracket(cv, sv, B, c);
  S = {__uint_as_float(__float_as_uint(S.h) ^ sign), __uint_as_float(__float_as_uint(S.l) ^ sign)};
}

__global__ void k_tet_volumes(const double* __restrict__ xyz, int nv, const int* __restrict__ tets,
                              int64_t nt, double* __restrict__ vol) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  int v[4];
  for (int a = 0; a < 4; ++a) v[a] = tets[a * nt + t];
  double e[3][3];
  for (int k = 0; k < 3; ++k)
    for (int d = 0; d < 3; ++d) e[k][d] = xyz[d * nv + v[k + 1]] - xyz[d * nv + v[0]];
  double det = e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) -
               e[0][1] * (e[1][0] * e[2][2] - e[1][2] * e[2][0]) +
               e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0]);
  vol[t] = fabs(det) / 6.0;
}

// int grad l_a . grad l_b over the tet, 10 symmetric entries at k * nt + t.
__global__ void k_stiffness_local(const double* __restrict__ xyz, int nv, const int* __restrict__ tets,
                                  int64_t nt, const double* __restrict__ vol, double* __restrict__ loc) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  int v[4];
  for (int a = 0; a < 4; ++a) v[a] = tets[a * nt + t];
  double e[3][3];
  for (int k = 0; k < 3; ++k)
    for (int d = 0; d < 3; ++d) e[k][d] = xyz[d * nv + v[k + 1]] - xyz[d * nv + v[0]];
  // rows of E^{-1}^T: gradient of l_{k+1} = (cofactor row k) / det
  double c[3][3];
  c[0][0] = e[1][1] * e[2][2] - e[1][2] * e[2][1];
  c[0][1] = e[1][2] * e[2][0] - e[1][0] * e[2][2];
  c[0][2] = e[1][0] * e[2][1] - e[1][1] * e[2][0];
  c[1][0] = e[2][1] * e[0][2] - e[2][2] * e[0][1];
  c[1][1] = e[2][2] * e[0][0] - e[2][0] * e[0][2];
  c[1][2] = e[2][0] * e[0][1] - e[2][1] * e[0][0];
  c[2][0] = e[0][1] * e[1][2] - e[0][2] * e[1][1];
  c[2][1] = e[0][2] * e[1][0] - e[0][0] * e[1][2];
  c[2][2] = e[0][0] * e[1][1] - e[0][1] * e[1][0];
  double det = e[0][0] * c[0][0] + e[0][1] * c[0][1] + e[0][2] * c[0][2];
  double g[4][3];
  for (int d = 0; d < 3; ++d) {
    g[1][d] = c[0][d] / det;
    g[2][d] = c[1][d] / det;
    g[3][d] = c[2][d] / det;
    g[0][d] = -(g[1][d] + g[2][d] + g[3][d]);
  }
  double V = vol[t];
  for (int a = 0; a < 4; ++a)
    for (int b = a; b < 4; ++b)
      loc[(int64_t)sym10(a, b) * nt + t] = V * (g[a][0] * g[b][0] + g[a][1] * g[b][1] + g[a][2] * g[b][2]);
}

// F, F' and F'' of a scheme in float-float.  The Taylor schemes by Horner's rule on u^2 with the
// ratios of consecutive coefficients (all terms of one sign, no cancellation):
//   F = u (1 + u^2/6 (1 + u^2/20 (1 + u^2/42))), F' = 1 + u^2/2 (1 + u^2/12 (1 + u^2/30)),
// cut at degree 3, 5 or 7; F'' is F one degree lower.  The sinh scheme from ff_sinh_cosh.
PBFB_FF(FX_R6, 1.0 / 6.0);
PBFB_FF(FX_R12, 1.0 / 12.0);
PBFB_FF(FX_R20, 1.0 / 20.0);
PBFB_FF(FX_R30, 1.0 / 30.0);
PBFB_FF(FX_R42, 1.0 / 42.0);

// 1 + u2 r (1 + ...): one Horner step on a float-float tail
__device__ __forceinline__ f2 ff_horner(f2 u2, f2 r, f2 tail) {
  return f2_add(f2{1.f, 0.f}, f2_mul(f2_mul(u2, r), tail));
}

template <int S>
__device__ __forceinline__ void ff_scheme(f2 u, const float4* __restrict__ tab, f2& F, f2& G, f2& H) {
  if (S == PBFB_HS) {
    ff_sinh_cosh(u, tab, F, G);
    H = F;
  } else if (S == PBFB_LINEAR) {
    F = u;
    G = f2{1.f, 0.f};
    H = f2{0.f, 0.f};
  } else {
    const f2 u2 = f2_mul(u, u);
    const f2 one{1.f, 0.f};
    const f2 half_u2{0.5f * u2.h, 0.5f * u2.l};
    // odd part: degree 3 -> u (1 + u2/6); 5 -> u (1 + u2/6 (1 + u2/20)); 7 -> one more factor
    const f2 o7 = S == PBFB_T7 ? ff_horner(u2, PBFB_FFV(FX_R42), one) : one;
    const f2 o5 = S == PBFB_T3 ? one : ff_horner(u2, PBFB_FFV(FX_R20), o7);
    F = f2_mul(u, ff_horner(u2, PBFB_FFV(FX_R6), o5));
    // F'': the odd series one degree lower
    const f2 p5 = S == PBFB_T7 ? ff_horner(u2, PBFB_FFV(FX_R20), one) : one;
    H = S == PBFB_T3 ? u : f2_mul(u, ff_horner(u2, PBFB_FFV(FX_R6), p5));
    // even part: 1 + u2/2 (1 + u2/12 (1 + u2/30)), cut at the scheme's degree - 1
    const f2 e6 = S == PBFB_T7 ? ff_horner(u2, PBFB_FFV(FX_R30), one) : one;
    const f2 e4 = S == PBFB_T3 ? one : ff_horner(u2, PBFB_FFV(FX_R12), e6);
    G = f2_add(one, f2_mul(half_u2, e4));
  }
}

// Jacobian (10 entries, k = 0..9) and load (4 entries) of F on one tet in float64.
__device__ __forceinline__ void element_sums_f64(int scheme, const double (&ua)[4], double (&J)[10],
                                                 double (&N)[4]) {
  for (int k = 0; k < 10; ++k) J[k] = 0.0;
  for (int a = 0; a < 4; ++a) N[a] = 0.0;
  for (int q = 0; q < QT; ++q) {
    double l0 = c_tet_l[q][0], l1 = c_tet_l[q][1], l2 = c_tet_l[q][2], l3 = c_tet_l[q][3];
    double uq = l0 * ua[0] + l1 * ua[1] + l2 * ua[2] + l3 * ua[3];
    double F, Fp, Fpp;
    scheme_F(scheme, uq, F, Fp, Fpp);
    double w = c_tet_w[q];
    double f = w * F, g = w * Fp;
    double l[4] = {l0, l1, l2, l3};
    for (int a = 0; a < 4; ++a) {
      N[a] += f * l[a];
      double gl = g * l[a];
      for (int b = a; b < 4; ++b) J[sym10(a, b)] += gl * l[b];
    }
  }
}

// The omega batch's three loads of one tet for one omega in float64.
__device__ __forceinline__ void omega_sums_f64(int scheme, const double (&ua)[4], const double (&da)[4], double om,
                                               double (&R0)[4], double (&R1)[4], double (&R2)[4]) {
  for (int a = 0; a < 4; ++a) R0[a] = R1[a] = R2[a] = 0.0;
  for (int q = 0; q < QT; ++q) {
    double l[4] = {c_tet_l[q][0], c_tet_l[q][1], c_tet_l[q][2], c_tet_l[q][3]};
    double uq = l[0] * ua[0] + l[1] * ua[1] + l[2] * ua[2] + l[3] * ua[3];
    double dq = l[0] * da[0] + l[1] * da[1] + l[2] * da[2] + l[3] * da[3];
    double F, Fp, Fpp;
    scheme_F(scheme, uq + om * dq, F, Fp, Fpp);
    double w = c_tet_w[q];
    double f0 = w * F, f1 = w * Fp * dq, f2 = w * Fpp * dq * dq;
    for (int a = 0; a < 4; ++a) {
      R0[a] += f0 * l[a];
      R1[a] += f1 * l[a];
      R2[a] += f2 * l[a];
    }
  }
}

// A slot's tet-local entries are read GB at a time: a vertex has 24 tets, a diagonal slot as many entries, and one
// load after another is a chain of L2 latencies.
constexpr int GB = 8;

__global__ void k_gather(int nslots, const int* __restrict__ ptr, const int* __restrict__ idx,
                         const double* __restrict__ local, const double* __restrict__ base, double scale,
                         double* __restrict__ out) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nslots) return;
  double acc = 0.0;
  const int k1 = ptr[s + 1];
  for (int k0 = ptr[s]; k0 < k1; k0 += GB) {
    double x[GB];
#pragma unroll
    for (int j = 0; j < GB; ++j) x[j] = k0 + j < k1 ? local[idx[k0 + j]] : 0.0;
#pragma unroll
    for (int j = 0; j < GB; ++j)
      if (k0 + j < k1) acc += x[j];
  }
  out[s] = (base ? base[s] : 0.0) + scale * acc;
}

// The Jacobian's slots (added to base) and, from there on, the nn load slots over float-float tet-local entries
// (the float-float element kernels' output): the sum in float-float, one conversion to float64 per slot.
// GB300, 408,000 tets: 29 + 9 us as two kernels entry by entry, 40 us in one.
__global__ void __launch_bounds__(256) k_gather_ff(int nj, const int* __restrict__ jptr, const int* __restrict__ jidx,
                                                   const float2* __restrict__ jloc, const double* __restrict__ base,
                                                   double* __restrict__ jout, int nn, const int* __restrict__ nptr,
                                                   const int* __restrict__ nidx, const float2* __restrict__ nloc,
                                                   double* __restrict__ nout) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  const bool j = s < nj;
  if (!j) s -= nj;
  if (!j && s >= nn) return;
  const int* ptr = j ? jptr : nptr;
  const int* idx = j ? jidx : nidx;
  const float2* local = j ? jloc : nloc;
  f2 acc{0.f, 0.f};
  const int k1 = ptr[s + 1];
  for (int k0 = ptr[s]; k0 < k1; k0 += GB) {
    float2 x[GB];
#pragma unroll
    for (int q = 0; q < GB; ++q) x[q] = k0 + q < k1 ? local[idx[k0 + q]] : make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < GB; ++q) acc = f2_add(acc, f2{x[q].x, x[q].y});
  }
  if (j)
    jout[s] = base[s] + f2_val(acc);
  else
    nout[s] = f2_val(acc);
}

constexpr int ELEM_T = 256;  // threads a block of the float-float element kernels (128: 47 and 64 us, 512: 54 and 79)

__device__ __forceinline__ float2 f2_store(f2 a) { return make_float2(a.h, a.l); }

// F, F' and F'' of a scheme in float64: e^u and e^-u from one reduction (exp_pm), the Taylor schemes by Horner's rule.
template <int S>
__device__ __forceinline__ void scheme_f64(double u, const double* __restrict__ tab, double& F, double& G, double& H) {
  if (S == PBFB_HS) {
    double ep, em;
    exp_pm(fabs(u), tab, ep, em);
    F = copysign(0.5 * (ep - em), u);
    G = 0.5 * (ep + em);
    H = F;
  } else if (S == PBFB_LINEAR) {
    F = u;
    G = 1.0;
    H = 0.0;
  } else {
    const double u2 = u * u;
    const double o7 = S == PBFB_T7 ? fma(u2, 1.0 / 42.0, 1.0) : 1.0;
    const double o5 = S == PBFB_T3 ? 1.0 : fma(u2 * (1.0 / 20.0), o7, 1.0);
    F = u * fma(u2 * (1.0 / 6.0), o5, 1.0);
    const double p5 = S == PBFB_T7 ? fma(u2, 1.0 / 20.0, 1.0) : 1.0;
    H = S == PBFB_T3 ? u : u * fma(u2 * (1.0 / 6.0), p5, 1.0);
    const double e6 = S == PBFB_T7 ? fma(u2, 1.0 / 30.0, 1.0) : 1.0;
    const double e4 = S == PBFB_T3 ? 1.0 : fma(u2 * (1.0 / 12.0), e6, 1.0);
    G = fma(u2 * 0.5, e4, 1.0);
  }
}

// The float64 loops' orbit sums hold where F stays finite.  Past |u| = 700 (upper word compared as integers; infinities
// and NaN are above) a tet takes the rule point by point, whose weights are all positive: sums past the range are then
// infinite with F's sign, where the second orbit's negative beta - alpha would make inf - inf of them.
constexpr int ORBIT_MAX_HI = 0x4085E000;
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }

__device__ __noinline__ void element_wide(int scheme, const double* ua4, double sc, int64_t nt, int64_t t,
                                          double* __restrict__ loc) {
  const double ua[4] = {ua4[0], ua4[1], ua4[2], ua4[3]};
  double J[10], N[4];
  element_sums_f64(scheme, ua, J, N);
  for (int k = 0; k < 10; ++k) loc[k * nt + t] = sc * J[k];
  for (int a = 0; a < 4; ++a) loc[(10 + a) * nt + t] = sc * N[a];
}

// Jacobian and load of F on one tet in float64 (layout k * nt + t: J at k = 0..9, N at k = 10..13), from the orbit
// sums of k_element_ff below.  The float64 pipe bounds it: about 400 operations a tet for the sinh scheme, 1000 with
// the 14 points one by one, the library's exponential and a division.
// GB300, 86,400 tets: 128 us so, 72 us now.  Against long double the loads' errors scatter alike (1.35e-16 of their
// terms' magnitudes, rms over the vertices, both forms); the products of weights, rounded once at compile time, shift
// all of them by 3e-17.
template <int S>
__global__ void __launch_bounds__(128) k_element_f64(const double* __restrict__ u, const int* __restrict__ tets,
                                                     int64_t nt, const double* __restrict__ vol, double coef,
                                                     const double* __restrict__ tab, double* __restrict__ loc) {
  constexpr double A1 = PBFB_T_A1, D1 = PBFB_T_B1 - PBFB_T_A1, A2 = PBFB_T_A2, D2 = PBFB_T_B2 - PBFB_T_A2;
  constexpr double C3 = PBFB_T_C3, E3 = PBFB_T_D3 - PBFB_T_C3, W1 = PBFB_T_W1, W2 = PBFB_T_W2, W3 = PBFB_T_W3;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double v[4];
  int vmax = 0;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    v[a] = u[tets[a * nt + t]];
    vmax = max(vmax, abs_hi(v[a]));
  }
  if (vmax >= ORBIT_MAX_HI) {
    element_wide(S, v, coef * vol[t], nt, t, loc);
    return;
  }
  const double su = (v[0] + v[1]) + (v[2] + v[3]);
  double n[4], h[4], D[4], g3[6], T, C;
  {
    double fs = 0.0, gs = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a) n[a] = h[a] = 0.0;
#pragma unroll
    for (int p = 0, P = 0; p < 3; ++p)
#pragma unroll
      for (int q = p + 1; q < 4; ++q, ++P) {
        double F, G, H;
        scheme_f64<S>(fma(E3, v[p] + v[q], C3 * su), tab, F, G, H);
        n[p] += F;
        n[q] += F;
        h[p] += G;
        h[q] += G;
        g3[P] = W3 * E3 * E3 * G;
        fs += F;
        gs += G;
      }
    T = W3 * C3 * fs;
    C = W3 * C3 * C3 * gs;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      n[a] *= W3 * E3;
      D[a] = W3 * E3 * E3 * h[a];
      h[a] *= W3 * C3 * E3;
    }
  }
  auto orbit = [&](double alpha, double delta, double w) {
    double fs = 0.0, gs = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      double F, G, H;
      scheme_f64<S>(fma(delta, v[a], alpha * su), tab, F, G, H);
      n[a] = fma(w * delta, F, n[a]);
      h[a] = fma(w * alpha * delta, G, h[a]);
      D[a] = fma(w * delta * delta, G, D[a]);
      fs += F;
      gs += G;
    }
    T = fma(w * alpha, fs, T);
    C = fma(w * alpha * alpha, gs, C);
  };
  orbit(A1, D1, W1);
  orbit(A2, D2, W2);
  const double s = coef * vol[t];
#pragma unroll
  for (int a = 0, P = 0; a < 4; ++a) {
    loc[sym10(a, a) * nt + t] = s * (C + fma(2.0, h[a], D[a]));
#pragma unroll
    for (int b = a + 1; b < 4; ++b, ++P) loc[sym10(a, b) * nt + t] = s * ((C + g3[P]) + (h[a] + h[b]));
    loc[(10 + a) * nt + t] = s * (T + n[a]);
  }
}

// Tets outside the float-float range take the float64 sums (kept out of line).
__device__ __noinline__ void element_fallback(int scheme, const double* ua4, double sc, int64_t nt, int64_t t,
                                              float2* __restrict__ loc) {
  const double ua[4] = {ua4[0], ua4[1], ua4[2], ua4[3]};
  double J[10], N[4];
  element_sums_f64(scheme, ua, J, N);
  for (int k = 0; k < 10; ++k) loc[k * nt + t] = f2_store(f2_split(sc * J[k]));
  for (int a = 0; a < 4; ++a) loc[(10 + a) * nt + t] = f2_store(f2_split(sc * N[a]));
}

// a quadrature point's value: as + delta v
__device__ __forceinline__ f2 ff_point(f2 as, f2 v, f2 delta) {
  const f2 q = f2_mul_raw(v, delta);
  const f2 s = f2_two(as.h, q.h);
  return f2_fast(s.h, __fadd_rn(s.l, __fadd_rn(as.l, q.l)));
}

// Jacobian and load of one tet in float-float (scheme S), from the orbit sums:
//   N_a  = sum_k W_k (alpha_k FS_k + delta_k f_{k,a}) + W_3 (c FS_3 + e sum_{P ∋ a} f_P)
//   J_ab = C + h_a + h_b + [a != b] W_3 e^2 g_{ab},  J_aa = C + 2 h_a + D_a
// with f = F, g = F' at the points, FS / GS the orbit sums, C = sum W alpha^2 GS,
// h_a = sum W alpha delta g_{k,a} (+ W_3 c e sum_{P ∋ a} g_P), D_a = sum W delta^2 g_{k,a}
// (+ W_3 e^2 sum_{P ∋ a} g_P): the 14-point sums of w F l_a and w F' l_a l_b regrouped.  The float32 pipes bound
// it (about 2900 operations a tet for the sinh scheme, a third of them the sinh and cosh).
// GB300, 408,000 tets: 77 -> 46 us (with ff_sinh_cosh's table, f2_split's integers and the sums normalised once).
template <int S>
__global__ void __launch_bounds__(ELEM_T) k_element_ff(const double* __restrict__ u, const int* __restrict__ tets,
                                                    int64_t nt, const double* __restrict__ vol, double coef,
                                                    const float4* __restrict__ tab, float2* __restrict__ loc) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double ua[4];
  int umax = 0;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    ua[a] = u[tets[a * nt + t]];
    umax = max(umax, __double2hiint(ua[a]) & 0x7fffffff);
  }
  const double sc = coef * vol[t];
  const f2 s = f2_split(sc);
  if (!(umax < FX_UMAX_HI && fabsf(s.h) <= 1e10f)) {  // |u_q| <= max |u_a| (convex combination)
    element_fallback(S, ua, sc, nt, t, loc);
    return;
  }
  f2 v[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) v[a] = f2_split(ua[a]);
  const f2 su = f2_add(f2_add(v[0], v[1]), f2_add(v[2], v[3]));
  f2 n[4], h[4], D[4], g3[6], T, C;
  {  // S22 orbit: pairs (0,1) (0,2) (0,3) (1,2) (1,3) (2,3); each vertex's pairs summed, then weighted
    const f2 cs = f2_mul(su, PBFB_FFV(OR_C3));
    f2 fs, gs;
#pragma unroll
    for (int p = 0, P = 0; p < 3; ++p)
#pragma unroll
      for (int q = p + 1; q < 4; ++q, ++P) {
        f2 F, G, H;
        ff_scheme<S>(ff_point(cs, f2_add(v[p], v[q]), PBFB_FFV(OR_E3)), tab, F, G, H);
        n[p] = p == 0 && q == 1 ? F : f2_sum(n[p], F);
        h[p] = p == 0 && q == 1 ? G : f2_sum(h[p], G);
        n[q] = p == 0 ? F : f2_sum(n[q], F);
        h[q] = p == 0 ? G : f2_sum(h[q], G);
        g3[P] = f2_mul_raw(G, PBFB_FFV(OR_WEE3));
        fs = P ? f2_sum(fs, F) : F;
        gs = P ? f2_sum(gs, G) : G;
      }
    T = f2_mul_raw(f2_norm(fs), PBFB_FFV(OR_WC3));
    C = f2_mul_raw(f2_norm(gs), PBFB_FFV(OR_WCC3));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const f2 g = f2_norm(h[i]);
      n[i] = f2_mul_raw(f2_norm(n[i]), PBFB_FFV(OR_WE3));
      h[i] = f2_mul_raw(g, PBFB_FFV(OR_WCE3));
      D[i] = f2_mul_raw(g, PBFB_FFV(OR_WEE3));
    }
  }
  // the S31 orbits
  auto orbit = [&](f2 alpha, f2 delta, f2 wa, f2 wd, f2 waa, f2 wad, f2 wdd) {
    const f2 as = f2_mul(su, alpha);
    f2 fs, gs;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f2 F, G, H;
      ff_scheme<S>(ff_point(as, v[i], delta), tab, F, G, H);
      f2_acc(n[i], f2_mul_raw(F, wd));
      f2_acc(h[i], f2_mul_raw(G, wad));
      f2_acc(D[i], f2_mul_raw(G, wdd));
      fs = i ? f2_sum(fs, F) : F;
      gs = i ? f2_sum(gs, G) : G;
    }
    f2_acc(T, f2_mul_raw(f2_norm(fs), wa));
    f2_acc(C, f2_mul_raw(f2_norm(gs), waa));
  };
  orbit(PBFB_FFV(OR_A1), PBFB_FFV(OR_D1), PBFB_FFV(OR_WA1), PBFB_FFV(OR_WD1), PBFB_FFV(OR_WAA1), PBFB_FFV(OR_WAD1),
        PBFB_FFV(OR_WDD1));
  orbit(PBFB_FFV(OR_A2), PBFB_FFV(OR_D2), PBFB_FFV(OR_WA2), PBFB_FFV(OR_WD2), PBFB_FFV(OR_WAA2), PBFB_FFV(OR_WAD2),
        PBFB_FFV(OR_WDD2));
#pragma unroll
  for (int a = 0, P = 0; a < 4; ++a) {
    loc[sym10(a, a) * nt + t] =
        f2_store(f2_mul(s, f2_norm(f2_sum(f2_sum(C, D[a]), f2{2.f * h[a].h, 2.f * h[a].l}))));
#pragma unroll
    for (int b = a + 1; b < 4; ++b, ++P)
      loc[sym10(a, b) * nt + t] = f2_store(f2_mul(s, f2_norm(f2_sum(f2_sum(C, g3[P]), f2_sum(h[a], h[b])))));
    loc[(10 + a) * nt + t] = f2_store(f2_mul(s, f2_norm(f2_sum(T, n[a]))));
  }
}

// Sparse part of the coupled operator: y = S x, L lanes per row (L = 4, 8 or 16).
template <int L>
__global__ void k_spmv(int nrows, const int* __restrict__ ptr, const int* __restrict__ col,
                       const double* __restrict__ val, const double* __restrict__ x, double* __restrict__ y) {
  int lane = threadIdx.x & (L - 1);
  int row = (blockIdx.x * blockDim.x + threadIdx.x) / L;
  const bool valid = row < nrows;  // all lanes reach the shuffles
  double acc = 0.0;
  if (valid)
    for (int k = ptr[row] + lane; k < ptr[row + 1]; k += L) acc += val[k] * __ldg(&x[col[k]]);
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o, L);
  if (lane == 0 && valid) y[row] = acc;
}

// Generic CSR y (+)= A x, 8 lanes per row.
__global__ void k_csr_acc(int nrows, const int* __restrict__ ptr, const int* __restrict__ col,
                          const double* __restrict__ val, const double* __restrict__ x, double* __restrict__ y,
                          int accumulate) {
  int lane = threadIdx.x & 7;
  int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 3;
  const bool valid = row < nrows;  // all lanes reach the shuffles
  double acc = 0.0;
  if (valid)
    for (int k = ptr[row] + lane; k < ptr[row + 1]; k += 8) acc += val[k] * x[col[k]];
  acc += __shfl_down_sync(0xffffffffu, acc, 4, 8);
  acc += __shfl_down_sync(0xffffffffu, acc, 2, 8);
  acc += __shfl_down_sync(0xffffffffu, acc, 1, 8);
  if (lane == 0 && valid) y[row] = accumulate ? y[row] + acc : acc;
}

// one omega of a tet with a value or a step past the orbit sums' range
__device__ __noinline__ void omega_wide(int scheme, const double* ua4, const double* da4, double om, double sc, int64_t nt,
                                        int64_t t, double* __restrict__ out) {
  const double ua[4] = {ua4[0], ua4[1], ua4[2], ua4[3]}, da[4] = {da4[0], da4[1], da4[2], da4[3]};
  double R0[4], R1[4], R2[4];
  omega_sums_f64(scheme, ua, da, om, R0, R1, R2);
  for (int a = 0; a < 4; ++a) {
    out[(0 * 4 + a) * nt + t] = sc * R0[a];
    out[(1 * 4 + a) * nt + t] = sc * R1[a];
    out[(2 * 4 + a) * nt + t] = sc * R2[a];
  }
}

// Omega batch in float64: per tet and omega, local load of F(w), of F'(w) du and of F''(w) du^2 at w = u + omega du
// from orbit sums; layout ((o * 3 + quantity) * 4 + a) * nt + t.  The float64 pipe bounds it.
// GB300, 86,400 tets, one omega: 135 us point by point, 83 us so.
template <int S>
__global__ void __launch_bounds__(128) k_omega_f64(const double* __restrict__ u, const double* __restrict__ du,
                                                   OmegaSet omegas, int nomega, const int* __restrict__ tets,
                                                   int64_t nt, const double* __restrict__ vol, double coef,
                                                   const double* __restrict__ tab, double* __restrict__ loc) {
  constexpr double A1 = PBFB_T_A1, D1 = PBFB_T_B1 - PBFB_T_A1, A2 = PBFB_T_A2, D2 = PBFB_T_B2 - PBFB_T_A2;
  constexpr double C3 = PBFB_T_C3, E3 = PBFB_T_D3 - PBFB_T_C3, W1 = PBFB_T_W1, W2 = PBFB_T_W2, W3 = PBFB_T_W3;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double ua[4], d[4];
  int dmax = 0;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int vtx = tets[a * nt + t];
    ua[a] = u[vtx];
    d[a] = du[vtx];
    dmax = max(dmax, abs_hi(d[a]));
  }
  const double sd = (d[0] + d[1]) + (d[2] + d[3]), s = coef * vol[t];
  for (int o = 0; o < nomega; ++o) {
    double* out = loc + (int64_t)o * 12 * nt;
    double w[4], n[3][4], T[3];
    int wmax = dmax;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      w[a] = fma(omegas.v[o], d[a], ua[a]);
      wmax = max(wmax, abs_hi(w[a]));
    }
    if (wmax >= ORBIT_MAX_HI) {
      omega_wide(S, ua, d, omegas.v[o], s, nt, t, out);
      continue;
    }
    const double sw = (w[0] + w[1]) + (w[2] + w[3]);
    auto point = [&](double wq, double dq, double (&x)[3]) {
      double G, H;
      scheme_f64<S>(wq, tab, x[0], G, H);
      x[1] = G * dq;
      x[2] = H * dq * dq;
    };
    {
      double sum[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int a = 0; a < 4; ++a) n[k][a] = 0.0;
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = p + 1; q < 4; ++q) {
          double x[3];
          point(fma(E3, w[p] + w[q], C3 * sw), fma(E3, d[p] + d[q], C3 * sd), x);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            n[k][p] += x[k];
            n[k][q] += x[k];
            sum[k] += x[k];
          }
        }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        T[k] = W3 * C3 * sum[k];
#pragma unroll
        for (int a = 0; a < 4; ++a) n[k][a] *= W3 * E3;
      }
    }
    auto orbit = [&](double alpha, double delta, double wt) {
      double sum[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        double x[3];
        point(fma(delta, w[a], alpha * sw), fma(delta, d[a], alpha * sd), x);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          n[k][a] = fma(wt * delta, x[k], n[k][a]);
          sum[k] += x[k];
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) T[k] = fma(wt * alpha, sum[k], T[k]);
    };
    orbit(A1, D1, W1);
    orbit(A2, D2, W2);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int a = 0; a < 4; ++a) out[(k * 4 + a) * nt + t] = s * (T[k] + n[k][a]);
  }
}

// Out-of-range omegas of a tet take the float64 loads (kept out of line).
__device__ __noinline__ void omega_fallback(int scheme, const double* ua4, const double* da4, double om, double sc,
                                            int64_t nt, int64_t t, float2* __restrict__ loc) {
  const double ua[4] = {ua4[0], ua4[1], ua4[2], ua4[3]}, da[4] = {da4[0], da4[1], da4[2], da4[3]};
  double R0[4], R1[4], R2[4];
  omega_sums_f64(scheme, ua, da, om, R0, R1, R2);
  for (int a = 0; a < 4; ++a) {
    loc[(0 * 4 + a) * nt + t] = f2_store(f2_split(sc * R0[a]));
    loc[(1 * 4 + a) * nt + t] = f2_store(f2_split(sc * R1[a]));
    loc[(2 * 4 + a) * nt + t] = f2_store(f2_split(sc * R2[a]));
  }
}

// Omega batch in float-float (scheme S): per tet and omega the loads of F(w), F'(w) d and F''(w) d^2 at
// w = u + omega du, each T + n_a from orbit sums (see k_element_ff); same layout as k_omega_f64.
// GB300, 408,000 tets, one omega: 106 -> 59 us.
template <int S>
__global__ void __launch_bounds__(ELEM_T) k_omega_ff(const double* __restrict__ u, const double* __restrict__ du,
                                                  OmegaSet omegas, int nomega, const int* __restrict__ tets,
                                                  int64_t nt, const double* __restrict__ vol, double coef,
                                                  const float4* __restrict__ tab, float2* __restrict__ loc) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double ua[4], da[4];
  f2 d[4];
  float dmax = 0.f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int vtx = tets[a * nt + t];
    ua[a] = u[vtx];
    da[a] = du[vtx];
    d[a] = f2_split(da[a]);
    dmax = fmaxf(dmax, fabsf(d[a].h));
  }
  const double sc = coef * vol[t];
  const f2 s = f2_split(sc);
  const bool scale_ok = fabsf(s.h) * (1.f + dmax) * (1.f + dmax) <= 1e10f;
  const f2 sd = f2_add(f2_add(d[0], d[1]), f2_add(d[2], d[3]));
  for (int o = 0; o < nomega; ++o) {
    const double om = omegas.v[o];
    float2* out = loc + (int64_t)o * 12 * nt;
    int wmax = 0;
    f2 w[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const double wa = fma(om, da[a], ua[a]);
      wmax = max(wmax, __double2hiint(wa) & 0x7fffffff);
      w[a] = f2_split(wa);
    }
    if (!(wmax < FX_UMAX_HI && scale_ok)) {
      omega_fallback(S, ua, da, om, sc, nt, t, out);
      continue;
    }
    const f2 sw = f2_add(f2_add(w[0], w[1]), f2_add(w[2], w[3]));
    f2 n[3][4], T[3], sum[3];
    // x = (F, F' d, F'' d^2) at one point
    auto point = [&](f2 wq, f2 dq, f2 (&x)[3]) {
      f2 F, G, H;
      ff_scheme<S>(wq, tab, F, G, H);
      x[0] = F;
      x[1] = f2_mul(G, dq);
      x[2] = f2_mul(f2_mul(H, dq), dq);
    };
    {  // S22 orbit: each vertex's pairs summed, then weighted
      const f2 cw = f2_mul(sw, PBFB_FFV(OR_C3)), cd = f2_mul(sd, PBFB_FFV(OR_C3));
#pragma unroll
      for (int p = 0, P = 0; p < 3; ++p)
#pragma unroll
        for (int q = p + 1; q < 4; ++q, ++P) {
          f2 x[3];
          point(ff_point(cw, f2_add(w[p], w[q]), PBFB_FFV(OR_E3)), ff_point(cd, f2_add(d[p], d[q]), PBFB_FFV(OR_E3)),
                x);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            n[k][p] = p == 0 && q == 1 ? x[k] : f2_sum(n[k][p], x[k]);
            n[k][q] = p == 0 ? x[k] : f2_sum(n[k][q], x[k]);
            sum[k] = P ? f2_sum(sum[k], x[k]) : x[k];
          }
        }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        T[k] = f2_mul_raw(f2_norm(sum[k]), PBFB_FFV(OR_WC3));
#pragma unroll
        for (int i = 0; i < 4; ++i) n[k][i] = f2_mul_raw(f2_norm(n[k][i]), PBFB_FFV(OR_WE3));
      }
    }
    auto orbit = [&](f2 alpha, f2 delta, f2 wa, f2 wd) {  // the S31 orbits
      const f2 aw = f2_mul(sw, alpha), ad = f2_mul(sd, alpha);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        f2 x[3];
        point(ff_point(aw, w[i], delta), ff_point(ad, d[i], delta), x);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          f2_acc(n[k][i], f2_mul_raw(x[k], wd));
          sum[k] = i ? f2_sum(sum[k], x[k]) : x[k];
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) f2_acc(T[k], f2_mul_raw(f2_norm(sum[k]), wa));
    };
    orbit(PBFB_FFV(OR_A1), PBFB_FFV(OR_D1), PBFB_FFV(OR_WA1), PBFB_FFV(OR_WD1));
    orbit(PBFB_FFV(OR_A2), PBFB_FFV(OR_D2), PBFB_FFV(OR_WA2), PBFB_FFV(OR_WD2));
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int a = 0; a < 4; ++a) out[(k * 4 + a) * nt + t] = f2_store(f2_mul(s, f2_norm(f2_sum(T[k], n[k][a]))));
  }
}

constexpr int RED_T = 256;

// Block sums of NV values per thread (NV <= 8).  A warp's lanes halve the values among them as they halve the lanes
// (xor 16: four sums a lane of eight values, xor 8: two, ...): 9 float64 additions a lane instead of 5 NV, which on
// this float64 pipe were the larger part of k_omega_dots.
template <int NV>
__device__ __forceinline__ void block_reduce_store(double (&v)[NV], double* out) {
  constexpr int P = NV == 1 ? 1 : (NV == 2 ? 2 : (NV <= 4 ? 4 : 8));
  __shared__ double sh[RED_T / 32][P];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double x[P];
#pragma unroll
  for (int k = 0; k < P; ++k) x[k] = k < NV ? v[k < NV ? k : 0] : 0.0;
  int o = 16;
#pragma unroll
  for (int h = P / 2; h > 0; h /= 2, o /= 2) {
    const bool up = lane & o;  // keeps the upper half of the values
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const double give = up ? x[k] : x[k + h], keep = up ? x[k + h] : x[k];
      x[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  for (; o > 0; o >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
  // value k is with the lanes whose upper log2(P) bits are k
  if (lane % (32 / P) == 0) sh[wid][lane / (32 / P)] = x[0];
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0.0;
    for (int w = 0; w < RED_T / 32; ++w) s += sh[w][threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// Per vertex: gather N(w), J(w) du, N''(w)[du,du] for one omega and accumulate the
// seven FEM-row dot products; one partial row of 7 per block.  FF: the tet-local entries are
// float-float pairs (summed in float-float, converted once per vertex).  The last row of blocks takes the three
// dots without an omega: p.c and c.c over the surface rows, p.p over all rows.  DL lanes a vertex.
// GB300, one omega: 72,036 vertices 21 -> 15 us, and 8 -> 3 us for the partials (a warp a column), without the
// three separate dots; 5202 vertices 6.2 us (DL = 1: 8.2).
template <bool FF, int DL>
__global__ void __launch_bounds__(RED_T) k_omega_dots(int nv, int n, const int* __restrict__ ptr,
                                                      const int* __restrict__ idx, const double* __restrict__ loc,
                                                      int64_t nt, const double* __restrict__ c,
                                                      const double* __restrict__ p, double* __restrict__ part) {
  int o = blockIdx.y;
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  if (o + 1 == gridDim.y) {
    for (int i = blockIdx.x * RED_T + threadIdx.x; i < n; i += gridDim.x * RED_T) {
      const double pi = p[i];
      acc[2] += pi * pi;
      if (i >= nv) {
        const double ci = c[i];
        acc[0] += pi * ci;
        acc[1] += ci * ci;
      }
    }
    block_reduce_store<7>(acc, part + ((int64_t)o * gridDim.x + blockIdx.x) * 7);
    return;
  }
  const double* L = loc + (int64_t)o * 12 * nt;
  const float2* L2 = reinterpret_cast<const float2*>(L);
  constexpr int GBD = DL == 1 ? GB : 6;
  const int lane = threadIdx.x % DL;
  const int nv_up = (nv + RED_T / DL - 1) / (RED_T / DL) * (RED_T / DL);  // whole warps in the shuffles
  for (int i = (blockIdx.x * RED_T + threadIdx.x) / DL; i < nv_up; i += gridDim.x * (RED_T / DL)) {
    const int k1 = i < nv ? ptr[i + 1] : 0;
    const int kb = i < nv ? ptr[i] + lane : 0;
    double nn[3] = {0, 0, 0};
    f2 a[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    for (int k0 = kb; k0 < k1; k0 += DL * GBD) {
      int e[GBD];
#pragma unroll
      for (int j = 0; j < GBD; ++j) e[j] = k0 + DL * j < k1 ? idx[k0 + DL * j] : -1;
      if (FF) {
        float2 x[3][GBD];
#pragma unroll
        for (int j = 0; j < GBD; ++j)
#pragma unroll
          for (int q = 0; q < 3; ++q) x[q][j] = e[j] >= 0 ? L2[4 * q * nt + e[j]] : make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < GBD; ++j)
#pragma unroll
          for (int q = 0; q < 3; ++q) a[q] = f2_add(a[q], f2{x[q][j].x, x[q][j].y});
      } else {
        double x[3][GBD];
#pragma unroll
        for (int j = 0; j < GBD; ++j)
#pragma unroll
          for (int q = 0; q < 3; ++q) x[q][j] = e[j] >= 0 ? L[4 * q * nt + e[j]] : 0.0;
#pragma unroll
        for (int j = 0; j < GBD; ++j)
#pragma unroll
          for (int q = 0; q < 3; ++q) nn[q] += x[q][j];
      }
    }
#pragma unroll
    for (int sh = 1; sh < DL; sh *= 2)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (FF)
          a[q] = f2_add(a[q], f2{__shfl_xor_sync(0xffffffffu, a[q].h, sh), __shfl_xor_sync(0xffffffffu, a[q].l, sh)});
        else
          nn[q] += __shfl_xor_sync(0xffffffffu, nn[q], sh);
      }
    if (lane || i >= nv) continue;
    if (FF)
      for (int q = 0; q < 3; ++q) nn[q] = f2_val(a[q]);
    double r = c[i] - nn[0], rp = -nn[1], rpp = -nn[2], pi = p[i];
    acc[0] += pi * r;     // p.r
    acc[1] += rp * r;     // r'.r
    acc[2] += rp * pi;    // r'.p
    acc[3] += rp * rp;    // r'.r'
    acc[4] += r * rpp;    // r.r''
    acc[5] += pi * rpp;   // p.r''
    acc[6] += r * r;      // r.r
  }
  block_reduce_store<7>(acc, part + ((int64_t)o * gridDim.x + blockIdx.x) * 7);
}

// Sum nb partial rows of width w (for each of gridDim.x problems), fixed order (one warp per problem and column)
__global__ void k_sum_partials(const double* __restrict__ part, int nb, int w, double* __restrict__ out) {
  const int o = blockIdx.x, k = threadIdx.x >> 5;
  const double s = warp_strided_sum(part + (int64_t)o * nb * w + k, nb, w);
  if ((threadIdx.x & 31) == 0) out[o * w + k] = s;
}

// Block partials of sum_t |T| sum_q W_q (u sinh u - 2 cosh u + 2) for u = u1 + u2 (even in u).  The float64 pipe
// bounds it: the points' values come from the rule's orbits (26 operations a tet for 14 points), e^u and e^-u
// from one reduction (exp_pm), no division.  GB300, 184,320 tets: 165 us with the library's exponential, a
// division and four products a point; 105 us so.
__global__ void __launch_bounds__(RED_T) k_ion_energy(const double* __restrict__ u1, const double* __restrict__ u2,
                                                      const int* __restrict__ tets, int64_t nt,
                                                      const double* __restrict__ vol, const double* __restrict__ tab,
                                                      double* __restrict__ part) {
  double acc[1] = {0.0};
  for (int64_t t = blockIdx.x * (int64_t)RED_T + threadIdx.x; t < nt; t += (int64_t)gridDim.x * RED_T) {
    double u[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int v = tets[a * nt + t];
      u[a] = u1[v] + u2[v];
    }
    const double su = (u[0] + u[1]) + (u[2] + u[3]);
    auto f = [&](double uq) {
      const double a = fabs(uq);
      double ep, em;
      exp_pm(a, tab, ep, em);
      return fma(0.5 * a, ep - em, 2.0 - (ep + em));
    };
    double s1 = 0.0, s2 = 0.0, s3 = 0.0;
    const double as1 = PBFB_T_A1 * su, as2 = PBFB_T_A2 * su, cs = PBFB_T_C3 * su;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s1 += f(fma(PBFB_T_B1 - PBFB_T_A1, u[i], as1));
      s2 += f(fma(PBFB_T_B2 - PBFB_T_A2, u[i], as2));
    }
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = p + 1; q < 4; ++q) s3 += f(fma(PBFB_T_D3 - PBFB_T_C3, u[p] + u[q], cs));
    acc[0] = fma(vol[t], fma(PBFB_T_W3, s3, fma(PBFB_T_W2, s2, PBFB_T_W1 * s1)), acc[0]);
  }
  block_reduce_store<1>(acc, part + blockIdx.x);
}

// Values of the sparse operator with J = 0 from the slot descriptors.
__global__ void k_fill_operator(int nnz, const int* __restrict__ kind, const int* __restrict__ ref,
                                const double* __restrict__ a1, const double* __restrict__ a1m, double eps_m,
                                double eps_s,
                                const double* __restrict__ mass_m, const double* __restrict__ corrV_m,
                                const double* __restrict__ corrK_m, const double* __restrict__ mass_s,
                                const double* __restrict__ corrV_s, const double* __restrict__ corrK_s,
                                double* __restrict__ base) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nnz) return;
  int r = ref[s];
  double v = 0.0;
  switch (kind[s]) {
    case 0: v = eps_s * a1[s] + (a1m ? eps_m * a1m[s] : 0.0); break;  // stiffness (Omega_i, Omega_m)
    case 1: v = eps_m * mass_m[r]; break;                      // eps_m R_m' M_m
    case 2: v = -eps_s * mass_s[r]; break;                     // -eps_s R_s' M_s
    case 3: v = 0.5 * mass_m[r] + corrK_m[r]; break;           // (M_m/2 + K_L) near part
    case 4: v = -corrV_m[r]; break;                            // -V_L near part
    case 5: v = 0.5 * mass_s[r] - corrK_s[r]; break;           // (M_s/2 - K_Y) near part
    case 6: v = corrV_s[r]; break;                             // V_Y near part
    case 7: v = 1.0; break;                                    // lam_m rows of Eq. fembem_matrix's
                                                               // solve (Gamma_m interior)
  }
  base[s] = v;
}

inline int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

int launch_tet_volumes(Mesh* m, const int* tets, int64_t nt, double* vol) {
  if (nt == 0) return PBFB_OK;
  k_tet_volumes<<<blocks_for(nt, 256), 256, 0, m->stream>>>(m->xyz.p, m->nv, tets, nt, vol);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_stiffness_local(Mesh* m, const int* tets, int64_t nt, const double* vol, double* loc10) {
  if (nt == 0) return PBFB_OK;
  k_stiffness_local<<<blocks_for(nt, 256), 256, 0, m->stream>>>(m->xyz.p, m->nv, tets, nt, vol, loc10);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_gather(Mesh* m, int nslots, const int* ptr, const int* idx, const double* local, const double* base,
                  double scale, double* out) {
  if (nslots == 0) return PBFB_OK;
  k_gather<<<blocks_for(nslots, 256), 256, 0, m->stream>>>(nslots, ptr, idx, local, base, scale, out);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_assemble_gather(Mesh* m, bool ff, double* N_out) {
  if (!ff) {
    PB_TRY(launch_gather(m, m->snnz, m->jg_ptr.p, m->jg_idx.p, m->tloc.p, m->s_base.p, 1.0, m->s_val.p));
    if (N_out)
      PB_TRY(launch_gather(m, m->nv, m->ng_ptr.p, m->ng_idx.p, m->tloc.p + 10 * m->nt, nullptr, 1.0, N_out));
    return PBFB_OK;
  }
  const float2* loc = reinterpret_cast<const float2*>(m->tloc.p);
  const int nn = N_out ? m->nv : 0;
  k_gather_ff<<<blocks_for((int64_t)m->snnz + nn, 256), 256, 0, m->stream>>>(
      m->snnz, m->jg_ptr.p, m->jg_idx.p, loc, m->s_base.p, m->s_val.p, nn, m->ng_ptr.p, m->ng_idx.p,
      loc + 10 * m->nt, N_out);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

// float-float tables of ff_sinh_cosh (uploaded once per mesh)
static int fx_table(Mesh* m) {
  if (m->fx_tab.n) return PBFB_OK;
  static const std::vector<float4> tab = [] {
    std::vector<float4> t(2 * FX_N);
    auto split = [](double v, float& h, float& l) {
      h = (float)v;
      l = (float)(v - (double)h);
    };
    for (int j = 0; j < FX_N; ++j) {
      const double v = j * FX_STEP;
      split(std::sinh(v), t[j].x, t[j].y);
      split(std::cosh(v), t[j].z, t[j].w);
      split(std::exp2((double)j / FX_N), t[FX_N + j].x, t[FX_N + j].y);
      split(std::exp2(-(double)j / FX_N), t[FX_N + j].z, t[FX_N + j].w);
    }
    return t;
  }();
  return m->fx_tab.upload(tab.data(), tab.size(), m->stream);
}

// The mixed precision runs the element kernels in float-float, the float64 precision in float64.
static bool use_ff(const Mesh* m, int scheme) {
  return m->precision != PBFB_FP64 && scheme >= PBFB_LINEAR && scheme <= PBFB_T7;
}

// f(integral_constant) of the scheme
template <class F>
static void with_scheme(int scheme, F f) {
  switch (scheme) {
    case PBFB_LINEAR: f(std::integral_constant<int, PBFB_LINEAR>()); break;
    case PBFB_T3: f(std::integral_constant<int, PBFB_T3>()); break;
    case PBFB_T5: f(std::integral_constant<int, PBFB_T5>()); break;
    case PBFB_T7: f(std::integral_constant<int, PBFB_T7>()); break;
    default: f(std::integral_constant<int, PBFB_HS>()); break;
  }
}

int launch_element_nl(Mesh* m, int scheme, const double* u, double coef, double* loc, bool* ff) {
  cudaEvent_t ev;
  *ff = use_ff(m, scheme);
  PB_TRY(*ff ? fx_table(m) : pair_tables(m, true));
  timer_begin(m, m->t_elem, &ev);
  with_scheme(scheme, [&](auto S) {
    if (*ff)
      k_element_ff<S()><<<blocks_for(m->nt, ELEM_T), ELEM_T, 0, m->stream>>>(
          u, m->tets.p, m->nt, m->vol.p, coef, m->fx_tab.p, reinterpret_cast<float2*>(loc));
    else
      k_element_f64<S()><<<blocks_for(m->nt, 128), 128, 0, m->stream>>>(u, m->tets.p, m->nt, m->vol.p, coef,
                                                                        m->pair_tab64.p, loc);
  });
  PB_LAUNCHED(m);
  timer_end(m, m->t_elem, ev, (double)m->nt);
  return PBFB_OK;
}

int launch_spmv(Mesh* m, const double* x, double* y) {
  cudaEvent_t ev;
  timer_begin(m, m->t_spmv, &ev);
  int n = m->n;
  const int L = m->spmv_lanes > 0 ? m->spmv_lanes : 8;
  const int B = m->spmv_block > 0 ? m->spmv_block : 256;
  const int g = blocks_for((int64_t)n * L, B);
  if (L == 4)
    k_spmv<4><<<g, B, 0, m->stream>>>(n, m->s_ptr.p, m->s_col.p, m->s_val.p, x, y);
  else if (L == 16)
    k_spmv<16><<<g, B, 0, m->stream>>>(n, m->s_ptr.p, m->s_col.p, m->s_val.p, x, y);
  else
    k_spmv<8><<<g, B, 0, m->stream>>>(n, m->s_ptr.p, m->s_col.p, m->s_val.p, x, y);
  PB_LAUNCHED(m);
  timer_end(m, m->t_spmv, ev, (double)m->snnz);
  return PBFB_OK;
}

int launch_csr_spmv(Mesh* m, int nrows, const int* ptr, const int* col, const double* val, const double* x,
                    double* y, bool accumulate) {
  if (nrows == 0) return PBFB_OK;
  k_csr_acc<<<blocks_for((int64_t)nrows * 8, 256), 256, 0, m->stream>>>(nrows, ptr, col, val, x, y,
                                                                        accumulate ? 1 : 0);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_omega_elements(Mesh* m, int scheme, const double* u, const double* du, const double* omegas_host,
                          int nomega, double coef, double* loc, bool* ff) {
  cudaEvent_t ev;
  *ff = use_ff(m, scheme);
  PB_TRY(*ff ? fx_table(m) : pair_tables(m, true));
  OmegaSet omegas;
  for (int o = 0; o < OMEGA_MAX; ++o) omegas.v[o] = o < nomega ? omegas_host[o] : 0.0;
  timer_begin(m, m->t_elem, &ev);
  with_scheme(scheme, [&](auto S) {
    if (*ff)
      k_omega_ff<S()><<<blocks_for(m->nt, ELEM_T), ELEM_T, 0, m->stream>>>(
          u, du, omegas, nomega, m->tets.p, m->nt, m->vol.p, coef, m->fx_tab.p, reinterpret_cast<float2*>(loc));
    else
      k_omega_f64<S()><<<blocks_for(m->nt, 128), 128, 0, m->stream>>>(u, du, omegas, nomega, m->tets.p, m->nt,
                                                                      m->vol.p, coef, m->pair_tab64.p, loc);
  });
  PB_LAUNCHED(m);
  timer_end(m, m->t_elem, ev, (double)m->nt * nomega);
  return PBFB_OK;
}

int launch_omega_dots(Mesh* m, int nomega, const double* loc, const double* c, const double* p, double* dots_dev,
                      bool ff) {
  // Two lanes a vertex while one block an SM holds them (72,036 vertices: 19.9 us against 15.2 with one lane; 5202:
  // 6.2 against 8.2); blocks for one omega: 4 an SM at most, an SM each from 4 omegas on (m->red holds 152 * 65).
  const int dl = 2 * m->n <= 152 * RED_T ? 2 : 1;
  const int nb = std::min(blocks_for((int64_t)dl * m->n, RED_T), 152 * std::max(1, 4 / nomega));
  dim3 grid(nb, nomega + 1);
  auto k = ff ? (dl == 2 ? k_omega_dots<true, 2> : k_omega_dots<true, 1>)
              : (dl == 2 ? k_omega_dots<false, 2> : k_omega_dots<false, 1>);
  k<<<grid, RED_T, 0, m->stream>>>(m->nv, m->n, m->ng_ptr.p, m->ng_idx.p, loc, m->nt, c, p, m->red.p);
  PB_LAUNCHED(m);
  k_sum_partials<<<nomega + 1, 32 * 7, 0, m->stream>>>(m->red.p, nb, 7, dots_dev);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_ion_energy(Mesh* m, const double* u1, const double* u2, double* out_dev) {
  const int nb = 4 * 152;  // 4 blocks an SM
  PB_TRY(pair_tables(m, true));
  k_ion_energy<<<nb, RED_T, 0, m->stream>>>(u1, u2, m->tets.p, m->nt, m->vol.p, m->pair_tab64.p, m->red.p);
  PB_LAUNCHED(m);
  return launch_sum_partials(m, nb, 1, out_dev);
}

int launch_sum_partials(Mesh* m, int nb, int w, double* out_dev) {
  k_sum_partials<<<1, 32 * w, 0, m->stream>>>(m->red.p, nb, w, out_dev);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_fill_operator(Mesh* m) {
  k_fill_operator<<<blocks_for(m->snnz, 256), 256, 0, m->stream>>>(
      m->snnz, m->s_kind.p, m->s_ref.p, m->a1.p, m->full ? m->a1m.p : nullptr, m->eps_m, m->eps_s, m->sm.mass.p, m->sm.corrV.p, m->sm.corrK.p,
      m->ss.mass.p, m->ss.corrV.p, m->ss.corrK.p, m->s_base.p);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

}  // namespace pbfb
