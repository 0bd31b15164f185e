// Direct far fields of the accurate precisions, by pairs of triangles: the quadrature-point sum
//   phi(x_i) = sum_{j != i} [ s_j + m_j . (x_i - y_j) (1 + kappa r) / r^2 ] exp(-kappa r) / r
// in float64 (PBFB_FP64) and in float-float arithmetic on the float32 pipes (PBFB_FLOAT2).
//
// What bounds these sums is the arithmetic per pair of points (the data of a whole surface are a few
// MB), so the kernels are built to need few operations per pair:
//   - every unordered pair of points is evaluated once for both directions: with g = exp(-kappa r) / r
//     and h = (1 + kappa r) exp(-kappa r) / r^3 it adds s_j g + m_j . (x_i - y_j) h to target i and
//     s_i g - m_i . (x_i - y_j) h to target j;
//   - the six points of a flat triangle share their normal, m_j = mu_j n_b, and n_b . (x - y_j) is the
//     distance D_b(x) of x from the triangle's plane whatever j: it is computed once per (point,
//     triangle), and the dipole part of a triangle is D_b(x) sum_j mu_j h_j.  Per pair of points that
//     leaves two products per direction, s g and mu h, instead of a three-term dot product and three;
//   - 1/r, 1/r^2 and 1/r^3 come from one hardware estimate y0 and one correction z = r^2 y0^2 - 1.
// A lane of a warp owns one target triangle, its NP packed pairs (float-float) or NQ points (float64)
// in registers, and walks over the source triangles of a tile of 32 held in the warp's own shared
// memory: at step k lane l takes triangle (l + k) mod 32, so the lanes add to different source-side
// sums (no atomics, fixed order, warp-synchronous).  Triangle tiles form G groups; a task is a pair of
// groups (rg <= cg), one of K parts of the 32 steps and, when a lane owns fewer than its triangle's six
// points, one share of them; it writes its own rows of partial sums, added in a fixed order by
// k_pairs_sum.  Tiles on the diagonal (I = J) are summed one-directionally with the coincident point
// masked.
//
// Measured on GB300 (one operator product, Laplace and Yukawa surface): float-float, 8000 triangles a
// surface, 7.58 + 11.12 ms for mutual pairs of points with a dipole vector each (97.7 and 145.7 float32 lane
// operations per ordered pair) to 3.9 + 5.7 ms (58 and 82 counted in the source; 82 to 86 % of the float32
// pipes' rate); float64, 3380 triangles, 14.9 + 33.6 ms one-directionally with the library's root and
// exponential to 7.0 + 11.6 ms (9.3 and 13.3 float64 operations per ordered pair counted in the source; the float64
// pipe 88 to 90 % busy).  Errors of V and K: float64 against long double (320 triangles) 0.9e-16 to 1.2e-16 (V, from
// 1.5e-16 to 2.1e-16) and 1.4e-16 to 1.8e-16 (K, from 3.4e-16 to 6.1e-16); float-float against 64 bits 2.5e-15 (V, from
// 4e-15) and 1.1e-14 (K, from 2e-14 to 7e-14).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "device_once.h"
#include "f32x2.cuh"
#include "fp64_math.cuh"
#include "pair_split.h"
#include "pbfb_internal.cuh"
#include "quad_tables.cuh"

namespace pbfb {

namespace {

constexpr int PT = PAIR_TILE;        // triangles per tile: one per lane
constexpr int PW = 4;                // warps (independent tasks) per block
constexpr int FF_GEO = 48;           // float rows of a tile: 18 hi, 18 lo coordinates, 3 hi, 3 lo normals, 6 plane offsets
constexpr int FF_SRC = 24;           // s hi, s lo, mu hi, mu lo of the 6 points
constexpr int D_GEO = 21;            // float64 rows: 18 coordinates, 3 normals
constexpr int D_SRC = 12;            // s, mu
constexpr int FF_HI = 657;           // exp(-k / 16): arguments are cut at 41, entries from 640 (x = 40) are 0
constexpr int FF_LO = 64;            // exp(-k / 1024)

// ---- float-float on pairs of float32 (per component the scalar operations' rounding)
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __fadd2_rn(a, neg(b)); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma_(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// an unevaluated sum h + l, |l| a few units of h's last place (not renormalised unless said)
template <class V>
struct Ff {
  V h, l;
};

template <class V>
__device__ __forceinline__ Ff<V> two_sum(V a, V b) {  // exact, Knuth
  const V s = add(a, b), bb = sub(s, a);
  return {s, add(sub(a, sub(s, bb)), sub(b, bb))};
}
template <class V>
__device__ __forceinline__ Ff<V> quick_sum(V a, V b) {  // exact for |a| >= |b|, Dekker
  const V s = add(a, b);
  return {s, sub(b, sub(s, a))};
}
// product, low part not renormalised
template <class V>
__device__ __forceinline__ Ff<V> prod(V ah, V al, V bh, V bl) {
  const V p = mul(ah, bh);
  return {p, fma_(al, bh, fma_(ah, bl, fma_(ah, bh, neg(p))))};
}
template <class V>
__device__ __forceinline__ void accumulate(Ff<V>& s, Ff<V> p) {
  const Ff<V> t = two_sum(s.h, p.h);
  s.h = t.h;
  s.l = add(s.l, add(t.l, p.l));
}
// a . b for a unit normal a and a difference vector b, renormalised components
template <class V>
__device__ __forceinline__ Ff<V> dot3(const V (&ah)[3], const V (&al)[3], const Ff<V> (&b)[3]) {
  const Ff<V> p0 = prod(ah[0], al[0], b[0].h, b[0].l), p1 = prod(ah[1], al[1], b[1].h, b[1].l),
              p2 = prod(ah[2], al[2], b[2].h, b[2].l);
  const Ff<V> s1 = two_sum(p0.h, p1.h), s2 = two_sum(s1.h, p2.h);
  return {s2.h, add(add(s1.l, s2.l), add(add(p0.l, p1.l), p2.l))};
}
__device__ __forceinline__ Ff<float2> norm2(const Ff<float2> (&d)[3]) {
  const float2 p0 = mul(d[0].h, d[0].h), p1 = mul(d[1].h, d[1].h), p2 = mul(d[2].h, d[2].h);
  const float2 e0 = fma_(d[0].h, d[0].h, neg(p0)), e1 = fma_(d[1].h, d[1].h, neg(p1)),
               e2 = fma_(d[2].h, d[2].h, neg(p2));
  const float2 c = fma_(d[2].h, d[2].l, fma_(d[1].h, d[1].l, mul(d[0].h, d[0].l)));
  const Ff<float2> s1 = two_sum(p0, p1), s2 = two_sum(s1.h, p2);
  return {s2.h, fma_(dup(2.f), c, add(add(s1.l, s2.l), add(add(e0, e1), e2)))};
}

// exp(-(xh + xl)), 0 <= xh, from tables of exp(-k / 16) and exp(-k / 1024): xh = k / 1024 + f exactly,
// |f| <= 2^-11, and exp(-f - xl) = 1 - f + q with q = -xl + f1^2 (1/2 - f1/6 + f1^2/24), f1 = f + xl
// (truncation 2^-62).  Arguments from 40 on give 0.
__device__ __forceinline__ Ff<float2> exp_neg(float2 xh, float2 xl, const float2* __restrict__ hi,
                                              const float2* __restrict__ lo) {
  const float2 magic = dup(12582912.f);  // 1.5 2^23: the sum's last place is 1
  const float2 x = make_float2(fminf(xh.x, 41.f), fminf(xh.y, 41.f));
  const float2 m = fma_(x, dup(1024.f), magic);
  const float2 kf = sub(m, magic);
  const float2 f = fma_(kf, dup(-1.f / 1024.f), x);
  const int k0 = __float_as_int(m.x) - 0x4B400000, k1 = __float_as_int(m.y) - 0x4B400000;
  const float2 a0 = hi[k0 >> 6], a1 = hi[k1 >> 6], b0 = lo[k0 & 63], b1 = lo[k1 & 63];
  const Ff<float2> T = prod(make_float2(a0.x, a1.x), make_float2(a0.y, a1.y), make_float2(b0.x, b1.x),
                            make_float2(b0.y, b1.y));
  const float2 f1 = add(f, xl);
  const float2 c = fma_(f1, fma_(f1, dup(1.f / 24.f), dup(-1.f / 6.f)), dup(0.5f));
  const float2 q = fma_(mul(f1, f1), c, neg(xl));
  const float2 t = mul(T.h, f), te = fma_(T.h, f, neg(t));
  const float2 E = sub(T.h, t);
  const float2 err = sub(sub(sub(T.h, E), t), te);
  return {E, add(fma_(T.h, q, err), fma_(neg(T.l), f, T.l))};
}

// g and h of a packed pair of targets from their difference vectors; coincident lanes (same) give 0.
// With y0 the hardware estimate of 1/r, t = y0^2 (+ te) and z = r^2 t - 1 (|z| < 2^-21), to z^2:
//   1/r = y0 (1 - z/2 + 3z^2/8), 1/r^2 = t (1 - z + z^2), 1/r^3 = y0 t (1 - 3z/2 + 15z^2/8).
template <bool YUK>
__device__ __forceinline__ void kernel_gh(const Ff<float2> (&d)[3], bool same_x, bool same_y,
                                          const float2* __restrict__ hi, const float2* __restrict__ lo, Ff<float2>& g,
                                          Ff<float2>& h) {
  const Ff<float2> r2 = norm2(d);
  float2 y = make_float2(rsqrt_approx(r2.h.x), rsqrt_approx(r2.h.y));
  if (same_x) y.x = 0.f;
  if (same_y) y.y = 0.f;
  const float2 t = mul(y, y), te = fma_(y, y, neg(t));
  const float2 z = fma_(r2.l, t, fma_(r2.h, te, fma_(r2.h, t, dup(-1.f)))), zz = mul(z, z);
  const float2 yl = mul(mul(y, dup(-0.5f)), fma_(zz, dup(-0.75f), z));
  if (YUK) {
    const Ff<float2> r = prod(r2.h, r2.l, y, yl);
    const Ff<float2> E = exp_neg(r.h, r.l, hi, lo);
    g = prod(y, yl, E.h, E.l);
    // (1 + r) e^-r / r^3 = (1/r^2) (e^-r / r + e^-r)
    const Ff<float2> w = two_sum(g.h, E.h);
    h = prod(t, fma_(neg(t), sub(z, zz), te), w.h, add(w.l, add(g.l, E.l)));
  } else {
    g = {y, yl};
    const float2 p = mul(y, t);
    h = {p, fma_(mul(p, fma_(zz, dup(-1.25f), z)), dup(-1.5f), fma_(y, te, fma_(y, t, neg(p))))};
  }
}

struct PairTask {
  int i0, i1, j0, j1;    // tile ranges of the two groups
  int k0, k1;            // steps of the 32
  int sub, pi, pj;       // share of the target points; rows of PI (targets) and PJ (sources)
  bool diag;
};

// task -> (group pair, part, share).  A point of group g has target sums from the groups c >= g and
// source sums from r <= g.  nsub = 1: both in G + 1 rows a part, c and r < g in the rows of those numbers and
// r = g in row G.  Else PI[part G + c] and PJ[(part nsub + sub) G + r].
__device__ __forceinline__ PairTask pair_task(int task, int nT, int tpg, int G, int K, int nsub) {
  PairTask T;
  T.sub = task % nsub;
  task /= nsub;
  const int part = task % K;
  task /= K;
  int rg = 0;
  while (task >= G - rg) {
    task -= G - rg;
    ++rg;
  }
  const int cg = rg + task;
  T.i0 = rg * tpg;
  T.i1 = min(nT, T.i0 + tpg);
  T.j0 = cg * tpg;
  T.j1 = min(nT, T.j0 + tpg);
  T.k0 = part * (PT / K);
  T.k1 = T.k0 + PT / K;
  T.diag = rg == cg;
  if (nsub == 1) {
    T.pi = part * (G + 1) + cg;
    T.pj = part * (G + 1) + (T.diag ? G : rg);
  } else {
    T.pi = part * G + cg;
    T.pj = (part * nsub + T.sub) * G + rg;
  }
  return T;
}

template <bool YUK, int NP>
__global__ void __launch_bounds__(32 * PW, NP == 3 ? 2 : 3)
    k_pairs_ff(int nt, int ntask, int nT, int tpg, int G, int K, const float* __restrict__ geo,
               const float* __restrict__ src, const float2* __restrict__ tab, double* PI,
               double* PJ) {
  __shared__ __align__(16) float s_tile[PW][(FF_GEO + FF_SRC) * PT];  // filled by float4 stores
  __shared__ float2 s_acc[PW][QS][PT];
  __shared__ float2 s_tab[YUK ? FF_HI + FF_LO : 1];
  if (YUK) {
    for (int k = threadIdx.x; k < FF_HI + FF_LO; k += 32 * PW) s_tab[k] = tab[k];
    __syncthreads();
  }
  const float2* hi = s_tab;
  const float2* lo = s_tab + (YUK ? FF_HI : 0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int task = blockIdx.x * PW + warp;
  if (task >= ntask) return;  // warps are independent from here on
  float* tile = s_tile[warp];
  float2(*acc_j)[PT] = s_acc[warp];
  const int nq = QS * nt;
  const PairTask T = pair_task(task, nT, tpg, G, K, 3 / NP);
  const int q0 = 2 * NP * T.sub;  // first of this lane's points
  for (int I = T.i0; I < T.i1; ++I) {
    const int ta = I * PT + lane;
    const bool va = ta < nt;
    const float* ga = geo + (size_t)I * FF_GEO * PT + lane;
    const float* sa = src + (size_t)I * FF_SRC * PT + lane;
    float2 xh[NP][3], xl[NP][3], ash[NP], asl[NP], amh[NP], aml[NP];
    float nh[3], nl[3];
    float2 ea[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int q = q0 + 2 * p;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        xh[p][c] = make_float2(ga[(6 * c + q) * PT], ga[(6 * c + q + 1) * PT]);
        xl[p][c] = make_float2(ga[(18 + 6 * c + q) * PT], ga[(18 + 6 * c + q + 1) * PT]);
      }
      ea[p] = make_float2(ga[(42 + q) * PT], ga[(43 + q) * PT]);
      if (!va) xh[p][0] = dup(2e15f);  // past the last triangle: far away (padding sources sit at 1e15), no strength
      ash[p] = make_float2(sa[q * PT], sa[(q + 1) * PT]);
      asl[p] = make_float2(sa[(6 + q) * PT], sa[(7 + q) * PT]);
      amh[p] = make_float2(sa[(12 + q) * PT], sa[(13 + q) * PT]);
      aml[p] = make_float2(sa[(18 + q) * PT], sa[(19 + q) * PT]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      nh[c] = ga[(36 + c) * PT];
      nl[c] = ga[(39 + c) * PT];
    }
    double acc[2 * NP];
#pragma unroll
    for (int p = 0; p < 2 * NP; ++p) acc[p] = 0.0;
    for (int J = T.diag ? I : T.j0; J < T.j1; ++J) {
      const bool dg = J == I;
      __syncwarp();
      {
        const float4* gs = reinterpret_cast<const float4*>(geo + (size_t)J * FF_GEO * PT);
        const float4* ss = reinterpret_cast<const float4*>(src + (size_t)J * FF_SRC * PT);
        float4* dst = reinterpret_cast<float4*>(tile);
        for (int e = lane; e < FF_GEO * PT / 4; e += 32) dst[e] = gs[e];
        for (int e = lane; e < FF_SRC * PT / 4; e += 32) dst[FF_GEO * PT / 4 + e] = ss[e];
#pragma unroll
        for (int q = 0; q < QS; ++q) acc_j[q][lane] = make_float2(0.f, 0.f);
      }
      __syncwarp();
      Ff<float2> out[NP];
#pragma unroll
      for (int p = 0; p < NP; ++p) out[p] = {dup(0.f), dup(0.f)};
      for (int k = T.k0; k < T.k1; ++k) {
        const int b = (lane + k) & (PT - 1);
        const float* tb = tile + b;
        const bool own = dg && k == 0;  // the lane's own triangle
        Ff<float2> S[NP], H[NP], Db[NP];
        // Unrolled as far as the instruction cache allows (the Yukawa pair is half as long again), with registers
        // for two blocks an SM: the longer run of independent pairs fills the float32 pipes better than a
        // third block.  8000 triangles, Laplace / Yukawa: not unrolled, three blocks 4.60 / 6.40 ms; 2, three
        // 4.36 / 6.06; 2, two 4.25 / 5.86; 3, two 4.14 / 5.78; 6, two 3.99 / 6.98.
#pragma unroll (YUK ? 3 : 6)
        for (int q = 0; q < QS; ++q) {
          float bh[3], bl[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            bh[c] = tb[(6 * c + q) * PT];
            bl[c] = tb[(18 + 6 * c + q) * PT];
          }
          const float* ts = tb + FF_GEO * PT;
          const float bsh = ts[q * PT], bsl = ts[(6 + q) * PT], bmh = ts[(12 + q) * PT], bml = ts[(18 + q) * PT];
          Ff<float2> Sj, Hj;  // source side: sums over this lane's points
          Ff<float> Da;
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            Ff<float2> d[3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
              d[c] = quick_sum(sub(xh[p][c], dup(bh[c])), sub(xl[p][c], dup(bl[c])));
            if (p == 0) {
              const Ff<float> d1[3] = {{d[0].h.x, d[0].l.x}, {d[1].h.x, d[1].l.x}, {d[2].h.x, d[2].l.x}};
              Da = dot3(nh, nl, d1);  // n_a . (x_i - y_j), whatever i
              Da.l = add(Da.l, sub(ea[0].x, tb[(42 + q) * PT]));
            }
            if (q == 0) {
              const float2 mh[3] = {dup(tb[36 * PT]), dup(tb[37 * PT]), dup(tb[38 * PT])};
              const float2 ml[3] = {dup(tb[39 * PT]), dup(tb[40 * PT]), dup(tb[41 * PT])};
              Db[p] = dot3(mh, ml, d);  // n_b . (x_i - y_j), whatever j
              Db[p].l = add(Db[p].l, sub(ea[p], dup(tb[42 * PT])));
              if (own) Db[p] = {dup(0.f), dup(0.f)};
            }
            Ff<float2> g, h;
            kernel_gh<YUK>(d, own && q == q0 + 2 * p, own && q == q0 + 2 * p + 1, hi, lo, g, h);
            const Ff<float2> sg = prod(g.h, g.l, dup(bsh), dup(bsl)), mh = prod(h.h, h.l, dup(bmh), dup(bml));
            if (q == 0) {
              S[p] = sg;
              H[p] = mh;
            } else {
              accumulate(S[p], sg);
              accumulate(H[p], mh);
            }
            const Ff<float2> sj = prod(g.h, g.l, ash[p], asl[p]), hj = prod(h.h, h.l, amh[p], aml[p]);
            if (p == 0) {
              Sj = sj;
              Hj = hj;
            } else {
              accumulate(Sj, sj);
              accumulate(Hj, hj);
            }
          }
          if (!dg) {
            Ff<float> s = two_sum(Sj.h.x, Sj.h.y), m = two_sum(Hj.h.x, Hj.h.y);
            s.l = add(s.l, add(Sj.l.x, Sj.l.y));
            m.l = add(m.l, add(Hj.l.x, Hj.l.y));
            accumulate(s, prod(-Da.h, -Da.l, m.h, m.l));
            const float2 o = acc_j[q][b];
            Ff<float> a{o.x, o.y};
            accumulate(a, s);
            acc_j[q][b] = make_float2(a.h, a.l);
          }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          accumulate(S[p], prod(H[p].h, H[p].l, Db[p].h, Db[p].l));
          accumulate(out[p], S[p]);
        }
        __syncwarp();  // the next step's lanes read these source-side sums
      }
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        acc[2 * p] += (double)out[p].h.x + (double)out[p].l.x;
        acc[2 * p + 1] += (double)out[p].h.y + (double)out[p].l.y;
      }
      // source-side sums of this tile pair: the first contributing I writes the row, later ones add; a
      // diagonal tile has none (it writes zeros where no earlier I did)
      const int tb = J * PT + lane;
      if (tb < nt && (!dg || I == T.i0)) {
        double* row = PJ + (size_t)T.pj * nq + QS * tb;
#pragma unroll
        for (int q = 0; q < QS; ++q) {
          const float2 o = acc_j[q][lane];
          const double v = (double)o.x + (double)o.y;
          row[q] = I == T.i0 ? v : row[q] + v;
        }
      }
    }
    if (va) {
      double* row = PI + (size_t)T.pi * nq + QS * ta + q0;
#pragma unroll
      for (int p = 0; p < 2 * NP; ++p) row[p] = acc[p];
    }
  }
}

// ---- float64

template <bool YUK>
__global__ void __launch_bounds__(32 * PW, 2)
    k_pairs_f64(int nt, int ntask, int nT, int tpg, int G, int K, const double* __restrict__ geo,
                const double* __restrict__ src, const double* __restrict__ tab, double kappa,
                double* PI, double* PJ) {
  extern __shared__ __align__(16) double smem[];  // tiles filled by double2 stores
  double* s_tab = smem;  // 2^(-k / 2048) (Yukawa)
  double* s_warp = smem + (YUK ? EXP2_TAB : 0);
  if (YUK) {
    for (int k = threadIdx.x; k < EXP2_TAB; k += 32 * PW) s_tab[k] = tab[k];
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int task = blockIdx.x * PW + warp;
  if (task >= ntask) return;
  double* tile = s_warp + warp * (D_GEO + D_SRC + QS) * PT;
  double* acc_j = tile + (D_GEO + D_SRC) * PT;
  const int nq = QS * nt;
  const double beta = kappa * 1.44269504088896340736;
  const PairTask T = pair_task(task, nT, tpg, G, K, 1);
  for (int I = T.i0; I < T.i1; ++I) {
    const int ta = I * PT + lane;
    const bool va = ta < nt;
    const double* ga = geo + (size_t)I * D_GEO * PT + lane;
    const double* sa = src + (size_t)I * D_SRC * PT + lane;
    double x[QS][3], as[QS], am[QS], n[3], acc[QS];
#pragma unroll
    for (int i = 0; i < QS; ++i) {
#pragma unroll
      for (int c = 0; c < 3; ++c) x[i][c] = ga[(6 * c + i) * PT];
      if (!va) x[i][0] = 2e150;
      as[i] = sa[(i) * PT];
      am[i] = sa[(6 + i) * PT];
      acc[i] = 0.0;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) n[c] = ga[(18 + c) * PT];
    for (int J = T.diag ? I : T.j0; J < T.j1; ++J) {
      const bool dg = J == I;
      __syncwarp();
      {
        const double2* gs = reinterpret_cast<const double2*>(geo + (size_t)J * D_GEO * PT);
        const double2* ss = reinterpret_cast<const double2*>(src + (size_t)J * D_SRC * PT);
        double2* dst = reinterpret_cast<double2*>(tile);
        for (int e = lane; e < D_GEO * PT / 2; e += 32) dst[e] = gs[e];
        for (int e = lane; e < D_SRC * PT / 2; e += 32) dst[D_GEO * PT / 2 + e] = ss[e];
#pragma unroll
        for (int q = 0; q < QS; ++q) acc_j[q * PT + lane] = 0.0;
      }
      __syncwarp();
      for (int k = T.k0; k < T.k1; ++k) {
        const int b = (lane + k) & (PT - 1);
        const double* tb = tile + b;
        const bool own = dg && k == 0;  // the lane's own triangle
        double H[QS], Db[QS];
#pragma unroll
        for (int i = 0; i < QS; ++i) H[i] = 0.0;
#pragma unroll 1
        for (int q = 0; q < QS; ++q) {
          const double y0 = tb[q * PT], y1 = tb[(6 + q) * PT], y2 = tb[(12 + q) * PT];
          const double bs = tb[(D_GEO + q) * PT], bm = tb[(D_GEO + 6 + q) * PT];
          double Sj = 0.0, Hj = 0.0, Da = 0.0;
#pragma unroll
          for (int i = 0; i < QS; ++i) {
            const double d0 = x[i][0] - y0, d1 = x[i][1] - y1, d2 = x[i][2] - y2;
            if (i == 0) Da = fma(n[2], d2, fma(n[1], d1, n[0] * d0));
            if (q == 0) Db[i] = own ? 0.0 : fma(tb[20 * PT], d2, fma(tb[19 * PT], d1, tb[18 * PT] * d0));
            const double r2 = fma(d2, d2, fma(d1, d1, d0 * d0));
            double y = rsqrt64(r2);
            if (own && q == i) y = 0.0;  // the coincident point
            const double yy = y * y;
            double g, h;
            if (YUK) {
              const double r = own && q == i ? 0.0 : r2 * y;
              g = y * exp2_neg(beta * r, s_tab);
              h = g * fma(kappa, y, yy);
            } else {
              g = y;
              h = y * yy;
            }
            acc[i] = fma(bs, g, acc[i]);
            H[i] = fma(bm, h, H[i]);
            Sj = fma(as[i], g, Sj);
            Hj = fma(am[i], h, Hj);
          }
          if (!dg) acc_j[q * PT + b] += fma(-Da, Hj, Sj);
        }
#pragma unroll
        for (int i = 0; i < QS; ++i) acc[i] = fma(Db[i], H[i], acc[i]);
        __syncwarp();
      }
      const int tb = J * PT + lane;
      if (tb < nt && (!dg || I == T.i0)) {
        double* row = PJ + (size_t)T.pj * nq + QS * tb;
#pragma unroll
        for (int q = 0; q < QS; ++q) row[q] = I == T.i0 ? acc_j[q * PT + lane] : row[q] + acc_j[q * PT + lane];
      }
    }
    if (va) {
      double* row = PI + (size_t)T.pi * nq + QS * ta;
#pragma unroll
      for (int i = 0; i < QS; ++i) row[i] = acc[i];
    }
  }
}

// out[i] = sum of point i's rows (pair_task), in a fixed order: SUM_Y threads a point, their sums added in thread
// order.  A chain of L2 latencies where rows are many (500 triangles: up to 768): 12.6 us with 8
// threads and one load at a time, 6.4 us with 16 and eight in flight.
constexpr int SUM_Y = 16;
__global__ void __launch_bounds__(32 * SUM_Y) k_pairs_sum(int nq, int per_group, int G, int K, int nsub,
                                                          const double* PI, const double* PJ,
                                                          double* __restrict__ out) {
  __shared__ double sh[SUM_Y][33];
  const int i = blockIdx.x * 32 + threadIdx.x, ty = threadIdx.y;
  double v = 0.0;
  // rows p G + c, p < np, lo <= c < hi, every SUM_Y-th of them; eight loads in flight
  auto rows = [&](const double* P, int np, int lo, int hi) {
    const int n = hi - lo, dp = SUM_Y / n, dc = SUM_Y - dp * n;
    int p = ty / n, c = lo + ty - p * n;
    while (p < np) {
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        x[u] = p < np ? P[((size_t)p * G + c) * nq + i] : 0.0;
        p += dp;
        c += dc;
        if (c >= hi) {
          c -= n;
          ++p;
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) v += x[u];
    }
  };
  if (i < nq) {
    if (nsub == 1) {
      rows(PI, 1, 0, K * (G + 1));
    } else {
      const int gi = i / per_group;
      rows(PI, K, gi, G);
      rows(PJ, K * nsub, 0, gi + 1);
    }
  }
  sh[ty][threadIdx.x] = v;
  __syncthreads();
  if (ty == 0 && i < nq) {
    for (int k = 1; k < SUM_Y; ++k) v += sh[k][threadIdx.x];
    out[i] = v;
  }
}

// ---- tile layouts: rows of 32 triangles, one thread per (padded) quadrature point

// coordinates relative to the surface centre times `scale` on the grids of ff_grid, triangles past the last at
// 1e15; unit normals; each point's distance from its rounded place along the normal, which keeps the plane
// distances those of the unrounded triangle
__global__ void k_pairs_geo_ff(int nt, int nT, const double* __restrict__ qx, const double* __restrict__ nrm,
                               double cx, double cy, double cz, double scale, double grid, float* __restrict__ geo) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nT * PT * QS) return;
  const int t = e / QS, q = e - t * QS, nq = QS * nt;
  float* row = geo + (size_t)(t / PT) * FF_GEO * PT + t % PT;
  const double c[3] = {cx, cy, cz};
  double off = 0.0;
  for (int d = 0; d < 3; ++d) {
    double yq = d == 0 ? 1e15 : 0.0, yl = 0.0;
    if (t < nt) {
      const double y = (qx[(size_t)d * nq + e] - c[d]) * scale, low = grid * 0x1p-24;
      yq = rint(y / grid) * grid;
      yl = rint((y - yq) / low) * low;
      off += nrm[(size_t)d * nt + t] * ((y - yq) - yl);
    }
    row[(6 * d + q) * PT] = (float)yq;
    row[(18 + 6 * d + q) * PT] = (float)yl;
    if (q == 0) {
      const double n = t < nt ? nrm[(size_t)d * nt + t] : 0.0;
      row[(36 + d) * PT] = (float)n;
      row[(39 + d) * PT] = (float)(n - (double)(float)n);
    }
  }
  row[(42 + q) * PT] = (float)off;
}
__global__ void k_pairs_geo_f64(int nt, int nT, const double* __restrict__ qx, const double* __restrict__ nrm,
                                double* __restrict__ geo) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nT * PT * QS) return;
  const int t = e / QS, q = e - t * QS, nq = QS * nt;
  double* row = geo + (size_t)(t / PT) * D_GEO * PT + t % PT;
  for (int d = 0; d < 3; ++d) {
    row[(6 * d + q) * PT] = t < nt ? qx[(size_t)d * nq + e] : (d == 0 ? 1e150 : 0.0);
    if (q == 0) row[(18 + d) * PT] = t < nt ? nrm[(size_t)d * nt + t] : 0.0;
  }
}

// strengths s_j = cs w_j lam_h(y_j) and mu_j = cd w_j u_h(y_j) (m_j = mu_j n)
template <bool F64>
__global__ void k_pairs_src(int nt, int nT, const int* __restrict__ tri, const int* __restrict__ vmap,
                            const double* __restrict__ lam, const double* __restrict__ u, int u_local,
                            const double* __restrict__ qw, double cs, double cd, float* __restrict__ srcf,
                            double* __restrict__ srcd) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nT * PT * QS) return;
  const int t = e / QS, q = e - t * QS;
  double s = 0.0, mu = 0.0;
  if (t < nt) {
    double lh = 0.0, uh = 0.0;
    for (int a = 0; a < 3; ++a) {
      const int v = tri[3 * t + a];
      const double b = c_tri_b[q][a];
      if (lam) lh += b * lam[v];
      if (u) uh += b * u[u_local ? v : vmap[v]];
    }
    const double w = qw[e];
    s = cs * w * lh;
    mu = cd * w * uh;
  }
  if (F64) {
    double* row = srcd + (size_t)(t / PT) * D_SRC * PT + t % PT;
    row[q * PT] = s;
    row[(6 + q) * PT] = mu;
  } else {
    float* row = srcf + (size_t)(t / PT) * FF_SRC * PT + t % PT;
    const float sh = (float)s, mh = (float)mu;
    row[q * PT] = sh;
    row[(6 + q) * PT] = (float)(s - (double)sh);
    row[(12 + q) * PT] = mh;
    row[(18 + q) * PT] = (float)(mu - (double)mh);
  }
}

inline int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

// exp(-k / 16) and exp(-k / 1024) as float-float pairs, 2^(-k / 2048) in float64 (host-computed, once per mesh)
int pair_tables(Mesh* m, bool f64) {
  if (f64) {
    if (m->pair_tab64.n) return PBFB_OK;
    std::vector<double> t(EXP2_TAB);
    for (int k = 0; k < EXP2_TAB; ++k) t[k] = std::exp2(-k / (double)EXP2_TAB);
    return m->pair_tab64.upload(t.data(), t.size(), m->stream);
  }
  if (m->pair_tab.n) return PBFB_OK;
  std::vector<float2> t(FF_HI + FF_LO);
  for (int k = 0; k < FF_HI + FF_LO; ++k) {
    const double v = k < FF_HI ? (k < 640 ? std::exp(-k / 16.0) : 0.0) : std::exp(-(k - FF_HI) / 1024.0);
    const float h = (float)v;
    t[k] = make_float2(h, (float)(v - (double)h));
  }
  return m->pair_tab.upload(t.data(), t.size(), m->stream);
}

// doubles of partial sums and their total, the larger of the two forms
size_t pair_work(int64_t nt) { return (pair_rows_max((int)nt) + 1) * QS * (size_t)nt; }

int launch_pairs(Mesh* m, Surface* s, const double* x, const double* lam, double cs, double cd, double kappa, bool f64,
                 double** val) {
  const int nt = s->nt, nq = s->nq;
  const bool yuk = kappa != 0.0;
  const int u_local = (x != nullptr && x == lam) ? 1 : 0;
  const double* uvec = cd != 0.0 ? x : nullptr;
  const double* lvec = cs != 0.0 ? lam : nullptr;
  const PairSplit S = pair_split(nt, pair_want(f64, m->tune_ff_bps), f64);
  const int nT = S.nT, npad = nT * PT * QS;
  PB_TRY(pair_tables(m, f64));
  PB_TRY(ensure(s->mval, (S.rows + 1) * nq));
  double* PI = s->mval.p;
  double* PJ = S.nsub == 1 ? PI : PI + (size_t)S.K * S.G * nq;
  double* out = PI + S.rows * nq;
  const int nb = blocks_for(S.ntask, PW);
  if (f64) {
    const bool geo = s->pgeo64.n == 0;
    if (geo) {
      PB_TRY(s->pgeo64.alloc((size_t)nT * D_GEO * PT));
      k_pairs_geo_f64<<<blocks_for(npad, 256), 256, 0, m->stream>>>(nt, nT, s->qx.p, s->nrm.p, s->pgeo64.p);
      PB_LAUNCHED(m);
    }
    if (!s->psrc64.n) PB_TRY(s->psrc64.alloc((size_t)nT * D_SRC * PT));
    k_pairs_src<true><<<blocks_for(npad, 256), 256, 0, m->stream>>>(nt, nT, s->tri.p, s->vmap.p, lvec, uvec, u_local,
                                                                    s->qw.p, cs, cd, nullptr, s->psrc64.p);
    PB_LAUNCHED(m);
  } else {
    const double scale = yuk ? kappa : 1.0;
    if (!s->pgeo.n) PB_TRY(s->pgeo.alloc((size_t)nT * FF_GEO * PT));
    if (s->pgeo_scale != scale) {
      k_pairs_geo_ff<<<blocks_for(npad, 256), 256, 0, m->stream>>>(nt, nT, s->qx.p, s->nrm.p, s->ctr[0], s->ctr[1],
                                                                   s->ctr[2], scale, ff_grid(s, scale),
                                                                   s->pgeo.p);
      PB_LAUNCHED(m);
      s->pgeo_scale = scale;
    }
    if (!s->psrc.n) PB_TRY(s->psrc.alloc((size_t)nT * FF_SRC * PT));
    // scaled lengths r' = kappa r: g = kappa g', D h = kappa D' h'; the factor goes into the strengths
    k_pairs_src<false><<<blocks_for(npad, 256), 256, 0, m->stream>>>(
        nt, nT, s->tri.p, s->vmap.p, lvec, uvec, u_local, s->qw.p, cs * scale, cd * scale * scale, s->psrc.p, nullptr);
    PB_LAUNCHED(m);
  }
  cudaEvent_t ev;
  KernelClassTimer& tm = f64 ? m->t_nbody64 : m->t_nbodyff;
  timer_begin(m, tm, &ev);
  if (f64) {
    const int smem = ((yuk ? EXP2_TAB : 0) + PW * (D_GEO + D_SRC + QS) * PT) * (int)sizeof(double);
    const void* fn = yuk ? (const void*)k_pairs_f64<true> : (const void*)k_pairs_f64<false>;
    int a_nt = nt, a_task = S.ntask, a_nT = nT, a_tpg = S.tpg, a_G = S.G, a_K = S.K;
    double a_kap = kappa;
    void* args[] = {&a_nt, &a_task, &a_nT, &a_tpg, &a_G, &a_K, &s->pgeo64.p, &s->psrc64.p, &m->pair_tab64.p, &a_kap,
                    &PI, &PJ};
    PB_CUDA(cudaLaunchKernel(fn, dim3(nb), dim3(32 * PW), args, smem, m->stream));
  } else {
    const void* fn = S.nsub == 1 ? (yuk ? (const void*)k_pairs_ff<true, 3> : (const void*)k_pairs_ff<false, 3>)
                                 : (yuk ? (const void*)k_pairs_ff<true, 1> : (const void*)k_pairs_ff<false, 1>);
    int a_nt = nt, a_task = S.ntask, a_nT = nT, a_tpg = S.tpg, a_G = S.G, a_K = S.K;
    void* args[] = {&a_nt, &a_task, &a_nT, &a_tpg, &a_G, &a_K, &s->pgeo.p, &s->psrc.p, &m->pair_tab.p, &PI, &PJ};
    PB_CUDA(cudaLaunchKernel(fn, dim3(nb), dim3(32 * PW), args, 0, m->stream));
  }
  PB_LAUNCHED(m);
  k_pairs_sum<<<blocks_for(nq, 32), dim3(32, SUM_Y), 0, m->stream>>>(nq, S.tpg * PT * QS, S.G, S.K, S.nsub, PI, PJ, out);
  PB_LAUNCHED(m);
  timer_end(m, tm, ev, (double)nq * (double)nq);
  *val = out;
  return PBFB_OK;
}

// Shared-memory limits of the float64 form, once per device (called by mesh creation, before any launch): later mesh
// creations leave the kernels' attributes alone while other host threads launch them
int init_pair_attributes() {
  static DeviceOnce once;
  int dev = 0;
  PB_CUDA(cudaGetDevice(&dev));
  return once.run(dev, []() -> int {
    const int smem = (EXP2_TAB + PW * (D_GEO + D_SRC + QS) * PT) * (int)sizeof(double);
    for (const void* f : {(const void*)k_pairs_f64<true>, (const void*)k_pairs_f64<false>})
      PB_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return PBFB_OK;
  });
}

}  // namespace pbfb
