// Boundary-element kernels: Galerkin P1 single- and double-layer operators of the
// Laplace kernel on Gamma_m (Eq. KV) and of the Yukawa kernel on Gamma_s (Sec. 2.2):
//   V_ij = int int psi_i(x) g(x,y) psi_j(y),  K_ij = int int psi_i(x) dg/dn_y(x,y) psi_j(y)
//   g = exp(-kappa r) / (4 pi r),  dg/dn_y = n_y.(x-y) (1 + kappa r) exp(-kappa r) / (4 pi r^3)
// (Laplace is kappa = 0).
//
// Matrix-free far field: every matvec evaluates all pairs of 6-point quadrature
// points of the surface (an N-body sum, coincident points excluded) and reduces the
// target potentials against the test functions.  Touching and close triangle pairs
// are corrected by a precomputed sparse matrix holding, per P1 pair (i, j), the
// difference between the accurate rule of the pair's class and the 6 x 6 rule (bem_corrections.cu):
//   identical / common edge / common vertex: Sauter-Schwab (Sauter & Schwab,
//     Boundary Element Methods, 2011, Sec. 5.2), 5 Gauss-Legendre points per variable;
//   near (no shared vertex, centroid distance < 2 max(h_tau, h_sigma)): 6 points on
//     the test triangle x 6 points on each of the 16 sub-triangles of the trial one.
#include <atomic>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "device_once.h"
#include "f32x2.cuh"
#include "fp64_math.cuh"
#include "pbfb_internal.cuh"
#include "quad_tables.cuh"
#include "solid_angle.h"

namespace pbfb {

namespace {

constexpr double INV4PI = 0.079577471545947667884;

// ---------------------------------------------------------------- geometry

__global__ void k_surface_geometry(const double* __restrict__ xyz, int nvtot, const int* __restrict__ tri,
                                   const int* __restrict__ vmap, int nt, double cx, double cy, double cz,
                                   double* __restrict__ qx, double* __restrict__ qw, double* __restrict__ nrm,
                                   double* __restrict__ area, float4* __restrict__ qpf) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double P[3][3];
  for (int a = 0; a < 3; ++a) {
    int v = vmap[tri[3 * t + a]];
    for (int d = 0; d < 3; ++d) P[a][d] = xyz[d * nvtot + v];
  }
  double e1[3], e2[3];
  for (int d = 0; d < 3; ++d) {
    e1[d] = P[1][d] - P[0][d];
    e2[d] = P[2][d] - P[0][d];
  }
  double c[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
  double nn = sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
  double A = 0.5 * nn;
  area[t] = A;
  for (int d = 0; d < 3; ++d) nrm[d * nt + t] = c[d] / nn;
  int nq = QS * nt;
  for (int q = 0; q < QS; ++q) {
    int j = QS * t + q;
    double y[3];
    for (int d = 0; d < 3; ++d) {
      y[d] = c_tri_b[q][0] * P[0][d] + c_tri_b[q][1] * P[1][d] + c_tri_b[q][2] * P[2][d];
      qx[d * nq + j] = y[d];
    }
    qw[j] = c_tri_w[q] * A;
    qpf[j] = make_float4((float)(y[0] - cx), (float)(y[1] - cy), (float)(y[2] - cz), 0.f);
  }
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------- far field

// Source data at every quadrature point j = 6 tau + q:
//   s_j = cs w_j lam_h(y_j)   (single layer),   m_j = cd w_j u_h(y_j) n_tau   (double layer)
__global__ void k_sources(int nt, const int* __restrict__ tri, const int* __restrict__ vmap,
                          const double* __restrict__ lam, const double* __restrict__ u, int u_local,
                          const double* __restrict__ qw, const double* __restrict__ nrm,
                          const float4* __restrict__ qpf, double cs, double cd, float4* __restrict__ spos,
                          float4* __restrict__ sdl) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  int nq = QS * nt;
  if (j >= nq) return;
  int t = j / QS, q = j - t * QS;
  double lh = 0.0, uh = 0.0;
  for (int a = 0; a < 3; ++a) {
    int v = tri[3 * t + a];
    double b = c_tri_b[q][a];
    if (lam) lh += b * lam[v];
    if (u) uh += b * u[u_local ? v : vmap[v]];
  }
  double w = qw[j];
  double sv = cs * w * lh, mu = cd * w * uh;
  double n0 = nrm[t], n1 = nrm[nt + t], n2 = nrm[2 * nt + t];
  float4 p = qpf[j];
  p.w = (float)sv;
  spos[j] = p;
  sdl[j] = make_float4((float)(mu * n0), (float)(mu * n1), (float)(mu * n2), 0.f);
}

// float32 N-body: targets = sources = the nq quadrature points.  Block = NT threads, each
// owning TPT targets (interleaved by NT); sources streamed through shared memory in tiles
// of NT; blockIdx.y selects a contiguous source range (split).  Each tile's float partial
// sum is added to a double accumulator.  Coincident points (target index == source
// index) are skipped; only tiles containing one of the thread's targets test for it.
template <int NT, int TPT, bool YUK>
__global__ void __launch_bounds__(NT) k_nbody_f32(int nq, const float4* __restrict__ tgt,
                                                  const float4* __restrict__ spos,
                                                  const float4* __restrict__ sdl, float kappa, int per_split,
                                                  double* __restrict__ out) {
  __shared__ float4 shp[NT];
  __shared__ float4 shd[NT];
  const int t0 = blockIdx.x * NT * TPT;
  int ti[TPT];
  float tx[TPT], ty[TPT], tz[TPT];
  double acc64[TPT];
#pragma unroll
  for (int k = 0; k < TPT; ++k) {
    ti[k] = t0 + k * NT + threadIdx.x;
    float4 p = tgt[ti[k] < nq ? ti[k] : 0];
    tx[k] = p.x;
    ty[k] = p.y;
    tz[k] = p.z;
    acc64[k] = 0.0;
  }
  const int sb = blockIdx.y * per_split;
  const int se = min(nq, sb + per_split);
  const float nk = -kappa * 1.4426950408889634f;  // -kappa log2(e)
  for (int s0 = sb; s0 < se; s0 += NT) {
    int j = s0 + threadIdx.x;
    if (j < se) {
      shp[threadIdx.x] = spos[j];
      shd[threadIdx.x] = sdl[j];
    } else {
      shp[threadIdx.x] = make_float4(1e18f, 1e18f, 1e18f, 0.f);
      shd[threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    const bool diag = (s0 < t0 + NT * TPT) && (s0 + NT > t0);
    float acc[TPT];
#pragma unroll
    for (int k = 0; k < TPT; ++k) acc[k] = 0.f;
    if (!diag) {
#pragma unroll 4
      for (int jj = 0; jj < NT; ++jj) {
        const float4 p = shp[jj];
        const float4 d = shd[jj];
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
          float dx = tx[k] - p.x, dy = ty[k] - p.y, dz = tz[k] - p.z;
          float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          float ri = rsqrt_approx(r2);
          float nd = fmaf(d.x, dx, fmaf(d.y, dy, d.z * dz));
          float ri2 = ri * ri;
          if (YUK) {
            float r = r2 * ri;
            float e = ex2_approx(nk * r);
            float kr1 = fmaf(kappa, r, 1.f);
            float tt = fmaf(nd * kr1, ri2, p.w);
            acc[k] = fmaf(tt, e * ri, acc[k]);
          } else {
            float tt = fmaf(nd, ri2, p.w);
            acc[k] = fmaf(tt, ri, acc[k]);
          }
        }
      }
    } else {
      for (int jj = 0; jj < NT; ++jj) {
        const float4 p = shp[jj];
        const float4 d = shd[jj];
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
          if (s0 + jj == ti[k]) continue;
          float dx = tx[k] - p.x, dy = ty[k] - p.y, dz = tz[k] - p.z;
          float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          float ri = rsqrt_approx(r2);
          float nd = fmaf(d.x, dx, fmaf(d.y, dy, d.z * dz));
          float ri2 = ri * ri;
          if (YUK) {
            float r = r2 * ri;
            float e = ex2_approx(nk * r);
            float kr1 = fmaf(kappa, r, 1.f);
            float tt = fmaf(nd * kr1, ri2, p.w);
            acc[k] = fmaf(tt, e * ri, acc[k]);
          } else {
            float tt = fmaf(nd, ri2, p.w);
            acc[k] = fmaf(tt, ri, acc[k]);
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < TPT; ++k) acc64[k] += (double)acc[k];
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < TPT; ++k)
    if (ti[k] < nq) out[(int64_t)blockIdx.y * nq + ti[k]] = acc64[k];
}

// Packed variant of k_nbody_f32: two targets per 64-bit register pair, evaluated with the
// Blackwell f32x2 instructions (add/sub/mul/fma on pairs of float32 values), which halve the
// instruction-issue slots of the pair arithmetic; the FP32 lanes do the same work.  Sources are
// staged pre-duplicated ((x,x),(y,y),...) so shared-memory loads give packed operands.  Tiles
// that contain one of the thread's own targets use the scalar path for the coincident-point test.
template <int NT, int NP, bool YUK>
__global__ void __launch_bounds__(NT) k_nbody_f32x2(int nq, const float4* __restrict__ tgt,
                                                    const float4* __restrict__ spos,
                                                    const float4* __restrict__ sdl, float kappa, int per_split,
                                                    double* __restrict__ out) {
  // per source: (x,x),(y,y) | (z,z),(s,s) | (mx,mx),(my,my) | (mz,mz),0
  __shared__ ulonglong2 sh[4][NT];
  __shared__ float4 shp[NT], shd[NT];  // scalar copies for the diagonal tiles
  constexpr int TPT = 2 * NP;
  const int t0 = blockIdx.x * NT * TPT;
  int ti[TPT];
  float txs[TPT], tys[TPT], tzs[TPT];
  f32x2 tx[NP], ty[NP], tz[NP], acc[NP];
  double acc64[TPT];
#pragma unroll
  for (int k = 0; k < TPT; ++k) {
    ti[k] = t0 + k * NT + threadIdx.x;
    float4 p = tgt[ti[k] < nq ? ti[k] : 0];
    txs[k] = p.x;
    tys[k] = p.y;
    tzs[k] = p.z;
    acc64[k] = 0.0;
  }
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    tx[k] = pk2(txs[2 * k], txs[2 * k + 1]);
    ty[k] = pk2(tys[2 * k], tys[2 * k + 1]);
    tz[k] = pk2(tzs[2 * k], tzs[2 * k + 1]);
  }
  const int sb = blockIdx.y * per_split;
  const int se = min(nq, sb + per_split);
  const float nk = -kappa * 1.4426950408889634f;
  const f32x2 nk2 = pk2(nk, nk), kap2 = pk2(kappa, kappa), one2 = pk2(1.f, 1.f);
  for (int s0 = sb; s0 < se; s0 += NT) {
    int j = s0 + threadIdx.x;
    float4 p, d;
    if (j < se) {
      p = spos[j];
      d = sdl[j];
    } else {
      p = make_float4(1e18f, 1e18f, 1e18f, 0.f);
      d = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    sh[0][threadIdx.x] = make_ulonglong2(pk2(p.x, p.x), pk2(p.y, p.y));
    sh[1][threadIdx.x] = make_ulonglong2(pk2(p.z, p.z), pk2(p.w, p.w));
    sh[2][threadIdx.x] = make_ulonglong2(pk2(d.x, d.x), pk2(d.y, d.y));
    sh[3][threadIdx.x] = make_ulonglong2(pk2(d.z, d.z), 0ull);
    shp[threadIdx.x] = p;
    shd[threadIdx.x] = d;
    __syncthreads();
    const bool diag = (s0 < t0 + NT * TPT) && (s0 + NT > t0);
    if (!diag) {
#pragma unroll
      for (int k = 0; k < NP; ++k) acc[k] = 0ull;
#pragma unroll 2
      for (int jj = 0; jj < NT; ++jj) {
        const ulonglong2 a0 = sh[0][jj], a1 = sh[1][jj], a2 = sh[2][jj], a3 = sh[3][jj];
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          f32x2 dx = sub2(tx[k], a0.x), dy = sub2(ty[k], a0.y), dz = sub2(tz[k], a1.x);
          f32x2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
          float ra, rb;
          upk2(r2, ra, rb);
          f32x2 ri = pk2(rsqrt_approx(ra), rsqrt_approx(rb));
          f32x2 nd = fma2(a3.x, dz, fma2(a2.y, dy, mul2(a2.x, dx)));
          f32x2 ri2 = mul2(ri, ri);
          if (YUK) {
            f32x2 r = mul2(r2, ri);
            float xa, xb;
            upk2(mul2(nk2, r), xa, xb);
            f32x2 e = pk2(ex2_approx(xa), ex2_approx(xb));
            f32x2 tt = fma2(mul2(nd, fma2(kap2, r, one2)), ri2, a1.y);
            acc[k] = fma2(tt, mul2(e, ri), acc[k]);
          } else {
            acc[k] = fma2(fma2(nd, ri2, a1.y), ri, acc[k]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        float a, b;
        upk2(acc[k], a, b);
        acc64[2 * k] += (double)a;
        acc64[2 * k + 1] += (double)b;
      }
    } else {
      float accs[TPT];
#pragma unroll
      for (int k = 0; k < TPT; ++k) accs[k] = 0.f;
      for (int jj = 0; jj < NT; ++jj) {
        const float4 p = shp[jj];
        const float4 d = shd[jj];
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
          if (s0 + jj == ti[k]) continue;
          float dx = txs[k] - p.x, dy = tys[k] - p.y, dz = tzs[k] - p.z;
          float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          float ri = rsqrt_approx(r2);
          float nd = fmaf(d.x, dx, fmaf(d.y, dy, d.z * dz));
          float ri2 = ri * ri;
          if (YUK) {
            float r = r2 * ri;
            float e = ex2_approx(nk * r);
            float kr1 = fmaf(kappa, r, 1.f);
            float tt = fmaf(nd * kr1, ri2, p.w);
            accs[k] = fmaf(tt, e * ri, accs[k]);
          } else {
            float tt = fmaf(nd, ri2, p.w);
            accs[k] = fmaf(tt, ri, accs[k]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < TPT; ++k) acc64[k] += (double)accs[k];
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < TPT; ++k)
    if (ti[k] < nq) out[(int64_t)blockIdx.y * nq + ti[k]] = acc64[k];
}

// Mutual float32 N-body for the GMRES operator: every unordered pair of points evaluated once
// for both directions, with one-warp blocks.  Block (rg, cg)
// is one warp; it holds 4 targets per lane (I * 128 + lane + 32 k) as two f32x2 pairs, streams
// the 128 points of tile J through shared memory, and at step s lane l takes point (l + s) mod
// 128, so the 32 lanes update distinct source-side sums (warp-synchronous, fixed order).  Pair
// (i, j): d = x_i - x_j, f = (1 + kappa r) / r^2, g = exp(-kappa r) / r;
//   to i: (s_j + (m_j . d) f) g,   to j: (s_i - (m_i . d) f) g.
constexpr int FM_T = 128;

template <bool YUK>
__global__ void __launch_bounds__(32) k_nbody_f32m(int nq, int G, const float4* __restrict__ spos,
                                                   const float4* __restrict__ sdl, float kappa,
                                                   double* __restrict__ PI, double* __restrict__ PJ) {
  __shared__ float4 sp[FM_T], sd[FM_T];
  __shared__ float accj[FM_T];
  int t = blockIdx.x, rg = 0;
  while (t >= G - rg) {
    t -= G - rg;
    ++rg;
  }
  const int cg = rg + t;
  const int nT = (nq + FM_T - 1) / FM_T;
  const int tpg = (nT + G - 1) / G;
  const int i0g = rg * tpg, i1g = min(nT, (rg + 1) * tpg);
  const int j0g = cg * tpg, j1g = min(nT, (cg + 1) * tpg);
  const int lane = threadIdx.x;
  const float nk = -kappa * 1.4426950408889634f;
  const f32x2 nk2 = pk2(nk, nk), kap2 = pk2(kappa, kappa), one2 = pk2(1.f, 1.f);
  for (int I = i0g; I < i1g; ++I) {
    float tx[4], ty[4], tz[4], ts[4], tmx[4], tmy[4], tmz[4];
    int ti[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ti[k] = I * FM_T + lane + 32 * k;
      const bool v = ti[k] < nq;
      const float4 p = v ? spos[ti[k]] : make_float4(2e15f, 0.f, 0.f, 0.f);
      const float4 d = v ? sdl[ti[k]] : make_float4(0.f, 0.f, 0.f, 0.f);
      tx[k] = p.x;
      ty[k] = p.y;
      tz[k] = p.z;
      ts[k] = p.w;
      tmx[k] = -d.x;  // negated: the source-side term needs -(m_i . d)
      tmy[k] = -d.y;
      tmz[k] = -d.z;
    }
    f32x2 TX[2], TY[2], TZ[2], TS[2], NMX[2], NMY[2], NMZ[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      TX[c] = pk2(tx[2 * c], tx[2 * c + 1]);
      TY[c] = pk2(ty[2 * c], ty[2 * c + 1]);
      TZ[c] = pk2(tz[2 * c], tz[2 * c + 1]);
      TS[c] = pk2(ts[2 * c], ts[2 * c + 1]);
      NMX[c] = pk2(tmx[2 * c], tmx[2 * c + 1]);
      NMY[c] = pk2(tmy[2 * c], tmy[2 * c + 1]);
      NMZ[c] = pk2(tmz[2 * c], tmz[2 * c + 1]);
    }
    double acc64[4] = {0.0, 0.0, 0.0, 0.0};
    for (int J = max(I, j0g); J < j1g; ++J) {
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int jl = J * FM_T + lane + 32 * k;
        if (jl < nq) {
          sp[lane + 32 * k] = spos[jl];
          sd[lane + 32 * k] = sdl[jl];
        } else {
          sp[lane + 32 * k] = make_float4(1e15f, 0.f, 0.f, 0.f);
          sd[lane + 32 * k] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        accj[lane + 32 * k] = 0.f;
      }
      __syncwarp();
      const int cnt = min(FM_T, nq - J * FM_T);
      if (J == I) {
        // diagonal tile: target side only, coincident point skipped
        float a[4] = {0.f, 0.f, 0.f, 0.f};
        for (int jj = 0; jj < cnt; ++jj) {
          const float4 p = sp[jj], d = sd[jj];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (jj == lane + 32 * k) continue;
            const float dx = tx[k] - p.x, dy = ty[k] - p.y, dz = tz[k] - p.z;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const float ri = rsqrt_approx(r2);
            const float nd = fmaf(d.x, dx, fmaf(d.y, dy, d.z * dz));
            const float ri2 = ri * ri;
            if (YUK) {
              const float r = r2 * ri;
              const float e = ex2_approx(nk * r);
              const float tt = fmaf(nd * fmaf(kappa, r, 1.f), ri2, p.w);
              a[k] = fmaf(tt, e * ri, a[k]);
            } else {
              a[k] = fmaf(fmaf(nd, ri2, p.w), ri, a[k]);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) acc64[k] += (double)a[k];
      } else {
        f32x2 acc[2] = {0ull, 0ull};
#pragma unroll 2
        for (int st = 0; st < FM_T; ++st) {
          const int jj = (lane + st) & (FM_T - 1);
          const float4 p = sp[jj], d = sd[jj];
          const f32x2 PX = pk2(p.x, p.x), PY = pk2(p.y, p.y), PZ = pk2(p.z, p.z), PS = pk2(p.w, p.w);
          const f32x2 MX = pk2(d.x, d.x), MY = pk2(d.y, d.y), MZ = pk2(d.z, d.z);
          float cj = 0.f;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const f32x2 dx = sub2(TX[c], PX), dy = sub2(TY[c], PY), dz = sub2(TZ[c], PZ);
            const f32x2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
            float ra, rb;
            upk2(r2, ra, rb);
            const f32x2 ri = pk2(rsqrt_approx(ra), rsqrt_approx(rb));
            const f32x2 ri2 = mul2(ri, ri);
            f32x2 f, g;
            if (YUK) {
              const f32x2 r = mul2(r2, ri);
              float xa, xb;
              upk2(mul2(nk2, r), xa, xb);
              const f32x2 e = pk2(ex2_approx(xa), ex2_approx(xb));
              f = mul2(fma2(kap2, r, one2), ri2);
              g = mul2(e, ri);
            } else {
              f = ri2;
              g = ri;
            }
            const f32x2 ndj = fma2(MZ, dz, fma2(MY, dy, mul2(MX, dx)));
            acc[c] = fma2(fma2(ndj, f, PS), g, acc[c]);
            const f32x2 ndi = fma2(NMZ[c], dz, fma2(NMY[c], dy, mul2(NMX[c], dx)));
            float u0, u1;
            upk2(mul2(fma2(ndi, f, TS[c]), g), u0, u1);
            cj += u0 + u1;
          }
          accj[jj] += cj;
          __syncwarp();
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float a0, a1;
          upk2(acc[c], a0, a1);
          acc64[2 * c] += (double)a0;
          acc64[2 * c + 1] += (double)a1;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int jl = J * FM_T + lane + 32 * k;
          if (jl < nq) PJ[(int64_t)rg * nq + jl] += (double)accj[lane + 32 * k];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (ti[k] < nq) PI[(int64_t)cg * nq + ti[k]] = acc64[k];
  }
}

// ---------------------------------------------------------------- float-float far field
//
// The Newton residual needs a far field accurate to float64 level, but the float64 rate of
// GB300 is 1/64 of its float32 rate.  These kernels evaluate the same pair sums in
// float-float arithmetic: every quantity is an unevaluated pair hi + lo of float32 values
// (about 48 significant bits), built from error-free transformations -- Knuth's TwoSum,
// Dekker's FastTwoSum (|a| >= |b|) and the FMA TwoProduct -- as in Ogita, Rump & Oishi,
// "Accurate sum and dot product" (SIAM J. Sci. Comput. 2005).  1/sqrt uses one Newton step
// from the hardware estimate; exp(-x) for the Yukawa kernel uses two float-float tables of
// exp(-k delta) (delta = 1/256) and a 5-term Taylor series for the remainder f < delta.
// The _rn intrinsics keep the compiler from contracting the transformations into FMAs.

constexpr int FF_TABLE_HI = 640;      // exp(-16 delta k1), k1 < 640: x up to 40
constexpr float FF_XMAX = 39.99f;      // exp(-40) ~ 4e-18: larger arguments give 0

__constant__ float2 c_ff_exp_lo[16];   // exp(-delta k0), k0 < 16

struct ff { float h, l; };

__device__ __forceinline__ ff two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff s = two_sum(a.h, b.h);
  float lo = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
  return fast_two_sum(s.h, lo);
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return fast_two_sum(p, e);
}
__device__ __forceinline__ ff ff_sq(ff a) {
  float p = __fmul_rn(a.h, a.h);
  float e = __fmaf_rn(a.h, a.h, -p);
  e = __fmaf_rn(__fadd_rn(a.h, a.h), a.l, e);
  return fast_two_sum(p, e);
}
// difference of two float-float coordinates whose high parts lie on a common grid q, fine enough
// that xh - yh is exact: (xh - yh) + (xl - yl) with |xl - yl| <= q <= |xh - yh| unless xh = yh,
// so a FastTwoSum renormalises it
__device__ __forceinline__ ff ff_diff(float xh, float xl, float yh, float yl) {
  return fast_two_sum(__fsub_rn(xh, yh), __fsub_rn(xl, yl));
}
// a.x + b.y + c.z for float-float vectors
__device__ __forceinline__ ff ff_dot3(ff a0, ff a1, ff a2, ff b0, ff b1, ff b2) {
  float p0 = __fmul_rn(a0.h, b0.h), p1 = __fmul_rn(a1.h, b1.h), p2 = __fmul_rn(a2.h, b2.h);
  float e0 = __fmaf_rn(a0.l, b0.h, __fmaf_rn(a0.h, b0.l, __fmaf_rn(a0.h, b0.h, -p0)));
  float e1 = __fmaf_rn(a1.l, b1.h, __fmaf_rn(a1.h, b1.l, __fmaf_rn(a1.h, b1.h, -p1)));
  float e2 = __fmaf_rn(a2.l, b2.h, __fmaf_rn(a2.h, b2.l, __fmaf_rn(a2.h, b2.h, -p2)));
  ff s1 = two_sum(p0, p1);
  ff s2 = two_sum(s1.h, p2);
  float lo = __fadd_rn(__fadd_rn(s1.l, s2.l), __fadd_rn(__fadd_rn(e0, e1), e2));
  return fast_two_sum(s2.h, lo);
}
// 1/sqrt(r) for r = rh + rl > 0: one Newton step y0 (1 - (r y0^2 - 1)/2) from the hardware estimate
__device__ __forceinline__ ff ff_rsqrt(ff r) {
  float y0 = rsqrtf(r.h);
  float t = __fmul_rn(y0, y0);
  float te = __fmaf_rn(y0, y0, -t);
  float a = __fmul_rn(r.h, t);
  float ae = __fmaf_rn(r.h, t, -a);
  float z = __fadd_rn(__fsub_rn(a, 1.0f), __fmaf_rn(r.l, t, __fmaf_rn(r.h, te, ae)));
  return fast_two_sum(y0, __fmul_rn(__fmul_rn(-0.5f, y0), z));
}
// exp(-x), 0 <= x (float-float); tab_hi in shared memory: exp(-16 k1 / 256)
__device__ __forceinline__ ff ff_expm(ff x, const float2* __restrict__ tab_hi) {
  if (x.h >= FF_XMAX) return {0.f, 0.f};
  int k = __float2int_rd(__fmul_rn(x.h, 256.0f));
  k = k < 0 ? 0 : k;
  ff f = fast_two_sum(__fsub_rn(x.h, __fmul_rn((float)k, 0.00390625f)), x.l);   // 0 <= f < 1/256 (+rounding)
  // exp(-f) = (1 - f) + f^2/2 + f^2 (-f/6 + f^2/24 - f^3/120)
  ff f2 = ff_sq(f);
  float p2 = __fmul_rn(f.h, __fmaf_rn(f.h, __fmaf_rn(f.h, -1.0f / 120.0f, 1.0f / 24.0f), -1.0f / 6.0f));
  ff one_minus = two_sum(1.0f, -f.h);
  one_minus = fast_two_sum(one_minus.h, __fsub_rn(one_minus.l, f.l));
  ff tail = fast_two_sum(__fmul_rn(0.5f, f2.h), __fmaf_rn(f2.h, p2, __fmul_rn(0.5f, f2.l)));
  ff ef = ff_add(one_minus, tail);
  float2 a = tab_hi[k >> 4];
  float2 b = c_ff_exp_lo[k & 15];
  return ff_mul(ff_mul(ef, ff{a.x, a.y}), ff{b.x, b.y});
}

// Float-float sources: 4 float4 per point: (y hi, s hi), (y lo, s lo), (m hi, 0), (m lo, 0),
// with y relative to the surface centre, s = cs w lam_h, m = cd w u_h n.  The coordinates' high
// parts lie on `grid` (a power of 2) with every difference of two of them exact in float32,
// the low parts are the remainders (|y lo| <= grid / 2).
__global__ void k_sources_ff(int nt, const int* __restrict__ tri, const int* __restrict__ vmap,
                             const double* __restrict__ lam, const double* __restrict__ u, int u_local,
                             const double* __restrict__ qw, const double* __restrict__ nrm,
                             const double* __restrict__ qx, double cx, double cy, double cz, double cs, double cd,
                             double grid, float4* __restrict__ src, float4* __restrict__ tgt) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  int nq = QS * nt;
  if (j >= nq) return;
  int t = j / QS, q = j - t * QS;
  double lh = 0.0, uh = 0.0;
  for (int a = 0; a < 3; ++a) {
    int v = tri[3 * t + a];
    double b = c_tri_b[q][a];
    if (lam) lh += b * lam[v];
    if (u) uh += b * u[u_local ? v : vmap[v]];
  }
  double w = qw[j];
  double sv = cs * w * lh, mu = cd * w * uh;
  double y[3] = {qx[j] - cx, qx[nq + j] - cy, qx[2 * nq + j] - cz};
  double mm[3] = {mu * nrm[t], mu * nrm[nt + t], mu * nrm[2 * nt + t]};
  float yh[3], yl[3], mh[3], ml[3];
  for (int d = 0; d < 3; ++d) {
    const double yq = rint(y[d] / grid) * grid;  // on the grid: exact in float32
    yh[d] = (float)yq;
    yl[d] = (float)(rint((y[d] - yq) / (grid * 0x1p-24)) * (grid * 0x1p-24));
    mh[d] = (float)mm[d];
    ml[d] = (float)(mm[d] - (double)mh[d]);
  }
  float sh = (float)sv, sl = (float)(sv - (double)sh);
  src[4 * j + 0] = make_float4(yh[0], yh[1], yh[2], sh);
  src[4 * j + 1] = make_float4(yl[0], yl[1], yl[2], sl);
  src[4 * j + 2] = make_float4(mh[0], mh[1], mh[2], 0.f);
  src[4 * j + 3] = make_float4(ml[0], ml[1], ml[2], 0.f);
  tgt[2 * j + 0] = make_float4(yh[0], yh[1], yh[2], 0.f);
  tgt[2 * j + 1] = make_float4(yl[0], yl[1], yl[2], 0.f);
}

// One pair in float-float: (s + nd (1 + kappa r) / r^2) exp(-kappa r) / r  (kappa = 0: Laplace)
template <bool YUK>
__device__ __forceinline__ ff ff_pair(const float4& ph, const float4& pl, const float4& mh, const float4& ml,
                                      const float (&th)[3], const float (&tl)[3], ff kap,
                                      const float2* __restrict__ tab) {
  ff d0 = ff_diff(th[0], tl[0], ph.x, pl.x);
  ff d1 = ff_diff(th[1], tl[1], ph.y, pl.y);
  ff d2 = ff_diff(th[2], tl[2], ph.z, pl.z);
  ff r2 = ff_dot3(d0, d1, d2, d0, d1, d2);
  ff ri = ff_rsqrt(r2);
  ff nd = ff_dot3(ff{mh.x, ml.x}, ff{mh.y, ml.y}, ff{mh.z, ml.z}, d0, d1, d2);
  ff ri2 = ff_sq(ri);
  if (YUK) {
    ff r = ff_mul(r2, ri);
    ff x = ff_mul(kap, r);
    ff e = ff_expm(x, tab);
    ff one_x = two_sum(1.0f, x.h);
    one_x = fast_two_sum(one_x.h, __fadd_rn(one_x.l, x.l));
    ff t = ff_add(ff{ph.w, pl.w}, ff_mul(ff_mul(nd, one_x), ri2));
    return ff_mul(t, ff_mul(e, ri));
  }
  ff t = ff_add(ff{ph.w, pl.w}, ff_mul(nd, ri2));
  return ff_mul(t, ri);
}

// Float-float N-body: same tiling as the float32 kernel (one target per thread); each tile's
// float-float partial sum is added to a float64 accumulator.
template <int NT, bool YUK>
__global__ void __launch_bounds__(NT) k_nbody_ff(int nq, const float4* __restrict__ tgt,
                                                 const float4* __restrict__ src, float kh, float kl,
                                                 const float2* __restrict__ tab_hi, int per_split,
                                                 double* __restrict__ out) {
  __shared__ float4 sh[4][NT];
  __shared__ float2 tab[YUK ? FF_TABLE_HI : 1];
  if (YUK)
    for (int k = threadIdx.x; k < FF_TABLE_HI; k += NT) tab[k] = tab_hi[k];
  const int i = blockIdx.x * NT + threadIdx.x;
  const int ii = i < nq ? i : 0;
  const float4 a = tgt[2 * ii], b = tgt[2 * ii + 1];
  const float th[3] = {a.x, a.y, a.z}, tl[3] = {b.x, b.y, b.z};
  const ff kap{kh, kl};
  const int sb = blockIdx.y * per_split;
  const int se = min(nq, sb + per_split);
  double acc64 = 0.0;
  for (int s0 = sb; s0 < se; s0 += NT) {
    int j = s0 + threadIdx.x;
    if (j < se) {
      for (int c = 0; c < 4; ++c) sh[c][threadIdx.x] = src[4 * j + c];
    }
    __syncthreads();
    const int cnt = min(NT, se - s0);
    ff acc{0.f, 0.f};
    for (int jj = 0; jj < cnt; ++jj) {
      if (s0 + jj == i) continue;
      ff v = ff_pair<YUK>(sh[0][jj], sh[1][jj], sh[2][jj], sh[3][jj], th, tl, kap, tab);
      acc = ff_add(acc, v);
    }
    acc64 += (double)acc.h + (double)acc.l;
    __syncthreads();
  }
  if (i < nq) out[(int64_t)blockIdx.y * nq + i] = acc64;
}

// out[i] = sum over c of PI[c][i] + sum over r of PJ[r][i] (fixed order)
__global__ void k_mutual_sum(int nq, int G, const double* __restrict__ PI, const double* __restrict__ PJ,
                             double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nq) return;
  double v = 0.0;
  for (int c = 0; c < G; ++c) v += PI[(int64_t)c * nq + i];
  for (int r = 0; r < G; ++r) v += PJ[(int64_t)r * nq + i];
  out[i] = v;
}

// val[0][j] = sum over the source splits of val[split][j] (fixed order)
__global__ void k_split_sum(int nq, int nsplit, double* __restrict__ val) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nq || nsplit <= 1) return;
  double v = val[j];
  for (int sp = 1; sp < nsplit; ++sp) v += val[(int64_t)sp * nq + j];
  val[j] = v;
}

// y[i] (+)= sum over incident (tau, a) of sum_q psi_a(x_q) w_q val[6 tau + q], plus the rows of `add` (the near
// field's, which would cost a launch of its own, 2.7 us of a 70 us product of 500 triangles); 8 lanes per vertex
__global__ void k_test_reduce(int nv, const int* __restrict__ ptr, const int* __restrict__ idx,
                              const double* __restrict__ val, const double* __restrict__ qw, RowAdd add,
                              int accumulate, double* __restrict__ y) {
  const int lane = threadIdx.x & 7;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 3;
  const bool valid = i < nv;  // all lanes reach the shuffles
  double acc = 0.0, cor = 0.0;
  const int b = valid ? ptr[i] : 0, e = valid ? ptr[i + 1] : 0;
  for (int k = b * QS + lane; k < e * QS; k += 8) {
    int ent = idx[k / QS], q = k % QS;
    int t = ent / 3, a = ent - 3 * t;
    int j = QS * t + q;
    acc += c_tri_b[q][a] * qw[j] * val[j];
  }
  if (add.ptr && valid) {
    const int k1 = add.ptr[i + 1];
    for (int k0 = add.ptr[i] + lane; k0 < k1; k0 += 32) {  // four entries a lane in flight
      double v[4], x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + 8 * u;
        v[u] = x[u] = 0.0;
        if (k < k1) {
          const int c = add.col[k];
          v[u] = add.val[k];
          if (add.half) v[u] = fma(0.5, add.half[k], v[u]);
          x[u] = add.x[add.map ? add.map[c] : c];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) cor = fma(v[u], x[u], cor);
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    acc += __shfl_down_sync(0xffffffffu, acc, o, 8);
    cor += __shfl_down_sync(0xffffffffu, cor, o, 8);
  }
  if (lane == 0 && valid) {
    acc = accumulate ? y[i] + acc : acc;
    y[i] = add.ptr ? acc + cor : acc;
  }
}

// The charges' Coulomb potential and its normal derivative's negative at the Gamma_m quadrature points,
//   C_j = sum_k z_k / |x_k - y_j|,   E_j = sum_k z_k n_j . (x_k - y_j) / |x_k - y_j|^3,
// once per set of charges: C gives the Coulomb data <u_coul, psi>, and both give the reaction energy of every
// solution, sum_k z_k phi(x_k) = (1 / 4 pi) sum_j (a_j C_j - c_j E_j) with a_j = w_j lam_h(y_j) and
// c_j = w_j u_h(y_j) (Eq. Esolv with Eq. Potential_in_Omega_m, the sums exchanged), so that an energy costs one
// pass over the points instead of one over all (charge, point) pairs.  The float64 pipe bounds it: a thread
// takes a triangle's six points, which share n . (x_k - y) (16.5 operations per pair with an own root); chunks
// of the charges (blockIdx.y) for enough blocks, added in chunk order.
// GB300, 8000 triangles, 200 charges: C alone 478 us with the library's root and division, and 461 us more for
// the potentials of both solutions at the charges in every energy (15,680 triangles, 1536 charges: 6.1 and 6.4
// ms); C and E together 5.4 ms there, and 4 us an energy.
constexpr int COUL_T = 128;
__global__ void __launch_bounds__(COUL_T) k_coulomb(int nt, const double* __restrict__ qx,
                                                    const double* __restrict__ nrm, int ncharge,
                                                    const double* __restrict__ cxyz, const double* __restrict__ cz,
                                                    double* __restrict__ part) {
  const int t = blockIdx.x * COUL_T + threadIdx.x;
  if (t >= nt) return;
  const int nq = QS * nt;
  double y[QS][3], C[QS], E[QS];
#pragma unroll
  for (int q = 0; q < QS; ++q) {
#pragma unroll
    for (int d = 0; d < 3; ++d) y[q][d] = qx[(size_t)d * nq + QS * t + q];
    C[q] = E[q] = 0.0;
  }
  const double n0 = nrm[t], n1 = nrm[nt + t], n2 = nrm[2 * nt + t];
  const int per = (ncharge + gridDim.y - 1) / gridDim.y;
  const int k1 = min(ncharge, (int)(blockIdx.y + 1) * per);
  for (int k = blockIdx.y * per; k < k1; ++k) {
    const double x0 = cxyz[k], x1 = cxyz[ncharge + k], x2 = cxyz[2 * ncharge + k], z = cz[k];
    double D = 0.0;
#pragma unroll
    for (int q = 0; q < QS; ++q) {
      const double d0 = x0 - y[q][0], d1 = x1 - y[q][1], d2 = x2 - y[q][2];
      if (q == 0) D = fma(n2, d2, fma(n1, d1, n0 * d0));
      const double ri = rsqrt64(fma(d2, d2, fma(d1, d1, d0 * d0)));
      const double zr = z * ri;
      C[q] += zr;
      E[q] = fma(D, zr * (ri * ri), E[q]);
    }
  }
  double* out = part + (size_t)blockIdx.y * 2 * nq + QS * t;
#pragma unroll
  for (int q = 0; q < QS; ++q) {
    out[q] = C[q];
    out[nq + q] = E[q];
  }
}

// out[i] = sum of the nchunk rows of part, in chunk order
__global__ void k_chunk_sum(int n, int nchunk, const double* __restrict__ part, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v = part[i];
  for (int c = 1; c < nchunk; ++c) v += part[(size_t)c * n + i];
  out[i] = v;
}

// Winding numbers of Gamma_m at the charges: sum over the triangles of their signed solid angles (half_solid_angle), as
// on the host (winding_numbers in mesh_setup.cu) with the same test for points on a triangle, all in float64, whose
// pipe bounds it.  A thread takes a charge, chunks of the triangles (blockIdx.y) give the blocks; a point on the
// surface makes its sum huge.
// GB300, the whole charges_set: 1536 charges on 15,680 triangles 35.5 ms with this check on 16 host cores, 10.2 ms so
// (8.6 with the angles in float32); 200 on 8000, 3.2 and 0.87 ms (0.71).
constexpr int WIND_T = 64;
constexpr double WIND_ON = 1e30;
__global__ void __launch_bounds__(WIND_T) k_winding(int nt, const int* __restrict__ tri, const int* __restrict__ vmap,
                                                    const double* __restrict__ xyz, int nvtot, int nq,
                                                    const double* __restrict__ q, double* __restrict__ part) {
  const int k = blockIdx.x * WIND_T + threadIdx.x;
  const double x = q[k < nq ? k : 0], y = q[nq + (k < nq ? k : 0)], z = q[2 * nq + (k < nq ? k : 0)];
  const int per = (nt + gridDim.y - 1) / gridDim.y;
  const int t1 = min(nt, (int)(blockIdx.y + 1) * per);
  double sum = 0.0;
  bool on = false;
  __shared__ double P[WIND_T][9];
  for (int t0 = blockIdx.y * per; t0 < t1; t0 += WIND_T) {
    __syncthreads();
    const int t = t0 + threadIdx.x;
    if (t < t1)
      for (int a = 0; a < 3; ++a) {
        const int v = vmap[tri[3 * t + a]];
        for (int d = 0; d < 3; ++d) P[threadIdx.x][3 * a + d] = xyz[(size_t)d * nvtot + v];
      }
    __syncthreads();
    const int cnt = min(WIND_T, t1 - t0);
    for (int i = 0; i < cnt; ++i) {
      const double* p = P[i];
      const double a0 = p[0] - x, a1 = p[1] - y, a2 = p[2] - z;
      const double b0 = p[3] - x, b1 = p[4] - y, b2 = p[5] - z;
      const double c0 = p[6] - x, c1 = p[7] - y, c2 = p[8] - z;
      const double ra2 = fma(a2, a2, fma(a1, a1, a0 * a0)), rb2 = fma(b2, b2, fma(b1, b1, b0 * b0)),
                   rc2 = fma(c2, c2, fma(c1, c1, c0 * c0));
      if (ra2 == 0.0 || rb2 == 0.0 || rc2 == 0.0) {
        on = true;
        continue;
      }
      sum += half_solid_angle(a0, a1, a2, b0, b1, b2, c0, c1, c2, ra2 * rsqrt64(ra2), rb2 * rsqrt64(rb2),
                              rc2 * rsqrt64(rc2), &on);
    }
  }
  if (k < nq) part[(size_t)blockIdx.y * nq + k] = on ? WIND_ON : sum;
}

// block partials of sum_j w_j (lam_h C_j - u_h E_j) for x_L and x_NL
constexpr int REAC_T = 256;
__global__ void __launch_bounds__(REAC_T) k_reaction_energy(
    int nt, const int* __restrict__ tri, const int* __restrict__ vmap, const double* __restrict__ qw,
    const double* __restrict__ ce, const double* __restrict__ lamL, const double* __restrict__ uL,
    const double* __restrict__ lamN, const double* __restrict__ uN, double* __restrict__ part) {
  const int nq = QS * nt;
  double acc[2] = {0.0, 0.0};
  for (int j = blockIdx.x * REAC_T + threadIdx.x; j < nq; j += gridDim.x * REAC_T) {
    const int t = j / QS, q = j - t * QS;
    double lL = 0.0, lU = 0.0, nL = 0.0, nU = 0.0;
    for (int a = 0; a < 3; ++a) {
      const int v = tri[3 * t + a], sv = vmap[v];
      const double b = c_tri_b[q][a];
      lL += b * lamL[v];
      lU += b * uL[sv];
      nL += b * lamN[v];
      nU += b * uN[sv];
    }
    const double w = qw[j], c = w * ce[j], e = w * ce[nq + j];
    acc[0] += lL * c - lU * e;
    acc[1] += nL * c - nU * e;
  }
  __shared__ double sh[2][REAC_T / 32];
  for (int k = 0; k < 2; ++k) {
    const double v = warp_sum(acc[k]);
    if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int w = 0; w < REAC_T / 32; ++w) s += sh[threadIdx.x][w];
    part[2 * (size_t)blockIdx.x + threadIdx.x] = s;
  }
}

inline int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

// Constant tables of the quadrature rules and of the float-float exponential, once per device (called by mesh
// creation, before any launch)
int init_quadrature() {
  static DeviceOnce once;
  int dev = 0;
  PB_CUDA(cudaGetDevice(&dev));
  return once.run(dev, []() -> int {
    PB_TRY(init_correction_rules());
    // float-float exp tables: exp(-k0 / 256), k0 < 16 (constant memory)
    float2 lo[16];
    for (int k = 0; k < 16; ++k) {
      double v = std::exp(-k / 256.0);
      float h = (float)v;
      lo[k] = make_float2(h, (float)(v - (double)h));
    }
    PB_CUDA(cudaMemcpyToSymbol(c_ff_exp_lo, lo, sizeof(lo)));
    // the copies run on the legacy stream, which a mesh's own (non-blocking) stream does not wait for
    PB_CUDA(cudaStreamSynchronize(cudaStreamLegacy));
    return PBFB_OK;
  });
}

// exp(-16 k1 / 256), k1 < FF_TABLE_HI, as float-float pairs (host-computed in float64)
int ff_exp_table(Mesh* m) {
  if (m->ff_tab.n) return PBFB_OK;
  std::vector<float2> t(FF_TABLE_HI);
  for (int k = 0; k < FF_TABLE_HI; ++k) {
    double v = std::exp(-16.0 * k / 256.0);
    float h = (float)v;
    t[k] = make_float2(h, (float)(v - (double)h));
  }
  PB_TRY(m->ff_tab.upload(t.data(), t.size(), m->stream));
  return PBFB_OK;
}

int test_reduce(Mesh* m, Surface* s, double* val, int nsplit, double* y, bool accumulate, const RowAdd* add) {
  if (nsplit > 1) {
    k_split_sum<<<blocks_for(s->nq, 256), 256, 0, m->stream>>>(s->nq, nsplit, val);
    PB_LAUNCHED(m);
  }
  k_test_reduce<<<blocks_for((int64_t)s->nv * 8, 128), 128, 0, m->stream>>>(
      s->nv, s->inc_ptr.p, s->inc_idx.p, val, s->qw.p, add ? *add : RowAdd{}, accumulate ? 1 : 0, y);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int launch_surface_geometry(Mesh* m, Surface* s) {
  k_surface_geometry<<<blocks_for(s->nt, 128), 128, 0, m->stream>>>(
      m->xyz.p, m->nv, s->tri.p, s->vmap.p, s->nt, s->ctr[0], s->ctr[1], s->ctr[2], s->qx.p, s->qw.p, s->nrm.p,
      s->area.p, s->qpf.p);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

constexpr int F32_NT = 128;

// Launch shape of the float32 far field: tuning knobs if set, else 2 targets per thread with
// the packed kernel and 32 blocks per SM of source splits for large surfaces (GB300 sweep on
// the multi-charge sphere), one target per thread unpacked for small ones.
// With explicit targets per thread and blocks_per_sm 0, *bps = 0 asks the caller for a source
// split that fills whole waves of resident blocks.
void f32_shape(const Mesh* m, int nq, int* tpt, int* packed, int* bps) {
  const bool big = nq >= 16384;
  *tpt = m->tune_tpt > 0 ? m->tune_tpt : (big ? 2 : 1);
  *packed = m->tune_tpt > 0 ? m->tune_packed : (big ? 1 : 0);
  if (*tpt < 2 && *packed == 1) *packed = 0;
  *bps = m->tune_bps > 0 ? m->tune_bps : (m->tune_tpt > 0 ? 0 : (big ? 32 : 16));
}

// resident blocks per SM of the split float32 kernel variant
static int f32_blocks_per_sm(int tpt, int packed, bool yuk) {
  constexpr int NT = F32_NT;
  const void* f = nullptr;
  if (packed) {
    if (tpt == 2) f = yuk ? (const void*)k_nbody_f32x2<NT, 1, true> : (const void*)k_nbody_f32x2<NT, 1, false>;
    else if (tpt == 8) f = yuk ? (const void*)k_nbody_f32x2<NT, 4, true> : (const void*)k_nbody_f32x2<NT, 4, false>;
    else f = yuk ? (const void*)k_nbody_f32x2<NT, 2, true> : (const void*)k_nbody_f32x2<NT, 2, false>;
  } else {
    if (tpt == 1) f = yuk ? (const void*)k_nbody_f32<NT, 1, true> : (const void*)k_nbody_f32<NT, 1, false>;
    else if (tpt == 2) f = yuk ? (const void*)k_nbody_f32<NT, 2, true> : (const void*)k_nbody_f32<NT, 2, false>;
    else if (tpt == 8) f = yuk ? (const void*)k_nbody_f32<NT, 8, true> : (const void*)k_nbody_f32<NT, 8, false>;
    else f = yuk ? (const void*)k_nbody_f32<NT, 4, true> : (const void*)k_nbody_f32<NT, 4, false>;
  }
  int per = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, NT, 0);
  return std::max(1, per);
}

void launch_nbody_f32(Mesh* m, Surface* s, double kappa, int tpt, int packed, int nsplit, int per,
                      const float4* spos, const float4* sdl, double* val) {
  constexpr int NT = F32_NT;
  const int nq = s->nq;
  const int ntb = blocks_for(nq, NT * tpt);
  dim3 grid(ntb, nsplit);
  const float kf = (float)kappa;
  const bool yuk = kappa != 0.0;
  const float4* q4 = s->qpf.p;
#define PB_NB(T)                                                                                    \
  if (yuk) k_nbody_f32<NT, T, true><<<grid, NT, 0, m->stream>>>(nq, q4, spos, sdl, kf, per, val);  \
  else k_nbody_f32<NT, T, false><<<grid, NT, 0, m->stream>>>(nq, q4, spos, sdl, kf, per, val);
#define PB_NB2(P)                                                                                   \
  if (yuk) k_nbody_f32x2<NT, P, true><<<grid, NT, 0, m->stream>>>(nq, q4, spos, sdl, kf, per, val); \
  else k_nbody_f32x2<NT, P, false><<<grid, NT, 0, m->stream>>>(nq, q4, spos, sdl, kf, per, val);
  if (packed) {
    switch (tpt) {
      case 2: PB_NB2(1) break;
      case 8: PB_NB2(4) break;
      default: PB_NB2(2) break;
    }
  } else {
    switch (tpt) {
      case 1: PB_NB(1) break;
      case 2: PB_NB(2) break;
      case 8: PB_NB(8) break;
      default: PB_NB(4) break;
    }
  }
#undef PB_NB
#undef PB_NB2
}

// y (+)= far-field part of the surface rows: for every test function psi_i,
//   sum_{x_q, y_p, q != p} psi_i(x_q) w_q [ g(x_q,y_p) s_p + dg/dn_y(x_q,y_p) m_p ]
// with s_p = cs w_p lam_h(y_p), m_p = cd w_p u_h(y_p) (kernel factors 1/(4 pi) included).
// lam indexed by local surface vertex; x (the shell part of the full vector, or a local
// surface vector when lam == x is a surface vector) indexed through vmap.
int launch_bem_far(Mesh* m, Surface* s, const double* x, const double* lam, double cs, double cd, double kappa,
                   int precision, double* y, bool accumulate, const RowAdd* add) {
  const int nq = s->nq;
  const bool yuk = kappa != 0.0;
  const int u_local = (x != nullptr && x == lam) ? 1 : 0;
  const double* uvec = (cd != 0.0) ? x : nullptr;
  const double* lvec = (cs != 0.0) ? lam : nullptr;
  if (precision == PBFB_FLOAT2) return launch_bem_far_ff(m, s, x, lam, cs, cd, kappa, y, accumulate, add);
  if (precision == PBFB_FP64) {
    double* v;
    PB_TRY(launch_pairs(m, s, x, lam, cs * INV4PI, cd * INV4PI, kappa, true, &v));
    return test_reduce(m, s, v, 1, y, accumulate, add);
  }
  k_sources<<<blocks_for(nq, 256), 256, 0, m->stream>>>(s->nt, s->tri.p, s->vmap.p, lvec, uvec, u_local, s->qw.p,
                                                        s->nrm.p, s->qpf.p, cs * INV4PI, cd * INV4PI, s->spos.p,
                                                        s->sdl.p);
  PB_LAUNCHED(m);
  cudaEvent_t ev;
  KernelClassTimer& tm = m->t_nbody;
  timer_begin(m, tm, &ev);
  int nsplit;
  double* vals = s->val.p;
  double tree_pairs = -1.0;
  if (use_tree(m, s)) {
    PB_TRY(launch_tree_far(m, s, kappa, s->spos.p, s->sdl.p, s->val.p, &tree_pairs));
    nsplit = 1;
  } else {
    int tpt, packed, bps;
    f32_shape(m, nq, &tpt, &packed, &bps);
    if (packed == 2) {
      // mutual pairs: G tile groups, G (G + 1) / 2 one-warp blocks (about bps per SM)
      const int nT = blocks_for(nq, FM_T);
      int G = (int)std::sqrt(2.0 * (bps > 0 ? bps : 32) * 152.0);
      G = std::max(1, std::min(G, nT));
      PB_TRY(ensure(s->mval, (size_t)(2 * G + 1) * nq));
      double* PI = s->mval.p;
      double* PJ = PI + (size_t)G * nq;
      double* out = PJ + (size_t)G * nq;
      PB_CUDA(cudaMemsetAsync(PI, 0, (size_t)2 * G * nq * sizeof(double), m->stream));
      const int nblk = G * (G + 1) / 2;
      if (yuk)
        k_nbody_f32m<true><<<nblk, 32, 0, m->stream>>>(nq, G, s->spos.p, s->sdl.p, (float)kappa, PI, PJ);
      else
        k_nbody_f32m<false><<<nblk, 32, 0, m->stream>>>(nq, G, s->spos.p, s->sdl.p, (float)kappa, PI, PJ);
      PB_LAUNCHED(m);
      k_mutual_sum<<<blocks_for(nq, 256), 256, 0, m->stream>>>(nq, G, PI, PJ, out);
      nsplit = 1;
      vals = out;
    } else {
      const int ntb = blocks_for(nq, F32_NT * tpt);
      if (bps == 0) {
        // whole waves: the largest split with at most 3 waves of resident blocks
        const int cap = f32_blocks_per_sm(tpt, packed, yuk) * 152;
        nsplit = std::max(1, std::min(3 * cap / ntb, blocks_for(nq, 4 * F32_NT)));
      } else {
        nsplit = std::max(1, std::min(blocks_for(bps * 152, ntb), blocks_for(nq, 4 * F32_NT)));
      }
      const int per = blocks_for(blocks_for(nq, nsplit), F32_NT) * F32_NT;
      nsplit = blocks_for(nq, per);
      if ((size_t)nsplit * nq > s->val.n) {
        set_error("far-field split buffer too small");
        return PBFB_ERR_STATE;
      }
      launch_nbody_f32(m, s, kappa, tpt, packed, nsplit, per, s->spos.p, s->sdl.p, s->val.p);
    }
  }
  PB_LAUNCHED(m);
  const double pairs = tree_pairs >= 0.0 ? tree_pairs : (double)nq * (double)nq;
  timer_end(m, tm, ev, pairs);
  m->nbody_flops += (yuk ? 24.0 : 18.0) * pairs;
  return test_reduce(m, s, vals, nsplit, y, accumulate, add);
}

int launch_bem_far_ff(Mesh* m, Surface* s, const double* x, const double* lam, double cs, double cd,
                      double kappa, double* y, bool accumulate, const RowAdd* add) {
  const int nq = s->nq;
  const bool yuk = kappa != 0.0;
  const int u_local = (x != nullptr && x == lam) ? 1 : 0;
  // by pairs of triangles; ff_kernel = 1 asks for the one-target-per-thread sum, which shares no pair formula with them
  // (a check of either by the other) and is slower at every size (K operator, Laplace / Yukawa: 20 triangles 44 / 71
  // against 36 / 40 us; 500, 119 / 241 and 58 / 68; 3920, 2.46 / 4.40 and 1.03 / 1.48 ms; 20,480, 66 / 119 and 26 /
  // 37), so that neither the built-in shapes nor the autotuner take it.  Lengths are scaled by kappa
  // there: a Yukawa kernel with kappa below 1e-8 (no physical ionic strength; the scaled 1/r^3 nears the end of
  // float32's range) takes the float64 form.
  if (m->tune_ff_kernel != 1) {
    double* v;
    PB_TRY(launch_pairs(m, s, x, lam, cs * INV4PI, cd * INV4PI, kappa, kappa > 0.0 && kappa < 1e-8, &v));
    return test_reduce(m, s, v, 1, y, accumulate, add);
  }
  PB_TRY(ff_exp_table(m));
  if (s->ffsrc.n < 4 * (size_t)nq) PB_TRY(s->ffsrc.alloc(4 * (size_t)nq));
  if (s->fftgt.n < 2 * (size_t)nq) PB_TRY(s->fftgt.alloc(2 * (size_t)nq));
  k_sources_ff<<<blocks_for(nq, 256), 256, 0, m->stream>>>(
      s->nt, s->tri.p, s->vmap.p, cs != 0.0 ? lam : nullptr, cd != 0.0 ? x : nullptr, u_local, s->qw.p, s->nrm.p,
      s->qx.p, s->ctr[0], s->ctr[1], s->ctr[2], cs * INV4PI, cd * INV4PI, ff_grid(s, 1.0), s->ffsrc.p, s->fftgt.p);
  PB_LAUNCHED(m);
  cudaEvent_t ev;
  timer_begin(m, m->t_nbodyff, &ev);
  constexpr int NT = 128;
  const int bps = m->tune_ff_bps > 0 ? m->tune_ff_bps : 8;
  const float kh = (float)kappa, kl = (float)(kappa - (double)kh);
  const int ntb = blocks_for(nq, NT);
  int nsplit = std::max(1, std::min(blocks_for(bps * 152, ntb), blocks_for(nq, 4 * NT)));
  const int per = blocks_for(blocks_for(nq, nsplit), NT) * NT;
  nsplit = blocks_for(nq, per);
  if ((size_t)nsplit * nq > s->val.n) {
    set_error("far-field split buffer too small");
    return PBFB_ERR_STATE;
  }
  dim3 grid(ntb, nsplit);
  if (yuk)
    k_nbody_ff<NT, true><<<grid, NT, 0, m->stream>>>(nq, s->fftgt.p, s->ffsrc.p, kh, kl, m->ff_tab.p, per, s->val.p);
  else
    k_nbody_ff<NT, false><<<grid, NT, 0, m->stream>>>(nq, s->fftgt.p, s->ffsrc.p, kh, kl, m->ff_tab.p, per, s->val.p);
  PB_LAUNCHED(m);
  timer_end(m, m->t_nbodyff, ev, (double)nq * (double)nq);
  return test_reduce(m, s, s->val.p, nsplit, y, accumulate, add);
}

int launch_coulomb(Mesh* m) {
  Surface* s = &m->sm;
  const int nb = blocks_for(s->nt, COUL_T);
  const int nchunk = std::max(1, std::min(m->nq, 4 * 152 / nb));
  PB_TRY(ensure(m->coul_ce, 2 * (size_t)s->nq));
  PB_TRY(ensure(s->mval, 2 * (size_t)nchunk * s->nq));
  k_coulomb<<<dim3(nb, nchunk), COUL_T, 0, m->stream>>>(s->nt, s->qx.p, s->nrm.p, m->nq, m->qxyz.p, m->qz.p,
                                                        s->mval.p);
  PB_LAUNCHED(m);
  k_chunk_sum<<<blocks_for(2 * (int64_t)s->nq, 256), 256, 0, m->stream>>>(2 * s->nq, nchunk, s->mval.p, m->coul_ce.p);
  PB_LAUNCHED(m);
  return test_reduce(m, s, m->coul_ce.p, 1, m->coul.p, false);
}

int launch_winding_numbers(Mesh* m, const double* soa, int nq, double* w) {
  Surface* s = &m->sm;
  const int nb = blocks_for(nq, WIND_T);
  const int nchunk = std::max(1, std::min(blocks_for(s->nt, WIND_T), 8 * 152 / nb));
  // the points, then the chunk sums
  PB_TRY(ensure(m->wind, (3 + (size_t)nchunk + 1) * nq));
  double* q = m->wind.p;
  double* part = q + 3 * (size_t)nq;
  double* out = part + (size_t)nchunk * nq;
  PB_CUDA(cudaMemcpyAsync(q, soa, 3 * (size_t)nq * sizeof(double), cudaMemcpyHostToDevice, m->stream));
  k_winding<<<dim3(nb, nchunk), WIND_T, 0, m->stream>>>(s->nt, s->tri.p, s->vmap.p, m->xyz.p, m->nv, nq, q, part);
  PB_LAUNCHED(m);
  k_chunk_sum<<<blocks_for(nq, 256), 256, 0, m->stream>>>(nq, nchunk, part, out);
  PB_LAUNCHED(m);
  PB_CUDA(cudaMemcpyAsync(w, out, nq * sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  PB_CUDA(cudaStreamSynchronize(m->stream));
  for (int k = 0; k < nq; ++k) w[k] = w[k] > 0.5 * WIND_ON ? 0.5 : 2.0 * w[k] / (4.0 * M_PI);
  return PBFB_OK;
}

// 4 pi times the reaction energies sum_k z_k phi(x_k) of x_L and x_NL: out_dev[0], out_dev[1]
int launch_reaction_energy(Mesh* m, const double* xL, const double* xNL, double* out_dev) {
  Surface* s = &m->sm;
  const int nb = std::min(152, blocks_for(s->nq, REAC_T));
  k_reaction_energy<<<nb, REAC_T, 0, m->stream>>>(s->nt, s->tri.p, s->vmap.p, s->qw.p, m->coul_ce.p, xL + s->col0, xL,
                                                  xNL + s->col0, xNL, m->red.p);
  PB_LAUNCHED(m);
  return launch_sum_partials(m, nb, 2, out_dev);
}

}  // namespace pbfb

// ---------------------------------------------------------------- allocation-free far field
//
// pbfb_bem_apply_noalloc (include/pbfb.h) computes what pbfb_bem_apply computes with the
// float32 far field, but keeps all of its working memory in the fixed array below instead
// of buffers owned by the mesh: float32 source records (two float4 per quadrature point)
// followed by the float64 partial potentials of at most NOALLOC_SPLITS source splits.
// The array is a device global of the library: every device that loads libpbfb holds it
// until the process exits.  Calls share it, so calls that run at the same time on the GPU
// (other streams, other threads) overwrite each other's data.  Every call writes all of
// the scratch it reads, so nothing has to be cleared between calls.

namespace pbfb {
namespace {

constexpr int NOALLOC_MAX_QP = 65536;   // quadrature points (6 per triangle): 10922 triangles
constexpr int NOALLOC_SPLITS = 8;
constexpr size_t NOALLOC_BYTES =
    (size_t)NOALLOC_MAX_QP * 2 * sizeof(float4) + (size_t)NOALLOC_SPLITS * NOALLOC_MAX_QP * sizeof(double);

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

// Device address of g_noalloc_scratch per device, looked up on the first call on that device.
// (In host code the symbol's name is only a host-side handle, not the device address.)  The
// entries are atomic: first calls from several host threads (server workers) may race to fill
// one; they all store the same address.
constexpr int NOALLOC_MAX_DEV = 64;
std::atomic<void*> g_noalloc_addr[NOALLOC_MAX_DEV];

int noalloc_scratch(int dev, unsigned char** out) {
  if (dev < 0 || dev >= NOALLOC_MAX_DEV) {
    set_error("bem_apply_noalloc: device ordinal %d out of range", dev);
    return PBFB_ERR_INVALID;
  }
  void* p = g_noalloc_addr[dev].load(std::memory_order_acquire);
  if (!p) {
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      set_error("bem_apply_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      return PBFB_ERR_CUDA;
    }
    g_noalloc_addr[dev].store(p, std::memory_order_release);
  }
  *out = (unsigned char*)p;
  return PBFB_OK;
}

}  // namespace

int bem_apply_noalloc(Mesh* m, int which, int op, const double* x, double* y) {
  Surface* s = which == PBFB_GAMMA_M ? &m->sm : &m->ss;
  const double kappa = which == PBFB_GAMMA_M ? 0.0 : m->kappa;
  const int nq = s->nq;
  if (nq > NOALLOC_MAX_QP) {
    set_error("bem_apply_noalloc: the surface has %d quadrature points; the fixed scratch holds at most %d "
              "(%d triangles)", nq, NOALLOC_MAX_QP, NOALLOC_MAX_QP / QS);
    return PBFB_ERR_INVALID;
  }
  unsigned char* base = nullptr;
  PB_TRY(noalloc_scratch(m->dev, &base));
  float4* spos = (float4*)base;
  float4* sdl = spos + NOALLOC_MAX_QP;
  double* val = (double*)(sdl + NOALLOC_MAX_QP);
  const double cs = op == 0 ? 1.0 : 0.0, cd = op == 1 ? 1.0 : 0.0;
  k_sources<<<blocks_for(nq, 256), 256, 0, m->stream>>>(s->nt, s->tri.p, s->vmap.p, cs != 0.0 ? x : nullptr,
                                                        cd != 0.0 ? x : nullptr, 1, s->qw.p, s->nrm.p, s->qpf.p,
                                                        cs * INV4PI, cd * INV4PI, spos, sdl);
  PB_LAUNCHED(m);
  // The split kernels and targets per thread of pbfb_bem_apply (launch_bem_far), with its split
  // rules (whole waves of resident blocks when blocks_per_sm is 0), capped at NOALLOC_SPLITS
  // source splits.  The mutual-pair variant (packed = 2) needs partial rows for every tile group,
  // more than the fixed array holds: it is replaced by the packed split kernel with the same
  // targets per thread, whose float32 sums run in another order.
  int tpt, packed, bps;
  f32_shape(m, nq, &tpt, &packed, &bps);
  if (packed == 2) {
    packed = tpt >= 2 ? 1 : 0;
    bps = 0;
  }
  const bool yuk = kappa != 0.0;
  const int ntb = blocks_for(nq, F32_NT * tpt);
  int nsplit;
  if (bps == 0) {
    const int cap = f32_blocks_per_sm(tpt, packed, yuk) * 152;
    nsplit = std::max(1, std::min(3 * cap / ntb, blocks_for(nq, 4 * F32_NT)));
  } else {
    nsplit = std::max(1, std::min(blocks_for(bps * 152, ntb), blocks_for(nq, 4 * F32_NT)));
  }
  nsplit = std::min(nsplit, NOALLOC_SPLITS);
  const int per = blocks_for(blocks_for(nq, nsplit), F32_NT) * F32_NT;
  nsplit = blocks_for(nq, per);
  launch_nbody_f32(m, s, kappa, tpt, packed, nsplit, per, spos, sdl, val);
  PB_LAUNCHED(m);
  const RowAdd near = near_rows(s, op, x);
  PB_TRY(test_reduce(m, s, val, nsplit, y, false, &near));
  return PBFB_OK;
}

}  // namespace pbfb
