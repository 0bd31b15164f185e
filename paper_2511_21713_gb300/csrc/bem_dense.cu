// Dense single-layer matrices of the two surfaces and their inverses, used on the surface
// rows of the block preconditioner of GMRES.  The paper solves every Newton increment
// (Sec. 2.4) with GMRES and does not state a preconditioner; this one is a design choice of
// this library.
//
// The diagonal blocks of the coupled operator on the unknowns lam_m and lam_s are -V_L
// (Gamma_m rows) and +V_Y (Gamma_s rows).  Scaling those rows by 1 / diag(V) leaves GMRES
// iterations growing with the condition number of V (like 1/h under refinement); applying
// V^-1 keeps them flat.  V is assembled densely in float32 from the same pieces as the
// matrix-free operator:
//   V = P^T G P + C
// with G the 6 x 6-point rule over all quadrature-point pairs (coincident points excluded),
// P the map from vertex values to weighted point values (w_q psi_i(x_q)), and C the sparse
// exact-minus-regular corrections of touching and near triangle pairs.  It is symmetrised
// and inverted in place by the sweep operator (Goodnight, "A tutorial on the SWEEP
// operator", The American Statistician 33, 1979) in pivot blocks of 64: sweeping every
// pivot of a symmetric positive definite matrix leaves -V^-1.
//
// Storage: row-major float32, leading dimension ld = n rounded up to 128; the padding rows
// and columns hold the identity, so every pivot block and update tile is full.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "device_once.h"
#include "f32x2.cuh"
#include "pbfb_internal.cuh"
#include "quad_tables.cuh"

namespace pbfb {

namespace {

constexpr int DW_T = 2;            // test triangles per block of the row kernel
constexpr int DW_S = 1536;         // trial triangles at a time
constexpr int DW_NT = 384;         // its threads
constexpr int DW_SMEM = 9 * DW_T * DW_S * (int)sizeof(float);
constexpr int SW_B = 64;           // sweep pivot block
constexpr int SW_TILE = 128;       // update tile (and ld granularity)
constexpr size_t DENSE_W_BYTES = size_t(256) << 20;  // float32 work matrix W, per chunk

// Rows (tau, a) of W = Pt^T G P for the triangles tau in [t0, t0 + gridDim.x DW_T): row 3 (tau - t0) + a, column j
// receives sum over (sigma, b) around vertex j with sigma >= tau of L_ab(tau, sigma), the pair tau = sigma halved
// (the other half of the symmetric G comes from the transpose in k_dense_sym), with
//   L_ab = sum_{q, p} w_q psi_a(x_q) g(x_q, y_p) psi_b(y_p) w_p / (4 pi)
// over the 6 x 6 points of the pair (coincident points left out).  A block takes DW_T test triangles and DW_S
// trial triangles at a time: thread sigma evaluates the 36 kernel values once (they serve three vertices on
// either side), contracts them to 3 x 3 and leaves those in shared memory; then a thread per vertex adds the
// entries of its triangles in incidence order.  The kernel's root (and exponential) on the special-function
// unit bounds it: 1 or 2 per point pair, about 8 float32 operations' time each.
// GB300, 3920 triangles (1962 vertices), Yukawa: 1279 us for G P evaluated once per (point, vertex), its weights
// multiplied in float64 each time, and 515 us for the second product; 287 us and 44 us so.
template <bool YUK>
__global__ void __launch_bounds__(DW_NT, 2) k_dense_rows(int nv, int nt, int t0, int t1, const float4* __restrict__ qpf,
                                                      const double* __restrict__ qw, const float* __restrict__ wq,
                                                      const int* __restrict__ inc_ptr,
                                                      const int* __restrict__ inc_idx, float nk,
                                                      float* __restrict__ W) {
  extern __shared__ float4 sm4[];
  float* L = reinterpret_cast<float*>(sm4);  // [DW_T][3 a][3 b][DW_S]
  __shared__ float4 tp[DW_T][QS];            // test points
  __shared__ float tw[DW_T][QS][3];          // w_q psi_a(x_q) / 4 pi
  const int tau0 = t0 + blockIdx.x * DW_T;
  if (threadIdx.x < DW_T * QS) {
    const int u = threadIdx.x / QS, q = threadIdx.x % QS;
    const int j = QS * min(tau0 + u, nt - 1) + q;
    tp[u][q] = qpf[j];
#pragma unroll
    for (int a = 0; a < 3; ++a) tw[u][q][a] = (float)(qw[j] * c_tri_b[q][a] * 0.079577471545947667884);
  }
  __syncthreads();
  for (int s0 = tau0; s0 < nt; s0 += DW_S) {
    const int s1 = min(nt, s0 + DW_S);
    for (int s = s0 + threadIdx.x; s < s1; s += DW_NT) {
      float y[QS][3], wb[QS][3];
#pragma unroll
      for (int p = 0; p < QS; ++p) {
        const float4 f = qpf[QS * s + p];
        y[p][0] = f.x;
        y[p][1] = f.y;
        y[p][2] = f.z;
#pragma unroll
        for (int b = 0; b < 3; ++b) wb[p][b] = wq[(size_t)b * QS * nt + QS * s + p];
      }
#pragma unroll 1
      for (int u = 0; u < DW_T; ++u) {
        const bool own = s == tau0 + u;
        float acc[3][3] = {};
#pragma unroll
        for (int q = 0; q < QS; ++q) {
          const float4 x = tp[u][q];
          float h[3] = {};
#pragma unroll
          for (int p = 0; p < QS; ++p) {
            const float dx = x.x - y[p][0], dy = x.y - y[p][1], dz = x.z - y[p][2];
            // the coincident point gets r2 = 1e-30 (finite terms) and weight 0
            const float r2 = fmaxf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)), 1e-30f);
            const float ir = rsqrt_approx(r2);
            float g = ir;
            if (YUK) g *= ex2_approx(nk * (r2 * ir));
            if (p == q && own) g = 0.f;
#pragma unroll
            for (int b = 0; b < 3; ++b) h[b] = fmaf(g, wb[p][b], h[b]);
          }
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float wa = tw[u][q][a];
#pragma unroll
            for (int b = 0; b < 3; ++b) acc[a][b] = fmaf(wa, h[b], acc[a][b]);
          }
        }
        const float f = own ? 0.5f : (s < tau0 + u ? 0.f : 1.f);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) L[((3 * u + a) * 3 + b) * DW_S + s - s0] = f * acc[a][b];
      }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < nv; j += DW_NT) {
      float v[3 * DW_T];
#pragma unroll
      for (int r = 0; r < 3 * DW_T; ++r) v[r] = 0.f;
      for (int e = inc_ptr[j]; e < inc_ptr[j + 1]; ++e) {
        const int ent = inc_idx[e], s = ent / 3, b = ent - 3 * s;
        if (s < s0 || s >= s1) continue;
#pragma unroll
        for (int r = 0; r < 3 * DW_T; ++r) v[r] += L[(3 * r + b) * DW_S + s - s0];
      }
#pragma unroll
      for (int r = 0; r < 3 * DW_T; ++r)
        if (tau0 + r / 3 < t1) {
          float* w = W + (size_t)(3 * (tau0 - t0) + r) * nv + j;
          *w = s0 > tau0 ? *w + v[r] : v[r];
        }
    }
    __syncthreads();
  }
}

// A[i][j] += sum over (tau, a) around vertex i with tau in [t0, t1) of W's row (tau, a)
__global__ void k_dense_fold(int nv, int ld, int t0, int t1, const float* __restrict__ W,
                             const int* __restrict__ inc_ptr, const int* __restrict__ inc_idx, float* __restrict__ A) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (j >= nv) return;
  float acc = 0.f;
  bool any = false;
  for (int e = inc_ptr[i]; e < inc_ptr[i + 1]; ++e) {
    const int ent = inc_idx[e], t = ent / 3, a = ent - 3 * t;
    if (t < t0 || t >= t1) continue;
    any = true;
    acc += W[(size_t)(3 * (t - t0) + a) * nv + j];
  }
  if (any) A[(size_t)i * ld + j] += acc;
}

// wq[b][j] = w_j psi_b(y_j)
__global__ void k_dense_weights(int nq, const double* __restrict__ qw, float* __restrict__ wq) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nq) return;
  for (int b = 0; b < 3; ++b) wq[(size_t)b * nq + j] = (float)(qw[j] * c_tri_b[j % QS][b]);
}

// zero, with the identity on the padding diagonal
__global__ void k_dense_init(int n, int ld, float* __restrict__ A) {
  const size_t tot = (size_t)ld * ld;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / ld), j = (int)(e - (size_t)i * ld);
    A[e] = (i == j && i >= n) ? 1.f : 0.f;
  }
}

// half of the sparse exact-minus-regular corrections, one thread per row
__global__ void k_dense_corr(int nv, int ld, const int* __restrict__ ptr, const int* __restrict__ col,
                             const double* __restrict__ corr, float* __restrict__ A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nv) return;
  for (int s = ptr[i]; s < ptr[i + 1]; ++s) A[(size_t)i * ld + col[s]] += 0.5f * (float)corr[s];
}

// A <- A + A^T by 32 x 32 tiles on and above the diagonal; a block writes a tile and its mirror image
__global__ void k_dense_sym(int n, int ld, float* __restrict__ A) {
  __shared__ float t[32][33], r[32][33];
  const int I = blockIdx.y, J = blockIdx.x;
  if (J < I) return;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int i = 32 * I + k, j = 32 * J + threadIdx.x;  // ld is a multiple of 128: the padding tiles exist
    t[k][threadIdx.x] = A[(size_t)i * ld + j];
    r[k][threadIdx.x] = A[(size_t)(32 * J + k) * ld + 32 * I + threadIdx.x];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int i = 32 * I + k, j = 32 * J + threadIdx.x;
    if (i < n && j < n) A[(size_t)i * ld + j] = t[k][threadIdx.x] + r[threadIdx.x][k];
    if (I != J && 32 * J + k < n && 32 * I + threadIdx.x < n)
      A[(size_t)(32 * J + k) * ld + 32 * I + threadIdx.x] = r[k][threadIdx.x] + t[threadIdx.x][k];
  }
}

// Sweep of the SW_B x SW_B pivot block at (k0, k0), scalar pivots in order, and the row panel of the pivot:
// P = A[K, :] (old values) and U = D P, D = -S the inverse of the block; the swept block S is written and a pivot
// that is not positive and finite flagged.  Only the tiles on and below the diagonal are kept current during the
// sweep (the matrix stays symmetric), so row K beyond its diagonal tile is read from column K: A[K][j] = A[j][K].
// The 64 dependent pivot steps bound it: every block sweeps the pivot block itself (no launch between the two
// halves), a thread keeping a 4 x 4 piece in registers and a step passing the pivot's row and column through
// one of two shared buffers, so that it needs one barrier; the panel's columns are loaded before.  A block takes
// 128 columns and nr of U's rows (blockIdx.y): fewer rows for more blocks on small matrices.
// GB300, ld = 2048, per step: 37.5 us for one block with four barriers a pivot and 15 us for the panel; 20.5 us
// together, and one launch gap less.
__global__ void __launch_bounds__(256) k_sweep_pivot_panel(int ld, int k0, int nr, const float* __restrict__ A,
                                                           float* __restrict__ S, float* __restrict__ P,
                                                           float* __restrict__ U, int* __restrict__ flag) {
  __shared__ float rowp[2][SW_B], colp[2][SW_B];
  __shared__ float sD[SW_B][SW_B];
  const int col = threadIdx.x & 127, half = threadIdx.x >> 7;
  const int j = blockIdx.x * 128 + col;  // ld is a multiple of 128
  const int kend = (k0 / SW_TILE + 1) * SW_TILE;  // end of the pivot's diagonal tile
  float pv[SW_B];
  if (j < kend) {
#pragma unroll
    for (int p = 0; p < SW_B; ++p) pv[p] = A[(size_t)(k0 + p) * ld + j];
  } else {
    const float4* c = reinterpret_cast<const float4*>(A + (size_t)j * ld + k0);
#pragma unroll
    for (int q = 0; q < SW_B / 4; ++q) {
      const float4 v = c[q];
      pv[4 * q] = v.x;
      pv[4 * q + 1] = v.y;
      pv[4 * q + 2] = v.z;
      pv[4 * q + 3] = v.w;
    }
  }
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;  // rows tr + 16 i, columns tc + 16 j
  float v[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) v[i][c] = A[(size_t)(k0 + tr + 16 * i) * ld + k0 + tc + 16 * c];
  bool bad = false;
#pragma unroll
  for (int pi = 0; pi < 4; ++pi)
#pragma unroll 1
    for (int pk = 0; pk < 16; ++pk) {
      const int p = 16 * pi + pk, buf = pk & 1;
      if (tr == pk)
#pragma unroll
        for (int c = 0; c < 4; ++c) rowp[buf][tc + 16 * c] = v[pi][c];
      if (tc == pk)
#pragma unroll
        for (int i = 0; i < 4; ++i) colp[buf][tr + 16 * i] = v[i][pi];
      __syncthreads();
      const float d = rowp[buf][p];
      bad = bad || !(d > 0.f) || !isfinite(d);
      const float inv = 1.f / d;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float x = colp[buf][tr + 16 * i];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[i][c] -= x * rowp[buf][tc + 16 * c] * inv;
      }
      if (tr == pk)
#pragma unroll
        for (int c = 0; c < 4; ++c) v[pi][c] = rowp[buf][tc + 16 * c] * inv;
      if (tc == pk)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i][pi] = colp[buf][tr + 16 * i] * inv;
      if (tr == pk && tc == pk) v[pi][pi] = -inv;
    }
  const bool first = blockIdx.x == 0 && blockIdx.y == 0;
  if (first && threadIdx.x == 0 && bad) atomicExch(flag, 1);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sD[tr + 16 * i][tc + 16 * c] = -v[i][c];
      if (first) S[(tr + 16 * i) * SW_B + tc + 16 * c] = v[i][c];
    }
  __syncthreads();
  if (blockIdx.y == 0 && half == 0)
#pragma unroll
    for (int p = 0; p < SW_B; ++p) P[(size_t)p * ld + j] = pv[p];
  for (int p = blockIdx.y * nr + half; p < (int)(blockIdx.y + 1) * nr; p += 2) {
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < SW_B; ++q) acc += sD[p][q] * pv[q];
    U[(size_t)p * ld + j] = acc;
  }
}

// Trailing update of one sweep step, 128 x 128 tiles on and below the diagonal (tile row >= tile
// column; the swept matrix is symmetric, the upper tiles are mirrored after the last step), 8 x 8
// per thread:
//   A[i][j] -= sum_p P[p][i] U[p][j]   (i, j outside K)
//   A[K][j] = U[:, j],  A[i][K] = U[:, i]^T,  A[K][K] = S
__global__ void __launch_bounds__(256) k_sweep_update(int ld, int k0, float* __restrict__ A,
                                                      const float* __restrict__ P, const float* __restrict__ U,
                                                      const float* __restrict__ S) {
  extern __shared__ float4 sm4[];
  float* Ps = reinterpret_cast<float*>(sm4);
  float* Us = Ps + SW_B * SW_TILE;
  const int tid = threadIdx.x;
  // blockIdx.x = I (I + 1) / 2 + J, J <= I
  int I = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((I + 1) * (I + 2) / 2 <= (int)blockIdx.x) ++I;
  while (I * (I + 1) / 2 > (int)blockIdx.x) --I;
  const int J = (int)blockIdx.x - I * (I + 1) / 2;
  const int i0 = I * SW_TILE, j0 = J * SW_TILE;
  for (int e = tid; e < SW_B * SW_TILE / 4; e += 256) {
    const int p = e / (SW_TILE / 4), c4 = e % (SW_TILE / 4);
    reinterpret_cast<float4*>(Ps)[e] = *reinterpret_cast<const float4*>(P + (size_t)p * ld + i0 + 4 * c4);
    reinterpret_cast<float4*>(Us)[e] = *reinterpret_cast<const float4*>(U + (size_t)p * ld + j0 + 4 * c4);
  }
  __syncthreads();
  const int ty = tid / 16, tx = tid % 16;
  float acc[8][8];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[r][c] = 0.f;
#pragma unroll 4
  for (int p = 0; p < SW_B; ++p) {
    float a[8];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float4 v = *reinterpret_cast<const float4*>(Ps + p * SW_TILE + 8 * ty + 4 * r);
      a[4 * r] = v.x;
      a[4 * r + 1] = v.y;
      a[4 * r + 2] = v.z;
      a[4 * r + 3] = v.w;
    }
    const float4 b0 = *reinterpret_cast<const float4*>(Us + p * SW_TILE + 4 * tx);
    const float4 b1 = *reinterpret_cast<const float4*>(Us + p * SW_TILE + 64 + 4 * tx);
    const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[r][c] += a[r] * b[c];
  }
  const bool slow = (k0 >= i0 && k0 < i0 + SW_TILE) || (k0 >= j0 && k0 < j0 + SW_TILE);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = i0 + 8 * ty + r;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = j0 + 64 * h + 4 * tx;
      float4* dst = reinterpret_cast<float4*>(A + (size_t)i * ld + j);
      float4 o = *dst;
      float v[4] = {o.x - acc[r][4 * h], o.y - acc[r][4 * h + 1], o.z - acc[r][4 * h + 2], o.w - acc[r][4 * h + 3]};
      if (slow) {
        const unsigned di = (unsigned)(i - k0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const unsigned dj = (unsigned)(j + c - k0);
          if (di < SW_B && dj < SW_B)
            v[c] = S[di * SW_B + dj];
          else if (di < SW_B)
            v[c] = U[(size_t)di * ld + j + c];
          else if (dj < SW_B)
            v[c] = U[(size_t)dj * ld + i];
        }
      }
      *dst = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// Upper tiles from the lower ones after the sweep: A[j][i] = A[i][j] for tile row I > tile column J,
// through a 32 x 33 shared-memory transpose; block = one 32 x 32 sub-tile of a lower tile.
__global__ void k_sweep_mirror(int ld, float* __restrict__ A) {
  __shared__ float t[32][33];
  const int nt = ld / 32;
  const int b = blockIdx.x;  // lower sub-tiles (I > J) in row-major order
  int I = (int)((sqrtf(8.f * (float)b + 1.f) + 1.f) * 0.5f);
  while (I * (I - 1) / 2 > b) --I;
  while ((I + 1) * I / 2 <= b) ++I;
  const int J = b - I * (I - 1) / 2;
  if (I >= nt || J >= I) return;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) t[r][threadIdx.x] = A[(size_t)(32 * I + r) * ld + 32 * J + threadIdx.x];
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) A[(size_t)(32 * J + r) * ld + 32 * I + threadIdx.x] = t[threadIdx.x][r];
}

// z[i] = scale * sum_j A[i][j] v[j], i < n: one warp per row, v staged in shared memory as float
__global__ void __launch_bounds__(256) k_dense_apply(int n, int ld, const float* __restrict__ A, double scale,
                                                     const double* __restrict__ v, double* __restrict__ z) {
  extern __shared__ float4 vs4[];
  float* vs = reinterpret_cast<float*>(vs4);
  for (int j = threadIdx.x; j < ld; j += 256) vs[j] = j < n ? (float)v[j] : 0.f;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;  // the whole warp leaves together
  const float4* row = reinterpret_cast<const float4*>(A + (size_t)i * ld);
  float acc = 0.f;
  for (int c = lane; c < ld / 4; c += 32) {
    const float4 a = row[c];
    const float4 x = vs4[c];
    acc += a.x * x.x + a.y * x.y + a.z * x.z + a.w * x.w;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) z[i] = scale * (double)acc;
}

// out[i * ld_out + j] = scale * A[i * ld + j], i, j < n
__global__ void k_dense_copy(int n, int ld, const float* __restrict__ A, float scale, float* __restrict__ out,
                             int ld_out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (j < n) out[(size_t)i * ld_out + j] = scale * A[(size_t)i * ld + j];
}

int ensure_f(DBuf<float>& b, size_t n) {
  if (b.n >= n) return PBFB_OK;
  return b.alloc(n);
}

}  // namespace

int dense_ld(int n) { return (n + SW_TILE - 1) / SW_TILE * SW_TILE; }

size_t dense_bytes(int n) {
  const size_t ld = (size_t)dense_ld(n);
  return ld * ld * 4;
}

size_t dense_work_bytes(int n, int nt) {
  const size_t ld = (size_t)dense_ld(n);
  return std::min(DENSE_W_BYTES, (size_t)3 * nt * n * 4) + (2 * SW_B * ld + SW_B * SW_B + 64 + (size_t)3 * QS * nt) * 4;
}

int build_dense_single_layer(Mesh* m, Surface* s, double kappa, bool invert) {
  const int n = s->nv, nt = s->nt;
  if (n < 1 || n > DENSE_V_MAX) {
    set_error("dense single layer: %d surface vertices (limit %d)", n, DENSE_V_MAX);
    return PBFB_ERR_INVALID;
  }
  if (s->kappa != kappa) {
    set_error("dense single layer: corrections were built for kappa %g, not %g", s->kappa, kappa);
    return PBFB_ERR_STATE;
  }
  const int ld = dense_ld(n);
  s->vinv_ok = false;
  PB_TRY(ensure_f(s->vinv, (size_t)ld * ld));
  s->vinv_ld = ld;
  // triangles per chunk of W (at most DENSE_W_BYTES of float32, released after the build)
  const int ct = (int)std::max<size_t>(1, std::min<size_t>(nt, DENSE_W_BYTES / ((size_t)3 * n * 4)));
  const size_t wlen = ((size_t)ct * 3 * n + 63) / 64 * 64;  // keeps the panels 256-byte aligned
  PB_TRY(ensure_f(m->dwork, wlen + 2 * (size_t)SW_B * ld + SW_B * SW_B + 3 * (size_t)s->nq));
  if (m->dflag.n < 1) PB_TRY(m->dflag.alloc(1));
  float* W = m->dwork.p;
  float* P = W + wlen;
  float* U = P + (size_t)SW_B * ld;
  float* S = U + (size_t)SW_B * ld;
  float* wq = S + SW_B * SW_B;
  float* A = s->vinv.p;
  cudaEvent_t ev;
  timer_begin(m, m->t_dense, &ev);
  k_dense_init<<<4 * 152, 256, 0, m->stream>>>(n, ld, A);
  PB_LAUNCHED(m);
  k_dense_weights<<<(s->nq + 255) / 256, 256, 0, m->stream>>>(s->nq, s->qw.p, wq);
  PB_LAUNCHED(m);
  const int gj = (n + 127) / 128;
  const float nk = (float)(-kappa * 1.44269504088896340736);
  for (int t0 = 0; t0 < nt; t0 += ct) {
    const int t1 = std::min(nt, t0 + ct);
    const auto fn = kappa != 0.0 ? k_dense_rows<true> : k_dense_rows<false>;
    fn<<<(t1 - t0 + DW_T - 1) / DW_T, DW_NT, DW_SMEM, m->stream>>>(n, nt, t0, t1, s->qpf.p, s->qw.p, wq, s->inc_ptr.p,
                                                                   s->inc_idx.p, nk, W);
    PB_LAUNCHED(m);
    k_dense_fold<<<dim3(gj, n), 128, 0, m->stream>>>(n, ld, t0, t1, W, s->inc_ptr.p, s->inc_idx.p, A);
    PB_LAUNCHED(m);
  }
  k_dense_corr<<<(n + 127) / 128, 128, 0, m->stream>>>(n, ld, s->c_ptr.p, s->c_col.p, s->corrV.p, A);
  PB_LAUNCHED(m);
  const int n32 = (n + 31) / 32;
  k_dense_sym<<<dim3(n32, n32), dim3(32, 8), 0, m->stream>>>(n, ld, A);
  PB_LAUNCHED(m);
  if (invert) {
    PB_CUDA(cudaMemsetAsync(m->dflag.p, 0, sizeof(int), m->stream));
    const int smem = 2 * SW_B * SW_TILE * (int)sizeof(float);  // attribute set by init_dense_attributes
    const int ntile = ld / SW_TILE;
    const int gu = ntile * (ntile + 1) / 2;  // tiles on and below the diagonal
    const int nr = ld <= 2432 ? 8 : (ld <= 4864 ? 16 : (ld <= 9728 ? 32 : SW_B));  // about a block an SM
    for (int k0 = 0; k0 < ld; k0 += SW_B) {
      k_sweep_pivot_panel<<<dim3(ld / 128, SW_B / nr), 256, 0, m->stream>>>(ld, k0, nr, A, S, P, U, m->dflag.p);
      PB_LAUNCHED(m);
      k_sweep_update<<<gu, 256, smem, m->stream>>>(ld, k0, A, P, U, S);
      PB_LAUNCHED(m);
    }
    const int l32 = ld / 32;
    k_sweep_mirror<<<l32 * (l32 - 1) / 2, dim3(32, 8), 0, m->stream>>>(ld, A);
    PB_LAUNCHED(m);
    PB_CUDA(cudaMemcpyAsync(m->pinned, m->dflag.p, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
  }
  timer_end(m, m->t_dense, ev, invert ? 2.0 * (double)ld * ld * ld : 0.0);
  PB_CUDA(cudaStreamSynchronize(m->stream));
  m->dwork.release();
  if (invert && reinterpret_cast<const int*>(m->pinned)[0] != 0) {
    set_error("dense single layer: a pivot of the float32 sweep was not positive");
    return PBFB_ERR_NONFINITE;
  }
  s->vinv_ok = invert;
  s->vinv_kappa = kappa;
  return PBFB_OK;
}

// Dynamic shared-memory limits of the dense kernels, set once per device by the first mesh
// creation, before any solve: the largest sweep tile pair, and the apply kernel's vector of
// dense_ld(DENSE_V_MAX) floats (every surface's fits).  Solves running on several host threads
// then never change a kernel's attributes while another thread launches or captures it, and a
// smaller matrix never lowers the limit a larger one needs.
int init_dense_attributes() {
  static DeviceOnce once;
  int dev = 0;
  PB_CUDA(cudaGetDevice(&dev));
  return once.run(dev, []() -> int {
    PB_CUDA(cudaFuncSetAttribute(k_sweep_update, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 2 * SW_B * SW_TILE * (int)sizeof(float)));
    for (const void* f : {(const void*)k_dense_rows<true>, (const void*)k_dense_rows<false>})
      PB_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM));
    PB_CUDA(cudaFuncSetAttribute(k_dense_apply, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 dense_ld(DENSE_V_MAX) * (int)sizeof(float)));
    return PBFB_OK;
  });
}

int launch_dense_apply(Mesh* m, Surface* s, double scale, const double* v, double* z) {
  if (!s->vinv_ok) {
    set_error("dense single-layer inverse not built");
    return PBFB_ERR_STATE;
  }
  const int smem = s->vinv_ld * (int)sizeof(float);  // within the limit of init_dense_attributes
  k_dense_apply<<<(s->nv + 7) / 8, 256, smem, m->stream>>>(s->nv, s->vinv_ld, s->vinv.p, scale, v, z);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

int dense_copy_out(Mesh* m, Surface* s, float scale, float* out, int ld_out) {
  k_dense_copy<<<dim3((s->nv + 127) / 128, s->nv), 128, 0, m->stream>>>(s->nv, s->vinv_ld, s->vinv.p, scale, out,
                                                                         ld_out);
  PB_LAUNCHED(m);
  return PBFB_OK;
}

}  // namespace pbfb
