// Near-field corrections of the boundary operators: for every ordered pair of touching or close triangles the
// accurate rule of its class minus the 6 x 6 rule that the far-field sum applies (Sec. 3's quadrature; classes
// in bem_kernels.cu), 3 x 3 values per pair for V and K.
//
// The float64 pipe bounds this (one operation per 64 float32 ones): once per mesh for Gamma_m, once per kappa
// for Gamma_s.  A warp per pair, and few operations per point:
//   - touching pairs (Sauter-Schwab, 5 Gauss points per variable): with the first three variables fixed the last
//     one, e, moves one of the two points along a straight line while the other stands still, so five points
//     share their difference vector D0 + e D1, their weight and the hat functions: per point three operations
//     for the difference, three for r^2, the root (and exponential), and five sums of g, e g, h, e h, e^2 h; the
//     3 x 3 moments follow once per five points.  The fixed and moving points of all triples are tables.
//   - n . (x - y) is linear in e (0 for a trial point that moves in its own plane);
//   - close pairs (6 x 96 points): five lanes per test point, whose plane distance and hats are constants.
// The 27 sums of a pair are added over the warp by halving exchanges (31 additions, lane l ends with value l).
// GB300, 2880 triangles (96,060 pairs): 24.5 ms with every point's map, weights, division, library root
// and exponential and nine sums per kernel, for either surface; 6.6 ms (Laplace) and 8.6 ms (Yukawa) so.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "fp64_math.cuh"
#include "pbfb_internal.cuh"
#include "quad_tables.cuh"

namespace pbfb {

namespace {

constexpr int NGL = 5;        // Gauss-Legendre points per Sauter-Schwab variable
constexpr int NSUB = 96;      // 16 sub-triangles x 6 points
constexpr int NTRIPLE = NGL * NGL * NGL;
constexpr int N_IDENT = 6 * NTRIPLE, N_EDGE = 5 * NTRIPLE, N_VERT = 2 * NTRIPLE;
constexpr int N_ROWS = N_IDENT + N_EDGE + N_VERT;
constexpr int CW = 4;         // warps (pairs) per block
constexpr double INV4PI = 0.079577471545947667884;

__constant__ double c_gl_x[NGL], c_gl_w[NGL];
// per triple: fixed point (f1, f2), moving point (a1 + e b1, a2 + e b2) on {0 <= s2 <= s1 <= 1}, the weight
// of the first three variables with the map's Jacobian, and whether the test point is the moving one
__device__ double d_row[7][N_ROWS];
__device__ unsigned char d_xmoves[N_ROWS];
// sub-triangle rule: barycentrics 1 and 2 and the weight times each of the three
__device__ double d_sub[5][NSUB];

// lane l's total over the warp of value l of v (all 32 lanes call): at each step a lane keeps the half of the
// values its number selects and adds its partner's
__device__ __forceinline__ double warp_scatter_sum(double (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double send = up ? v[i] : v[i + o];
      v[i] = (up ? v[i + o] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return v[0];
}

// g = exp(-kappa r) / r and h = (1 + kappa r) exp(-kappa r) / r^3
template <bool YUK>
__device__ __forceinline__ void kernel_gh(double r2, double kappa, double beta, const double* __restrict__ tab,
                                          double& g, double& h) {
  const double y = rsqrt64(r2), yy = y * y;
  if (YUK) {
    g = y * exp2_neg(beta * (r2 * y), tab);
    h = g * fma(kappa, y, yy);
  } else {
    g = y;
    h = y * yy;
  }
}

// One warp per pair.  Outputs, per pair, 9 entries in stored local vertex order (a of the test triangle, b of
// the trial one): corrV/corrK = accurate rule - 6 x 6 rule (coincident points excluded, plane distances from the
// trial triangle's first point as the far field takes them), fullV = accurate single-layer value (for the
// operator diagonal), mass = P1 mass entries (identical pairs only).
template <bool YUK>
__global__ void __launch_bounds__(32 * CW) k_pair_corrections(
    int npair, const int* __restrict__ pt_, const int* __restrict__ ps_, const int* __restrict__ cls_,
    const int* __restrict__ perm_, const int* __restrict__ tri, const int* __restrict__ vmap,
    const double* __restrict__ xyz, int nvtot, const double* __restrict__ nrm, const double* __restrict__ area,
    const double* __restrict__ qx, const double* __restrict__ qw, int nt, double kappa,
    const double* __restrict__ tab, double* __restrict__ corrV, double* __restrict__ corrK,
    double* __restrict__ fullV, double* __restrict__ mass) {
  __shared__ double s_E[CW][2][2][3];   // [trial, test][P1 - P0, P2 - P1] in rule order
  __shared__ double s_b6[QS][3];        // the 6-point rule's barycentrics
  __shared__ double s_out[CW][27];
  if (threadIdx.x < 3 * QS) s_b6[threadIdx.x / 3][threadIdx.x % 3] = c_tri_b[threadIdx.x / 3][threadIdx.x % 3];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pair = blockIdx.x * CW + w;
  if (pair >= npair) return;  // warps are independent from here on
  const int t = pt_[pair], s = ps_[pair], cls = cls_[pair];
  const int* pm = perm_ + 6 * (size_t)pair;
  const double beta = kappa * 1.44269504088896340736;
  double ns[3];
  for (int d = 0; d < 3; ++d) ns[d] = nrm[(size_t)d * nt + s];
  if (lane < 12) {
    const int which = lane / 6, k = (lane / 3) % 2, d = lane % 3, tr = which ? t : s, o = which ? 0 : 3;
    const double* X = xyz + (size_t)d * nvtot;
    s_E[w][which][k][d] = X[vmap[tri[3 * tr + pm[o + k + 1]]]] - X[vmap[tri[3 * tr + pm[o + k]]]];
  }
  __syncwarp();
  const double At = area[t], As = area[s];
  // v: 0..8 the accurate single layer (moments or hats), 9..17 the double layer's, 18..26 the 6 x 6 single layer;
  // the 6 x 6 double layer is taken off v[9..17] of close pairs and kept in rd for the moments of touching ones
  double v[32], rd[9];
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = 0.0;
#pragma unroll
  for (int k = 0; k < 9; ++k) rd[k] = 0.0;
  if (cls != PAIR_NEAR) {
    const int r0 = cls == PAIR_IDENTICAL ? 0 : (cls == PAIR_EDGE ? N_IDENT : N_IDENT + N_EDGE);
    const int r1 = r0 + (cls == PAIR_IDENTICAL ? N_IDENT : (cls == PAIR_EDGE ? N_EDGE : N_VERT));
    // n . E of the test triangle's edges: 0 for edges that lie in the trial plane
    double nE1 = 0.0, nE2 = 0.0;
    if (cls == PAIR_VERTEX)
      nE1 = fma(ns[2], s_E[w][1][0][2], fma(ns[1], s_E[w][1][0][1], ns[0] * s_E[w][1][0][0]));
    if (cls != PAIR_IDENTICAL)
      nE2 = fma(ns[2], s_E[w][1][1][2], fma(ns[1], s_E[w][1][1][1], ns[0] * s_E[w][1][1][0]));
    for (int r = r0 + lane; r < r1; r += 32) {
      const double f1 = d_row[0][r], f2 = d_row[1][r], a1 = d_row[2][r], b1 = d_row[3][r], a2 = d_row[4][r],
                   b2 = d_row[5][r], W = d_row[6][r];
      const int xm = d_xmoves[r];
      double D0[3], D1[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double m1 = s_E[w][xm][0][d], m2 = s_E[w][xm][1][d];
        D0[d] = fma(-f2, s_E[w][1 - xm][1][d], fma(-f1, s_E[w][1 - xm][0][d], fma(a2, m2, a1 * m1)));
        D1[d] = fma(b2, m2, b1 * m1);
      }
      double G0 = 0.0, G1 = 0.0, H0 = 0.0, H1 = 0.0, H2 = 0.0;
#pragma unroll
      for (int k = 0; k < NGL; ++k) {
        const double e = c_gl_x[k], we = c_gl_w[k], wee = we * e;
        const double d0 = fma(e, D1[0], D0[0]), d1 = fma(e, D1[1], D0[1]), d2 = fma(e, D1[2], D0[2]);
        double g, h;
        kernel_gh<YUK>(fma(d2, d2, fma(d1, d1, d0 * d0)), kappa, beta, tab, g, h);
        G0 = fma(we, g, G0);
        G1 = fma(wee, g, G1);
        H0 = fma(we, h, H0);
        H1 = fma(wee, h, H1);
        H2 = fma(wee * e, h, H2);
      }
      // n . (x - y) = n0 + e n1, x measured from the shared rule vertex 0
      const double n0 = xm ? fma(a2, nE2, a1 * nE1) : fma(f2, nE2, f1 * nE1);
      const double n1 = xm ? fma(b2, nE2, b1 * nE1) : 0.0;
      const double L0 = W * fma(n1, H1, n0 * H0), L1 = W * fma(n1, H2, n0 * H1);
      G0 *= W;
      G1 *= W;
      // moments 1, s1, s2 of both points: those of the moving one from the sums
      const double gm[3] = {G0, fma(b1, G1, a1 * G0), fma(b2, G1, a2 * G0)};
      const double lm[3] = {L0, fma(b1, L1, a1 * L0), fma(b2, L1, a2 * L0)};
      const double ff[3] = {1.0, f1, f2};
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const double gi = xm ? gm[i] : gm[j], li = xm ? lm[i] : lm[j], fj = xm ? ff[j] : ff[i];
          v[3 * i + j] = fma(gi, fj, v[3 * i + j]);
          v[9 + 3 * i + j] = fma(li, fj, v[9 + 3 * i + j]);
        }
    }
    const double jac = 4.0 * At * As * INV4PI;
#pragma unroll
    for (int k = 0; k < 18; ++k) v[k] *= jac;
  } else if (lane < 5 * QS) {
    // test point q of this lane against every fifth sub-rule point; rule order = stored order
    const int q = lane / 5;
    const double bq[3] = {s_b6[q][0], s_b6[q][1], s_b6[q][2]};
    double X[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double* P = xyz + (size_t)d * nvtot;
      const double p0 = P[vmap[tri[3 * t]]], q0 = P[vmap[tri[3 * s]]];
      // X - Ps0
      X[d] = fma(bq[1], s_E[w][1][0][d], fma(bq[2], s_E[w][1][0][d] + s_E[w][1][1][d], p0 - q0));
    }
    const double nd = fma(ns[2], X[2], fma(ns[1], X[1], ns[0] * X[0]));
    double G[3] = {0.0, 0.0, 0.0}, H[3] = {0.0, 0.0, 0.0};
    for (int p = lane % 5; p < NSUB; p += 5) {
      // Y - Ps0 = c1 (P1 - P0) + c2 (P2 - P1), c1 = b1 + b2, c2 = b2
      const double c1 = d_sub[0][p], c2 = d_sub[1][p];
      const double d0 = fma(-c2, s_E[w][0][1][0], fma(-c1, s_E[w][0][0][0], X[0]));
      const double d1 = fma(-c2, s_E[w][0][1][1], fma(-c1, s_E[w][0][0][1], X[1]));
      const double d2 = fma(-c2, s_E[w][0][1][2], fma(-c1, s_E[w][0][0][2], X[2]));
      double g, h;
      kernel_gh<YUK>(fma(d2, d2, fma(d1, d1, d0 * d0)), kappa, beta, tab, g, h);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const double wb = d_sub[2 + b][p];
        G[b] = fma(wb, g, G[b]);
        H[b] = fma(wb, h, H[b]);
      }
    }
    const double f = c_tri_w[q] * At * As * INV4PI;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        v[3 * a + b] = f * bq[a] * G[b];
        v[9 + 3 * a + b] = f * nd * bq[a] * H[b];
      }
  }
  // 6 x 6 rule in stored order (what the far-field sum adds), coincident points excluded
  const int nqt = QS * nt;
  for (int k = lane; k < QS * QS; k += 32) {
    const int q = k / QS, p = k - q * QS;
    if (t == s && q == p) continue;
    const double x0 = qx[QS * t + q], x1 = qx[nqt + QS * t + q], x2 = qx[2 * nqt + QS * t + q];
    const int j = QS * s + p, j0 = QS * s;
    const double d0 = x0 - qx[j], d1 = x1 - qx[nqt + j], d2 = x2 - qx[2 * nqt + j];
    double g, h;
    kernel_gh<YUK>(fma(d2, d2, fma(d1, d1, d0 * d0)), kappa, beta, tab, g, h);
    const double D = t == s ? 0.0
                            : fma(ns[2], x2 - qx[2 * nqt + j0], fma(ns[1], x1 - qx[nqt + j0], ns[0] * (x0 - qx[j0])));
    const double W = qw[QS * t + q] * qw[j] * INV4PI;
    g *= W;
    h *= W * D;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const double bb = s_b6[q][a] * s_b6[p][b];
        v[18 + 3 * a + b] = fma(g, bb, v[18 + 3 * a + b]);
        rd[3 * a + b] = fma(h, bb, rd[3 * a + b]);
      }
  }
  // touching pairs: moments (1, s1, s2) x (1, s1, s2) -> hats (1 - s1, s1 - s2, s2) in rule order, per lane, so that
  // the 6 x 6 double layer (stored order) can be taken off before the warp sum
  if (cls != PAIR_NEAR) {
#pragma unroll
    for (int o = 0; o < 18; o += 9) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        v[o + j] -= v[o + 3 + j];
        v[o + 3 + j] -= v[o + 6 + j];
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        v[o + 3 * i] -= v[o + 3 * i + 1];
        v[o + 3 * i + 1] -= v[o + 3 * i + 2];
      }
    }
  }
  {
    // rule order (a, b) -> stored order (pm[a], pm[3 + b]): the 6 x 6 entries permuted to rule order instead
    const int p0 = pm[0], p1 = pm[1], s0 = pm[3], s1 = pm[4], p2 = pm[2], s2 = pm[5];
    auto pick = [](const double(&r)[9], int i) {
      double x = r[0];
#pragma unroll
      for (int k = 1; k < 9; ++k) x = i == k ? r[k] : x;
      return x;
    };
    const int pa[3] = {p0, p1, p2}, pb[3] = {s0, s1, s2};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) v[9 + 3 * a + b] -= pick(rd, 3 * pa[a] + pb[b]);
  }
  const double tot = warp_scatter_sum(v);
  if (lane < 27) s_out[w][lane] = tot;
  __syncwarp();
  if (lane < 9) {
    const int a = lane / 3, b = lane % 3;
    const int so = 3 * pm[a] + pm[3 + b];
    const size_t o = 9 * (size_t)pair + so;
    fullV[o] = s_out[w][lane];
    corrV[o] = s_out[w][lane] - s_out[w][18 + so];
    corrK[o] = s_out[w][9 + lane];
    mass[9 * (size_t)pair + lane] = cls == PAIR_IDENTICAL ? At * (a == b ? 2.0 : 1.0) / 12.0 : 0.0;
  }
}

// Gauss-Legendre nodes on [-1, 1] by Newton's method on the three-term recurrence of
// P_n, mapped to [0, 1].
void gauss_legendre01(int n, double* x01, double* w01) {
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    double pp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      pp = n * (z * p1 - p0) / (z * z - 1.0);
      double dz = p1 / pp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      pp = n * (z * p1 - p0) / (z * z - 1.0);
    }
    x01[i] = 0.5 * (1.0 - z);
    w01[i] = 1.0 / ((1.0 - z * z) * pp * pp);  // (2 / ((1 - z^2) P'^2)) / 2
  }
}

// One row of a touching class's table: the fixed point, the moving one as a + e b, the weight of the triple.
struct Row {
  double f1, f2, a1, b1, a2, b2, W;
  int xmoves;
};

// Sauter-Schwab maps (Sauter & Schwab, Boundary Element Methods, 2011, Sec. 5.2) with the last variable e left
// free: in every region it moves one of the two points.
std::vector<Row> touching_rows(const double* x, const double* w) {
  std::vector<Row> R;
  auto triples = [&](auto f) {
    for (int i = 0; i < NGL; ++i)
      for (int j = 0; j < NGL; ++j)
        for (int k = 0; k < NGL; ++k) {
          Row r = f(x[i], x[j], x[k]);
          r.W *= w[i] * w[j] * w[k];
          R.push_back(r);
        }
  };
  // identical: three maps (first point, second point), each also with the two exchanged
  for (int swap = 0; swap < 2; ++swap) {
    triples([&](double xi, double p, double q) {
      return Row{xi, xi * (1 - p + p * q), xi, -xi * p * q, xi * (1 - p), 0.0, xi * xi * xi * p * p * q, swap};
    });
    triples([&](double xi, double p, double q) {
      return Row{xi * (1 - p * q), xi * p * (1 - q), xi, 0.0, xi * p * (1 - q), xi * p * q, xi * xi * xi * p * p * q,
                 1 - swap};
    });
    triples([&](double xi, double p, double q) {
      return Row{xi, xi * p * (1 - q), xi, -xi * p * q, xi * p, -xi * p * q, xi * xi * xi * p * p * q, 1 - swap};
    });
  }
  // common edge: five maps
  triples([&](double xi, double p, double q) {
    return Row{xi * (1 - p * q), xi * p * (1 - q), xi, 0.0, 0.0, xi * p, xi * xi * xi * p * p, 1};
  });
  triples([&](double xi, double p, double q) {
    return Row{xi, xi * p, xi, -xi * p * q, xi * p * q, -xi * p * q, xi * xi * xi * p * p * q, 0};
  });
  triples([&](double xi, double p, double q) {
    return Row{xi * (1 - p * q), xi * p * (1 - q), xi, 0.0, 0.0, xi * p * q, xi * xi * xi * p * p * q, 0};
  });
  triples([&](double xi, double p, double q) {
    return Row{xi, xi * p, xi, -xi * p * q, xi * p * q, -xi * p * q, xi * xi * xi * p * p * q, 1};
  });
  triples([&](double xi, double p, double q) {
    return Row{xi, xi * p * q, xi, -xi * p * q, xi * p, -xi * p * q, xi * xi * xi * p * p * q, 1};
  });
  // common vertex: two maps
  triples([&](double xi, double p, double q) {
    return Row{xi, xi * p, xi * q, 0.0, 0.0, xi * q, xi * xi * xi * q, 0};
  });
  triples([&](double xi, double p, double q) {
    return Row{xi, xi * p, xi * q, 0.0, 0.0, xi * q, xi * xi * xi * q, 1};
  });
  return R;
}

}  // namespace

// tables of the accurate rules on the current device (called by init_quadrature, once per device)
int init_correction_rules() {
  double x[NGL], w[NGL];
  gauss_legendre01(NGL, x, w);
  PB_CUDA(cudaMemcpyToSymbol(c_gl_x, x, sizeof(x)));
  PB_CUDA(cudaMemcpyToSymbol(c_gl_w, w, sizeof(w)));
  const std::vector<Row> R = touching_rows(x, w);
  std::vector<double> rows(7 * (size_t)N_ROWS);
  std::vector<unsigned char> xm(N_ROWS);
  for (int r = 0; r < N_ROWS; ++r) {
    const double c[7] = {R[r].f1, R[r].f2, R[r].a1, R[r].b1, R[r].a2, R[r].b2, R[r].W};
    for (int k = 0; k < 7; ++k) rows[(size_t)k * N_ROWS + r] = c[k];
    xm[r] = (unsigned char)R[r].xmoves;
  }
  PB_CUDA(cudaMemcpyToSymbol(d_row, rows.data(), rows.size() * sizeof(double)));
  PB_CUDA(cudaMemcpyToSymbol(d_xmoves, xm.data(), xm.size()));
  // 6-point rule on the 16 congruent sub-triangles of the 4-fold uniform refinement
  double sub[5][NSUB];
  int k = 0;
  const int m = 4;
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m - i; ++j) {
      const int cnt = (i + j < m - 1) ? 2 : 1;
      for (int up = 0; up < cnt; ++up) {
        const int li[2][3][2] = {{{i, j}, {i + 1, j}, {i, j + 1}}, {{i + 1, j}, {i + 1, j + 1}, {i, j + 1}}};
        for (int q = 0; q < QS; ++q) {
          double b1 = 0.0, b2 = 0.0;
          for (int c = 0; c < 3; ++c) {
            b1 += h_tri_b[q][c] * (li[up][c][0] / (double)m);
            b2 += h_tri_b[q][c] * (li[up][c][1] / (double)m);
          }
          const double wq = h_tri_w[q] / (m * m);
          sub[0][k] = b1 + b2;
          sub[1][k] = b2;
          sub[2][k] = wq * (1.0 - b1 - b2);
          sub[3][k] = wq * b1;
          sub[4][k] = wq * b2;
          ++k;
        }
      }
    }
  PB_CUDA(cudaMemcpyToSymbol(d_sub, sub, sizeof(sub)));
  return PBFB_OK;
}

int launch_pair_corrections(Mesh* m, Surface* s, double kappa) {
  if (s->npair == 0) return PBFB_OK;
  if (kappa != 0.0) PB_TRY(pair_tables(m, true));
  const int blocks = (s->npair + CW - 1) / CW;
  const auto fn = kappa != 0.0 ? k_pair_corrections<true> : k_pair_corrections<false>;
  fn<<<blocks, 32 * CW, 0, m->stream>>>(s->npair, s->pair_t.p, s->pair_s.p, s->pair_cls.p, s->pair_perm.p, s->tri.p,
                                        s->vmap.p, m->xyz.p, m->nv, s->nrm.p, s->area.p, s->qx.p, s->qw.p, s->nt,
                                        kappa, m->pair_tab64.p, s->pairV.p, s->pairK.p, s->pairVfull.p, m->red2.p);
  PB_LAUNCHED(m);
  // per-slot sums (fixed order): corrections, mass, V diagonal
  PB_TRY(launch_gather(m, s->cnnz, s->cg_ptr.p, s->cg_idx.p, s->pairV.p, nullptr, 1.0, s->corrV.p));
  PB_TRY(launch_gather(m, s->cnnz, s->cg_ptr.p, s->cg_idx.p, s->pairK.p, nullptr, 1.0, s->corrK.p));
  PB_TRY(launch_gather(m, s->cnnz, s->cg_ptr.p, s->cg_idx.p, m->red2.p, nullptr, 1.0, s->mass.p));
  PB_TRY(launch_gather(m, s->nv, s->dg_ptr.p, s->dg_idx.p, s->pairVfull.p, nullptr, 1.0, s->diagV.p));
  return PBFB_OK;
}

}  // namespace pbfb
