// The cell matrices by direct Gauss sums in every cell, for contexts with the FP32 preconditioner: the
// 27-point form at the lowest order with an LU of each velocity block, the (p+3)^3-point form at degree
// p with a pivoted Gauss-Jordan inverse of the whole mixed matrix.
//
// assemble.cu and ho_cells.cu form the same matrices 6 and 17 times faster, and equal to rounding
// (1e-14 of a row's scale). In FP64 the solutions then agree to 1e-10. With the FP32 preconditioner they
// do not: a last-bit difference in S changes the FP32 rounding of every preconditioner call, and on
// tall columns or at degree 2 and 3 the iterations amplify that to the size of the forward error that
// the tolerance leaves (3e-4 of lambda on C8 x 66 at 1e-6, 6e-9 at degree 3 at 1e-10). Contexts with
// that precision keep the bits of this form.
//
// Paper (arXiv 2210.11797): as assemble.cu and ho_cells.cu.
#include <cmath>
#include <cstring>
#include <vector>

#include "assemble.cuh"
#include "device_common.cuh"
#include "hmg_internal.cuh"
#include "ho_common.cuh"
#include "ho_reference.cuh"

namespace hmg {

// Trilinear shape function values and derivatives at the 27 Gauss points (3 per direction):
// [q][v] = {N_v, dN_v/dxi, dN_v/deta, dN_v/dzeta}, q = qi + 3 qj + 9 qk, vertex v = (v&1,
// v>>1&1, v>>2). They depend on the point only, so they are formed once on the host (with the
// same expressions and order of operations a per-cell evaluation would use) instead of in
// every cell.
__constant__ double c_shape[27][8][4];

static int upload_shape_functions(Ctx *c) {
  static thread_local double h[27][8][4];
  const double gq = std::sqrt(15.0) / 10.0;
  const double gx[3] = {0.5 - gq, 0.5, 0.5 + gq};
  for (int q = 0; q < 27; ++q) {
    const double xi = gx[q % 3], eta = gx[(q / 3) % 3], zeta = gx[q / 9];
    for (int v = 0; v < 8; ++v) {
      const int av = v & 1, bv = (v >> 1) & 1, cv = (v >> 2) & 1;
      const double fx = av ? xi : 1.0 - xi, fy = bv ? eta : 1.0 - eta, fz = cv ? zeta : 1.0 - zeta;
      const double sx = av ? 1.0 : -1.0, sy = bv ? 1.0 : -1.0, sz = cv ? 1.0 : -1.0;
      h[q][v][0] = fx * fy * fz;
      h[q][v][1] = sx * fy * fz;
      h[q][v][2] = fx * sy * fz;
      h[q][v][3] = fx * fy * sz;
    }
  }
  HMG_CUDA(c, cudaMemcpyToSymbol(c_shape, h, sizeof(h)));
  return HMG_OK;
}

// Corner of the column at reference (xi, eta) in {0,1}^2: (0,0)->0, (1,0)->1, (1,1)->2, (0,1)->3.
__device__ __forceinline__ int corner_of(int a, int b) { return b ? (a ? 2 : 3) : (a ? 1 : 0); }

// Geometry and coefficients of one cell; writes its CellRec.
//  M_K(f,g) = sum_q w_q / det J_q * s_f s_g [ (J^T J)_{d_f d_g} + c22 (r.J)_{d_f} (r.J)_{d_g} ],
// where the RT0 reference function of face f is s_f(xi) e_{d_f} (outward unit flux) and the
// contravariant Piola map gives v_f = J s_f e_{d_f} / det J.
__global__ void __launch_bounds__(128) gauss_cell_kernel(const CellArgs a, double *__restrict__ rec) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= a.ncell) return;
  const int c = (int)(K / a.L), k = (int)(K - (int64_t)c * a.L);
  const double z0 = a.z[k], z1 = a.z[k + 1];
  double vx[8], vy[8], vz[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const int ci = corner_of(v & 1, (v >> 1) & 1);
    const double *cp = a.corners + 12 * (int64_t)c + 3 * ci;
    const double h = (v >> 2) ? z1 : z0;
    if (a.geometry == 1) {
      const double s = a.radius + h;
      vx[v] = cp[0] * s; vy[v] = cp[1] * s; vz[v] = cp[2] * s;
    } else {
      vx[v] = cp[0]; vy[v] = cp[1]; vz[v] = h;
    }
  }
  const int L1 = a.L + 1;
  const double th0 = a.theta_lev[(int64_t)c * L1 + k], th1 = a.theta_lev[(int64_t)c * L1 + k + 1];
  const double pi0 = a.exner_lev[(int64_t)c * L1 + k], pi1 = a.exner_lev[(int64_t)c * L1 + k + 1];
  const double dz = z1 - z0;
  const bool helm = a.sc.preset == 1;
  const double c22 = helm ? 0.0
                          : -a.sc.tau_u * a.sc.tau_theta * a.sc.dt * a.sc.dt * a.sc.cp *
                                ((pi1 - pi0) / dz) * ((th1 - th0) / dz);
  const int dir[6] = {1, 0, 1, 0, 2, 2};
  const double gq = sqrt(15.0) / 10.0;
  const double gx[3] = {0.5 - gq, 0.5, 0.5 + gq};
  const double gw[3] = {5.0 / 18.0, 8.0 / 18.0, 5.0 / 18.0};
  double M[21], Cor[15];
#pragma unroll
  for (int i = 0; i < 21; ++i) M[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 15; ++i) Cor[i] = 0.0;
  // Coriolis vector tau_u dt 2 Omega about z (Eq. gh-u); none for the Helmholtz preset
  const double cz = helm ? 0.0 : a.sc.tau_u * a.sc.dt * 2.0 * a.sc.omega;
  double vol = 0.0;
  for (int q = 0; q < 27; ++q) {
    const int qi = q % 3, qj = (q / 3) % 3, qk = q / 9;
    const double xi = gx[qi], eta = gx[qj], zeta = gx[qk];
    const double w = gw[qi] * gw[qj] * gw[qk];
    double J[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    double x[3] = {0, 0, 0};
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const double n = c_shape[q][v][0];
      const double d0 = c_shape[q][v][1], d1 = c_shape[q][v][2], d2 = c_shape[q][v][3];
      x[0] += n * vx[v]; x[1] += n * vy[v]; x[2] += n * vz[v];
      J[0][0] += vx[v] * d0; J[0][1] += vx[v] * d1; J[0][2] += vx[v] * d2;
      J[1][0] += vy[v] * d0; J[1][1] += vy[v] * d1; J[1][2] += vy[v] * d2;
      J[2][0] += vz[v] * d0; J[2][1] += vz[v] * d1; J[2][2] += vz[v] * d2;
    }
    const double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                       J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                       J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
    double r[3];
    if (a.geometry == 1) {
      const double inv = 1.0 / sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
      r[0] = x[0] * inv; r[1] = x[1] * inv; r[2] = x[2] * inv;
    } else {
      r[0] = 0.0; r[1] = 0.0; r[2] = 1.0;
    }
    const double wd = w / det;
    // H[d][e] = w / det * (G[d][e] + c22 (r.J)_d (r.J)_e), G = J^T J: 6 distinct entries,
    // formed once per point; each of the 21 entries of M then costs a multiply and an FMA
    double rJ[3], H[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) rJ[d] = r[0] * J[0][d] + r[1] * J[1][d] + r[2] * J[2][d];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int e = d; e < 3; ++e) {
        const double g = J[0][d] * J[0][e] + J[1][d] * J[1][e] + J[2][d] * J[2][e];
        H[d][e] = H[e][d] = wd * fma(c22 * rJ[d], rJ[e], g);
      }
    const double s[6] = {eta - 1.0, xi, eta, xi - 1.0, zeta - 1.0, zeta};
    int idx = 0;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
#pragma unroll
      for (int g = f; g < 6; ++g) {
        M[idx] = fma(s[f], s[g] * H[dir[f]][dir[g]], M[idx]);
        ++idx;
      }
    }
    if (cz != 0.0) {
      // v_f . (c x v_g) = s_f s_g c . (J_dg x J_df) / det^2: X[d][e] = (c x-products of the
      // columns of J), antisymmetric; c = (0, 0, cz)
      double X[3][3];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int e = 0; e < 3; ++e) X[d][e] = wd * cz * (J[0][e] * J[1][d] - J[1][e] * J[0][d]);
      int ci = 0;
#pragma unroll
      for (int f = 0; f < 6; ++f)
#pragma unroll
        for (int g = f + 1; g < 6; ++g) {
          Cor[ci] = fma(s[f], s[g] * X[dir[f]][dir[g]], Cor[ci]);
          ++ci;
        }
    }
    vol += w * det;
  }
  // cell centre: one-point volume |K|_1 and zhat.v_f
  double Jc[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}}, xc[3] = {0, 0, 0};
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const double sx = (v & 1) ? 1.0 : -1.0, sy = ((v >> 1) & 1) ? 1.0 : -1.0, sz = ((v >> 2) & 1) ? 1.0 : -1.0;
    xc[0] += 0.125 * vx[v]; xc[1] += 0.125 * vy[v]; xc[2] += 0.125 * vz[v];
    Jc[0][0] += 0.25 * sx * vx[v]; Jc[0][1] += 0.25 * sy * vx[v]; Jc[0][2] += 0.25 * sz * vx[v];
    Jc[1][0] += 0.25 * sx * vy[v]; Jc[1][1] += 0.25 * sy * vy[v]; Jc[1][2] += 0.25 * sz * vy[v];
    Jc[2][0] += 0.25 * sx * vz[v]; Jc[2][1] += 0.25 * sy * vz[v]; Jc[2][2] += 0.25 * sz * vz[v];
  }
  const double vol1 = Jc[0][0] * (Jc[1][1] * Jc[2][2] - Jc[1][2] * Jc[2][1]) -
                      Jc[0][1] * (Jc[1][0] * Jc[2][2] - Jc[1][2] * Jc[2][0]) +
                      Jc[0][2] * (Jc[1][0] * Jc[2][1] - Jc[1][1] * Jc[2][0]);
  double rc[3];
  if (a.geometry == 1) {
    const double inv = 1.0 / sqrt(xc[0] * xc[0] + xc[1] * xc[1] + xc[2] * xc[2]);
    rc[0] = xc[0] * inv; rc[1] = xc[1] * inv; rc[2] = xc[2] * inv;
  } else {
    rc[0] = 0.0; rc[1] = 0.0; rc[2] = 1.0;
  }
  double rJc[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) rJc[d] = rc[0] * Jc[0][d] + rc[1] * Jc[1][d] + rc[2] * Jc[2][d];
  const double sc_[6] = {-0.5, 0.5, 0.5, -0.5, -0.5, 0.5};
  // single-valued theta on each face: vertical faces average the two columns' layer means
  const double mean_own = 0.5 * (th0 + th1);
  double theta[6];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int oc = a.col_nbr[4 * (int64_t)c + f];
    const double mo = 0.5 * (a.theta_lev[(int64_t)oc * L1 + k] + a.theta_lev[(int64_t)oc * L1 + k + 1]);
    theta[f] = 0.5 * (mean_own + mo);
  }
  theta[4] = th0;
  theta[5] = th1;
  double *out = rec + (int64_t)K * kCellData;
  double kk, m;
  double b[6];
  if (helm) {
    kk = 1.0;
    m = a.sc.sigma * vol1;
#pragma unroll
    for (int f = 0; f < 6; ++f) { theta[f] = 1.0; b[f] = 1.0; }
  } else {
    kk = a.sc.tau_u * a.sc.dt * a.sc.cp;
    const double dlog = ((th1 - th0) / dz) / mean_own;
    const double base = a.sc.tau_rho * a.sc.dt * vol1 / vol;   // M3^rho M3^-1 D
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const double zv = sc_[f] * rJc[dir[f]] / vol1;               // (zhat.v_f)(x_c)
      b[f] = base + a.sc.tau_theta * a.sc.dt * (vol1 * dlog) * zv; // + q32
    }
    m = (1.0 - a.sc.kappa) / a.sc.kappa * vol1 / a.exner[K];
  }
#pragma unroll
  for (int i = 0; i < 21; ++i) out[CellRec::M + i] = M[i];
#pragma unroll
  for (int i = 0; i < 15; ++i) out[CellRec::CORI + i] = Cor[i];
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    out[CellRec::B + f] = b[f];
    out[CellRec::KTH + f] = kk * theta[f];
  }
  out[CellRec::MPI] = m;
  // lumped mass share: |M(f,f)| + |M(f, opposite f)|
  const double Mff[6] = {M[0], M[6], M[11], M[15], M[18], M[20]};
  const double Mopp[6] = {M[2], M[8], M[2], M[8], M[19], M[19]};  // (0,2) (1,3) (4,5)
#pragma unroll
  for (int f = 0; f < 6; ++f) out[CellRec::LUMP + f] = fabs(Mff[f]) + fabs(Mopp[f]);
}

__device__ __forceinline__ double mget(const double *M, int f, int g) {
  if (f > g) { int t = f; f = g; g = t; }
  return M[f * 6 - f * (f - 1) / 2 + (g - f)];
}

// A_K = [[M, g], [b^T, m]] with g = -KTH (Eq. hybrid-A). A_K^-1 by block elimination:
// M^-1 from the LU factors of the equilibrated velocity block D M D (D = diag(M)^-1/2; its
// symmetric part is positive definite, the Coriolis part antisymmetric), y = M^-1 g,
// z = M^-T b, pressure Schur complement s = m - b.y, then
// A^-1 = [[M^-1 + y z^T / s, -y / s], [-z^T / s, 1 / s]]. The rows of
// A_K span ~20 orders of magnitude on the sphere; this form keeps every entry within a few
// ulps of its row's scale, where pivoting on A_K itself can lose 1e-12.
// Outputs: Ainv entry-major ((7 i + j) * ncell + K). A non-positive pivot (M not positive definite) or
// s == 0 sets *singular.
__global__ void __launch_bounds__(128) gauss_condense_kernel(int64_t ncell, const double *__restrict__ rec,
                                                       double *__restrict__ Ainv,
                                                       int *__restrict__ singular) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= ncell) return;
  const double *r = rec + K * kCellData;
  // M_K = symmetric part (21 stored) + Coriolis part (antisymmetric, 15 stored)
  auto mfull = [&](int f, int g) {
    double v = mget(r + CellRec::M, f, g);
    if (f < g) v += r[CellRec::CORI + f * 6 - f * (f + 1) / 2 + (g - f - 1)];
    else if (f > g) v -= r[CellRec::CORI + g * 6 - g * (g + 1) / 2 + (f - g - 1)];
    return v;
  };
  double d[6], A[6][6];
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const double mff = fabs(mget(r + CellRec::M, f, f));
    if (!(mff > 0.0)) { atomicExch(singular, 1); return; }
    d[f] = 1.0 / sqrt(mff);
  }
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) A[i][j] = d[i] * mfull(i, j) * d[j];
  // LU of the equilibrated D M D without pivoting (its symmetric part is positive definite,
  // so every pivot is positive; with no rotation this is the symmetric case), in place
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (!(A[k][k] > 0.0)) { atomicExch(singular, 1); return; }
    const double inv = 1.0 / A[k][k];
#pragma unroll
    for (int i = k + 1; i < 6; ++i) {
      const double l = A[i][k] * inv;
      A[i][k] = l;
#pragma unroll
      for (int j = k + 1; j < 6; ++j) A[i][j] -= l * A[k][j];
    }
  }
  // M^-1 = D (LU)^-1 D, column by column
  double Mi[6][6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    double y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      double t = i == c ? 1.0 : 0.0;
#pragma unroll
      for (int q = 0; q < i; ++q) t -= A[i][q] * y[q];
      y[i] = t;
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
      double t = y[i];
#pragma unroll
      for (int q = i + 1; q < 6; ++q) t -= A[i][q] * y[q];
      y[i] = t / A[i][i];
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) Mi[i][c] = d[i] * y[i] * d[c];
  }
  double kth[6], g[6], b[6], y[6], z[6];
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    kth[f] = r[CellRec::KTH + f];
    g[f] = -kth[f];
    b[f] = r[CellRec::B + f];
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double ty = 0.0, tz = 0.0;
#pragma unroll
    for (int j = 0; j < 6; ++j) { ty += Mi[i][j] * g[j]; tz += Mi[j][i] * b[j]; }   // y = M^-1 g, z = M^-T b
    y[i] = ty;
    z[i] = tz;
  }
  double s = r[CellRec::MPI];
#pragma unroll
  for (int j = 0; j < 6; ++j) s -= b[j] * y[j];
  if (s == 0.0) { atomicExch(singular, 1); return; }
  const double is = 1.0 / s;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const double a = Mi[i][j] + y[i] * z[j] * is;
      Ainv[(int64_t)(7 * i + j) * ncell + K] = a;
    }
    Ainv[(int64_t)(7 * i + 6) * ncell + K] = -y[i] * is;
    Ainv[(int64_t)(42 + i) * ncell + K] = -z[i] * is;
  }
  Ainv[(int64_t)48 * ncell + K] = is;
}

// b, the lumped mass shares, k theta and M3^Pi of the cell records, face-major
__global__ void gauss_out_kernel(int64_t ncell, const double *__restrict__ rec, const CellOut q) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= ncell) return;
  const double *r = rec + K * kCellData;
  CellCo o;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    o.b[f] = r[CellRec::B + f];
    o.kth[f] = r[CellRec::KTH + f];
    o.lump[f] = r[CellRec::LUMP + f];
  }
  o.m = r[CellRec::MPI];
  store_cell(q, o, ncell, K);
}

int gauss_setup(Ctx *c, int64_t ncell, double **rec) {
  int st;
  if ((st = upload_shape_functions(c))) return st;
  if (cudaMalloc(rec, (size_t)ncell * kCellData * sizeof(double)) != cudaSuccess) {
    *rec = nullptr;
    cudaGetLastError();
    return fail(c, HMG_ERR_OUT_OF_MEMORY, "device allocation of the cell records failed");
  }
  return HMG_OK;
}

int gauss_cells(Ctx *c, const CellArgs &a, const CellOut &q, double *rec, double *Ainv) {
  gauss_cell_kernel<<<grid_for(a.ncell, 128), 128, 0, c->stream>>>(a, rec);
  gauss_out_kernel<<<grid_for(a.ncell, 256), 256, 0, c->stream>>>(a.ncell, rec, q);
  if (Ainv) gauss_condense_kernel<<<grid_for(a.ncell, 128), 128, 0, c->stream>>>(a.ncell, rec, Ainv, c->asm_flag);
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

// ---- degree p ---------------------------------------------------------------------------------
template <int P>
struct HoGauss {   // reference tables: velocity values, pressure values, weights, points, G, facet weights
  using H = Ho<P>;
  static constexpr int Q = H::NQ1 * H::NQ1 * H::NQ1;
  static constexpr int TV = 0, TPHI = TV + Q * H::NU, TW = TPHI + Q * H::NP, TX = TW + Q, TG = TX + 3 * Q,
                       TC = TG + H::NU * H::NP, TAB = TC + H::NB;
};

// lagrange1d with the roundings of its derivative's sum spelled out: which of its last products are
// fused into the sum is otherwise the host compiler's choice, by its inlining, and moves the last bits
// of G. (All of them up to n = 4; at n = 5 not those of the last node and of nodes 2, 3 for i = 4.)
static void gauss_lagrange1d(const double *nodes, int n, double x, double *val, double *der) {
  for (int i = 0; i < n; ++i) {
    double v = 1.0, d = 0.0;
    for (int j = 0; j < n; ++j)
      if (j != i) v *= (x - nodes[j]) / (nodes[i] - nodes[j]);
    for (int m = 0; m < n; ++m) {
      if (m == i) continue;
      double t = 1.0 / (nodes[i] - nodes[m]), last = 1.0;
      for (int j = 0; j < n; ++j)
        if (j != i && j != m) {
          t *= last;
          last = (x - nodes[j]) / (nodes[i] - nodes[j]);
        }
      if (n < 5 || (m < 4 && (i < 4 || m < 2))) {
        d = std::fma(t, last, d);
      } else {
        const volatile double r = t * last;
        d += r;
      }
    }
    val[i] = v;
    der[i] = d;
  }
}

// the RT_p basis (value of its one nonzero component and its divergence) and the DG_p basis at
// the Q Gauss points, G(f, j) = -int phi_j div v_f, and the facet weights of C_K
template <int P>
static void ho_gauss_tables(std::vector<double> &tab) {
  using H = Ho<P>;
  using G = HoGauss<P>;
  tab.assign(G::TAB, 0.0);
  double gl[H::NT], glw[H::NT], gll[P + 2], qx[H::NQ1], qw[H::NQ1];
  gauss_legendre01(H::NT, gl, glw);
  gauss_lobatto01(P + 2, gll);
  gauss_legendre01(H::NQ1, qx, qw);
  const std::vector<HoDof> dofs = ho_dofs<P>();
  for (int a = 0; a < H::NQ1; ++a)
    for (int b = 0; b < H::NQ1; ++b)
      for (int c = 0; c < H::NQ1; ++c) {
        const int q = (a * H::NQ1 + b) * H::NQ1 + c;
        const double x[3] = {qx[a], qx[b], qx[c]};
        double tv[3][H::NT], td[3][H::NT], nv[3][P + 2], nd[3][P + 2];
        for (int k = 0; k < 3; ++k) {
          gauss_lagrange1d(gl, H::NT, x[k], tv[k], td[k]);
          gauss_lagrange1d(gll, P + 2, x[k], nv[k], nd[k]);
        }
        const double wq = qw[a] * qw[b] * qw[c];
        tab[G::TW + q] = wq;
        for (int k = 0; k < 3; ++k) tab[G::TX + 3 * q + k] = x[k];
        double phi[H::NP];
        for (int ii = 0; ii < H::NT; ++ii)
          for (int jj = 0; jj < H::NT; ++jj)
            for (int kk = 0; kk < H::NT; ++kk) phi[(ii * H::NT + jj) * H::NT + kk] = tv[0][ii] * tv[1][jj] * tv[2][kk];
        for (int j = 0; j < H::NP; ++j) tab[G::TPHI + q * H::NP + j] = phi[j];
        for (int i = 0; i < H::NU; ++i) {
          const HoDof &o = dofs[i];
          const int t1 = o.d == 0 ? 1 : 0, t2 = o.d == 2 ? 1 : 2;
          const double tan = tv[t1][o.b] * tv[t2][o.c];
          tab[G::TV + q * H::NU + i] = o.sign * nv[o.d][o.a] * tan;
          // divergence: the derivative of the one nonzero component along its own coordinate
          const double dv = o.sign * nd[o.d][o.a] * tan;
          for (int j = 0; j < H::NP; ++j) {
            double &g = tab[G::TG + i * H::NP + j];
            g = std::fma(-(wq * dv), phi[j], g);
          }
        }
      }
  for (int s = 0; s < H::NT; ++s)
    for (int t = 0; t < H::NT; ++t) tab[G::TC + s * H::NT + t] = glw[s] * glw[t];
}

template <int P>
__device__ __forceinline__ int ho_comp(int i) {   // the nonzero component of velocity dof i
  using H = Ho<P>;
  if (i < H::NF) {
    const int f = i / H::NB;
    return f == 0 || f == 2 ? 1 : (f == 1 || f == 3 ? 0 : 2);
  }
  return (i - H::NF) / H::NINT;
}

struct HoGaussArgs {
  int geometry, ncol, L;
  int64_t ncell;
  double radius, sigma;
  const double *corners, *z;
};

// Shared memory of the cell kernel: the mixed matrix when it fits (p <= 2), then the per-point
// metric terms and the elimination's vectors.
template <int P>
struct HoGaussSmem {
  static constexpr bool IN_SMEM = P <= 2;
  static constexpr size_t MAT = IN_SMEM ? sizeof(double) * Ho<P>::N * Ho<P>::N : 0;
  static constexpr size_t BYTES =
      MAT + sizeof(double) * (HoGauss<P>::Q * 7 + 3 * Ho<P>::N + 24) + sizeof(int) * (Ho<P>::N + 8);
};

// A_K = [[M, G], [-G^T, Mp]] by the (p+3)^3 Gauss rule (M with the contravariant Piola map,
// Mp = sigma int phi_i phi_j), then A_K^-1 by in-place Gauss-Jordan elimination with partial
// pivoting of the symmetrically equilibrated D A_K D, D = |diag A_K|^-1/2: A^-1 = D (D A D)^-1 D.
// The row interchanges are undone at the end as column interchanges in reverse order. One cell
// per block; the matrix lives in shared memory for p <= 2 and in its output slot (global memory)
// at p = 3. m[K] = sigma |K|_1 (the one-point volume), H 1 of the coarse operator.
template <int P>
__global__ void __launch_bounds__(256)
    ho_gauss_cell_kernel(const HoGaussArgs a, const double *__restrict__ tab, double *__restrict__ Ainv,
                   double *__restrict__ mK, int *singular) {
  using H = Ho<P>;
  using G = HoGauss<P>;
  using SM = HoGaussSmem<P>;
  constexpr int N = H::N;
  extern __shared__ __align__(16) unsigned char ho_smem[];
  const int64_t K = blockIdx.x;
  double *Ag = SM::IN_SMEM ? reinterpret_cast<double *>(ho_smem) : Ainv + K * (int64_t)(N * N);
  double *Kq = reinterpret_cast<double *>(ho_smem + SM::MAT);   // [Q][6] (w / det) J^T J
  double *wd = Kq + 6 * G::Q;                                     // [Q] sigma w det
  double *dsc = wd + G::Q, *fac = dsc + N, *rowk = fac + N;
  double *X = rowk + N;                                           // [8][3] corners
  int *perm = reinterpret_cast<int *>(X + 24);
  int *piv = perm + N;
  __shared__ double bestv[8];
  __shared__ int besti[8];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int c = (int)(K / a.L), k = (int)(K - (int64_t)c * a.L);
  if (tid < 8) {
    const int va = tid & 1, vb = (tid >> 1) & 1, vc = (tid >> 2) & 1;
    const int corner = va == 0 ? (vb == 0 ? 0 : 3) : (vb == 0 ? 1 : 2);
    const double *cp = a.corners + (4 * (int64_t)c + corner) * 3;
    const double h = a.z[k + vc];
    if (a.geometry == 1) {
      for (int i = 0; i < 3; ++i) X[3 * tid + i] = cp[i] * (a.radius + h);
    } else {
      X[3 * tid] = cp[0];
      X[3 * tid + 1] = cp[1];
      X[3 * tid + 2] = h;
    }
  }
  __syncthreads();
  auto jacobian = [&](double xi, double eta, double zeta, double J[3][3]) {
    for (int i = 0; i < 3; ++i) J[i][0] = J[i][1] = J[i][2] = 0.0;
    for (int v = 0; v < 8; ++v) {
      const int va = v & 1, vb = (v >> 1) & 1, vc = (v >> 2) & 1;
      const double fx = va ? xi : 1.0 - xi, fy = vb ? eta : 1.0 - eta, fz = vc ? zeta : 1.0 - zeta;
      const double gx = va ? 1.0 : -1.0, gy = vb ? 1.0 : -1.0, gz = vc ? 1.0 : -1.0;
      const double dn[3] = {gx * fy * fz, fx * gy * fz, fx * fy * gz};
      for (int i = 0; i < 3; ++i)
        for (int d = 0; d < 3; ++d) J[i][d] += X[3 * v + i] * dn[d];
    }
  };
  auto det3 = [](const double J[3][3]) {
    return J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) - J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
           J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
  };
  for (int q = tid; q <= G::Q; q += nthr) {
    if (q < G::Q) {
      const double *xq = tab + G::TX + 3 * q;
      double J[3][3];
      jacobian(xq[0], xq[1], xq[2], J);
      const double det = det3(J), w = tab[G::TW + q];
      double GG[3][3];
      for (int p = 0; p < 3; ++p)
        for (int r = 0; r < 3; ++r) GG[p][r] = J[0][p] * J[0][r] + J[1][p] * J[1][r] + J[2][p] * J[2][r];
      const double s = w / det;
      Kq[6 * q] = s * GG[0][0];
      Kq[6 * q + 1] = s * GG[1][1];
      Kq[6 * q + 2] = s * GG[2][2];
      Kq[6 * q + 3] = s * GG[0][1];
      Kq[6 * q + 4] = s * GG[0][2];
      Kq[6 * q + 5] = s * GG[1][2];
      wd[q] = a.sigma * w * det;
    } else {
      double J[3][3];
      jacobian(0.5, 0.5, 0.5, J);
      mK[K] = a.sigma * det3(J);
    }
  }
  __syncthreads();
  const double *tv = tab + G::TV, *tp = tab + G::TPHI, *tg = tab + G::TG;
  for (int idx = tid; idx < N * N; idx += nthr) {
    const int i = idx / N, j = idx - i * N;
    double v = 0.0;
    if (i < H::NU && j < H::NU) {
      const int di = ho_comp<P>(i), dj = ho_comp<P>(j);
      const int kk = di == dj ? di : (di + dj == 1 ? 3 : (di + dj == 2 ? 4 : 5));
      for (int q = 0; q < G::Q; ++q)
        v = fma(__ldg(tv + q * H::NU + i) * __ldg(tv + q * H::NU + j), Kq[6 * q + kk], v);
    } else if (i < H::NU) {
      v = __ldg(tg + i * H::NP + (j - H::NU));
    } else if (j < H::NU) {
      v = -__ldg(tg + j * H::NP + (i - H::NU));
    } else {
      for (int q = 0; q < G::Q; ++q)
        v = fma(wd[q] * __ldg(tp + q * H::NP + (i - H::NU)), __ldg(tp + q * H::NP + (j - H::NU)), v);
    }
    Ag[idx] = v;
  }
  __syncthreads();
  for (int i = tid; i < N; i += nthr) dsc[i] = 1.0 / sqrt(fabs(Ag[(int64_t)i * N + i]));
  __syncthreads();
  for (int idx = tid; idx < N * N; idx += nthr) {
    const int i = idx / N, j = idx - i * N;
    Ag[idx] *= dsc[i] * dsc[j];
  }
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31, nwarp = nthr >> 5;
  for (int col = 0; col < N; ++col) {
    // pivot: the largest |A[r][col]|, r >= col (the first such row on ties)
    double bv = -1.0;
    int bi = col;
    for (int r = col + tid; r < N; r += nthr) {
      const double v = fabs(Ag[(int64_t)r * N + col]);
      if (v > bv) { bv = v; bi = r; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
    }
    if (lane == 0) { bestv[warp] = bv; besti[warp] = bi; }
    __syncthreads();
    if (tid == 0) {
      double v = bestv[0];
      int p = besti[0];
      for (int w = 1; w < nwarp; ++w)
        if (bestv[w] > v || (bestv[w] == v && besti[w] < p)) { v = bestv[w]; p = besti[w]; }
      if (!(v > 0.0)) atomicExch(singular, 1);
      piv[0] = p;
      perm[col] = p;
    }
    __syncthreads();
    const int p = piv[0];
    if (p != col)
      for (int j = tid; j < N; j += nthr) {
        const double t = Ag[(int64_t)col * N + j];
        Ag[(int64_t)col * N + j] = Ag[(int64_t)p * N + j];
        Ag[(int64_t)p * N + j] = t;
      }
    __syncthreads();
    for (int r = tid; r < N; r += nthr) fac[r] = Ag[(int64_t)r * N + col];
    __syncthreads();
    const double pinv = 1.0 / fac[col];
    for (int j = tid; j < N; j += nthr) {
      const double v = (j == col ? 1.0 : Ag[(int64_t)col * N + j]) * pinv;
      Ag[(int64_t)col * N + j] = v;
      rowk[j] = v;
    }
    __syncthreads();
    for (int idx = tid; idx < N * N; idx += nthr) {
      const int r = idx / N, j = idx - r * N;
      if (r != col) Ag[idx] = fma(-fac[r], rowk[j], j == col ? 0.0 : Ag[idx]);
    }
    __syncthreads();
  }
  for (int col = N - 1; col >= 0; --col) {   // undo the row interchanges: columns, in reverse
    const int p = perm[col];
    if (p != col)
      for (int r = tid; r < N; r += nthr) {
        const double t = Ag[(int64_t)r * N + col];
        Ag[(int64_t)r * N + col] = Ag[(int64_t)r * N + p];
        Ag[(int64_t)r * N + p] = t;
      }
    __syncthreads();
  }
  double *out = Ainv + K * (int64_t)(N * N);
  for (int idx = tid; idx < N * N; idx += nthr) {
    const int i = idx / N, j = idx - i * N;
    out[idx] = dsc[i] * Ag[idx] * dsc[j];
  }
}

template <int P>
int ho_gauss_cell_matrices(Ctx *c) {
  const Level &f = c->lv[0];
  HoData &h = c->ho;
  int st;
  if (!h.gtab) {
    std::vector<double> tab;
    ho_gauss_tables<P>(tab);
    if ((st = dev_alloc(c, &h.gtab, tab.size()))) return st;
    HMG_CUDA(c, cudaMemcpy(h.gtab, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice));
  }
  h.cw = h.gtab + HoGauss<P>::TC;   // (host compilers may contract the quadrature rule's sums differently in another file)
  const HoGaussArgs a{f.geometry, f.ncol, f.nlev, f.ncell, f.radius, c->sc.sigma, f.corners, f.z};
  const size_t smem = HoGaussSmem<P>::BYTES;
  HMG_CUDA(c, cudaFuncSetAttribute(ho_gauss_cell_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ho_gauss_cell_kernel<P><<<(unsigned)f.ncell, 256, smem, c->stream>>>(a, h.gtab, h.Ainv, h.m, h.flag);
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

template int ho_gauss_cell_matrices<1>(Ctx *);
template int ho_gauss_cell_matrices<2>(Ctx *);
template int ho_gauss_cell_matrices<3>(Ctx *);

}  // namespace hmg
