// The mixed cell matrices of degree p = 1, 2, 3 and their inverses: A_K = [[M, G], [-G^T, Mp]] by the
// (p+3)^3 Gauss rule (M with the contravariant Piola map, Mp = sigma int phi_i phi_j).
//
// Paper (arXiv 2210.11797): Sec. 2.2 (spaces of degree p, n = p + 3 Gauss points per direction),
// Sec. 2.4 (static condensation: A_K is inverted cell by cell).
//
// The trilinear map of an extruded cell is x = C(xi, eta) s(zeta) (C the bilinear corner map, s = R + z;
// on the plane x = (C, z), s = 1), so with h = w / D, D = (C_xi x C_eta) . C, every Gauss sum is a sum
// over the horizontal points of a column times one over the vertical points of a level, and with the
// tensor-product basis every block is a Kronecker product (horizontal functions x vertical nodes):
//   xi and eta components:  M_hh = H_hh (x) D,    H_hh = sum h C_d . C_d' f f', D = diag(w_c) / dz
//   with zeta:              M_hz = H_hz (x) V,    H_hz = sum h (C_d . C) f g,   V = sum w T_c N_n / s
//   zeta:                   M_zz = H_zz (x) V_zz, H_zz = sum h |C|^2 g g',      V_zz = dz sum w N N' / s^2
//   pressure:               Mp = sigma H_p (x) V_p
// D is diagonal because the Gauss-Legendre nodal basis is orthogonal. So M^-1 by block elimination takes
// one NH x NH inverse per column (H_hh^-1), Q = M_hh^-1 M_hz = Q_c (x) Q_l with Q_c = H_hh^-1 H_hz and
// Q_l = D^-1 V, and per cell only the inverse of S_z = H_zz (x) V_zz - K_c (x) W_l (NZ = 12, 36, 80 rows):
//   M^-1 = [[H_hh^-1 (x) D^-1 + Q S_z^-1 Q^T, -Q S_z^-1], [-S_z^-1 Q^T, S_z^-1]].
// The pressure is eliminated with X = M^-1 G (G has 3 (p+2) nonzeros per column),
// Sigma = Mp + G^T X, Y = X Sigma^-1: A^-1 = [[M^-1 - Y X^T, -Y], [Y^T, Sigma^-1]].
// All three inverted matrices are symmetric positive definite (sigma > 0): Gauss-Jordan without
// pivoting, a non-positive pivot is reported as a singular cell.
#include <vector>

#include "device_common.cuh"
#include "hmg_internal.cuh"
#include "ho_common.cuh"
#include "ho_reference.cuh"

namespace hmg {

// the one-dimensional bases at the Gauss points, the nonzeros G(f, j) = -int phi_j div v_f (the
// Gauss-Legendre nodes across the component match), the facet weights of C_K, and the dof order
template <int P>
static void ho_tables(std::vector<double> &tab, std::vector<int> &itab) {
  using H = Ho<P>;
  tab.assign(H::TAB, 0.0);
  itab.assign(H::ITAB, 0);
  double gl[H::NT], glw[H::NT], gll[H::NV], qx[H::NQ1], qw[H::NQ1], div[H::NV][H::NT] = {};
  gauss_legendre01(H::NT, gl, glw);
  gauss_lobatto01(H::NV, gll);
  gauss_legendre01(H::NQ1, qx, qw);
  for (int q = 0; q < H::NQ1; ++q) {
    double tv[H::NT], td[H::NT], nv[H::NV], nd[H::NV];
    lagrange1d(gl, H::NT, qx[q], tv, td);
    lagrange1d(gll, H::NV, qx[q], nv, nd);
    for (int i = 0; i < H::NT; ++i) tab[H::TL + q * H::NT + i] = tv[i];
    for (int i = 0; i < H::NV; ++i) tab[H::TN + q * H::NV + i] = nv[i];
    tab[H::TW + q] = qw[q];
    tab[H::TX + q] = qx[q];
    for (int a = 0; a < H::NV; ++a)
      for (int j = 0; j < H::NT; ++j) div[a][j] += qw[q] * nd[a] * tv[j];
  }
  for (int i = 0; i < H::NT; ++i) tab[H::TGW + i] = glw[i];
  for (int s = 0; s < H::NT; ++s)
    for (int t = 0; t < H::NT; ++t) tab[H::TC + s * H::NT + t] = glw[s] * glw[t];
  const std::vector<HoDof> dofs = ho_dofs<P>();
  int count[H::NP] = {};
  for (int i = 0; i < H::NU; ++i) {
    const HoDof &o = dofs[i];
    const int place = o.d < 2 ? ((o.d * H::NV + o.a) * H::NT + o.b) * H::NT + o.c
                              : H::NH * H::NT + (o.b * H::NT + o.c) * H::NV + o.a;
    itab[H::IO + place] = i | (o.sign < 0.0 ? 1 << 30 : 0);
    for (int m = 0; m < H::NT; ++m) {   // the pressure nodes with the dof's nodes across its direction
      const int ii = o.d == 0 ? m : o.b, jj = o.d == 0 ? o.b : (o.d == 1 ? m : o.c), kk = o.d == 2 ? m : o.c;
      const int j = (ii * H::NT + jj) * H::NT + kk, e = j * H::NG + count[j]++;
      tab[H::TGV + e] = -o.sign * div[o.a][m] * glw[o.b] * glw[o.c];
      itab[H::IG + e] = i;
    }
  }
}

struct HoCellArgs {
  int geometry, ncol, L;
  double radius, sigma;
  const double *corners, *z;
  const double *tab;
  const int *itab;
  double *ctab, *ltab;
};

// In-place inverse of a symmetric positive definite N x N matrix in shared memory by Gauss-Jordan
// elimination without pivoting, by the whole block (T >= N threads); v: 2 N scratch values. Two
// barriers and N^2 FMAs per pivot: bound by the FP64 issue rate from N = 36 up.
template <int N, int T>
__device__ __forceinline__ void block_spd_inverse(double *a, double *v, int *singular) {
  static_assert(T >= N, "a thread per row");
  const int tid = threadIdx.x;
  double *col = v, *row = v + N;
  for (int k = 0; k < N; ++k) {
    __syncthreads();
    if (tid < N) {
      const double p = a[k * N + k], inv = 1.0 / p;
      if (tid == 0 && !(p > 0.0)) atomicExch(singular, 1);
      col[tid] = a[tid * N + k];
      row[tid] = tid == k ? inv : a[k * N + tid] * inv;
    }
    __syncthreads();
    for (int e = tid; e < N * N; e += T) {
      const int i = e / N, j = e - i * N;
      a[e] = i == k ? row[j] : fma(-col[i], row[j], j == k ? 0.0 : a[e]);
    }
  }
  __syncthreads();
}

// The geometry sums of one column (one block per column): H_hh^-1, Q_c, H_zz, K_c, H_p and D at the
// centre. They depend on the mesh only and serve every level of the column.
constexpr int kHoColThreads = 128;

template <int P>
constexpr int kHoColSmem = 7 * Ho<P>::NQ1 * Ho<P>::NQ1 + (Ho<P>::NH + Ho<P>::NM) * Ho<P>::NQ1 * Ho<P>::NQ1 +
                           Ho<P>::NH * Ho<P>::NH + 2 * Ho<P>::NH * Ho<P>::NM + 2 * Ho<P>::NH;

template <int P>
__global__ void __launch_bounds__(kHoColThreads) ho_column_kernel(const HoCellArgs a, int *singular) {
  using H = Ho<P>;
  constexpr int Q = H::NQ1 * H::NQ1, NH = H::NH, NM = H::NM, NT = H::NT, NV = H::NV;
  extern __shared__ __align__(16) double hc_smem[];
  double *g = hc_smem, *fh = g + 7 * Q, *fm = fh + NH * Q, *Hh = fm + NM * Q, *Hz = Hh + NH * NH, *Qc = Hz + NH * NM,
         *v = Qc + NH * NM;
  const int c = blockIdx.x, tid = threadIdx.x;
  const bool sphere = a.geometry == 1;
  const double *cp = a.corners + 12 * (int64_t)c;
  double *out = a.ctab + (int64_t)c * H::CTAB;
  // point q < Q: horizontal Gauss point (q / NQ1, q % NQ1); q = Q: the centre
  for (int q = tid; q <= Q; q += kHoColThreads) {
    const int qi = q / H::NQ1, qj = q - qi * H::NQ1;
    const double xi = q < Q ? a.tab[H::TX + qi] : 0.5, eta = q < Q ? a.tab[H::TX + qj] : 0.5;
    double C[3], Cx[3], Ce[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const bool used = sphere || i < 2;
      const double c0 = used ? cp[i] : 0.0, c1 = used ? cp[3 + i] : 0.0, c2 = used ? cp[6 + i] : 0.0,
                   c3 = used ? cp[9 + i] : 0.0, p1 = c1 - c0, p2 = c3 - c0, p3 = (c2 - c3) - p1;
      Cx[i] = fma(eta, p3, p1);
      Ce[i] = fma(xi, p3, p2);
      C[i] = fma(xi, Cx[i], fma(eta, p2, c0));
    }
    auto dot = [](const double (&x)[3], const double (&y)[3]) { return fma(x[2], y[2], fma(x[1], y[1], x[0] * y[0])); };
    const double n2 = Cx[0] * Ce[1] - Cx[1] * Ce[0];
    double D = n2;
    if (sphere)
      D = fma(n2, C[2], fma(Cx[2] * Ce[0] - Cx[0] * Ce[2], C[1], (Cx[1] * Ce[2] - Cx[2] * Ce[1]) * C[0]));
    if (q == Q) {
      out[H::CD] = D;
      continue;
    }
    const double w = a.tab[H::TW + qi] * a.tab[H::TW + qj], h = w / D;
    g[q] = h * dot(Cx, Cx);
    g[Q + q] = h * dot(Cx, Ce);
    g[2 * Q + q] = h * dot(Ce, Ce);
    g[3 * Q + q] = sphere ? h * dot(Cx, C) : 0.0;
    g[4 * Q + q] = sphere ? h * dot(Ce, C) : 0.0;
    g[5 * Q + q] = sphere ? h * dot(C, C) : h;
    g[6 * Q + q] = w * D;
  }
  for (int e = tid; e < (NH + NM) * Q; e += kHoColThreads) {
    const int f = e / Q, q = e - f * Q, qi = q / H::NQ1, qj = q - qi * H::NQ1;
    if (f < NH) {   // N_a along the component, T_b across
      const int d = f / (NV * NT), r = f - d * NV * NT, n = r / NT, b = r - n * NT;
      fh[e] = a.tab[H::TN + (d == 0 ? qi : qj) * NV + n] * a.tab[H::TL + (d == 0 ? qj : qi) * NT + b];
    } else {
      const int m = f - NH, b = m / NT, cc = m - b * NT;
      fh[e] = a.tab[H::TL + qi * NT + b] * a.tab[H::TL + qj * NT + cc];   // (fm follows fh)
    }
  }
  __syncthreads();
  auto sum = [&](const double *w, const double *x, const double *y) {
    double s = 0.0;
    for (int q = 0; q < Q; ++q) s = fma(w[q] * x[q], y[q], s);
    return s;
  };
  for (int e = tid; e < NH * NH; e += kHoColThreads) {
    const int i = e / NH, j = e - i * NH, di = i / (NV * NT), dj = j / (NV * NT);
    Hh[e] = sum(g + (di + dj) * Q, fh + i * Q, fh + j * Q);
  }
  for (int e = tid; e < NH * NM; e += kHoColThreads) {
    const int i = e / NM, m = e - i * NM;
    Hz[e] = sum(g + (3 + i / (NV * NT)) * Q, fh + i * Q, fm + m * Q);
  }
  for (int e = tid; e < NM * NM; e += kHoColThreads) {
    const int i = e / NM, j = e - i * NM;
    out[H::CZZ + e] = sum(g + 5 * Q, fm + i * Q, fm + j * Q);
    out[H::CP + e] = sum(g + 6 * Q, fm + i * Q, fm + j * Q);
  }
  block_spd_inverse<NH, kHoColThreads>(Hh, v, singular);
  for (int e = tid; e < NH * NH; e += kHoColThreads) out[H::CHI + e] = Hh[e];
  for (int e = tid; e < NH * NM; e += kHoColThreads) {
    const int i = e / NM, m = e - i * NM;
    double s = 0.0;
    for (int j = 0; j < NH; ++j) s = fma(Hh[i * NH + j], Hz[j * NM + m], s);
    Qc[e] = s;
    out[H::CQ + e] = s;
  }
  __syncthreads();
  for (int e = tid; e < NM * NM; e += kHoColThreads) {
    const int i = e / NM, j = e - i * NM;
    double s = 0.0;
    for (int q = 0; q < NH; ++q) s = fma(Hz[q * NM + i], Qc[q * NM + j], s);
    out[H::CK + e] = s;
  }
}

// The sums of one level (one thread per level).
template <int P>
__global__ void ho_level_kernel(const HoCellArgs a) {
  using H = Ho<P>;
  constexpr int NT = H::NT, NV = H::NV;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.L) return;
  const bool sphere = a.geometry == 1;
  const double s0 = sphere ? a.radius + a.z[k] : a.z[k], dz = (sphere ? a.radius + a.z[k + 1] : a.z[k + 1]) - s0;
  double *o = a.ltab + (int64_t)k * H::LTAB;
  auto at = [&](int q) { return sphere ? fma(a.tab[H::TX + q], dz, s0) : 1.0; };
  auto tl = [&](int q, int i) { return a.tab[H::TL + q * NT + i]; };
  auto tn = [&](int q, int i) { return a.tab[H::TN + q * NV + i]; };
  double V[NT][NV];
  for (int i = 0; i < NT; ++i) {
    o[H::LD + i] = dz / a.tab[H::TGW + i];
    for (int n = 0; n < NV; ++n) {
      double s = 0.0;
      for (int q = 0; q < H::NQ1; ++q) s += a.tab[H::TW + q] * tl(q, i) * tn(q, n) / at(q);
      V[i][n] = s;
      o[H::LQ + i * NV + n] = o[H::LD + i] * s;
    }
    for (int j = 0; j < NT; ++j) {
      double s = 0.0;
      for (int q = 0; q < H::NQ1; ++q) s += a.tab[H::TW + q] * (at(q) * at(q)) * tl(q, i) * tl(q, j);
      o[H::LP + i * NT + j] = dz * s;
    }
  }
  for (int n = 0; n < NV; ++n)
    for (int m = 0; m < NV; ++m) {
      double s = 0.0, w = 0.0;
      for (int q = 0; q < H::NQ1; ++q) s += a.tab[H::TW + q] / (at(q) * at(q)) * tn(q, n) * tn(q, m);
      for (int i = 0; i < NT; ++i) w += V[i][n] * o[H::LQ + i * NV + m];
      o[H::LZZ + n * NV + m] = dz * s;
      o[H::LW + n * NV + m] = w;
    }
  const double sc = sphere ? fma(0.5, dz, s0) : 1.0;
  o[H::LV] = sc * sc * dz;
}

// Shared memory of the cell kernel, in doubles. First half: T = Q S_z^-1 (sphere), S_z and the
// half-applied Kronecker products; second half: X (a column of X contiguous) and Sigma.
template <int P>
struct HoCellShape {
  using H = Ho<P>;
  static constexpr int THREADS = P == 3 ? 256 : (P == 2 ? 128 : 64);
  static constexpr int NHT = H::NH * H::NT, TSZ = NHT * H::NZ, U0 = H::NM * H::NT * H::NZ;
  static constexpr int FIRST = TSZ + H::NZ * H::NZ + U0, SECOND = H::NP * H::NU + H::NP * H::NP;
  static constexpr int V2 = 2 * (H::NZ > H::NP ? H::NZ : H::NP);
  static constexpr int VEC = V2 > H::NF + H::NP ? V2 : H::NF + H::NP;
  static_assert(NHT * H::NM * H::NT <= H::NZ * H::NZ + U0, "the right-applied product takes S_z's place");
  static constexpr int doubles(bool sphere) {
    return VEC + (sphere && FIRST > SECOND ? FIRST : (H::NZ * H::NZ > SECOND ? H::NZ * H::NZ : SECOND));
  }
};

// A_K^-1 of one cell per block (the header comment has the algebra), the rank-NP update M^-1 - Y X^T on
// 4 x 4 tiles of the symmetric matrix, its operands in shared memory (X) and in the block's own output
// rows (Y, in L2). About NU^2 NP / 2 + NU NP^2 + NZ^3 + NP^3 FMAs: 3.9 M at p = 3 against 40 M for the
// Gauss points and the pivoted Gauss-Jordan inverse of the whole matrix that this replaced, and bound
// by the FP64 issue rate like it.
template <int P>
__global__ void __launch_bounds__(HoCellShape<P>::THREADS)
    ho_cell_kernel(const HoCellArgs a, int64_t ncell, double *Ainv, double *__restrict__ mK, double *__restrict__ sk1,
                   int *singular) {
  using H = Ho<P>;
  using SH = HoCellShape<P>;
  constexpr int T = SH::THREADS, N = H::N, NU = H::NU, NP = H::NP, NZ = H::NZ, NT = H::NT, NV = H::NV, NM = H::NM,
                NH = H::NH, NHT = SH::NHT, NG = H::NG;
  extern __shared__ __align__(16) double hk_smem[];
  const int64_t K = blockIdx.x;
  const int tid = threadIdx.x, c = (int)(K / a.L), k = (int)(K - (int64_t)c * a.L);
  const bool sphere = a.geometry == 1;
  const double *ct = a.ctab + (int64_t)c * H::CTAB, *lt = a.ltab + (int64_t)k * H::LTAB;
  const int *io = a.itab + H::IO, *gi = a.itab + H::IG;
  const double *gv = a.tab + H::TGV;
  double *A = Ainv + K * (int64_t)(N * N);
  double *v = hk_smem, *Tm = v + SH::VEC, *Sz = Tm + (sphere ? SH::TSZ : 0), *U = Sz + NZ * NZ;
  if (tid == 0) {
    mK[K] = a.sigma * (ct[H::CD] * lt[H::LV]);
    if (!(a.sigma > 0.0)) atomicExch(singular, 1);
  }
  for (int e = tid; e < NZ * NZ; e += T) {
    const int i = e / NZ, j = e - i * NZ, mi = i / NV, mj = j / NV, n = (i - mi * NV) * NV + (j - mj * NV);
    double s = ct[H::CZZ + mi * NM + mj] * lt[H::LZZ + n];
    if (sphere) s = fma(-ct[H::CK + mi * NM + mj], lt[H::LW + n], s);
    Sz[e] = s;
  }
  block_spd_inverse<NZ, T>(Sz, v, singular);
  // M^-1 into the output, dofs in output order
  auto put = [&](int i, int j, double x) {   // tensor-product places i, j
    const int oi = io[i], oj = io[j];
    A[(int64_t)(oi & 0xffff) * N + (oj & 0xffff)] = ((oi ^ oj) >> 30) & 1 ? -x : x;
  };
  for (int e = tid; e < NZ * NZ; e += T) put(NHT + e / NZ, NHT + e % NZ, Sz[e]);
  if (sphere) {
    for (int e = tid; e < NM * NT * NZ; e += T) {   // U = (1 (x) Q_l) S_z^-1
      const int r = e / NZ, z = e - r * NZ, m = r / NT, cc = r - m * NT;
      double s = 0.0;
#pragma unroll
      for (int n = 0; n < NV; ++n) s = fma(lt[H::LQ + cc * NV + n], Sz[(m * NV + n) * NZ + z], s);
      U[e] = s;
    }
    __syncthreads();
    for (int e = tid; e < NHT * NZ; e += T) {   // T = (Q_c (x) 1) U
      const int r = e / NZ, z = e - r * NZ, h = r / NT, cc = r - h * NT;
      double s = 0.0;
#pragma unroll
      for (int m = 0; m < NM; ++m) s = fma(ct[H::CQ + h * NM + m], U[(m * NT + cc) * NZ + z], s);
      Tm[e] = s;
      put(r, NHT + z, -s);
      put(NHT + z, r, -s);
    }
    __syncthreads();
    U = Sz;
    for (int e = tid; e < NHT * NM * NT; e += T) {   // U = T (1 (x) Q_l^T)
      const int r = e / (NM * NT), q = e - r * NM * NT, m = q / NT, cc = q - m * NT;
      double s = 0.0;
#pragma unroll
      for (int n = 0; n < NV; ++n) s = fma(Tm[r * NZ + m * NV + n], lt[H::LQ + cc * NV + n], s);
      U[e] = s;
    }
    __syncthreads();
  }
  for (int e = tid; e < NHT * NHT; e += T) {
    const int r = e / NHT, q = e - r * NHT, h = r / NT, cr = r - h * NT, hq = q / NT, cq = q - hq * NT;
    double s = cr == cq ? ct[H::CHI + h * NH + hq] * lt[H::LD + cr] : 0.0;
    if (sphere) {
#pragma unroll
      for (int m = 0; m < NM; ++m) s = fma(U[r * NM * NT + m * NT + cq], ct[H::CQ + hq * NM + m], s);
    }
    put(r, q, s);
  }
  if (!sphere)
    for (int e = tid; e < NHT * NZ; e += T) {
      put(e / NZ, NHT + e % NZ, 0.0);
      put(NHT + e % NZ, e / NZ, 0.0);
    }
  __syncthreads();
  // X = M^-1 G (M^-1 is symmetric: its rows are read along their length), Sigma = Mp + G^T X
  double *X = v + SH::VEC, *Sg = X + NP * NU;
  for (int e = tid; e < NP * NU; e += T) {
    const int j = e / NU, i = e - j * NU;
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < NG; ++q) s = fma(gv[j * NG + q], A[(int64_t)gi[j * NG + q] * N + i], s);
    X[e] = s;
  }
  __syncthreads();
  for (int e = tid; e < NP * NP; e += T) {
    const int j = e / NP, q = e - j * NP, mj = j / NT, mq = q / NT;
    double s = a.sigma * (ct[H::CP + mj * NM + mq] * lt[H::LP + (j - mj * NT) * NT + (q - mq * NT)]);
#pragma unroll
    for (int r = 0; r < NG; ++r) s = fma(gv[j * NG + r], X[q * NU + gi[j * NG + r]], s);
    Sg[e] = s;
  }
  block_spd_inverse<NP, T>(Sg, v, singular);
  for (int e = tid; e < NP * NP; e += T) A[(int64_t)(NU + e / NP) * N + NU + e % NP] = Sg[e];
  for (int j = tid; j < NP; j += T) {   // Mp 1
    double s = 0.0, w = 0.0;
#pragma unroll
    for (int m = 0; m < NM; ++m) s += ct[H::CP + (j / NT) * NM + m];
#pragma unroll
    for (int n = 0; n < NT; ++n) w += lt[H::LP + (j % NT) * NT + n];
    v[H::NF + j] = a.sigma * s * w;
  }
  // Y = X Sigma^-1 into the pressure rows (and -Y into the pressure columns)
  constexpr int R = NU / 4, CJ = P == 2 ? 3 : 4, W = NP / CJ;
  static_assert(4 * R == NU && CJ * W == NP, "whole tiles");
  for (int e = tid; e < R * W; e += T) {
    const int ti = e % R, tj = e / R;
    double acc[4][CJ];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < CJ; ++r) acc[q][r] = 0.0;
#pragma unroll 2
    for (int m = 0; m < NP; ++m) {
      double x[4], s[CJ];
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = X[m * NU + ti + R * q];
#pragma unroll
      for (int r = 0; r < CJ; ++r) s[r] = Sg[m * NP + tj + W * r];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < CJ; ++r) acc[q][r] = fma(x[q], s[r], acc[q][r]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < CJ; ++r) {
        const int i = ti + R * q, j = tj + W * r;
        A[(int64_t)(NU + j) * N + i] = acc[q][r];
        A[(int64_t)i * N + NU + j] = -acc[q][r];
      }
  }
  __syncthreads();
  // S_K 1 summed over each facet's nodes, for Gamma: G 1 = -C 1, so A [0; 1] = [-C 1; Mp 1] and
  // S_K 1 = C (A^-1)_uu C 1 = C (A^-1)_up Mp 1, without the cancellation of summing S_K's rows
  for (int q = tid; q < H::NF; q += T) {
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < NP; ++j) s = fma(-A[(int64_t)(NU + j) * N + q], v[H::NF + j], s);
    v[q] = a.tab[H::TC + q % H::NB] * s;
  }
  __syncthreads();
  if (tid < 6) {
    double s = 0.0;
    for (int n = 0; n < H::NB; ++n) s += v[tid * H::NB + n];
    sk1[tid * ncell + K] = s;
  }
  // the velocity block: tiles (ti >= tj) of rows ti + R q and columns tj + R r, and their mirror image
  for (int e = tid; e < R * (R + 1) / 2; e += T) {
    int ti = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= e) ++ti;
    while (ti * (ti + 1) / 2 > e) --ti;
    const int tj = e - ti * (ti + 1) / 2;
    double acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[q][r] = A[(int64_t)(ti + R * q) * N + tj + R * r];
#pragma unroll 2
    for (int m = 0; m < NP; ++m) {
      double y[4], x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = A[(int64_t)(NU + m) * N + ti + R * q];
#pragma unroll
      for (int r = 0; r < 4; ++r) x[r] = X[m * NU + tj + R * r];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = fma(-y[q], x[r], acc[q][r]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = ti + R * q, j = tj + R * r;
        A[(int64_t)i * N + j] = acc[q][r];
        A[(int64_t)j * N + i] = acc[q][r];
      }
  }
}

static HoCellArgs ho_cell_args(const Ctx *c) {
  const Level &f = c->lv[0];
  const HoData &h = c->ho;
  return HoCellArgs{f.geometry, f.ncol, f.nlev, f.radius, c->sc.sigma, f.corners, f.z, h.tab, h.itab, h.ctab, h.ltab};
}

template <int P>
static int ho_make_tables(Ctx *c) {
  using H = Ho<P>;
  const Level &f = c->lv[0];
  HoData &h = c->ho;
  int st;
  std::vector<double> tab;
  std::vector<int> itab;
  ho_tables<P>(tab, itab);
  if ((st = dev_alloc(c, &h.tab, tab.size()))) return st;
  if ((st = dev_alloc(c, &h.itab, itab.size()))) return st;
  if ((st = dev_alloc(c, &h.ctab, (size_t)H::CTAB * f.ncol))) return st;
  if ((st = dev_alloc(c, &h.ltab, (size_t)H::LTAB * f.nlev))) return st;
  HMG_CUDA(c, cudaMemcpy(h.tab, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice));
  HMG_CUDA(c, cudaMemcpy(h.itab, itab.data(), sizeof(int) * itab.size(), cudaMemcpyHostToDevice));
  const HoCellArgs a = ho_cell_args(c);
  ho_column_kernel<P><<<f.ncol, kHoColThreads, sizeof(double) * kHoColSmem<P>, c->stream>>>(a, h.flag);
  ho_level_kernel<P><<<grid_for(f.nlev, 32), 32, 0, c->stream>>>(a);
  HMG_CUDA(c, cudaGetLastError());
  int sing = 0;
  HMG_CUDA(c, cudaMemcpyAsync(&sing, h.flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  HMG_CUDA(c, cudaStreamSynchronize(c->stream));
  if (sing) return fail(c, HMG_ERR_INVALID_ARG, "a degree-p cell matrix A_K is singular");
  return HMG_OK;
}

template <int P>
int ho_cell_matrices(Ctx *c, double *sk1) {
  using SH = HoCellShape<P>;
  const Level &f = c->lv[0];
  HoData &h = c->ho;
  int st;
  if (!h.tab && (st = ho_make_tables<P>(c))) return st;   // (a failure here frees the layout)
  const int smem = (int)sizeof(double) * SH::doubles(f.geometry == 1);
  HMG_CUDA(c, cudaFuncSetAttribute(ho_cell_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  ho_cell_kernel<P><<<(unsigned)f.ncell, SH::THREADS, smem, c->stream>>>(ho_cell_args(c), f.ncell, h.Ainv, h.m, sk1,
                                                                        h.flag);
  HMG_CUDA(c, cudaGetLastError());
  h.cw = h.tab + Ho<P>::TC;
  return HMG_OK;
}

template int ho_cell_matrices<1>(Ctx *, double *);
template int ho_cell_matrices<2>(Ctx *, double *);
template int ho_cell_matrices<3>(Ctx *, double *);

}  // namespace hmg

