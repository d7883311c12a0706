// Assembly kernels (setup phase): per-cell local matrices by Gauss quadrature, local
// condensation, the rows of the trace operator S, the pressure operator H on every
// multigrid level, Thomas factors of the column systems and the coarse scaling Gamma.
//
// Paper (arXiv 2210.11797): Sec. 2.2 Eq. bilinear_forms and the quadrature rule (3 Gauss
// points per direction for volume terms at p = 0; one-point cell-centre rule for q32,
// m3^rho, m3^Pi); Eq. 2x2system (B = Q32 + M3^rho M3^-1 D); Sec. 2.4 Eqs. hybrid-A,
// hybrid-K, hybrid-S (S = C^T A^-1 K); Sec. 2.3 Eq. elliptic_pressure_system
// (H = -B Mlump^-1 G + M3^Pi); Sec. 2.5 Eq. scaling_matrix (Gamma).
#include "assemble.cuh"
#include "device_common.cuh"
#include "hmg_internal.cuh"

namespace hmg {

// ---- the geometry of an extruded column, factorised -----------------------------------------
// A vertex at height z over corner c is c (R + z) on the sphere and (c_x, c_y, z) on the plane, so
// the trilinear map is x = C(xi, eta) s(zeta) with the bilinear corner map C and s = R + z (on the
// plane the two parts sit in different components and s = 1). The columns of J are then C_xi s,
// C_eta s and C dz, det J = s^2 dz D with D = (C_xi x C_eta) . C, the local vertical is
// C / |C|, and every integrand of M_K is a function of (xi, eta) times one of zeta: the 27-point
// Gauss sums are products of a 9-point sum per column and a 3-point sum per level. With
// q_d = C_d . C and h = 9-point weight / D:
//   vertical faces f, g:   M(f, g) = (A_fg + c22 B_fg) / dz,   A = sum h s_f s_g C_df . C_dg,
//                          B = sum h s_f s_g q_df q_dg / |C|^2
//   f and bottom / top z:  M(f, z) = (1 + c22) V1_z U_f,       U = sum h s_f q_df, V1 = sum w s_z / s
//   bottom / top:          M(z, z') = (1 + c22) dz V2_zz' W,   W = sum h |C|^2, V2 = sum w s_z s_z' / s^2
// and the antisymmetric Coriolis part likewise from (C_e x C_d) . z.
//
// On the sphere one thing does not factorise: the columns of J are differences of vertex coordinates
// of size R, so as the 27-point form evaluates them (rounded products c (R + z), an FMA chain over the
// eight vertices) they carry a rounding of about 1e-9 m: 3e-11 of a 33 m layer in the vertical column,
// and as much of the vertical part of the horizontal ones, which M(f, z) consists of. Results are kept
// on that form: the cell evaluates the same chains (the vertical column depends on (xi, eta) only, the
// xi column on (eta, zeta), the eta column on (xi, zeta): nine values each), takes their differences
// e, e_xi, e_eta from C dz, C_xi s, C_eta s and adds the first-order terms to the sums (in FP32: they
// are 1e-10 of the sums, so FP32 leaves 1e-17; the second order is 1e-21; the horizontal parts of e_xi
// and e_eta are 1e-14 of theirs and are left out). Without the correction M is off from the 27-point
// form by up to 1e-10 of an entry, with it by 1e-14 of the row's scale.
//
// Evaluating the 27 points in every cell cost about 6,700 FP64 operations per cell (22.2 ms for the
// 1.66M cells of C96 x 30 with rotation, and 3.0 ms for the condensation; all FP64 issue); here a column
// costs about 1,000 and a cell of the finest level about 1,000, most of them for the chains (coarser
// levels, which need neither M(f, z) nor its correction: 480), and the finest level's geometry and
// condensation together take 4.5 ms, at the FP64 issue rate.
struct Col {   // per-column sums [ncol][N]; face pairs f <= g in row-major order (10 of them)
  static constexpr int A = 0, B = 10, U = 20, XU = 24;   // XU: (C x C_d) . z part of M(f, z) per cz
  static constexpr int X = 28;     // 4: Coriolis pairs (0,1) (0,3) (1,2) (2,3) per cz / dz
  static constexpr int W = 32, DC = 33, DD = 34;         // D at the centre, sum w D
  static constexpr int RJ = 35;    // 3: (r . C_xi), (r . C_eta), |C| at the centre
  static constexpr int C = 38;     // 30: C at the nine points and the centre
  static constexpr int CD = 68;    // 18: C_xi at the three eta, C_eta at the three xi
  // 36 floats: sum over xi of h s_f C at the three eta for faces 1 and 3, over eta at the three xi for 0, 2
  static constexpr int K = 86;
  static constexpr int N = 104;
};
struct Lev {   // per-level sums [L][N]
  static constexpr int V1 = 0;     // 2: bottom, top
  static constexpr int V2 = 2;     // 3: bottom-bottom, bottom-top, top-top
  static constexpr int R = 5;      // s_centre^2 / sum w s^2: the ratio of the one-point and Gauss volumes
  static constexpr int S = 6;      // s_centre
  static constexpr int S0 = 7, S1 = 8;   // s at the bottom and the top (R + z)
  static constexpr int DZ = 9, IDZ = 10; // the layer's depth in the map (s1 - s0) and its inverse
  static constexpr int IZ = 11;    // 1 / (z1 - z0), of the background's vertical differences
  static constexpr int SQ = 12;    // 3: s at the Gauss points
  static constexpr int WQ = 15;    // 6 floats: w (zeta - 1) / s^2 and w zeta / s^2 there
  static constexpr int N = 18;
};

// the three Gauss points and weights on [0, 1]: 1/2 -+ sqrt(15) / 10
constexpr double kGq = 0.3872983346207417, kG0 = 0.5 - kGq, kG2 = 0.5 + kGq, kW0 = 5.0 / 18.0, kW1 = 8.0 / 18.0;
__constant__ double c_gx[3] = {kG0, 0.5, kG2}, c_gw[3] = {kW0, kW1, kW0};
__constant__ float c_gxf[3] = {(float)kG0, 0.5f, (float)kG2}, c_gwf[3] = {(float)kW0, (float)kW1, (float)kW0};
// bilinear weights of the corners (0,0), (1,0), (0,1), (1,1) at the nine points and the centre
#define HMG_BILINEAR(x, y) {(1.0 - x) * (1.0 - y), x * (1.0 - y), (1.0 - x) * y, x * y}
__constant__ double c_bilinear[10][4] = {
    HMG_BILINEAR(kG0, kG0), HMG_BILINEAR(0.5, kG0), HMG_BILINEAR(kG2, kG0), HMG_BILINEAR(kG0, 0.5),
    HMG_BILINEAR(0.5, 0.5), HMG_BILINEAR(kG2, 0.5), HMG_BILINEAR(kG0, kG2), HMG_BILINEAR(0.5, kG2),
    HMG_BILINEAR(kG2, kG2), HMG_BILINEAR(0.5, 0.5)};
#undef HMG_BILINEAR

// One thread per column, then one per level (blocks past the columns).
__global__ void __launch_bounds__(64) column_kernel(const CellArgs a, double *__restrict__ ctab,
                                                    double *__restrict__ ltab) {
  const double *gx = c_gx, *gw = c_gw;
  const int ncb = (a.ncol + (int)blockDim.x - 1) / (int)blockDim.x;
  if ((int)blockIdx.x >= ncb) {
    const int k = ((int)blockIdx.x - ncb) * blockDim.x + threadIdx.x;
    if (k >= a.L) return;
    const double z0 = a.z[k], z1 = a.z[k + 1];
    const bool sph = a.geometry == 1;
    const double s0 = sph ? a.radius + z0 : z0, s1 = sph ? a.radius + z1 : z1, dz = s1 - s0;
    double v1[2] = {0, 0}, v2[3] = {0, 0, 0}, s2 = 0.0;
    for (int q = 0; q < 3; ++q) {
      const double s = sph ? fma(gx[q], dz, s0) : 1.0, w = gw[q], is = 1.0 / s;
      const double m = (gx[q] - 1.0) * is, p = gx[q] * is;
      v1[0] = fma(w, m, v1[0]);
      v1[1] = fma(w, p, v1[1]);
      v2[0] = fma(w * m, m, v2[0]);
      v2[1] = fma(w * m, p, v2[1]);
      v2[2] = fma(w * p, p, v2[2]);
      s2 = fma(w * s, s, s2);
      double *o = ltab + (int64_t)k * Lev::N;
      o[Lev::SQ + q] = s;
      float *of = reinterpret_cast<float *>(o + Lev::WQ) + 2 * q;
      of[0] = (float)(w * m * is);
      of[1] = (float)(w * p * is);
    }
    const double sc = sph ? fma(0.5, dz, s0) : 1.0;
    double *o = ltab + (int64_t)k * Lev::N;
    for (int i = 0; i < 2; ++i) o[Lev::V1 + i] = v1[i];
    for (int i = 0; i < 3; ++i) o[Lev::V2 + i] = v2[i];
    o[Lev::R] = sc * sc / s2;
    o[Lev::S] = sc;
    o[Lev::S0] = s0;
    o[Lev::S1] = s1;
    o[Lev::DZ] = dz;
    o[Lev::IDZ] = 1.0 / dz;
    o[Lev::IZ] = 1.0 / (z1 - z0);
    return;
  }
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.ncol) return;
  const bool sphere = a.geometry == 1;
  // C = p0 + xi p1 + eta p2 + xi eta p3 from the corners (0,0), (1,0), (1,1), (0,1)
  const double *cp = a.corners + 12 * (int64_t)c;
  double p0[3], p1[3], p2[3], p3[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const bool used = sphere || i < 2;
    const double c0 = used ? cp[i] : 0.0, c1 = used ? cp[3 + i] : 0.0, c2 = used ? cp[6 + i] : 0.0,
                 c3 = used ? cp[9 + i] : 0.0;
    p0[i] = c0;
    p1[i] = c1 - c0;
    p2[i] = c3 - c0;
    p3[i] = (c2 - c3) - (c1 - c0);
  }
  double *o = ctab + (int64_t)c * Col::N;
  double A[10], B[10], U[4], XU[4], X[4], W = 0.0, DD = 0.0;
#pragma unroll
  for (int i = 0; i < 10; ++i) A[i] = B[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i) U[i] = XU[i] = X[i] = 0.0;
  float *kf = reinterpret_cast<float *>(o + Col::K);
#pragma unroll 1
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      o[Col::CD + 3 * q + i] = fma(gx[q], p3[i], p1[i]);
      o[Col::CD + 9 + 3 * q + i] = fma(gx[q], p3[i], p2[i]);
#pragma unroll
      for (int j = 0; j < 4; ++j) kf[3 * (q + 3 * j) + i] = 0.f;
    }
  auto at = [&](double xi, double eta, double (&C)[3], double (&Cx)[3], double (&Ce)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Cx[i] = fma(eta, p3[i], p1[i]);
      Ce[i] = fma(xi, p3[i], p2[i]);
      C[i] = fma(xi, Cx[i], fma(eta, p2[i], p0[i]));
    }
  };
  auto dot = [](const double (&u)[3], const double (&v)[3]) { return fma(u[2], v[2], fma(u[1], v[1], u[0] * v[0])); };
  // (C_xi x C_eta) . C on the sphere, the third component of C_xi x C_eta on the plane
  auto triple = [&](const double (&C)[3], const double (&Cx)[3], const double (&Ce)[3]) {
    const double n2 = Cx[0] * Ce[1] - Cx[1] * Ce[0];
    if (!sphere) return n2;
    const double n0 = Cx[1] * Ce[2] - Cx[2] * Ce[1], n1 = Cx[2] * Ce[0] - Cx[0] * Ce[2];
    return fma(n2, C[2], fma(n1, C[1], n0 * C[0]));
  };
#pragma unroll 1
  for (int q = 0; q < 9; ++q) {
    const double xi = gx[q % 3], eta = gx[q / 3], w = gw[q % 3] * gw[q / 3];
    double C[3], Cx[3], Ce[3];
    at(xi, eta, C, Cx, Ce);
#pragma unroll
    for (int i = 0; i < 3; ++i) o[Col::C + 3 * q + i] = C[i];
    const double D = triple(C, Cx, Ce), h = w / D;
    DD = fma(w, D, DD);
    const double g00 = h * dot(Cx, Cx), g01 = h * dot(Cx, Ce), g11 = h * dot(Ce, Ce);
    // pairs (0,0) (0,1) (0,2) (0,3) (1,1) (1,2) (1,3) (2,2) (2,3) (3,3); s = eta-1, xi, eta, xi-1
    const double s[4] = {eta - 1.0, xi, eta, xi - 1.0};
    const double x01 = h * (Ce[0] * Cx[1] - Ce[1] * Cx[0]);   // (C_eta x C_xi) . z = X[xi][eta]
    double b00 = 0.0, b01 = 0.0, b11 = 0.0;
    if (sphere) {
      const double cc = dot(C, C), qx = dot(C, Cx), qe = dot(C, Ce), hr = h / cc;
      const double hx = hr * qx;
      b00 = hx * qx;
      b01 = hx * qe;
      b11 = hr * qe * qe;
      W = fma(h, cc, W);
      const double yx = h * (C[0] * Cx[1] - C[1] * Cx[0]), ye = h * (C[0] * Ce[1] - C[1] * Ce[0]);
      U[0] = fma(s[0], h * qe, U[0]);
      U[1] = fma(s[1], h * qx, U[1]);
      U[2] = fma(s[2], h * qe, U[2]);
      U[3] = fma(s[3], h * qx, U[3]);
      XU[0] = fma(s[0], ye, XU[0]);
      XU[1] = fma(s[1], yx, XU[1]);
      XU[2] = fma(s[2], ye, XU[2]);
      XU[3] = fma(s[3], yx, XU[3]);
      const int face[4] = {1, 3, 0, 2};
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 3; ++i) kf[3 * ((j < 2 ? q / 3 : q % 3) + 3 * j) + i] += (float)(h * s[face[j]] * C[i]);
    } else {
      W += h;
    }
    int i = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int g = f; g < 4; ++g) {
        const double ss = s[f] * s[g];
        const bool df = (f & 1) == 0, dg = (g & 1) == 0;   // even faces: eta direction
        A[i] = fma(ss, df && dg ? g11 : (df || dg ? g01 : g00), A[i]);
        B[i] = fma(ss, df && dg ? b11 : (df || dg ? b01 : b00), B[i]);
        ++i;
      }
    // X[d_f][d_g] for f < g: (0,1) eta-xi, (0,3) eta-xi, (1,2) xi-eta, (2,3) eta-xi
    X[0] = fma(s[0] * s[1], -x01, X[0]);
    X[1] = fma(s[0] * s[3], -x01, X[1]);
    X[2] = fma(s[1] * s[2], x01, X[2]);
    X[3] = fma(s[2] * s[3], -x01, X[3]);
  }
#pragma unroll
  for (int i = 0; i < 10; ++i) { o[Col::A + i] = A[i]; o[Col::B + i] = B[i]; }
#pragma unroll
  for (int i = 0; i < 4; ++i) { o[Col::U + i] = U[i]; o[Col::XU + i] = XU[i]; o[Col::X + i] = X[i]; }
  double C[3], Cx[3], Ce[3];
  at(0.5, 0.5, C, Cx, Ce);
  const double Dc = triple(C, Cx, Ce), nc = sphere ? sqrt(dot(C, C)) : 1.0;
#pragma unroll
  for (int i = 0; i < 3; ++i) o[Col::C + 27 + i] = C[i];
  o[Col::W] = W;
  o[Col::DC] = Dc;
  o[Col::DD] = DD;
  o[Col::RJ] = sphere ? dot(C, Cx) / nc : 0.0;
  o[Col::RJ + 1] = sphere ? dot(C, Ce) / nc : 0.0;
  o[Col::RJ + 2] = nc;
}

// The geometry of one cell with its vertical weight c22 = -tau_u tau_theta dt^2 c_p d_z Pi d_z theta:
// M_K and the volumes. XPART: also the Coriolis part.
struct CellGeo {
  double hh[10];            // M(f, g) between vertical faces, symmetric part
  double xx[4];             // its Coriolis part on (0,1) (0,3) (1,2) (2,3)
  double us[4][2], px[4];   // M(f, z) = us_fz + V1_z px_f, M(z, f) = us_fz - V1_z px_f
  double wz;                // M(z, z') = wz V2_zz'
  double vol1, ratio;       // |K|_1 and |K|_1 / |K|
  double rj[3];             // zhat . J_d at the centre
};

__device__ __forceinline__ int pair4(int f, int g) {   // index of (f, g), f <= g, in Col::A and Col::B
  return f * 4 - f * (f - 1) / 2 + (g - f);
}

template <bool XPART>
__device__ __forceinline__ void cell_geometry(const CellArgs &a, const double *__restrict__ t,
                                              const double *__restrict__ l, int c, double c22, double cz,
                                              CellGeo &o) {
  const double dz = l[Lev::DZ], idz = l[Lev::IDZ], kap = 1.0 + c22, sc = l[Lev::S];
#pragma unroll
  for (int i = 0; i < 10; ++i) o.hh[i] = fma(c22, t[Col::B + i], t[Col::A + i]) * idz;
  if (XPART) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o.xx[i] = cz * idz * t[Col::X + i];
      o.us[i][0] = kap * l[Lev::V1] * t[Col::U + i];
      o.us[i][1] = kap * l[Lev::V1 + 1] * t[Col::U + i];
      o.px[i] = cz * t[Col::XU + i];
    }
  }
  o.wz = kap * dz * t[Col::W];
  o.vol1 = sc * sc * dz * t[Col::DC];
  o.ratio = t[Col::DC] / t[Col::DD] * l[Lev::R];
  o.rj[0] = sc * t[Col::RJ];
  o.rj[1] = sc * t[Col::RJ + 1];
  o.rj[2] = dz * t[Col::RJ + 2];
  if (a.geometry != 1) return;
  // vertices as rounded by the map, corners in the order (0,0), (1,0), (0,1), (1,1)
  double xb[3][4], xt[3][4];
  float p0[3], p1[3], p2[3], p3[3];
  {
    const double *cp = a.corners + 12 * (int64_t)c, s0 = l[Lev::S0], s1 = l[Lev::S1];
    const int at[4] = {0, 1, 3, 2};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double cc[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        cc[v] = cp[3 * at[v] + i];
        xb[i][v] = cc[v] * s0;
        xt[i][v] = cc[v] * s1;
      }
      p0[i] = (float)cc[0];
      p1[i] = (float)(cc[1] - cc[0]);
      p2[i] = (float)(cc[2] - cc[0]);
      p3[i] = (float)((cc[3] - cc[2]) - (cc[1] - cc[0]));
    }
  }
  // e = (the chain sum_v X_v dN_v / dzeta) - C dz at point q, over dz
  const float fi = (float)idz;
  auto rounding = [&](int q, float (&e)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double s = -(xb[i][0] * c_bilinear[q][0]);
#pragma unroll
      for (int v = 1; v < 4; ++v) s = fma(-xb[i][v], c_bilinear[q][v], s);
#pragma unroll
      for (int v = 0; v < 4; ++v) s = fma(xt[i][v], c_bilinear[q][v], s);
      e[i] = (float)fma(-t[Col::C + 3 * q + i], dz, s) * fi;
    }
  };
  auto dot = [](const float (&u)[3], const float (&v)[3]) { return fmaf(u[2], v[2], fmaf(u[1], v[1], u[0] * v[0])); };
  auto at = [&](float xi, float eta, float (&C)[3], float (&Cx)[3], float (&Ce)[3], float (&n)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Cx[i] = fmaf(eta, p3[i], p1[i]);
      Ce[i] = fmaf(xi, p3[i], p2[i]);
      C[i] = fmaf(xi, Cx[i], fmaf(eta, p2[i], p0[i]));
    }
    n[0] = Cx[1] * Ce[2] - Cx[2] * Ce[1];
    n[1] = Cx[2] * Ce[0] - Cx[0] * Ce[2];
    n[2] = Cx[0] * Ce[1] - Cx[1] * Ce[0];
  };
  const float fc22 = (float)c22, fkap = (float)kap, fcz = (float)cz;
  float dh[10], dx[4], du[4], dp[4], dw = 0.f, dv = 0.f, dd = 0.f;
#pragma unroll
  for (int i = 0; i < 10; ++i) dh[i] = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) dx[i] = du[i] = dp[i] = 0.f;
  float C[3], Cx[3], Ce[3], n[3], e[3];
#pragma unroll 1
  for (int q = 0; q < 9; ++q) {
    const float xi = c_gxf[q % 3], eta = c_gxf[q / 3], w = c_gwf[q % 3] * c_gwf[q / 3];
    rounding(q, e);
    at(xi, eta, C, Cx, Ce, n);
    const float D = dot(n, C), h = w / D, cc = dot(C, C), ic = 1.f / cc, ne = dot(n, e), tau = ne / D, ce = dot(C, e);
    const float qx = dot(C, Cx), qe = dot(C, Ce), ht = -h * tau, cr = fc22 * ic;
    dv = fmaf(w, ne, dv);
    dd = fmaf(w, D, dd);
    dw = fmaf(h, 2.f * ce - tau * cc, dw);
    const float m00 = ht * (dot(Cx, Cx) + cr * qx * qx), m01 = ht * (dot(Cx, Ce) + cr * qx * qe),
                m11 = ht * (dot(Ce, Ce) + cr * qe * qe);
    const float s[4] = {eta - 1.f, xi, eta, xi - 1.f};
    int i = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int g = f; g < 4; ++g) {
        const bool df = (f & 1) == 0, dg = (g & 1) == 0;
        dh[i] = fmaf(s[f] * s[g], df && dg ? m11 : (df || dg ? m01 : m00), dh[i]);
        ++i;
      }
    if (XPART) {
      const float x01 = ht * fcz * (Ce[0] * Cx[1] - Ce[1] * Cx[0]);
      dx[0] = fmaf(s[0] * s[1], -x01, dx[0]);
      dx[1] = fmaf(s[0] * s[3], -x01, dx[1]);
      dx[2] = fmaf(s[1] * s[2], x01, dx[2]);
      dx[3] = fmaf(s[2] * s[3], -x01, dx[3]);
      const float ux = h * (dot(Cx, e) + cr * qx * ce - tau * fkap * qx), ue = h * (dot(Ce, e) + cr * qe * ce - tau * fkap * qe);
      const float yx = h * fcz * (e[0] * Cx[1] - e[1] * Cx[0] - tau * (C[0] * Cx[1] - C[1] * Cx[0])),
                  ye = h * fcz * (e[0] * Ce[1] - e[1] * Ce[0] - tau * (C[0] * Ce[1] - C[1] * Ce[0]));
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        du[f] = fmaf(s[f], f & 1 ? ux : ue, du[f]);
        dp[f] = fmaf(s[f], f & 1 ? yx : ye, dp[f]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 10; ++i) o.hh[i] = fma((double)dh[i], idz, o.hh[i]);
  if (XPART) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o.xx[i] = fma((double)dx[i], idz, o.xx[i]);
      o.px[i] += (double)dp[i];
    }
    // e_xi at (eta, zeta) for faces 1 and 3, e_eta at (xi, zeta) for faces 0 and 2
    float dz1[4][2];
#pragma unroll
    for (int f = 0; f < 4; ++f) dz1[f][0] = dz1[f][1] = 0.f;
#pragma unroll 1
    for (int q = 0; q < 9; ++q) {
      const int hq = q % 3, vq = q / 3;
      const double sv = l[Lev::SQ + vq];
      const float *wq = reinterpret_cast<const float *>(l + Lev::WQ) + 2 * vq;
      const float w0 = wq[0], w1 = wq[1];
      const double *bw = c_bilinear[q];
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        float ed[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          double s = 0.0;
#pragma unroll
          for (int v = 0; v < 8; ++v) {   // v = va + 2 vb + 4 vc; the sign by va (xi) or vb (eta)
            const int va = v & 1, vb = (v >> 1) & 1, vc = v >> 2;
            const double x = vc ? xt[i][v & 3] : xb[i][v & 3], w = bw[(d == 0 ? vb : va) + 2 * vc];
            s = fma((d == 0 ? va : vb) ? x : -x, w, s);
          }
          ed[i] = (float)fma(-t[Col::CD + 9 * d + 3 * hq + i], sv, s);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float *kk = reinterpret_cast<const float *>(t + Col::K) + 3 * (hq + 3 * (2 * d + j));
          const float m = fmaf(ed[2], kk[2], fmaf(ed[1], kk[1], ed[0] * kk[0]));
          const int f = d == 0 ? 1 + 2 * j : 2 * j;
          dz1[f][0] = fmaf(w0, m, dz1[f][0]);
          dz1[f][1] = fmaf(w1, m, dz1[f][1]);
        }
      }
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      o.us[f][0] += (double)fmaf(fkap, dz1[f][0], du[f] * (float)l[Lev::V1]);
      o.us[f][1] += (double)fmaf(fkap, dz1[f][1], du[f] * (float)l[Lev::V1 + 1]);
    }
  }
  o.wz = fma(kap * dz, (double)dw, o.wz);
  rounding(9, e);
  at(0.5f, 0.5f, C, Cx, Ce, n);
  const float tc = dot(n, e) / dot(n, C), rc = dot(C, e) / dot(C, C);
  o.ratio = fma(o.ratio, (double)(tc - dv / dd), o.ratio);
  o.vol1 = fma(o.vol1, (double)tc, o.vol1);
  o.rj[2] = fma(o.rj[2], (double)rc, o.rj[2]);
}

template <bool XPART>
__device__ __forceinline__ void cell_coefficients(const CellArgs &a, const double *__restrict__ t,
                                                  const double *__restrict__ l, int c, int k, double cz,
                                                  CellGeo &g, CellCo &o) {
  const int L1 = a.L + 1;
  if (a.sc.preset == 1) {
    cell_geometry<XPART>(a, t, l, c, 0.0, 0.0, g);
    o.m = a.sc.sigma * g.vol1;
#pragma unroll
    for (int f = 0; f < 6; ++f) o.kth[f] = o.b[f] = 1.0;
  } else {
    const double *th = a.theta_lev + (int64_t)c * L1 + k, *pi = a.exner_lev + (int64_t)c * L1 + k;
    const double iz = l[Lev::IZ], th0 = th[0], th1 = th[1], dth = (th1 - th0) * iz, mean = 0.5 * (th0 + th1);
    const double c22 = -a.sc.tau_u * a.sc.tau_theta * a.sc.dt * a.sc.dt * a.sc.cp * ((pi[1] - pi[0]) * iz) * dth;
    cell_geometry<XPART>(a, t, l, c, c22, cz, g);
    const double kk = a.sc.tau_u * a.sc.dt * a.sc.cp;
    // single-valued theta on each face: vertical faces average the two columns' layer means
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const double *tn = a.theta_lev + (int64_t)__ldg(a.col_nbr + 4 * (int64_t)c + f) * L1 + k;
      o.kth[f] = kk * (0.5 * (mean + 0.5 * (tn[0] + tn[1])));
    }
    o.kth[4] = kk * th0;
    o.kth[5] = kk * th1;
    const double base = a.sc.tau_rho * a.sc.dt * g.ratio;   // M3^rho M3^-1 D
    // q32: tau_theta dt |K|_1 (d_z theta / theta) (zhat.v_f)(x_c), zhat.v_f = +-1/2 zhat.J_d / |K|_1
    const double q = 0.5 * a.sc.tau_theta * a.sc.dt * (dth / mean);
    o.b[0] = fma(-q, g.rj[1], base);
    o.b[1] = fma(q, g.rj[0], base);
    o.b[2] = fma(q, g.rj[1], base);
    o.b[3] = fma(-q, g.rj[0], base);
    o.b[4] = fma(-q, g.rj[2], base);
    o.b[5] = fma(q, g.rj[2], base);
    o.m = (1.0 - a.sc.kappa) / a.sc.kappa * g.vol1 / a.exner[(int64_t)c * a.L + k];
  }
  const double m02 = fabs(g.hh[pair4(0, 2)]), m13 = fabs(g.hh[pair4(1, 3)]);
  o.lump[0] = fabs(g.hh[pair4(0, 0)]) + m02;
  o.lump[1] = fabs(g.hh[pair4(1, 1)]) + m13;
  o.lump[2] = fabs(g.hh[pair4(2, 2)]) + m02;
  o.lump[3] = fabs(g.hh[pair4(3, 3)]) + m13;
  const double wz = fabs(g.wz), mp = fabs(l[Lev::V2 + 1]);
  o.lump[4] = wz * (l[Lev::V2] + mp);
  o.lump[5] = wz * (l[Lev::V2 + 2] + mp);
}

__device__ __forceinline__ double coriolis(const CellArgs &a) {   // tau_u dt 2 Omega (Eq. gh-u)
  return a.sc.preset == 1 ? 0.0 : a.sc.tau_u * a.sc.dt * 2.0 * a.sc.omega;
}

__global__ void __launch_bounds__(128) cell_kernel(const CellArgs a, const double *__restrict__ ctab,
                                                   const double *__restrict__ ltab, const CellOut q) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= a.ncell) return;
  const int c = (int)((unsigned)K / (unsigned)a.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)a.L);
  CellGeo g;
  CellCo o;
  cell_coefficients<false>(a, ctab + (int64_t)c * Col::N, ltab + k * Lev::N, c, k, 0.0, g, o);
  store_cell(q, o, a.ncell, K);
}

// The whole record of each finest-level cell (configuration 1's 2x2 system reads M_K itself).
__global__ void __launch_bounds__(128) record_kernel(const CellArgs a, const double *__restrict__ ctab,
                                                     const double *__restrict__ ltab, double *__restrict__ rec) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= a.ncell) return;
  const int c = (int)((unsigned)K / (unsigned)a.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)a.L);
  const double *t = ctab + (int64_t)c * Col::N, *l = ltab + k * Lev::N;
  CellGeo q;
  CellCo o;
  cell_coefficients<true>(a, t, l, c, k, coriolis(a), q, o);
  double *r = rec + K * kCellData;
  int im = 0, ic = 0;
#pragma unroll
  for (int f = 0; f < 6; ++f)
#pragma unroll
    for (int g = f; g < 6; ++g) {
      double v, x = 0.0;
      if (g < 4) {
        v = q.hh[pair4(f, g)];
        if ((f + g) & 1) x = q.xx[f == 0 ? g / 2 : f + 1];   // (0,1) (0,3) (1,2) (2,3)
      } else if (f < 4) {
        v = q.us[f][g - 4];
        x = l[Lev::V1 + g - 4] * q.px[f];
      } else {
        v = q.wz * l[Lev::V2 + (f - 4) + (g - 4)];
      }
      r[CellRec::M + im++] = v;
      if (g > f) r[CellRec::CORI + ic++] = x;
    }
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    r[CellRec::B + f] = o.b[f];
    r[CellRec::KTH + f] = o.kth[f];
    r[CellRec::LUMP + f] = o.lump[f];
  }
  r[CellRec::MPI] = o.m;
}

// A_K = [[M, g], [b^T, m]] with g = -KTH (Eq. hybrid-A), inverted by block elimination. The velocity
// block is M = [[H, U], [V, W]] over the vertical faces (H 4 x 4) and bottom / top (W 2 x 2):
//   Q = H^-1 U, P = V H^-1, Z = (W - V Q)^-1, M^-1 = [[H^-1 + Q Z P, -Q Z], [-Z P, Z]],
// with H^-1 by Gauss-Jordan without pivoting (the symmetric part of M is positive definite, the
// Coriolis part antisymmetric, so every pivot is positive). Then y = M^-1 g, z = M^-T b, the
// pressure Schur complement s = m - b.y and A^-1 = [[M^-1 + y z^T / s, -y / s], [-z^T / s, 1 / s]].
// The rows of A_K span ~20 orders of magnitude on the sphere; this form keeps every entry within a
// few ulps of its row's scale, where pivoting on A_K itself can lose 1e-12. About 400 FP64
// operations and 7 divides per cell instead of about 600 and 43 for a 6 x 6 LU of the equilibrated
// block and six pairs of triangular solves (no-pivot elimination does not depend on the scaling).
// Outputs: Ainv entry-major ((7 i + j) * ncell + K) and the cell's coefficients for the pressure
// operator. A non-positive pivot (M not positive definite) or s == 0 sets *singular.
__global__ void __launch_bounds__(128) condense_kernel(const CellArgs a, const double *__restrict__ ctab,
                                                       const double *__restrict__ ltab,
                                                       double *__restrict__ Ainv, const CellOut out,
                                                       int *__restrict__ singular) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= a.ncell) return;
  const int64_t C = a.ncell;
  const int c = (int)((unsigned)K / (unsigned)a.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)a.L);
  const double *t = ctab + (int64_t)c * Col::N, *l = ltab + k * Lev::N;
  CellGeo geo;
  CellCo o;
  cell_coefficients<true>(a, t, l, c, k, coriolis(a), geo, o);
  store_cell(out, o, C, K);
  double h[4][4];
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int g = f; g < 4; ++g) {
      const double v = geo.hh[pair4(f, g)];
      if ((f + g) & 1) {
        const double x = geo.xx[f == 0 ? g / 2 : f + 1];   // (0,1) (0,3) (1,2) (2,3)
        h[f][g] = v + x;
        h[g][f] = v - x;
      } else {
        h[f][g] = h[g][f] = v;
      }
    }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (!(h[p][p] > 0.0)) { atomicExch(singular, 1); return; }
    const double inv = 1.0 / h[p][p];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j != p) h[p][j] *= inv;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i == p) continue;
      const double f = h[i][p];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j != p) h[i][j] = fma(-f, h[p][j], h[i][j]);
      h[i][p] = -f * inv;
    }
    h[p][p] = inv;
  }
  double Q[4][2], P[2][4], w[2][2];
  {
    double U[4][2], V[2][4];
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const double x = l[Lev::V1 + e] * geo.px[f];
        U[f][e] = geo.us[f][e] + x;
        V[e][f] = geo.us[f][e] - x;
      }
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          s0 = fma(h[f][g], U[g][e], s0);
          s1 = fma(V[e][g], h[g][f], s1);
        }
        Q[f][e] = s0;
        P[e][f] = s1;
      }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        double v = geo.wz * l[Lev::V2 + i + j];
#pragma unroll
        for (int g = 0; g < 4; ++g) v = fma(-V[i][g], Q[g][j], v);
        w[i][j] = v;
      }
  }
  if (!(w[0][0] > 0.0)) { atomicExch(singular, 1); return; }
  const double i0 = 1.0 / w[0][0], lw = w[1][0] * i0, uw = w[0][1] * i0, piv = fma(-lw, w[0][1], w[1][1]);
  if (!(piv > 0.0)) { atomicExch(singular, 1); return; }
  double Mi[6][6];   // M^-1
  Mi[5][5] = 1.0 / piv;
  Mi[4][5] = -uw * Mi[5][5];
  Mi[5][4] = -lw * Mi[5][5];
  Mi[4][4] = fma(-uw, Mi[5][4], i0);
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      Mi[f][4 + e] = -fma(Q[f][1], Mi[5][4 + e], Q[f][0] * Mi[4][4 + e]);
      Mi[4 + e][f] = -fma(Mi[4 + e][5], P[1][f], Mi[4 + e][4] * P[0][f]);
    }
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int g = 0; g < 4; ++g) Mi[f][g] = fma(-Mi[f][5], P[1][g], fma(-Mi[f][4], P[0][g], h[f][g]));
  double y[6], z[6];   // y = M^-1 g (g = -kth), z = M^-T b
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      s0 = fma(-Mi[i][j], o.kth[j], s0);
      s1 = fma(Mi[j][i], o.b[j], s1);
    }
    y[i] = s0;
    z[i] = s1;
  }
  double s = o.m;
#pragma unroll
  for (int j = 0; j < 6; ++j) s = fma(-o.b[j], y[j], s);
  if (s == 0.0) { atomicExch(singular, 1); return; }
  const double is = 1.0 / s;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double yi = y[i] * is;
#pragma unroll
    for (int j = 0; j < 6; ++j) Ainv[(int64_t)(7 * i + j) * C + K] = fma(yi, z[j], Mi[i][j]);
    Ainv[(int64_t)(7 * i + 6) * C + K] = -yi;
    Ainv[(int64_t)(42 + i) * C + K] = -z[i] * is;
  }
  Ainv[(int64_t)48 * C + K] = is;
}

struct RowArgs {
  int L;
  int64_t NH, NT, ncell;
  const int32_t *stencil, *edge_fc, *col_edges, *col_nbr, *col_nbr_face;
};

// Rows of S: the sum of the (at most two) cells' S_K rows, in the slot order of s_row.
// S_K = (A_K^-1)_uu diag(KTH) is formed here, entry by entry: storing it cost 36 doubles per cell
// written and read (0.96 GB at C96 x 30).
__global__ void trace_rows_kernel(const RowArgs a, const double *__restrict__ Ainv,
                                  const double *__restrict__ kth, double *__restrict__ S) {
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row >= a.NT) return;
  const int64_t C = a.ncell, T = a.NT;
  double v[kSlots];
  auto sk = [&](int64_t K, int i, int j) {   // (rounded before any sum: a contracted sum would depend on the row)
    return __dmul_rn(Ainv[(int64_t)(7 * i + j) * C + K], kth[(int64_t)j * C + K]);
  };
  if (row < a.NH) {
    const int e = (int)((unsigned)row / (unsigned)a.L), k = (int)((unsigned)row - (unsigned)e * (unsigned)a.L);
    const int c1 = a.stencil[8 * (int64_t)e], c2 = a.stencil[8 * (int64_t)e + 1];
    const int i1 = a.edge_fc[2 * (int64_t)e], i2 = a.edge_fc[2 * (int64_t)e + 1];
    const int64_t K1 = (int64_t)c1 * a.L + k, K2 = (int64_t)c2 * a.L + k;
    v[0] = sk(K1, i1, i1) + sk(K2, i2, i2);
    for (int m = 1; m <= 3; ++m) v[m] = sk(K1, i1, (i1 + m) & 3);
    v[4] = sk(K1, i1, 4);
    v[5] = sk(K1, i1, 5);
    for (int m = 1; m <= 3; ++m) v[5 + m] = sk(K2, i2, (i2 + m) & 3);
    v[9] = sk(K2, i2, 4);
    v[10] = sk(K2, i2, 5);
  } else {
    const unsigned zr = (unsigned)(row - a.NH), L1 = (unsigned)a.L + 1u;
    const int c = (int)(zr / L1), k = (int)(zr - (unsigned)c * L1);
    for (int m = 0; m < kSlots; ++m) v[m] = 0.0;
    double self_a = 0.0, self_b = 0.0;
    if (k < a.L) {
      const int64_t Ka = (int64_t)c * a.L + k;
      self_a = sk(Ka, 4, 4);
      for (int i = 0; i < 4; ++i) v[1 + i] = sk(Ka, 4, i);
      v[5] = sk(Ka, 4, 5);
    }
    if (k > 0) {
      const int64_t Kb = (int64_t)c * a.L + k - 1;
      self_b = sk(Kb, 5, 5);
      for (int i = 0; i < 4; ++i) v[6 + i] = sk(Kb, 5, i);
      v[10] = sk(Kb, 5, 4);
    }
    v[0] = self_a + self_b;
  }
#pragma unroll
  for (int m = 0; m < kSlots; ++m) S[m * T + row] = v[m];
}

// Thomas factors of every column system, the relaxation folded in: the S^zz_j of Algorithm 1 (rows
// k = 0..L: sub = slot 10, diag = slot 0, sup = slot 5) and the H_z of every multigrid level. For
// pivot p_k = d_k - s_k cp_{k-1}: w = omega / p_k, l = s_k / p_k (s_k the sub-diagonal) and
// cp = u_k / p_k (u_k the super-diagonal). The sweeps then do y_k = r_k w_k - l_k y_{k-1},
// x_k = y_k - cp_k x_{k+1} (one FMA per row each), and x += is omega (tridiagonal)^-1 r. One launch
// for all systems, a block per cpb columns: the three diagonals staged in shared memory with
// coalesced loads, one lane per column on the serial chain of divides (whole warps on it, as the
// FP64 pipe is occupied per warp), the factors stored coalesced. A launch per system with one thread
// per column straight from global memory took 0.24 ms for the five systems of C96 x 30, four of them
// waiting on the strided loads of a few warps; this takes 0.09 ms.
struct FactorJob {
  const double *sub, *diag, *sup;   // [ncol][n], sub ignored at k = 0
  double *w, *l, *cp;
  double omega;
  int n, ncol, cpb, blk0;           // blocks blk0 .. of the launch
};
struct FactorJobs {
  FactorJob j[kMaxLevels + 1];
  int count;
};

__global__ void __launch_bounds__(128) factor_kernel(const FactorJobs jobs) {
  extern __shared__ double fsm[];
  int id = jobs.count - 1;
  while (id > 0 && (int)blockIdx.x < jobs.j[id].blk0) --id;
  const FactorJob &q = jobs.j[id];
  const int n = q.n, ld = n | 1, c0 = ((int)blockIdx.x - q.blk0) * q.cpb, nc = min(q.cpb, q.ncol - c0);
  double *sub = fsm, *diag = sub + q.cpb * ld, *sup = diag + q.cpb * ld;
  const int64_t base = (int64_t)c0 * n;
  for (int i = threadIdx.x; i < nc * n; i += blockDim.x) {
    const int o = (i / n) * ld + i % n;
    sub[o] = __ldg(q.sub + base + i);
    diag[o] = __ldg(q.diag + base + i);
    sup[o] = __ldg(q.sup + base + i);
  }
  __syncthreads();
  if ((int)threadIdx.x < nc) {
    const int o = (int)threadIdx.x * ld;
    double cp = 0.0;
    for (int k = 0; k < n; ++k) {
      const double sb = k > 0 ? sub[o + k] : 0.0;
      const double inv = 1.0 / (diag[o + k] - sb * cp);
      cp = sup[o + k] * inv;
      diag[o + k] = q.omega * inv;
      sub[o + k] = sb * inv;
      sup[o + k] = cp;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nc * n; i += blockDim.x) {
    const int o = (i / n) * ld + i % n;
    q.w[base + i] = diag[o];
    q.l[base + i] = sub[o];
    q.cp[base + i] = sup[o];
  }
}

// hw = omega / diag(S^hh) (the Jacobi part of Algorithm 1)
__global__ void jacobi_factor_kernel(int64_t n, const double *__restrict__ S, double omega, double *__restrict__ hw) {
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row < n) hw[row] = omega / S[row];
}

struct HArgs {
  int L, ncol;
  int64_t ncell;
  const int32_t *col_nbr, *col_nbr_face;
};

// Row of H = -B Mlump^-1 G + M3^Pi for cell K (7-point): coupling across face f is
// -b_K(f) k theta_f / Mlump_f with Mlump_f the sum of both cells' shares (k theta_f is single-valued);
// the diagonal is M3^Pi plus b_K(f) k theta_f / Mlump_f over the interior faces. One divide per face.
__global__ void pressure_rows_kernel(const HArgs a, const CellOut q, double *__restrict__ H) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= a.ncell) return;
  const int c = (int)((unsigned)K / (unsigned)a.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)a.L);
  const int64_t C = a.ncell;
  auto b = [&](int f) { return (f < 3 ? q.b[0] : q.b[1])[(f % 3) * C + K]; };
  auto lump = [&](int f, int64_t cell) { return (f < 3 ? q.lump[0] : q.lump[1])[(f < 3 ? f : f - 3) * C + cell]; };
  double diag = q.m[K];
  auto face = [&](int f, int nf, int64_t nb) {
    const double h = b(f) * q.kth[f * C + K] / (lump(f, K) + lump(nf, nb));
    diag += h;
    H[(1 + f) * C + K] = -h;
  };
#pragma unroll
  for (int f = 0; f < 4; ++f)
    face(f, __ldg(a.col_nbr_face + 4 * (int64_t)c + f), (int64_t)__ldg(a.col_nbr + 4 * (int64_t)c + f) * a.L + k);
  if (k > 0) face(4, 5, K - 1);
  else H[5 * C + K] = 0.0;
  if (k < a.L - 1) face(5, 4, K + 1);
  else H[6 * C + K] = 0.0;
  H[K] = diag;
}

// Gamma_K = (H 1)_K / (P^T S P 1)_K (Eq. scaling_matrix). H 1 = M3^Pi 1: G annihilates
// constants on every interior facet (its two cells contribute -k theta and +k theta with the
// same single-valued theta), so the numerator is the cell's M3^Pi, free of the cancellation
// of summing H's row. P 1 = 1; S 1 on each face is the sum of S_K 1 over the (one or two) cells
// sharing it, and S_K 1 = m (A^-1)_{u,p}: from G_K = -K_K 1, A [0; -1] = [K_K 1; -m], so the row sums
// follow without the cancellation of summing S_K's entries. P^T weights 1/2 on interior faces and 1
// on ground and lid faces.
__global__ void gamma_kernel(const RowArgs a, const double *__restrict__ Ainv, const double *__restrict__ m,
                             double *__restrict__ gamma) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= a.ncell) return;
  const int c = (int)((unsigned)K / (unsigned)a.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)a.L);
  const int64_t C = a.ncell;
  auto sk1 = [&](int f, int64_t cell) { return __dmul_rn(m[cell], Ainv[(int64_t)(7 * f + 6) * C + cell]); };
  double ps1 = 0.0;
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int nb = __ldg(a.col_nbr + 4 * (int64_t)c + f), nf = __ldg(a.col_nbr_face + 4 * (int64_t)c + f);
    ps1 += 0.5 * (sk1(f, K) + sk1(nf, (int64_t)nb * a.L + k));
  }
  ps1 += k == 0 ? sk1(4, K) : 0.5 * (sk1(4, K) + sk1(5, K - 1));
  ps1 += k == a.L - 1 ? sk1(5, K) : 0.5 * (sk1(5, K) + sk1(4, K + 1));
  gamma[K] = m[K] / ps1;
}

__global__ void to_float_kernel(const double *__restrict__ in, float *__restrict__ out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

static int to_float(Ctx *c, const double *in, float **out, int64_t n) {
  if (!*out) {
    int st = dev_alloc(c, out, (size_t)n);
    if (st) return st;
  }
  to_float_kernel<<<grid_for(n, 256) > 4096 ? 4096 : grid_for(n, 256), 256, 0, c->stream>>>(in, *out, n);
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

// The FP32 preconditioner's copies of the assembled lowest-order operators (S, Gamma, H on every
// level, then the factors with their copies through build_factors), made from the FP64 data on
// the device: for a context that switches to precision mixed without room for the direct sums' operators.
int make_fp32(Ctx *c) {
  const Level &f = c->lv[0];
  int st;
  if ((st = to_float(c, c->S, &c->S32, (int64_t)kSlots * f.ntrace))) return st;
  if ((st = to_float(c, c->gamma, &c->gamma32, f.ncell))) return st;
  for (int l = 0; l < c->nmg; ++l) {
    Level &lv = c->lv[l];
    if ((st = to_float(c, lv.H, &lv.H32, (int64_t)kHCoef * lv.ncell))) return st;
  }
  c->have_fp32 = true;
  if ((st = build_factors(c))) c->have_fp32 = false;
  return st;
}

// Relaxation-weighted Thomas factors of S^zz, 1/diag S^hh and H_z on every level for the
// current omega and mg_omega (and their FP32 copies when those exist). Rebuilt whenever
// either relaxation weight changes.
int build_factors(Ctx *c) {
  const Level &f = c->lv[0];
  FactorJobs jobs{};
  int blocks = 0;
  size_t smem = 0;
  auto add = [&](const double *sub, const double *diag, const double *sup, double *w, double *l, double *cp,
                 double omega, int n, int ncol) {
    const int cmax = 2048 / (n | 1), cpb = cmax < 1 ? 1 : (cmax < 32 ? cmax : 32);   // three arrays within 48 KB
    jobs.j[jobs.count++] = FactorJob{sub, diag, sup, w, l, cp, omega, n, ncol, cpb, blocks};
    blocks += (ncol + cpb - 1) / cpb;
    const size_t need = sizeof(double) * 3 * cpb * (n | 1);
    smem = need > smem ? need : smem;
  };
  const double *Sz = c->S + f.nth;
  add(Sz + 10 * f.ntrace, Sz, Sz + 5 * f.ntrace, c->Sz_w, c->Sz_l, c->Sz_cp, c->opt.omega, f.nlev + 1, f.ncol);
  for (int l = 0; l < c->nmg; ++l) {
    Level &lv = c->lv[l];
    add(lv.H + 5 * lv.ncell, lv.H, lv.H + 6 * lv.ncell, lv.Hz_w, lv.Hz_l, lv.Hz_cp, c->opt.mg_omega, lv.nlev, lv.ncol);
  }
  factor_kernel<<<blocks, 128, smem, c->stream>>>(jobs);
  jacobi_factor_kernel<<<grid_for(f.nth, 256), 256, 0, c->stream>>>(f.nth, c->S, c->opt.omega, c->Sh_w);
  HMG_CUDA(c, cudaGetLastError());
  int st;
  if (c->have_fp32) {
    if ((st = to_float(c, c->Sz_w, &c->Sz_w32, f.ntz))) return st;
    if ((st = to_float(c, c->Sz_l, &c->Sz_l32, f.ntz))) return st;
    if ((st = to_float(c, c->Sz_cp, &c->Sz_cp32, f.ntz))) return st;
    if ((st = to_float(c, c->Sh_w, &c->Sh_w32, f.nth))) return st;
    for (int l = 0; l < c->nmg; ++l) {
      Level &lv = c->lv[l];
      if ((st = to_float(c, lv.Hz_w, &lv.Hz_w32, lv.ncell))) return st;
      if ((st = to_float(c, lv.Hz_l, &lv.Hz_l32, lv.ncell))) return st;
      if ((st = to_float(c, lv.Hz_cp, &lv.Hz_cp32, lv.ncell))) return st;
    }
  }
  c->factor_omega = c->opt.omega;
  c->factor_mg_omega = c->opt.mg_omega;
  return HMG_OK;
}

// The per-cell data between the kernels lives in the Krylov vectors (at least ntrace + ncell > 4 C
// doubles each, idle here: whatever used them before is earlier on this stream): level 0 in r, rhat,
// p, v and s, each coarser level (at most C / 4 cells) in turn in t and phat.
static CellOut cell_buffers(Ctx *c, int l) {
  const int64_t C = c->lv[l].ncell;
  CellOut q;
  if (l == 0) {
    q.b[0] = c->r;
    q.b[1] = c->rhat;
    q.lump[0] = c->p;
    q.lump[1] = c->v;
    q.kth = c->kth;
    q.m = c->s;
  } else {
    q.b[0] = c->t;
    q.b[1] = c->t + 3 * C;
    q.lump[0] = c->t + 6 * C;
    q.lump[1] = c->t + 9 * C;
    q.kth = c->phat;
    q.m = c->phat + 6 * C;
  }
  return q;
}

static int assemble_levels(Ctx *c, double *rec) {
  Level &f = c->lv[0];
  const int64_t C = f.ncell, T = f.ntrace;
  int st;
  if ((st = dev_make(c, &c->S, (size_t)kSlots * T))) return st;
  if ((st = dev_make(c, &c->Sz_w, (size_t)f.ntz))) return st;
  if ((st = dev_make(c, &c->Sz_l, (size_t)f.ntz))) return st;
  if ((st = dev_make(c, &c->Sz_cp, (size_t)f.ntz))) return st;
  if ((st = dev_make(c, &c->Sh_w, (size_t)f.nth))) return st;
  if ((st = dev_make(c, &c->Ainv, (size_t)49 * C))) return st;
  if ((st = dev_make(c, &c->kth, (size_t)6 * C))) return st;
  if ((st = dev_make(c, &c->gamma, (size_t)C))) return st;
  if ((st = dev_make(c, &c->asm_flag, 1))) return st;
  HMG_CUDA(c, cudaMemsetAsync(c->asm_flag, 0, sizeof(int), c->stream));
  for (int l = 0; l < c->nmg; ++l) {
    Level &lv = c->lv[l];
    const CellArgs a{lv.geometry, lv.ncol, lv.nlev, lv.ncell, lv.radius, lv.corners, lv.z,
                     lv.theta_lev, lv.exner_lev, lv.exner, lv.col_nbr, c->sc};
    if (!rec && !lv.geo_ready) {   // the sums depend on the mesh only, which a context keeps
      if ((st = dev_make(c, &lv.ctab, (size_t)Col::N * lv.ncol))) return st;
      if ((st = dev_make(c, &lv.ltab, (size_t)Lev::N * lv.nlev))) return st;
      column_kernel<<<grid_for(lv.ncol, 64) + grid_for(lv.nlev, 64), 64, 0, c->stream>>>(a, lv.ctab, lv.ltab);
      HMG_CUDA(c, cudaGetLastError());
      lv.geo_ready = true;
    }
    if ((st = dev_make(c, &lv.H, (size_t)kHCoef * lv.ncell))) return st;
    if ((st = dev_make(c, &lv.Hz_w, (size_t)lv.ncell))) return st;
    if ((st = dev_make(c, &lv.Hz_l, (size_t)lv.ncell))) return st;
    if ((st = dev_make(c, &lv.Hz_cp, (size_t)lv.ncell))) return st;
    const CellOut q = cell_buffers(c, l);
    if (rec) {
      if ((st = gauss_cells(c, a, q, rec, l == 0 ? c->Ainv : nullptr))) return st;
    } else if (l == 0) condense_kernel<<<grid_for(C, 128), 128, 0, c->stream>>>(a, lv.ctab, lv.ltab, c->Ainv, q, c->asm_flag);
    else cell_kernel<<<grid_for(lv.ncell, 128), 128, 0, c->stream>>>(a, lv.ctab, lv.ltab, q);
    const HArgs ha{lv.nlev, lv.ncol, lv.ncell, lv.col_nbr, lv.col_nbr_face};
    pressure_rows_kernel<<<grid_for(lv.ncell, 256), 256, 0, c->stream>>>(ha, q, lv.H);
    HMG_CUDA(c, cudaGetLastError());
    if (l == 0) {
      const RowArgs ra{f.nlev, f.nth, T, C, f.edge_stencil, f.edge_fc, f.col_edges, f.col_nbr, f.col_nbr_face};
      trace_rows_kernel<<<grid_for(T, 256), 256, 0, c->stream>>>(ra, c->Ainv, c->kth, c->S);
      gamma_kernel<<<grid_for(C, 256), 256, 0, c->stream>>>(ra, c->Ainv, q.m, c->gamma);
      HMG_CUDA(c, cudaGetLastError());
      if (c->opt.precond == HMG_PRECOND_SCHUR) {   // configuration 1 (FP64) needs M_K itself
        double *mk = nullptr;
        HMG_CUDA(c, cudaMalloc(&mk, (size_t)C * kCellData * sizeof(double)));
        record_kernel<<<grid_for(C, 128), 128, 0, c->stream>>>(a, lv.ctab, lv.ltab, mk);
        st = build_mixed(c, mk);
        const cudaError_t e = cudaStreamSynchronize(c->stream);
        cudaFree(mk);
        if (st) return st;
        HMG_CUDA(c, e);
      }
    }
  }
  if (c->opt.precision == HMG_PRECISION_MIXED && !c->have_fp32) {
    if ((st = to_float(c, c->S, &c->S32, (int64_t)kSlots * T))) return st;
    if ((st = to_float(c, c->gamma, &c->gamma32, C))) return st;
    for (int l = 0; l < c->nmg; ++l) {
      Level &lv = c->lv[l];
      if ((st = to_float(c, lv.H, &lv.H32, (int64_t)kHCoef * lv.ncell))) return st;
    }
    c->have_fp32 = true;
  }
  if ((st = build_factors(c))) return st;
  int sing = 0;
  HMG_CUDA(c, cudaMemcpyAsync(&sing, c->asm_flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  HMG_CUDA(c, cudaStreamSynchronize(c->stream));
  if (sing) return fail(c, HMG_ERR_INVALID_ARG, "a velocity mass block M_K is not positive definite or A_K is singular");
  return HMG_OK;
}

int assemble_all(Ctx *c) {
  if (c->opt.precision != HMG_PRECISION_MIXED) return assemble_levels(c, nullptr);
  // contexts with the FP32 preconditioner: direct Gauss sums (gauss_cells.cu says why)
  double *rec = nullptr;
  int st = gauss_setup(c, c->lv[0].ncell, &rec);
  if (!st) st = assemble_levels(c, rec);
  if (rec) {
    cudaStreamSynchronize(c->stream);   // (an error return may leave kernels that use it in flight)
    cudaFree(rec);
  }
  return st;
}

}  // namespace hmg
