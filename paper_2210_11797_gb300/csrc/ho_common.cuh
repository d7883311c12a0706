// The degree-p spaces' sizes and table layouts and the access to the mesh, shared by the degree-p
// translation units (higher_order.cu: the operator and its preconditioner, ho_cells.cu: the cell
// matrices).
#pragma once

#include "hmg_internal.cuh"

namespace hmg {

template <int P>
struct Ho {
  static constexpr int NT = P + 1;                    // Gauss-Legendre nodes per direction
  static constexpr int NB = NT * NT;                  // nodes (trace rows) per facet
  static constexpr int NF = 6 * NB;                   // facet dofs: the hybridised cell matrix is NF x NF
  static constexpr int NU = 3 * NT * NT * (P + 2);    // RT_p dofs
  static constexpr int NP = NT * NT * NT;             // DG_p dofs
  static constexpr int N = NU + NP;                   // the mixed cell matrix
  static constexpr int NQ1 = P + 3;                   // volume Gauss points per direction
  static constexpr int SLOTS = 2 * NF;                // S coefficients stored per trace row
  static constexpr int NINT = P * NT * NT;            // interior dofs per component
  static constexpr int NV = P + 2;                    // Gauss-Lobatto nodes along a component's direction
  static constexpr int NH = 2 * NV * NT;              // horizontal functions of the xi and eta components
  static constexpr int NM = NT * NT;                  // of the zeta component, and of the pressure
  static constexpr int NZ = NM * NV;                  // zeta-component dofs (NU = NH NT + NZ)
  static constexpr int NG = 3 * NV;                   // nonzeros of a column of G
  // reference tables: Gauss-Legendre and Gauss-Lobatto bases at the Gauss points, its weights and
  // points, the Gauss-Legendre weights, the nonzeros of G, the facet weights
  static constexpr int TL = 0, TN = TL + NQ1 * NT, TW = TN + NQ1 * NV, TX = TW + NQ1, TGW = TX + NQ1, TGV = TGW + NT,
                       TC = TGV + NG * NP, TAB = TC + NB;
  // integer tables: the row of each nonzero of G; the velocity dof at each place of the
  // tensor-product order (horizontal function, vertical node), its basis function's sign in bit 30
  static constexpr int IG = 0, IO = IG + NG * NP, ITAB = IO + NU;
  // geometry sums per column (H_hh^-1, Q_c = H_hh^-1 H_hz, H_zz, K_c = H_zh Q_c, H_p) and per level
  // (1 / D, Q_l = D^-1 V, V_zz, W_l = V^T Q_l, V_p), and the one-point volume's factors
  static constexpr int CHI = 0, CQ = CHI + NH * NH, CZZ = CQ + NH * NM, CK = CZZ + NM * NM, CP = CK + NM * NM,
                       CD = CP + NM * NM, CTAB = CD + 1;
  static constexpr int LD = 0, LQ = LD + NT, LZZ = LQ + NT * NV, LW = LZZ + NV * NV, LP = LW + NV * NV,
                       LV = LP + NT * NT, LTAB = LV + 1;
  // the sweep's line part: lanes per column (a group of LPC >= NB lanes of one warp; lane n < NB
  // computes component n of each block product) and columns per warp (p = 2: three groups of
  // nine, five lanes idle)
  static constexpr int LPC = P == 1 ? 4 : (P == 2 ? 9 : 16);
  static constexpr int CPW = 32 / LPC;
};

// ---- mesh access ------------------------------------------------------------------------------
struct HoGeo {
  int L, ncol;
  int64_t NH;                 // rows of the vertical facets (NB nedge L)
  int64_t nhf, nzf;           // vertical and horizontal facets
  const int32_t *col_edges, *stencil, *edge_fc;
  const int8_t *own;          // [ncol][4] 1 if the column owns the edge of that face
};

// trace row of local facet dof q of cell (c, k)
template <int P>
__device__ __forceinline__ int64_t ho_gid(const HoGeo &g, int c, int k, int q) {
  using H = Ho<P>;
  const int f = q / H::NB, r = q - f * H::NB, s = r / H::NT, t = r - s * H::NT;
  if (f < 4) {
    const int64_t e = g.col_edges[4 * (int64_t)c + f];
    const int sg = g.own[4 * (int64_t)c + f] ? s : P - s;
    return H::NB * (e * g.L + k) + H::NT * sg + t;
  }
  const int kk = k + (f == 5 ? 1 : 0);
  return g.NH + H::NB * ((int64_t)c * (g.L + 1) + kk) + H::NT * s + t;
}

// The one or two cells of facet F: A (and B), their local faces, and whether a node's local s is
// reversed in B (vertical facets: B traverses the edge backwards).
struct HoFacet {
  int cA, kA, fA, cB, kB, fB;   // cB < 0: a ground or lid facet (one cell)
  bool flipB;
};

__device__ __forceinline__ HoFacet ho_facet(const HoGeo &g, int64_t F) {
  HoFacet r;
  if (F < g.nhf) {   // (facets number less than 2^31: 32-bit index arithmetic)
    const unsigned Fu = (unsigned)F, Lu = (unsigned)g.L;
    const int e = (int)(Fu / Lu), k = (int)(Fu - (unsigned)e * Lu);
    r.cA = g.stencil[8 * (int64_t)e];
    r.cB = g.stencil[8 * (int64_t)e + 1];
    r.fA = g.edge_fc[2 * (int64_t)e];
    r.fB = g.edge_fc[2 * (int64_t)e + 1];
    r.kA = r.kB = k;
    r.flipB = true;
  } else {
    const unsigned zf = (unsigned)(F - g.nhf), L1 = (unsigned)g.L + 1u;
    const int c = (int)(zf / L1), k = (int)(zf - (unsigned)c * L1);
    r.cA = c;
    r.flipB = false;
    if (k < g.L) {
      r.kA = k;
      r.fA = 4;                                  // the facet is the bottom of the cell above
      r.cB = k > 0 ? c : -1;
      r.kB = k - 1;
      r.fB = 5;
    } else {
      r.kA = g.L - 1;
      r.fA = 5;                                  // the lid: the top of the last cell
      r.cB = -1;
      r.kB = 0;
      r.fB = 0;
    }
  }
  return r;
}

// ho_cells.cu: A_K^-1 of every cell into ho.Ainv, (H 1)_K into ho.m and S_K 1 summed over each facet into
// sk1 [6][ncell], from the reference tables and the mesh's geometry sums (made on the first call of a
// layout); *ho.flag set when a cell is singular
template <int P>
int ho_cell_matrices(Ctx *c, double *sk1);
// gauss_cells.cu: A_K^-1 and (H 1)_K by direct Gauss sums and a pivoted elimination
template <int P>
int ho_gauss_cell_matrices(Ctx *c);

}  // namespace hmg
