// The per-cell data shared by the two forms of the lowest-order assembly (assemble.cu, gauss_cells.cu).
#pragma once

#include "hmg_internal.cuh"

namespace hmg {

struct CellArgs {
  int geometry, ncol, L;
  int64_t ncell;
  double radius;
  const double *corners, *z, *theta_lev, *exner_lev, *exner;
  const int32_t *col_nbr;
  hmg_scalars sc;
};

// The coefficients of one cell: the diagonal of K_K, the pressure-row couplings, M3^Pi and this
// cell's share |M(f,f)| + |M(f, opposite f)| of the lumped mass of each face.
struct CellCo {
  double kth[6], b[6], m, lump[6];
};

// What the pressure operator needs of each cell, face-major [f][ncell] (level 0: written by
// condense_kernel). Pointers may lie in different buffers.
struct CellOut {
  double *b[2], *lump[2];   // faces 0-2 and 3-5
  double *kth, *m;
};

__device__ __forceinline__ void store_cell(const CellOut &q, const CellCo &o, int64_t C, int64_t K) {
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    q.b[f / 3][(f % 3) * C + K] = o.b[f];
    q.lump[f / 3][(f % 3) * C + K] = o.lump[f];
    q.kth[f * C + K] = o.kth[f];
  }
  q.m[K] = o.m;
}

// gauss_cells.cu: the record buffer of the largest level (the caller frees it after a synchronisation),
// then per level the cell data by 27-point sums in every cell, and A_K^-1 where Ainv is not null
// (c->asm_flag set when a cell is singular)
int gauss_setup(Ctx *c, int64_t ncell, double **rec);
int gauss_cells(Ctx *c, const CellArgs &a, const CellOut &q, double *rec, double *Ainv);

}  // namespace hmg
