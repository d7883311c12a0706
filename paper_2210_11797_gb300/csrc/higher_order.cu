// The hybridised system of degree p = 1, 2, 3 (broken RT_p velocity, DG_p pressure, Q_p trace
// multipliers: (p+1)^2 per facet) for the constant-coefficient Helmholtz form of the operator,
// and its non-nested two-level preconditioner with the piecewise-constant coarse space.
//
// Paper (arXiv 2210.11797): Sec. 2.2 (spaces of degree p, n = p + 3 Gauss points per
// direction), Sec. 2.4 (Eqs. hybrid-S, hybrid-rhs, hybrid-recovery), Sec. 4.1 and the table
// of unknowns per cell (hybridised cell matrices of 24 x 24, 54 x 54 and 96 x 96, mixed cell
// matrices of 44 x 44, 135 x 135 and 304 x 304 at p = 1, 2, 3), Algorithm 1 (here on facet
// blocks and block-tridiagonal columns), Algorithm 2 with the DG0 coarse space of Sec. 2.5
// (P lambda = {{Pi}}, Restrict = P^T, Eq. scaling_matrix) and the lowest-order pressure
// multigrid as its coarse solve.
//
// Numbering (NT = p + 1, NB = NT^2 nodes per facet, NF = 6 NB facet dofs per cell). Cell dofs:
// the RT_p dofs (NF facet dofs, face f = e0..e3, bottom, top, node (s, t) at NB f + NT s + t,
// each the cell's outward normal flux at a Gauss-Legendre node of the facet; then the
// 3 p NT^2 interior dofs, component-major), then the NT^3 DG_p dofs. Trace rows: NB per facet,
// facet-major: vertical facet (edge e, level k) at NB (e L + k), horizontal facet (column c,
// interface k) at NH + NB (c (L + 1) + k), node (s, t) at + NT s + t; on a vertical facet s
// counts along the edge in the traversal of its owner column (the other column's local s is
// p - s).
#include <type_traits>

#include "device_common.cuh"
#include "hmg_internal.cuh"
#include "ho_common.cuh"
#include "precond.cuh"

namespace hmg {

// The row kernels take whole facets per block (p = 2: 28 facets of nine rows) and kHoR rows of one facet
// per thread: the lanes of a warp read consecutive coefficients of a slot, and the rows of a facet share
// its x values. One thread per facet with NB accumulators leaves most of the GPU idle on small meshes (16 x
// 16 x 16 cells at p = 3: 49 blocks on 152 SMs, S apply 266 us); on large ones FP32 takes it (below).
constexpr int kHoRowThreads = 256;
template <int P>
constexpr int kHoFacets = kHoRowThreads / Ho<P>::NB;   // facets per block
template <int P>
constexpr int kHoRows = kHoFacets<P> * Ho<P>::NB;      // rows per block
// rows per thread (consecutive rows of one facet, which share its x values) and threads per block
template <int P, typename T>
constexpr int kHoR = P == 2 ? (sizeof(T) == 4 ? 3 : 1) : 16 / (int)sizeof(T);
template <int P, typename T>
constexpr int kHoThreads = (kHoRows<P> / kHoR<P, T> + 31) / 32 * 32;

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int NLEFT>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(NLEFT) : "memory");
}
template <int BYTES>   // 4, 8 or 16, both addresses aligned to it
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem),
               "n"(BYTES)
               : "memory");
}

// acc (+/-)= sum over the stored slots of row NB F + n times x, in slot order: cell A's NF facet dofs,
// then cell B's without the shared facet (merged into A's slots when S was assembled). OFFD leaves out
// the couplings inside the smoother's diagonal block D of Algorithm 1 (acc - (S - D) x): on a
// vertical facet its own nodes, on a horizontal facet the horizontal facets of its column (A's
// bottom and top, B's bottom).
// A thread takes R consecutive rows of the facet. A facet's coefficients come through shared memory by
// cp.async, one facet ahead of the products, into this thread's part of buf ([NB][threads][R]; no barrier, a
// thread reads what it copied): a slot is refilled as soon as it is read. In FP32 x is an internal work
// vector (256-byte aligned), read NT values at a time. With plain loads the compiler keeps few of them in flight, and a mesh of one wave
// pays their latency for each facet. p = 3, 16 x 16 x 16 cells: FP32 sweep rows 46-54 us with plain loads and
// a row per thread, 30 now (118 MB), FP32 residual 33 and 28, FP64 S apply 83 and 79 (FP64 issue alone: 64).
// R is one 16-byte copy; at p = 2 (nine rows) FP64 takes 1 (S apply on 56 x 56 x 32 cells 470 us, 545 at 3).
template <int R, typename T>
__device__ __forceinline__ void ho_copy(T *smem, const T *gmem) {   // R values, 16 bytes at once where they are
  if constexpr (R * sizeof(T) == 16) cp_async<16>(smem, gmem);
  else
#pragma unroll
    for (int r = 0; r < R; ++r) cp_async<sizeof(T)>(smem + r, gmem + r);
}
template <int R, typename T>
__device__ __forceinline__ void ho_take(T (&v)[R], const T *smem) {
  if constexpr (R * sizeof(T) == 16) {
    const int4 u = *reinterpret_cast<const int4 *>(smem);
    memcpy(v, &u, 16);
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = smem[r];
  }
}
template <int P, bool NEG, bool OFFD, typename TS>
__device__ __forceinline__ void ho_row(const TS *__restrict__ S, const TS *__restrict__ x, const HoGeo &g, int64_t T,
                                       int64_t F, int n, TS (&acc)[kHoR<P, TS>], TS *buf) {
  using H = Ho<P>;
  constexpr int NB = H::NB, NT = H::NT, R = kHoR<P, TS>, STEP = kHoThreads<P, TS> * R;
  const HoFacet fc = ho_facet(g, F);
  const bool vert = F < g.nhf;
  const TS *s0 = S + (int64_t)NB * F + n;
  auto next = [&](int j) {   // the first facet from slot group j on that the row takes, or 12
    for (; j < 12; ++j) {
      const int f = j < 6 ? j : j - 6;
      if (OFFD && !vert && f >= 4) continue;
      if (j < 6 ? !(OFFD && vert && f == fc.fA) : fc.cB >= 0 && f != fc.fB) break;
    }
    return j;
  };
  int nj = next(0);   // (every row takes a facet of its first cell)
#pragma unroll
  for (int q = 0; q < NB; ++q) ho_copy<R>(buf + q * STEP, s0 + ((int64_t)nj * NB + q) * T);
#pragma unroll 1
  for (int j = 0; j < 12; ++j) {
    if (j != nj) continue;
    const int f = j < 6 ? j : j - 6;
    const int64_t c = j < 6 ? fc.cA : fc.cB;
    const int k = j < 6 ? fc.kA : fc.kB;
    const TS *xf;         // the facet's first value in the cell's traversal, step per s
    int ds = NT;
    if (f < 4) {
      const int64_t e = __ldg(g.col_edges + 4 * c + f);
      xf = x + NB * (e * g.L + k);
      if (!__ldg(g.own + 4 * c + f)) {
        xf += NT * P;
        ds = -NT;
      }
    } else {
      xf = x + g.NH + NB * (c * (g.L + 1) + k + (f == 5 ? 1 : 0));
    }
    TS v[NB];
#pragma unroll
    for (int q = 0; q < NT; ++q) {
      const TS *xq = xf + q * ds;
      if constexpr (NT == 4 && sizeof(TS) == 4) {
        const float4 u = __ldg(reinterpret_cast<const float4 *>(xq));
        v[4 * q] = u.x; v[4 * q + 1] = u.y; v[4 * q + 2] = u.z; v[4 * q + 3] = u.w;
      } else if constexpr (NT == 2 && sizeof(TS) == 4) {
        const float2 u = __ldg(reinterpret_cast<const float2 *>(xq));
        v[2 * q] = u.x; v[2 * q + 1] = u.y;
      } else {
#pragma unroll
        for (int t = 0; t < NT; ++t) v[q * NT + t] = __ldg(xq + t);
      }
    }
    cp_async_commit();
    cp_async_wait<0>();
    nj = next(j + 1);
    const TS *s = s0 + (int64_t)nj * NB * T;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      TS a[R];
      ho_take<R>(a, buf + q * STEP);
      if (nj < 12) ho_copy<R>(buf + q * STEP, s + (int64_t)q * T);
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fma(NEG ? -a[r] : a[r], v[q], acc[r]);
    }
  }
}

// The same products, negative, for all NB rows of a facet by one thread, in FP32: a slot's coefficients in
// 16-byte loads where NB allows, and each x value read once for NB products. It needs a facet for every
// thread of the chip: kHoFacetRows.
template <int P, bool OFFD>
__device__ __forceinline__ void ho_facet_rows(const float *__restrict__ S, const float *__restrict__ x, const HoGeo &g,
                                              int64_t T, int64_t F, float (&acc)[Ho<P>::NB]) {
  using H = Ho<P>;
  constexpr int NB = H::NB, U = P == 1 ? 4 : 2;
  const HoFacet fc = ho_facet(g, F);
  const bool vert = F < g.nhf;
  const float *Sr = S + (int64_t)NB * F;
  auto cell = [&](int c, int k, int skip) {
#pragma unroll U
    for (int q = 0; q < H::NF; ++q) {
      if (q / NB == skip || (OFFD && !vert && q / NB >= 4)) continue;
      const float xv = __ldg(x + ho_gid<P>(g, c, k, q));
      const float *s = Sr + (int64_t)q * T;
      if constexpr (NB % 4 == 0) {
#pragma unroll
        for (int n = 0; n < NB; n += 4) {
          const float4 v = __ldcs(reinterpret_cast<const float4 *>(s + n));
          acc[n] = fmaf(-v.x, xv, acc[n]);
          acc[n + 1] = fmaf(-v.y, xv, acc[n + 1]);
          acc[n + 2] = fmaf(-v.z, xv, acc[n + 2]);
          acc[n + 3] = fmaf(-v.w, xv, acc[n + 3]);
        }
      } else {
#pragma unroll
        for (int n = 0; n < NB; ++n) acc[n] = fmaf(-__ldcs(s + n), xv, acc[n]);
      }
    }
  };
  cell(fc.cA, fc.kA, OFFD && vert ? fc.fA : -1);
  Sr += (int64_t)H::NF * T;
  if (fc.cB >= 0) cell(fc.cB, fc.kB, fc.fB);
}
// FP32 rows from which a facet per thread is the faster form: where the facet form's latency (2 NF times NB
// products of one thread) meets the other's time per row. Measured as sweeps (us each with their line
// solves, by rows / by facets) and residuals: p = 1 sweeps 42 / 46 at 0.61 M rows, 51 / 49 at 0.80 M, 271 / 239
// at 6.4 M, its residual always by rows (34 / 43 at 0.80 M, 173 / 186 at 6.4 M); p = 2 two sweeps and a
// residual 284 / 290 at 0.71 M, 322 / 310 at 0.85 M; p = 3 773 / 778 at 1.89 M, 969 / 824 at 2.48 M. Both
// forms add a row's products in the same order.
template <int P>
constexpr int64_t kHoFacetRows = P == 1 ? 700'000 : (P == 2 ? 780'000 : 1'950'000);

// ---- assembly -------------------------------------------------------------------------------
// own[c][f] = 1 where column c owns the edge of its face f (each entry written by one edge)
__global__ void ho_own_kernel(const int32_t *__restrict__ stencil, const int32_t *__restrict__ edge_fc, int nedge,
                              int8_t *__restrict__ own) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nedge) return;
  own[4 * (int64_t)stencil[8 * (int64_t)e] + edge_fc[2 * (int64_t)e]] = 1;
  own[4 * (int64_t)stencil[8 * (int64_t)e + 1] + edge_fc[2 * (int64_t)e + 1]] = 0;
}

// Rows of S = sum_K C_K^T A_K^-1 C_K (C_K diagonal on the facet dofs: w_s w_t of the node): row
// NB F + n holds, in slots 0 .. NF - 1, C A_A^-1 C restricted to the facet dofs of cell A (row:
// the node's local index in A), and in slots NF .. 2 NF - 1 the same of cell B, whose
// shared-facet entries are added into A's slots (and stored as 0).
template <int P>
__global__ void ho_rows_kernel(const HoGeo g, int64_t T, const double *__restrict__ Cw,
                               const double *__restrict__ Ainv, double *__restrict__ S) {
  using H = Ho<P>;
  constexpr int N = H::N;
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row >= T) return;
  const int64_t F = row / H::NB;
  const int n = (int)(row - F * H::NB), s = n / H::NT, t = n - s * H::NT;
  const HoFacet fc = ho_facet(g, F);
  const int qa = H::NB * fc.fA + n;
  const double *IA = Ainv + ((int64_t)fc.cA * g.L + fc.kA) * (int64_t)(N * N) + (int64_t)qa * N;
  for (int q = 0; q < H::NF; ++q) S[(int64_t)q * T + row] = Cw[n] * Cw[q % H::NB] * IA[q];
  if (fc.cB >= 0) {
    const int sb = fc.flipB ? P - s : s;
    const int nb = H::NT * sb + t;
    const int qb = H::NB * fc.fB + nb;
    const double *IB = Ainv + ((int64_t)fc.cB * g.L + fc.kB) * (int64_t)(N * N) + (int64_t)qb * N;
    for (int q = 0; q < H::NF; ++q) {
      const double w = Cw[nb] * Cw[q % H::NB] * IB[q];
      if (q / H::NB == fc.fB) {   // the shared facet: the same trace row as A's node
        const int r = q % H::NB, sq = r / H::NT, tq = r - sq * H::NT;
        const int sa = fc.flipB ? P - sq : sq;
        S[(int64_t)(H::NB * fc.fA + H::NT * sa + tq) * T + row] += w;
        S[(int64_t)(H::NF + q) * T + row] = 0.0;
      } else {
        S[(int64_t)(H::NF + q) * T + row] = w;
      }
    }
  } else {
    for (int q = 0; q < H::NF; ++q) S[(int64_t)(H::NF + q) * T + row] = 0.0;
  }
}

// Gauss-Jordan elimination with partial pivoting by one warp: W [NB][2 NB] (shared memory) holds
// [A | I] on entry and [I | A^-1] on return; lane j < 2 NB owns column j. Every lane finds the
// same pivot (they read the same values), so the branches are uniform. False if A is singular.
template <int NB>
__device__ bool warp_gauss_jordan(double *W, int lane) {
  constexpr int W2 = 2 * NB;
  static_assert(W2 <= 32, "one lane per column");
  for (int c = 0; c < NB; ++c) {
    int p = c;
    double best = fabs(W[c * W2 + c]);
    for (int r = c + 1; r < NB; ++r) {
      const double v = fabs(W[r * W2 + c]);
      if (v > best) { best = v; p = r; }
    }
    if (!(best > 0.0)) return false;
    if (p != c && lane < W2) {
      const double t = W[c * W2 + lane];
      W[c * W2 + lane] = W[p * W2 + lane];
      W[p * W2 + lane] = t;
    }
    __syncwarp();
    const double inv = 1.0 / W[c * W2 + c];
    double fr[NB];   // column c, read before its owner lane changes it
#pragma unroll
    for (int r = 0; r < NB; ++r) fr[r] = W[r * W2 + c];
    __syncwarp();
    if (lane < W2) {
      const double pv = W[c * W2 + lane] * inv;
      W[c * W2 + lane] = pv;
#pragma unroll
      for (int r = 0; r < NB; ++r)
        if (r != c) W[r * W2 + lane] = fma(-fr[r], pv, W[r * W2 + lane]);
    }
    __syncwarp();
  }
  return true;
}

constexpr int kHoFacWarps = 4;   // warps per block of the factor kernels

// omega times the inverse of each vertical facet's NB x NB block of S (the Jacobi part of
// Algorithm 1), entry (n, m) at hw[NB^2 F + NB m + n] (the rows of a facet, one lane each, read one run
// per m); one warp per facet. The facet block lives in the slots of cell A's face (A owns the edge, so
// its local nodes are the facet's).
template <int P>
__global__ void __launch_bounds__(32 * kHoFacWarps)
    ho_hfactor_kernel(const HoGeo g, int64_t T, const double *__restrict__ S, double omega,
                      double *__restrict__ hw, int *singular) {
  constexpr int NB = Ho<P>::NB, W2 = 2 * NB;
  __shared__ double Wsh[kHoFacWarps][NB * W2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t F = (int64_t)blockIdx.x * kHoFacWarps + warp;
  if (F >= g.nhf) return;   // whole warps leave
  double *W = Wsh[warp];
  const HoFacet fc = ho_facet(g, F);
  for (int e = lane; e < NB * NB; e += 32) {
    const int n = e / NB, m = e - n * NB;
    W[n * W2 + m] = S[(int64_t)(NB * fc.fA + m) * T + NB * F + n];
    W[n * W2 + NB + m] = n == m ? 1.0 : 0.0;
  }
  __syncwarp();
  if (!warp_gauss_jordan<NB>(W, lane) && lane == 0) atomicExch(singular, 1);
  for (int e = lane; e < NB * NB; e += 32) {
    const int n = e / NB, m = e - n * NB;
    hw[(int64_t)NB * NB * F + NB * m + n] = omega * W[n * W2 + NB + m];
  }
}

// Block Thomas factors of each column's block-tridiagonal S^zz (blocks D_k, L_k = coupling of
// facet k to k - 1, U_k to k + 1): G_0 = D_0, G_k = D_k - L_k G_{k-1}^-1 U_{k-1}; stored per
// horizontal facet: omega G_k^-1, G_k^-1 L_k, G_k^-1 U_k ([nzf][3][NB][NB], each transposed: entry
// (n, m) at m NB + n, so that the NB lanes of a column read one contiguous run per m), so that
// omega (S^zz)^-1 r is y_k = (omega G_k^-1) r_k - (G_k^-1 L_k) y_{k-1}, x_k = y_k - (G_k^-1 U_k) x_{k+1}.
// Slots: the cell above (c, k) is A for k < L: its bottom (face 4) is this facet, its top (face 5)
// facet k + 1; the cell below (c, k - 1) is B, its bottom facet k - 1. The lid row's A is the
// cell below: its top is this facet, its bottom the facet below. One warp per column.
template <int P>
__global__ void __launch_bounds__(32 * kHoFacWarps)
    ho_zfactor_kernel(const HoGeo g, int64_t T, const double *__restrict__ S, double omega,
                      double *__restrict__ zf, int *singular) {
  using H = Ho<P>;
  constexpr int NB = H::NB, NB2 = NB * NB, W2 = 2 * NB;
  extern __shared__ double zsh[];   // per warp: GU, Lk, U [NB2] and W [NB][2 NB]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x * kHoFacWarps + warp;
  if (c >= g.ncol) return;   // whole warps leave
  double *GU = zsh + warp * (3 * NB2 + NB * W2), *Lk = GU + NB2, *U = Lk + NB2, *W = U + NB2;
  const int L = g.L;
  bool ok = true;
  for (int k = 0; k <= L; ++k) {
    const int64_t F = (int64_t)c * (L + 1) + k, row0 = g.NH + NB * F;
    for (int e = lane; e < NB2; e += 32) {
      const int n = e / NB, m = e - n * NB;
      const double *r = S + row0 + n;
      if (k < L) {
        W[n * W2 + m] = r[(int64_t)(4 * NB + m) * T];
        U[e] = r[(int64_t)(5 * NB + m) * T];
        Lk[e] = k > 0 ? r[(int64_t)(H::NF + 4 * NB + m) * T] : 0.0;
      } else {
        W[n * W2 + m] = r[(int64_t)(5 * NB + m) * T];
        Lk[e] = r[(int64_t)(4 * NB + m) * T];
        U[e] = 0.0;
      }
      W[n * W2 + NB + m] = n == m ? 1.0 : 0.0;
    }
    __syncwarp();
    if (k > 0) {
      for (int e = lane; e < NB2; e += 32) {   // G_k = D_k - L_k (G_{k-1}^-1 U_{k-1})
        const int n = e / NB, m = e - n * NB;
        double s = W[n * W2 + m];
        for (int j = 0; j < NB; ++j) s = fma(-Lk[n * NB + j], GU[j * NB + m], s);
        W[n * W2 + m] = s;
      }
      __syncwarp();
    }
    if (!warp_gauss_jordan<NB>(W, lane)) ok = false;
    double *o = zf + 3 * NB2 * F;   // facet-major: 3 NB^2 contiguous factors, each matrix transposed
    for (int e = lane; e < NB2; e += 32) {
      const int n = e / NB, m = e - n * NB;
      double sl = 0.0, su = 0.0;
      for (int j = 0; j < NB; ++j) {
        sl = fma(W[n * W2 + NB + j], Lk[j * NB + m], sl);
        su = fma(W[n * W2 + NB + j], U[j * NB + m], su);
      }
      o[m * NB + n] = omega * W[n * W2 + NB + m];
      o[NB2 + m * NB + n] = sl;
      o[2 * NB2 + m * NB + n] = su;
      GU[e] = su;   // (row-major, for the next level's G; nothing reads GU in this loop)
    }
    __syncwarp();
  }
  if (!ok && lane == 0) atomicExch(singular, 1);
}

// ---- the operator, the right-hand side and the recovery --------------------------------------
// y = S x, kHoR rows per thread; MODE 1, 2, 3 fuse the inner products of the Krylov loop as the
// lowest-order S apply does (3: (b - S x, b - S x), no y): a facet's products are summed in row order by
// one thread into fs[F] (and fs[nF + F]), which ho_reduce_kernel adds up.
template <int P, int MODE>
__global__ void __launch_bounds__(kHoThreads<P, double>)
    ho_spmv_kernel(const HoGeo g, int64_t T, const double *__restrict__ S, const double *__restrict__ x,
                   double *__restrict__ y, const double *__restrict__ w, double *__restrict__ fs) {
  constexpr int NB = Ho<P>::NB, FB = kHoFacets<P>, R = kHoR<P, double>;
  __shared__ __align__(16) double ss[NB * kHoThreads<P, double> * R];
  __shared__ double sv[MODE ? kHoRows<P> : 1], sw[MODE == 1 || MODE == 2 ? kHoRows<P> : 1];
  const int i = threadIdx.x, i0 = i * R;
  const int64_t row = (int64_t)blockIdx.x * kHoRows<P> + i0, F = (int64_t)blockIdx.x * FB + i0 / NB;
  if (i0 < kHoRows<P> && row < T) {
    double v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = MODE == 3 ? __ldg(w + row + r) : 0.0;
    ho_row<P, MODE == 3, false>(S, x, g, T, F, i0 % NB, v, ss + i0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (MODE != 3) y[row + r] = v[r];
      if (MODE) sv[i0 + r] = v[r];
      if (MODE == 1 || MODE == 2) sw[i0 + r] = __ldg(w + row + r);
    }
  }
  if (MODE) {
    __syncthreads();
    const int64_t f = (int64_t)blockIdx.x * FB + i, nF = g.nhf + g.nzf;
    if (i < FB && f < nF) {
      double a0 = 0.0, a1 = 0.0;
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        const double v = sv[i * NB + n];
        if (MODE == 1) a0 = fma(sw[i * NB + n], v, a0);
        if (MODE == 2) a0 = fma(v, sw[i * NB + n], a0);
        if (MODE == 2) a1 = fma(v, v, a1);
        if (MODE == 3) a0 = fma(v, v, a0);
      }
      fs[f] = a0;
      if (MODE == 2) fs[nF + f] = a1;
    }
  }
}

// The sums of the facets' partial products: a warp adds 256 facets (eight per lane, then a shuffle
// tree) into part[slot][group]; the last block adds the groups into scal. Fixed order, and the order of
// block_sum and finalize_kernel over blocks of 256 facets.
template <int NV>
__global__ void __launch_bounds__(256)
    ho_reduce_kernel(const double *__restrict__ fs, int64_t nF, int slot0, int slot1, double *part,
                     unsigned int *counter, double *scal) {
  __shared__ double sh[NV][32];
  __shared__ bool is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ng = (int)((nF + 255) / 256), grp = blockIdx.x * 8 + warp;
  if (grp < ng) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      double f[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int64_t F = (int64_t)grp * 256 + lane + 32 * j;
        f[j] = F < nF ? fs[q * nF + F] : 0.0;
      }
      double v = f[0];
#pragma unroll
      for (int j = 1; j < 8; ++j) v += f[j];
      v = warp_sum(v);
      if (lane == 0) part[(int64_t)(q ? slot1 : slot0) * kMaxRedBlocks + grp] = v;
    }
  }
  __threadfence();   // every warp's partials before the block's ticket
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(&counter[slot0], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int slot = q ? slot1 : slot0;
    const double s = sum_partials<256>(part + (int64_t)slot * kMaxRedBlocks, ng, sh[q]);
    if (threadIdx.x == 0) scal[slot] = s;
  }
  if (threadIdx.x == 0) counter[slot0] = 0u;
}

template <int P>
static HoGeo ho_geo(const Ctx *c) {
  const Level &f = c->lv[0];
  HoGeo g;
  g.L = f.nlev;
  g.ncol = f.ncol;
  g.nhf = (int64_t)f.nedge * f.nlev;
  g.nzf = (int64_t)f.ncol * (f.nlev + 1);
  g.NH = (int64_t)Ho<P>::NB * g.nhf;
  g.col_edges = f.col_edges;
  g.stencil = f.edge_stencil;
  g.edge_fc = f.edge_fc;
  g.own = c->ho.own;
  return g;
}

// ---- products with A_K^-1 ----------------------------------------------------------------------
// One thread per row of A_K^-1, each row's dot product in column order; the rows of all cells in one
// index space, so that no lane idles (p = 1: 44 rows per cell, 24 for the right-hand side). A warp stages
// its 32 rows 16 columns at a time through shared memory (cp.async, two tiles in flight): one thread per
// row straight from global memory touched 32 lines per load (p = 3, 4,096 cells: recovery 1,402 us, 0.3
// of HBM bandwidth; now bound by the FP64 rate of its 378 M FMAs).
constexpr int kHoTile = 16, kHoDotThreads = 256;

// The rows of cell K that a product takes (all N, or the NF facet dofs) and its shared memory: the
// block's cells' vectors, then per warp the row addresses and two tiles.
template <int P, bool REC>
struct HoDot {
  using H = Ho<P>;
  static constexpr int ROWS = REC ? H::N : H::NF, CELLS = (kHoDotThreads - 1) / ROWS + 2, LD = kHoTile + 1;
  static constexpr int WARP = 32 + 2 * 32 * LD;   // doubles per warp
  static constexpr int SMEM = (int)sizeof(double) * (CELLS * H::N + (kHoDotThreads / 32) * WARP);
};

// REC: X_K = A_K^-1 (R_K - C_K lambda_K) into o0 = u [ncell][NU], o1 = pi [ncell][NP]. Otherwise
// (A_K^-1 R_K)_q on the facet dofs q < NF, into o0 (q < NF / 2) and o1, NF / 2 per cell each.
template <int P, bool REC>
__global__ void __launch_bounds__(kHoDotThreads)
    ho_dot_kernel(const HoGeo g, int64_t ncell, const double *__restrict__ cw, const double *__restrict__ Ainv,
                  const double *__restrict__ lam, const double *__restrict__ Ru, const double *__restrict__ Rp,
                  double *__restrict__ o0, double *__restrict__ o1) {
  using H = Ho<P>;
  using D = HoDot<P, REC>;
  constexpr int N = H::N, LD = D::LD, NTILE = (N + kHoTile - 1) / kHoTile, HF = H::NF / 2;
  extern __shared__ __align__(16) double hd_smem[];
  const int lane = threadIdx.x & 31;
  const int64_t first = (int64_t)blockIdx.x * kHoDotThreads, total = ncell * D::ROWS, idx = first + threadIdx.x;
  const int64_t K0 = first / D::ROWS;
  double *r = hd_smem;
  double *wsm = r + D::CELLS * N + (threadIdx.x >> 5) * D::WARP, *tile = wsm + 32;
  const double **rows = reinterpret_cast<const double **>(wsm);
  for (int e = threadIdx.x; e < D::CELLS * N; e += kHoDotThreads) {
    const int64_t K = K0 + e / N;
    const int j = e % N;
    if (K >= ncell) break;
    double v = j < H::NU ? Ru[K * H::NU + j] : Rp[K * H::NP + (j - H::NU)];
    if (REC && j < H::NF) {
      const int c = (int)((unsigned)K / (unsigned)g.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)g.L);
      v = fma(-cw[j % H::NB], lam[ho_gid<P>(g, c, k, j)], v);
    }
    r[e] = v;
  }
  const int64_t K = idx / D::ROWS;
  const int q = (int)(idx - K * D::ROWS);
  rows[lane] = idx < total ? Ainv + K * (int64_t)(N * N) + (int64_t)q * N : nullptr;
  __syncthreads();
  static_assert(kHoTile == 16, "two rows per warp load");
  auto stage = [&](int j) {
    double *t = tile + (j & 1) * 32 * LD;
    const int sub = lane & (kHoTile - 1), col = j * kHoTile + sub;
#pragma unroll
    for (int s = 0; s < 32; s += 2) {
      const int rr = s + (lane >> 4);
      const double *row = rows[rr];
      if (row && col < N) cp_async<8>(t + rr * LD + sub, row + col);
    }
    cp_async_commit();
  };
  stage(0);
  double v = 0.0;
  const double *rk = r + (int)(K - K0) * N;
  for (int j = 0; j < NTILE; ++j) {
    if (j + 1 < NTILE) {
      stage(j + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const double *t = tile + (j & 1) * 32 * LD + lane * LD, *rj = rk + j * kHoTile;
    const int m = N - j * kHoTile < kHoTile ? N - j * kHoTile : kHoTile;
    if (idx < total) {
      if (m == kHoTile) {
#pragma unroll
        for (int s = 0; s < kHoTile; ++s) v = fma(t[s], rj[s], v);
      } else {
        for (int s = 0; s < m; ++s) v = fma(t[s], rj[s], v);
      }
    }
    __syncwarp();   // the tile is staged again two steps on
  }
  if (idx >= total) return;
  if (REC) {
    if (q < H::NU) o0[K * H::NU + q] = v;
    else o1[K * H::NP + (q - H::NU)] = v;
  } else {
    if (q < HF) o0[K * HF + q] = v;
    else o1[K * HF + q - HF] = v;
  }
}

// The recovery at p = 1 on small meshes: a thread per row that reads its row of A_K^-1 itself. Its short
// rows (44 columns) cost less there than the staging, whose shared memory leaves three blocks per SM: 28 x
// 28 x 16 cells 86 us (staged 91), 40 x 40 x 16 149 (152), 64 x 64 x 16 344 (332).
constexpr int64_t kHoDirectCells = 40'000;
template <int P>
__global__ void ho_recover_direct_kernel(const HoGeo g, int64_t ncell, const double *__restrict__ cw,
                                         const double *__restrict__ Ainv, const double *__restrict__ lam,
                                         const double *__restrict__ Ru, const double *__restrict__ Rp,
                                         double *__restrict__ u, double *__restrict__ pi) {
  using H = Ho<P>;
  constexpr int N = H::N;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= ncell * N) return;
  const int64_t K = idx / N;
  const int i = (int)(idx - K * N);
  const int c = (int)((unsigned)K / (unsigned)g.L), k = (int)((unsigned)K - (unsigned)c * (unsigned)g.L);
  const double *I = Ainv + K * (int64_t)(N * N) + (int64_t)i * N;
  double v = 0.0;
  for (int j = 0; j < H::NU; ++j) {
    double r = Ru[K * H::NU + j];
    if (j < H::NF) r = fma(-cw[j % H::NB], lam[ho_gid<P>(g, c, k, j)], r);
    v = fma(I[j], r, v);
  }
  for (int j = 0; j < H::NP; ++j) v = fma(I[H::NU + j], Rp[K * H::NP + j], v);
  if (i < H::NU) u[K * H::NU + i] = v;
  else pi[K * H::NP + (i - H::NU)] = v;
}

template <int P, bool REC>
static int ho_launch_dot(Ctx *c, const double *lam, const double *Ru, const double *Rp, double *o0, double *o1) {
  using D = HoDot<P, REC>;
  const int64_t C = c->lv[0].ncell;
  HMG_CUDA(c, cudaFuncSetAttribute(ho_dot_kernel<P, REC>, cudaFuncAttributeMaxDynamicSharedMemorySize, D::SMEM));
  ho_dot_kernel<P, REC><<<grid_for(C * D::ROWS, kHoDotThreads), kHoDotThreads, D::SMEM, c->stream>>>(
      ho_geo<P>(c), C, c->ho.cw, c->ho.Ainv, lam, Ru, Rp, o0, o1);
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

// B_lambda row NB F + n: the sum over the facet's cells of C_K (A_K^-1 R_K) at the node's local dof, from the
// products of ho_dot_kernel, or (p = 1) by a thread per row that reads its rows of A_K^-1 itself: with 44
// columns the second launch and the products' way through memory cost more than the staging saves (24 x 24
// x 10 cells 31 us, 41 staged; 128 x 128 x 32 1.25 and 1.32 ms; p = 2 and 3 gain from 16 x 16 x 16 on, 96
// and 92 us, 465 and 274).
template <int P>
__global__ void ho_rhs_direct_kernel(const HoGeo g, int64_t T, const double *__restrict__ cw,
                                     const double *__restrict__ Ainv, const double *__restrict__ Ru,
                                     const double *__restrict__ Rp, double *__restrict__ B) {
  using H = Ho<P>;
  constexpr int N = H::N;
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row >= T) return;
  const int64_t F = row / H::NB;
  const int n = (int)(row - F * H::NB), s = n / H::NT, t = n - s * H::NT;
  const HoFacet fc = ho_facet(g, F);
  auto cell = [&](int cc, int kk, int q) {
    const int64_t K = (int64_t)cc * g.L + kk;
    const double *I = Ainv + K * (int64_t)(N * N) + (int64_t)q * N;
    double v = 0.0;
    for (int j = 0; j < H::NU; ++j) v = fma(I[j], Ru[K * H::NU + j], v);
    for (int j = 0; j < H::NP; ++j) v = fma(I[H::NU + j], Rp[K * H::NP + j], v);
    return v;
  };
  double v = cell(fc.cA, fc.kA, H::NB * fc.fA + n);
  if (fc.cB >= 0) v += cell(fc.cB, fc.kB, H::NB * fc.fB + H::NT * (fc.flipB ? P - s : s) + t);
  B[row] = cw[n] * v;
}

template <int P>
__global__ void ho_rhs_kernel(const HoGeo g, int64_t T, const double *__restrict__ cw, const double *__restrict__ d0,
                              const double *__restrict__ d1, double *__restrict__ B) {
  using H = Ho<P>;
  constexpr int HF = H::NF / 2;
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row >= T) return;
  const int64_t F = row / H::NB;
  const int n = (int)(row - F * H::NB), s = n / H::NT, t = n - s * H::NT;
  const HoFacet fc = ho_facet(g, F);
  auto cell = [&](int cc, int kk, int q) {
    const int64_t K = (int64_t)cc * g.L + kk;
    return q < HF ? d0[K * HF + q] : d1[K * HF + q - HF];
  };
  double v = cell(fc.cA, fc.kA, H::NB * fc.fA + n);
  if (fc.cB >= 0) v += cell(fc.cB, fc.kB, H::NB * fc.fB + H::NT * (fc.flipB ? P - s : s) + t);
  B[row] = cw[n] * v;
}

// ---- Algorithm 1 at p >= 1 ------------------------------------------------------------------------
// lam_out = lam_in + omega D^-1 (b - S lam_in) (ZERO: lam_in = 0), evaluated as
// (1 - omega) lam_in + omega D^-1 (b - (S - D) lam_in): equal in exact arithmetic, without the
// couplings of a row inside D. Two launches per sweep. Part 1, kHoR rows per thread as the S apply (in
// FP32 a facet from kHoFacetRows on): the residual rows r = b - (S - D) lam_in; on a vertical facet the NB x NB block Jacobi step
// lam_out = keep lam_in + (omega D_F^-1) r at once (the facet's r in shared memory), on a horizontal
// facet r is parked in lam_out's rows (ZERO: vertical facets only, r = b). Part 2, the line
// solves: each column's r staged in shared memory, the block Thomas recurrences with LPC lanes
// per column (lane n < NB computes component n of each NB x NB product from its rows of the
// stored factors; the lanes of a column sit in one warp and meet at __syncwarp between the
// steps), lam_out = keep lam_in + omega (S^zz_c)^-1 r. T is the arithmetic and coefficient
// type (double, or float in the FP32 preconditioner, whose b is the FP64 Krylov residual and
// whose last sweep writes FP64).
template <int P, bool ZERO, typename T = double, typename Tb = double, typename Tin = double, typename Tout = double>
__global__ void __launch_bounds__(ZERO ? kHoRowThreads : kHoThreads<P, T>)
    ho_sweep_rows_kernel(const HoGeo g, int64_t TT, const T *__restrict__ S, const T *__restrict__ hw,
                         const Tb *__restrict__ b, const Tin *__restrict__ lam_in,
                         Tout *__restrict__ lam_out, double keep) {
  constexpr int NB = Ho<P>::NB, R = ZERO ? 1 : kHoR<P, T>, STEP = kHoThreads<P, T> * kHoR<P, T>;
  constexpr bool AHEAD = !ZERO && sizeof(T) == 4;         // (FP64 is bound by its issue rate)
  __shared__ T sr[kHoRows<P>];
  __shared__ __align__(16) T sf[AHEAD ? NB * STEP : 1];   // the rows of omega D_F^-1, copied behind the products
  __shared__ __align__(16) T ss[ZERO ? 1 : NB * STEP];
  const int i0 = threadIdx.x * R, n = i0 % NB;
  const int64_t row = (int64_t)blockIdx.x * kHoRows<P> + i0, F = (int64_t)blockIdx.x * kHoFacets<P> + i0 / NB;
  const bool act = i0 < kHoRows<P> && row < (ZERO ? g.NH : TT);
  const T *f = hw + (int64_t)NB * NB * F + n;
  T v[R];
  if (act) {
    if (AHEAD && F < g.nhf) {
#pragma unroll
      for (int m = 0; m < NB; ++m) ho_copy<R>(sf + m * STEP + i0, f + NB * m);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = (T)__ldg(b + row + r);
    if constexpr (!ZERO) ho_row<P, true, true>(S, lam_in, g, TT, F, n, v, ss + i0);
#pragma unroll
    for (int r = 0; r < R; ++r) sr[i0 + r] = v[r];
  }
  __syncthreads();
  if (!act) return;
  if (F < g.nhf) {
    const T *rf = sr + (i0 - n);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ZERO ? (T)0 : (T)keep * (T)lam_in[row + r];
    if (AHEAD) {
      cp_async_commit();
      cp_async_wait<0>();
    }
#pragma unroll
    for (int m = 0; m < NB; ++m) {
      T a[R];
      if constexpr (AHEAD) ho_take<R>(a, sf + m * STEP + i0);
      else
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = __ldg(f + NB * m + r);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = fma(a[r], rf[m], v[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) lam_out[row + r] = (Tout)v[r];
}

// Part 2's ring of factor blocks: levels in flight and values per column of a slot (padded by NB, so that
// the columns of a warp meet different banks).
template <int P>
struct HoLines {
  static constexpr int DEPTH = P == 1 ? 8 : (P == 2 ? 6 : 4);
  static constexpr int NB2 = Ho<P>::NB * Ho<P>::NB, STRIDE = 2 * NB2 + Ho<P>::NB;
};

// v = p[0 .. NB - 1] in shared memory, in 16-byte reads where a block is a multiple of them
template <int NB, typename T>
__device__ __forceinline__ void ho_block(T (&v)[NB], const T *p) {
  constexpr int W = 16 / (int)sizeof(T);
  if constexpr (NB % W == 0) {
#pragma unroll
    for (int q = 0; q < NB; q += W) {
      const int4 u = *reinterpret_cast<const int4 *>(p + q);
      memcpy(v + q, &u, 16);
    }
  } else {
#pragma unroll
    for (int q = 0; q < NB; ++q) v[q] = p[q];
  }
}

// One warp of recurrences per block of CPW columns, and a second one that feeds it. The recurrences are
// serial over the levels (2 L + 1 steps of NB-term dot products), so a step must not wait for its factors:
// they stream through shared memory by cp.async, DEPTH - 1 steps ahead, and the copies' instructions are
// the other warp's. Loaded one step ahead into registers, four warps per block, the kernel took 1.1 us per
// step, one memory latency (37 us per sweep at p = 1 on 64 x 64 x 16 cells, 40 us at p = 3 in FP32 on
// 16 x 16 x 16); with the copies issued by the same warp 22 and 19 us;
// now 20 and 16.5 (at p = 1 the FP64 pipe's twelve FMAs per step and warp, 3.4 warps per SM, are half of it).
// Part 2; r is read from src (lam_out after part 1, b for a sweep from zero)
template <int P, bool ZERO, typename T = double, typename Ts = double, typename Tin = double, typename Tout = double>
__global__ void __launch_bounds__(64)
    ho_sweep_lines_kernel(const HoGeo g, int cpb, const T *__restrict__ zf, const Ts *src,
                          const Tin *__restrict__ lam_in, Tout *lam_out, double keep) {
  using H = Ho<P>;
  using W = HoLines<P>;
  constexpr int NB = H::NB, NB2 = NB * NB, LPC = H::LPC, D = W::DEPTH, CS = W::STRIDE;
  // the widest copy that every matrix of every facet is aligned to
  constexpr int VB = (NB2 * sizeof(T)) % 16 == 0 ? 16 : (int)sizeof(T), VN = VB / (int)sizeof(T);
  extern __shared__ __align__(16) unsigned char ho_lines_smem[];
  T *ring = reinterpret_cast<T *>(ho_lines_smem);   // [D][CPW][CS]
  T *sr = ring + D * H::CPW * CS;                   // [cpb][L+1][NB]
  const int L1 = g.L + 1, lane = threadIdx.x & 31;
  const bool feeds = threadIdx.x >= 32;
  const int c0 = blockIdx.x * cpb, nc = min(cpb, g.ncol - c0);
  const int64_t base = g.NH + (int64_t)NB * c0 * L1;
  // step s of the two passes: the forward step of level s, then the backward step of level 2 L1 - 2 - s
  const int steps = 2 * L1 - 1;
  auto stage = [&](int s) {
    if (s < steps) {
      T *slot = ring + (s % D) * (H::CPW * CS);
      const bool fwd = s < L1;
      const T *f = zf + 3 * NB2 * ((int64_t)c0 * L1 + (fwd ? s : 2 * L1 - 2 - s)) + (fwd ? 0 : 2 * NB2);
      const int per = (fwd ? 2 * NB2 : NB2) / VN;
      for (int cc = 0; cc < nc; ++cc, f += 3 * NB2 * (int64_t)L1)
        for (int e = lane; e < per; e += 32) cp_async<VB>(slot + cc * CS + e * VN, f + e * VN);
    }
    cp_async_commit();
  };
  if (feeds)
#pragma unroll
    for (int s = 0; s < D; ++s) stage(s);
  for (int i = threadIdx.x; i < nc * L1 * NB; i += 64) sr[i] = (T)src[base + i];
  const int cc = lane / LPC, n = lane - cc * LPC;
  const bool act = cc < nc && n < NB;
  T *r = sr + NB * (act ? cc : 0) * L1;
  // a step's factors and what does not depend on the step before it are taken one step ahead:
  // forward v = (omega G_k^-1) r_k, backward v = y_k
  T f[NB], v = (T)0;
  auto load = [&](int s) {
    const T *q = ring + (s % D) * (H::CPW * CS) + (act ? cc * CS + n : 0);   // this lane's rows (transposed)
    if (s < L1) {
      T rk[NB];
      ho_block<NB>(rk, r + NB * s);
      v = (T)0;
#pragma unroll
      for (int m = 0; m < NB; ++m) v = fma(q[NB * m], rk[m], v);
      q += NB2;
    } else {
      v = r[NB * (2 * L1 - 2 - s) + (act ? n : 0)];
    }
#pragma unroll
    for (int m = 0; m < NB; ++m) f[m] = q[NB * m];
  };
  cp_async_wait<D - 1>();
  __syncthreads();
  if (!feeds) load(0);
  for (int s = 0; s < steps; ++s) {
    if (!feeds) {
      if (s < L1) {
        // forward: y_k = (omega G_k^-1) r_k - (G_k^-1 L_k) y_{k-1}, y written over r
        T u = (T)0;
        if (s > 0) {
          T y[NB];
          ho_block<NB>(y, r + NB * (s - 1));
#pragma unroll
          for (int m = 0; m < NB; ++m) u = fma(-f[m], y[m], u);
        }
        if (act) r[NB * s + n] = v + u;
      } else {
        // backward: x_k = y_k - (G_k^-1 U_k) x_{k+1}, x written over y
        const int k = 2 * L1 - 2 - s;
        T x[NB], u = v;
        ho_block<NB>(x, r + NB * (k + 1));
#pragma unroll
        for (int m = 0; m < NB; ++m) u = fma(-f[m], x[m], u);
        if (act) r[NB * k + n] = u;
      }
    }
    cp_async_wait<D - 2>();   // the next step's factors (the feeding warp's copies)
    __syncthreads();
    if (feeds) stage(s + D);  // (its slot was read before this barrier)
    else if (s + 1 < steps) load(s + 1);
  }
  for (int i = threadIdx.x; i < nc * L1 * NB; i += 64)
    lam_out[base + i] = (Tout)(ZERO ? sr[i] : fma((T)keep, (T)lam_in[base + i], sr[i]));
}

// Part 2 at p = 2 in FP32: one warp per block, each lane's factor rows loaded one step ahead into
// registers. A block of 81 floats is aligned to four bytes only, so that the ring takes a 4-byte copy and a
// shared-memory read per factor. 88 x 88 x 32 cells: a zero-start sweep 153 us with the
// ring and 108 so, 56 x 56 x 32: 75 and 69, 16 x 16 x 16: 31 and 29; one warp per block against four
// (few columns then leave SMs without a block) 69 and 74 us on 56 x 56 x 32.
template <int P, bool ZERO, typename T, typename Ts, typename Tout>
__global__ void __launch_bounds__(32)
    ho_sweep_lines_regs_kernel(const HoGeo g, int cpb, const T *__restrict__ zf, const Ts *src,
                               const T *__restrict__ lam_in, Tout *lam_out, double keep) {
  using H = Ho<P>;
  constexpr int NB = H::NB, NB2 = NB * NB, LPC = H::LPC;
  extern __shared__ __align__(16) unsigned char ho_lines_smem[];
  T *sr = reinterpret_cast<T *>(ho_lines_smem);   // [cpb][L+1][NB]
  const int L1 = g.L + 1, lane = threadIdx.x, c0 = blockIdx.x * cpb, nc = min(cpb, g.ncol - c0);
  const int64_t base = g.NH + (int64_t)NB * c0 * L1;
#pragma unroll 4
  for (int i = lane; i < nc * L1 * NB; i += 32) sr[i] = (T)src[base + i];
  __syncwarp();
  const int cc = lane / LPC, n = lane - cc * LPC;
  const bool act = cc < nc && n < NB;   // (the other lanes follow the first column)
  T *r = sr + NB * (act ? cc : 0) * L1;
  const T *f0 = zf + 3 * NB2 * ((int64_t)(c0 + (act ? cc : 0)) * L1) + (act ? n : 0);   // this lane's rows (transposed)
  // forward: y_k = (omega G_k^-1) r_k - (G_k^-1 L_k) y_{k-1}, y written over r
  T fa[NB], fb[NB];
#pragma unroll
  for (int m = 0; m < NB; ++m) { fa[m] = __ldg(f0 + NB * m); fb[m] = __ldg(f0 + NB2 + NB * m); }
  for (int k = 0; k < L1; ++k) {
    const T *f = f0 + 3 * NB2 * min(k + 1, L1 - 1);
    T na[NB], nb[NB], v = (T)0, u = (T)0;
#pragma unroll
    for (int m = 0; m < NB; ++m) { na[m] = __ldg(f + NB * m); nb[m] = __ldg(f + NB2 + NB * m); }
#pragma unroll
    for (int m = 0; m < NB; ++m) v = fma(fa[m], r[NB * k + m], v);
    if (k > 0) {
#pragma unroll
      for (int m = 0; m < NB; ++m) u = fma(-fb[m], r[NB * (k - 1) + m], u);
    }
    __syncwarp();
    if (act) r[NB * k + n] = v + u;
    __syncwarp();
#pragma unroll
    for (int m = 0; m < NB; ++m) { fa[m] = na[m]; fb[m] = nb[m]; }
  }
  // backward: x_k = y_k - (G_k^-1 U_k) x_{k+1}, x written over y (row k only by its own lane)
  const T *fu = f0 + 2 * NB2;
#pragma unroll
  for (int m = 0; m < NB; ++m) fa[m] = __ldg(fu + 3 * NB2 * max(L1 - 2, 0) + NB * m);
  for (int k = L1 - 2; k >= 0; --k) {
    const T *f = fu + 3 * NB2 * max(k - 1, 0);
    T na[NB], v = act ? r[NB * k + n] : (T)0;
#pragma unroll
    for (int m = 0; m < NB; ++m) na[m] = __ldg(f + NB * m);
#pragma unroll
    for (int m = 0; m < NB; ++m) v = fma(-fa[m], r[NB * (k + 1) + m], v);
    if (act) r[NB * k + n] = v;
    __syncwarp();
#pragma unroll
    for (int m = 0; m < NB; ++m) fa[m] = na[m];
  }
#pragma unroll 4
  for (int i = lane; i < nc * L1 * NB; i += 32)
    lam_out[base + i] = (Tout)(ZERO ? sr[i] : fma((T)keep, (T)lam_in[base + i], sr[i]));
}

// R = b - S lam (Algorithm 2 line 3), kHoR rows per thread. ZSWEEP: lam is one sweep from zero,
// lam = omega D^-1 b, so R = (1 - omega) b - (S - D) lam (equal in exact arithmetic).
template <int P, bool ZSWEEP, typename T = double>
__global__ void __launch_bounds__(kHoThreads<P, T>)
    ho_residual_kernel(const HoGeo g, int64_t TT, const T *__restrict__ S, const double *__restrict__ b,
                       const T *__restrict__ lam, T *__restrict__ R_out, double keep) {
  constexpr int NB = Ho<P>::NB, R = kHoR<P, T>;
  __shared__ __align__(16) T ss[NB * kHoThreads<P, T> * R];
  const int i0 = threadIdx.x * R;
  const int64_t row = (int64_t)blockIdx.x * kHoRows<P> + i0, F = (int64_t)blockIdx.x * kHoFacets<P> + i0 / NB;
  if (i0 >= kHoRows<P> || row >= TT) return;
  T v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const T bv = (T)__ldg(b + row + r);
    v[r] = ZSWEEP ? (T)keep * bv : bv;
  }
  ho_row<P, true, ZSWEEP>(S, lam, g, TT, F, i0 % NB, v, ss + i0);
#pragma unroll
  for (int r = 0; r < R; ++r) R_out[row + r] = v[r];
}

// Part 1 of a sweep and the residual in FP32 with a facet per thread (kHoFacetRows). The Jacobi step goes
// through shared memory, a thread per row, so that the factors and the results are coalesced; at p = 1 a
// thread takes its facet's four rows in 16-byte loads instead (128 x 128 x 32 cells: the sweep 261 us
// through shared memory, 240 so).
template <int P, typename Tout>
__global__ void __launch_bounds__(kHoRowThreads)
    ho_sweep_facets_kernel(const HoGeo g, int64_t TT, const float *__restrict__ S, const float *__restrict__ hw,
                           const double *__restrict__ b, const float *__restrict__ lam_in, Tout *__restrict__ lam_out,
                           double keep) {
  constexpr int NB = Ho<P>::NB, LD = NB | 1;
  __shared__ float sr[P == 1 ? 1 : kHoRowThreads * LD];
  const int64_t F0 = (int64_t)blockIdx.x * kHoRowThreads, F = F0 + threadIdx.x, nF = g.nhf + g.nzf;
  if (F < nF) {
    float acc[NB];
#pragma unroll
    for (int n = 0; n < NB; ++n) acc[n] = (float)__ldg(b + NB * F + n);
    ho_facet_rows<P, true>(S, lam_in, g, TT, F, acc);
    if constexpr (P == 1) {
      if (F < g.nhf) {
        const float4 l = __ldg(reinterpret_cast<const float4 *>(lam_in + NB * F));
        float v[4] = {(float)keep * l.x, (float)keep * l.y, (float)keep * l.z, (float)keep * l.w};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float4 w = __ldg(reinterpret_cast<const float4 *>(hw + NB * NB * F) + m);
          v[0] = fmaf(w.x, acc[m], v[0]);
          v[1] = fmaf(w.y, acc[m], v[1]);
          v[2] = fmaf(w.z, acc[m], v[2]);
          v[3] = fmaf(w.w, acc[m], v[3]);
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[n] = v[n];
      }
#pragma unroll
      for (int n = 0; n < NB; ++n) lam_out[NB * F + n] = (Tout)acc[n];
    } else {
#pragma unroll
      for (int n = 0; n < NB; ++n) sr[threadIdx.x * LD + n] = acc[n];
    }
  }
  if constexpr (P == 1) return;
  __syncthreads();
  const int rows = NB * (int)min((int64_t)kHoRowThreads, nF - F0);
  for (int e = threadIdx.x; e < rows; e += kHoRowThreads) {
    const int f = e / NB, n = e - f * NB;
    const float *rf = sr + f * LD;
    const int64_t row = NB * F0 + e;
    float v = rf[n];
    if (F0 + f < g.nhf) {
      const float *w = hw + (int64_t)NB * NB * (F0 + f) + n;
      v = (float)keep * lam_in[row];
#pragma unroll
      for (int m = 0; m < NB; ++m) v = fmaf(__ldg(w + NB * m), rf[m], v);
    }
    lam_out[row] = (Tout)v;
  }
}

template <int P, bool ZSWEEP>
__global__ void __launch_bounds__(kHoRowThreads)
    ho_residual_facets_kernel(const HoGeo g, int64_t TT, const float *__restrict__ S, const double *__restrict__ b,
                              const float *__restrict__ lam, float *__restrict__ R, double keep) {
  constexpr int NB = Ho<P>::NB;
  const int64_t F = (int64_t)blockIdx.x * kHoRowThreads + threadIdx.x;
  if (F >= g.nhf + g.nzf) return;
  float acc[NB];
#pragma unroll
  for (int n = 0; n < NB; ++n) {
    const float bv = (float)__ldg(b + NB * F + n);
    acc[n] = ZSWEEP ? (float)keep * bv : bv;
  }
  ho_facet_rows<P, ZSWEEP>(S, lam, g, TT, F, acc);
#pragma unroll
  for (int n = 0; n < NB; ++n) R[NB * F + n] = acc[n];
}

// bbar_K = Gamma_K (P^T R)_K (Algorithm 2 lines 4-5): P is constant on a facet (all its nodes)
// and averages the facet's cells, so P^T sums the cell's facet nodes with weight 1/2 (1 on
// ground and lid facets)
template <int P, typename T = double>
__global__ void ho_restrict_kernel(const HoGeo g, int64_t ncell, const T *__restrict__ R,
                                   const T *__restrict__ gamma, T *__restrict__ bbar) {
  using H = Ho<P>;
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= ncell) return;
  const int c = (int)(K / g.L), k = (int)(K - (int64_t)c * g.L);
  T s = (T)0;
  for (int q = 0; q < H::NF; ++q) {
    const int f = q / H::NB;
    const bool boundary = (f == 4 && k == 0) || (f == 5 && k == g.L - 1);
    s = fma(boundary ? (T)1 : (T)0.5, R[ho_gid<P>(g, c, k, q)], s);
  }
  bbar[K] = gamma ? gamma[K] * s : s;
}

// lam_out = lam_in + P dPi (Algorithm 2 line 7), one thread per row
template <int P, typename T = double>
__global__ void ho_prolong_kernel(const HoGeo g, int64_t TT, const T *__restrict__ lam_in,
                                  const T *__restrict__ dpi, T *__restrict__ lam_out) {
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row >= TT) return;
  const HoFacet fc = ho_facet(g, row / Ho<P>::NB);
  const T a = dpi[(int64_t)fc.cA * g.L + fc.kA];
  lam_out[row] = fc.cB >= 0 ? fma((T)0.5, a + dpi[(int64_t)fc.cB * g.L + fc.kB], lam_in[row]) : lam_in[row] + a;
}

// the FP32 preconditioner's copies of the degree-p operator and factors; the last step's FP32
// result widened to FP64
template <typename Ta, typename Tb>
__global__ void ho_convert_kernel(const Ta *__restrict__ x, Tb *__restrict__ y, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = (Tb)x[i];
}

// Gamma = (H 1) / (P^T S P 1) (Eq. scaling_matrix): P^T sums a facet's nodes with weight 1/2 (1 on
// ground and lid facets), S 1 on a facet is the sum over its cells of S_K 1 (sk1 [6][ncell], summed over
// the facet's nodes).
__global__ void ho_gamma_kernel(int64_t ncell, int L, const int32_t *__restrict__ nbr,
                                const int32_t *__restrict__ nbr_face, const double *__restrict__ m,
                                const double *__restrict__ sk1, double *__restrict__ gamma) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K >= ncell) return;
  const int c = (int)(K / L), k = (int)(K - (int64_t)c * L);
  double s = 0.0;
#pragma unroll
  for (int f = 0; f < 4; ++f)
    s += 0.5 * (sk1[f * ncell + K] + sk1[nbr_face[4 * (int64_t)c + f] * ncell + (int64_t)nbr[4 * (int64_t)c + f] * L + k]);
  s += k == 0 ? sk1[4 * ncell + K] : 0.5 * (sk1[4 * ncell + K] + sk1[5 * ncell + K - 1]);
  s += k == L - 1 ? sk1[5 * ncell + K] : 0.5 * (sk1[5 * ncell + K] + sk1[4 * ncell + K + 1]);
  gamma[K] = m[K] / s;
}

__global__ void ho_fill_kernel(double *__restrict__ x, int64_t n, double v) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) x[i] = v;
}

__global__ void ho_gamma_div_kernel(int64_t ncell, const double *__restrict__ m, double *__restrict__ gamma) {
  const int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (K < ncell) gamma[K] = m[K] / gamma[K];   // gamma holds P^T S P 1 on entry
}

// ---- host side ------------------------------------------------------------------------------------
int64_t ho_trace_size(const Ctx *c, int p) {
  const Level &f = c->lv[0];
  return (int64_t)(p + 1) * (p + 1) * ((int64_t)f.nedge * f.nlev + (int64_t)f.ncol * (f.nlev + 1));
}

template <int P>
static int ho_build_factors(Ctx *c) {
  HoData &h = c->ho;
  const HoGeo g = ho_geo<P>(c);
  constexpr int NB = Ho<P>::NB;
  int *sing = h.flag;
  HMG_CUDA(c, cudaMemsetAsync(sing, 0, sizeof(int), c->stream));
  const size_t zsmem = sizeof(double) * kHoFacWarps * (3 * NB * NB + 2 * NB * NB);
  ho_hfactor_kernel<P><<<grid_for(g.nhf, kHoFacWarps), 32 * kHoFacWarps, 0, c->stream>>>(g, h.T, h.S, c->opt.omega,
                                                                                      h.hw, sing);
  ho_zfactor_kernel<P><<<grid_for(g.ncol, kHoFacWarps), 32 * kHoFacWarps, zsmem, c->stream>>>(
      g, h.T, h.S, c->opt.omega, h.zf, sing);
  HMG_CUDA(c, cudaGetLastError());
  if (h.have_fp32) {   // the FP32 preconditioner's copies of the factors follow them
    const int64_t nh = (int64_t)NB * NB * g.nhf, nz = (int64_t)3 * NB * NB * g.nzf;
    ho_convert_kernel<double, float><<<grid_for(nh, 256), 256, 0, c->stream>>>(h.hw, h.hw32, nh);
    ho_convert_kernel<double, float><<<grid_for(nz, 256), 256, 0, c->stream>>>(h.zf, h.zf32, nz);
    HMG_CUDA(c, cudaGetLastError());
  }
  int s = 0;
  HMG_CUDA(c, cudaMemcpyAsync(&s, sing, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  HMG_CUDA(c, cudaStreamSynchronize(c->stream));
  if (s) return fail(c, HMG_ERR_INVALID_ARG, "a smoother block of the degree-p trace operator is singular");
  h.factor_omega = c->opt.omega;
  return HMG_OK;
}

// The FP32 copies of S, Gamma and the smoother factors (allocated once per layout)
template <int P>
static int ho_build_fp32(Ctx *c) {
  using H = Ho<P>;
  HoData &h = c->ho;
  const HoGeo g = ho_geo<P>(c);
  const int64_t C = c->lv[0].ncell, nS = (int64_t)H::SLOTS * h.T;
  const int64_t nh = (int64_t)H::NB * H::NB * g.nhf, nz = (int64_t)3 * H::NB * H::NB * g.nzf;
  int st;
  if ((st = dev_make(c, &h.S32, (size_t)nS))) return st;
  if ((st = dev_make(c, &h.hw32, (size_t)nh))) return st;
  if ((st = dev_make(c, &h.zf32, (size_t)nz))) return st;
  if ((st = dev_make(c, &h.gamma32, (size_t)C))) return st;
  ho_convert_kernel<double, float><<<grid_for(nS, 256), 256, 0, c->stream>>>(h.S, h.S32, nS);
  ho_convert_kernel<double, float><<<grid_for(nh, 256), 256, 0, c->stream>>>(h.hw, h.hw32, nh);
  ho_convert_kernel<double, float><<<grid_for(nz, 256), 256, 0, c->stream>>>(h.zf, h.zf32, nz);
  ho_convert_kernel<double, float><<<grid_for(C, 256), 256, 0, c->stream>>>(h.gamma, h.gamma32, C);
  HMG_CUDA(c, cudaGetLastError());
  h.have_fp32 = true;
  return HMG_OK;
}

void ho_free(Ctx *c) {
  HoData &h = c->ho;
  if (h.flag) drop_graph(c);   // captured launches hold these buffers (flag is the first of them to be made)
  double **bufs[] = {&h.tab, &h.gtab, &h.ctab, &h.ltab, &h.S, &h.Ainv, &h.hw, &h.zf, &h.gamma, &h.m, &h.fs};
  for (double **b : bufs) {
    dev_free(c, *b);
    *b = nullptr;
  }
  dev_free(c, h.itab);
  h.itab = nullptr;
  dev_free(c, h.own);
  h.own = nullptr;
  dev_free(c, h.flag);
  h.flag = nullptr;
  float **f32[] = {&h.S32, &h.hw32, &h.zf32, &h.gamma32};
  for (float **b : f32) {
    dev_free(c, *b);
    *b = nullptr;
  }
  h.cw = nullptr;
  h.have_fp32 = false;
  h.degree = 0;
  h.ncell = 0;
  h.T = 0;
}

template <int P>
static int ho_launch_spmv_p(Ctx *c, const double *x, double *y, int mode, const double *w, int slot0, int slot1);

template <int P>
static int ho_assemble_p(Ctx *c) {
  using H = Ho<P>;
  const Level &f = c->lv[0];
  HoData &h = c->ho;
  const int64_t C = f.ncell;
  int st;
  if (C > 0x7fffffff) return fail(c, HMG_ERR_INVALID_ARG, "too many cells for one launch");
  if (h.degree != P || h.ncell != C || h.T != ho_trace_size(c, P)) {   // (re)allocate for this degree and mesh
    ho_free(c);
    if ((st = dev_alloc(c, &h.flag, 1))) return st;
    const int64_t T = ho_trace_size(c, P);
    if ((st = dev_alloc(c, &h.S, (size_t)H::SLOTS * T))) return st;
    if ((st = dev_alloc(c, &h.Ainv, (size_t)H::N * H::N * C))) return st;
    if ((st = dev_alloc(c, &h.hw, (size_t)H::NB * H::NB * f.nedge * f.nlev))) return st;
    if ((st = dev_alloc(c, &h.zf, (size_t)3 * H::NB * H::NB * f.ncol * (f.nlev + 1)))) return st;
    if ((st = dev_alloc(c, &h.gamma, (size_t)C))) return st;
    if ((st = dev_alloc(c, &h.m, (size_t)C))) return st;
    if ((st = dev_alloc(c, &h.own, (size_t)4 * f.ncol))) return st;
    if ((st = dev_alloc(c, &h.fs, (size_t)2 * (T / H::NB)))) return st;
    h.degree = P;
    h.ncell = C;
    h.T = T;
  }
  h.factor_omega = 0.0;
  h.have_fp32 = false;
  HMG_CUDA(c, cudaMemsetAsync(h.own, 0, 4 * (size_t)f.ncol, c->stream));
  ho_own_kernel<<<grid_for(f.nedge, 256), 256, 0, c->stream>>>(f.edge_stencil, f.edge_fc, f.nedge, h.own);
  HMG_CUDA(c, cudaMemsetAsync(h.flag, 0, sizeof(int), c->stream));
  double *sk1 = static_cast<double *>(c->w1);   // 6 C doubles of at least NB (3 C + ncol)
  const bool gauss = c->opt.precision == HMG_PRECISION_MIXED;   // (gauss_cells.cu says why)
  if ((st = gauss ? ho_gauss_cell_matrices<P>(c) : ho_cell_matrices<P>(c, sk1))) return st;
  int sing = 0;
  HMG_CUDA(c, cudaMemcpyAsync(&sing, h.flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  HMG_CUDA(c, cudaStreamSynchronize(c->stream));
  if (sing) return fail(c, HMG_ERR_INVALID_ARG, "a degree-p cell matrix A_K is singular");
  const HoGeo g = ho_geo<P>(c);
  ho_rows_kernel<P><<<grid_for(h.T, 256), 256, 0, c->stream>>>(g, h.T, h.cw, h.Ainv, h.S);
  HMG_CUDA(c, cudaGetLastError());
  if (gauss) {   // P^T S P 1 by the operator itself (P 1 = 1)
    double *ones = sk1, *s1 = static_cast<double *>(c->w2);
    ho_fill_kernel<<<grid_for(h.T, 256), 256, 0, c->stream>>>(ones, h.T, 1.0);
    if ((st = ho_launch_spmv_p<P>(c, ones, s1, 0, nullptr, 0, 0))) return st;
    ho_restrict_kernel<P, double><<<grid_for(C, 64), 64, 0, c->stream>>>(g, C, s1, nullptr, h.gamma);
    ho_gamma_div_kernel<<<grid_for(C, 256), 256, 0, c->stream>>>(C, h.m, h.gamma);
  } else {
    ho_gamma_kernel<<<grid_for(C, 256), 256, 0, c->stream>>>(C, f.nlev, f.col_nbr, f.col_nbr_face, h.m, sk1, h.gamma);
  }
  HMG_CUDA(c, cudaGetLastError());
  if ((st = ho_build_factors<P>(c))) return st;
  if (c->opt.precision == HMG_PRECISION_MIXED) return ho_build_fp32<P>(c);
  return HMG_OK;
}

template <int P>
static int ho_launch_spmv_p(Ctx *c, const double *x, double *y, int mode, const double *w, int slot0, int slot1) {
  const HoData &h = c->ho;
  const HoGeo g = ho_geo<P>(c);
  const int64_t nF = g.nhf + g.nzf;
  if (grid_for(nF, 256) > (unsigned)kMaxRedBlocks)
    return fail(c, HMG_ERR_INVALID_ARG, "too many facets for one reduction");
  const unsigned grid = grid_for(h.T, kHoRows<P>);
  Prof prof(c, kCompApply);
  switch (mode) {
    case 0: ho_spmv_kernel<P, 0><<<grid, kHoThreads<P, double>, 0, c->stream>>>(g, h.T, h.S, x, y, w, h.fs); break;
    case 1: ho_spmv_kernel<P, 1><<<grid, kHoThreads<P, double>, 0, c->stream>>>(g, h.T, h.S, x, y, w, h.fs); break;
    case 2: ho_spmv_kernel<P, 2><<<grid, kHoThreads<P, double>, 0, c->stream>>>(g, h.T, h.S, x, y, w, h.fs); break;
    default: ho_spmv_kernel<P, 3><<<grid, kHoThreads<P, double>, 0, c->stream>>>(g, h.T, h.S, x, y, w, h.fs); break;
  }
  const unsigned rg = grid_for(nF, 2048);
  if (mode == 2) ho_reduce_kernel<2><<<rg, 256, 0, c->stream>>>(h.fs, nF, slot0, slot1, c->part, c->counter, c->scal);
  else if (mode) ho_reduce_kernel<1><<<rg, 256, 0, c->stream>>>(h.fs, nF, slot0, 0, c->part, c->counter, c->scal);
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

template <int P>
static int ho_trace_rhs_p(Ctx *c, const double *Ru, const double *Rp, double *B) {
  const HoData &h = c->ho;
  Prof prof(c, kCompRhs);
  if constexpr (P == 1) {
    ho_rhs_direct_kernel<P><<<grid_for(h.T, 128), 128, 0, c->stream>>>(ho_geo<P>(c), h.T, h.cw, h.Ainv, Ru, Rp, B);
    HMG_CUDA(c, cudaGetLastError());
    return HMG_OK;
  }
  // the cells' products pass through the preconditioner's work vectors (T >= 3 NB C = NF / 2 C doubles each)
  double *d0 = static_cast<double *>(c->w1), *d1 = static_cast<double *>(c->w2);
  int st;
  if ((st = ho_launch_dot<P, false>(c, nullptr, Ru, Rp, d0, d1))) return st;
  ho_rhs_kernel<P><<<grid_for(h.T, 256), 256, 0, c->stream>>>(ho_geo<P>(c), h.T, h.cw, d0, d1, B);
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

template <int P>
static int ho_reconstruct_p(Ctx *c, const double *lam, const double *Ru, const double *Rp, double *u, double *pi) {
  const int64_t C = c->lv[0].ncell;
  if constexpr (P == 1) {
    if (first_form(c, C < kHoDirectCells)) {
      ho_recover_direct_kernel<P><<<grid_for(C * Ho<P>::N, 128), 128, 0, c->stream>>>(ho_geo<P>(c), C, c->ho.cw, c->ho.Ainv,
                                                                                       lam, Ru, Rp, u, pi);
      HMG_CUDA(c, cudaGetLastError());
      return HMG_OK;
    }
  }
  return ho_launch_dot<P, true>(c, lam, Ru, Rp, u, pi);
}

// The FP64 operator or the FP32 preconditioner's copies
template <typename T> struct HoPrec;
template <> struct HoPrec<double> {
  static const double *S(const HoData &h) { return h.S; }
  static const double *hw(const HoData &h) { return h.hw; }
  static const double *zf(const HoData &h) { return h.zf; }
  static const double *gamma(const HoData &h) { return h.gamma; }
};
template <> struct HoPrec<float> {
  static const float *S(const HoData &h) { return h.S32; }
  static const float *hw(const HoData &h) { return h.hw32; }
  static const float *zf(const HoData &h) { return h.zf32; }
  static const float *gamma(const HoData &h) { return h.gamma32; }
};

// One sweep of Algorithm 1 in arithmetic T: b (the Krylov residual, FP64) and lam_in (Tin) in,
// lam_out (Tout) out.
template <int P, bool ZERO, typename T = double, typename Tin = double, typename Tout = double>
static int ho_sweep(Ctx *c, const double *b, const Tin *lam_in, Tout *lam_out) {
  using H = Ho<P>;
  const HoData &h = c->ho;
  const HoGeo g = ho_geo<P>(c);
  // columns per block of the line part: one warp of CPW columns, and the block's rows (NB (L + 1)
  // values per column) within 48 KB beside the ring
  const int cap = (int)((48 * 1024) / (sizeof(T) * H::NB * (g.L + 1)));
  if (cap < 1) return fail(c, HMG_ERR_INVALID_ARG, "too many layers for the degree-p line smoother");
  const int cpb = cap < H::CPW ? cap : H::CPW;
  const unsigned nzb = (unsigned)((g.ncol + cpb - 1) / cpb);
  const size_t rows = sizeof(T) * H::NB * cpb * (g.L + 1), ring = sizeof(T) * HoLines<P>::DEPTH * H::CPW * HoLines<P>::STRIDE;
  const double keep = 1.0 - h.factor_omega;
  Prof prof(c, ZERO ? kCompPresmooth : kCompSweep, 2);
  bool by_row = true;
  if constexpr (!ZERO && sizeof(T) == 4) {
    by_row = first_form(c, h.T < kHoFacetRows<P>);
    if (!by_row)
      ho_sweep_facets_kernel<P, Tout><<<grid_for(g.nhf + g.nzf, kHoRowThreads), kHoRowThreads, 0, c->stream>>>(
          g, h.T, HoPrec<T>::S(h), HoPrec<T>::hw(h), b, lam_in, lam_out, keep);
  }
  if (by_row)
    ho_sweep_rows_kernel<P, ZERO, T, double, Tin, Tout>
        <<<grid_for(ZERO ? g.NH : h.T, kHoRows<P>), ZERO ? kHoRowThreads : kHoThreads<P, T>, 0, c->stream>>>(
            g, h.T, HoPrec<T>::S(h), HoPrec<T>::hw(h), b, lam_in, lam_out, keep);
  auto lines = [&](auto kern, int threads, size_t smem, const auto *src) {
    const cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                           : cudaSuccess;
    if (e == cudaSuccess) kern<<<nzb, threads, smem, c->stream>>>(g, cpb, HoPrec<T>::zf(h), src, lam_in, lam_out, keep);
    return e;
  };
  using Ts = std::conditional_t<ZERO, double, Tout>;
  const Ts *src;
  if constexpr (ZERO) src = b;
  else src = lam_out;
  if constexpr (P == 2 && sizeof(T) == 4)
    HMG_CUDA(c, lines(ho_sweep_lines_regs_kernel<P, ZERO, T, Ts, Tout>, 32, rows, src));
  else
    HMG_CUDA(c, lines(ho_sweep_lines_kernel<P, ZERO, T, Ts, Tin, Tout>, 64, ring + rows, src));
  HMG_CUDA(c, cudaGetLastError());
  return HMG_OK;
}

template <int P>
static int ho_line_smooth_p(Ctx *c, const double *b, double *lam, int nsweeps) {
  int st;
  if ((st = ho_refactor_if_needed(c))) return st;
  double *cur = lam, *nxt = static_cast<double *>(c->w3);
  for (int i = 0; i < nsweeps; ++i) {
    if ((st = ho_sweep<P, false>(c, b, cur, nxt))) return st;
    double *t = cur;
    cur = nxt;
    nxt = t;
  }
  if (cur != lam)
    HMG_CUDA(c, cudaMemcpyAsync(lam, cur, sizeof(double) * c->ho.T, cudaMemcpyDeviceToDevice, c->stream));
  return HMG_OK;
}

// z = M^-1 r: configuration 3c (Algorithm 2, the V-cycle of the lowest-order pressure operator as
// the coarse solve), configuration 2 (n_smooth sweeps of Algorithm 1 from zero) or none. T = float
// is the FP32 preconditioner: its coefficients, work vectors and V-cycle in FP32, r read and z
// written in FP64 (the Krylov vectors).
template <int P, typename T>
static int ho_precond_p(Ctx *c, const double *r, double *z) {
  const HoData &h = c->ho;
  const HoGeo g = ho_geo<P>(c);
  const int64_t TT = h.T, C = c->lv[0].ncell;
  int st;
  if (sizeof(T) == 4 && !h.have_fp32) return fail(c, HMG_ERR_NOT_READY, "the FP32 copies of the degree-p operator are missing");
  T *w1 = static_cast<T *>(c->w1), *w2 = static_cast<T *>(c->w2), *w3 = static_cast<T *>(c->w3);
  if (c->opt.precond == HMG_PRECOND_NONE) {
    HMG_CUDA(c, cudaMemcpyAsync(z, r, sizeof(double) * TT, cudaMemcpyDeviceToDevice, c->stream));
    return HMG_OK;
  }
  if (c->opt.precond == HMG_PRECOND_LINESMOOTH) {
    const int n = c->opt.n_smooth;
    if (n == 1) return ho_sweep<P, true, T, T, double>(c, r, nullptr, z);
    if ((st = ho_sweep<P, true, T, T, T>(c, r, nullptr, w1))) return st;
    T *cur = w1, *nxt = w2;
    for (int i = 1; i < n; ++i) {
      if (i == n - 1) return ho_sweep<P, false, T, T, double>(c, r, cur, z);
      if ((st = ho_sweep<P, false, T, T, T>(c, r, cur, nxt))) return st;
      T *t = cur;
      cur = nxt;
      nxt = t;
    }
    return HMG_OK;
  }
  // lines 1-2: presmoothing from zero
  if (c->opt.n_pre >= 1) {
    if ((st = ho_sweep<P, true, T, T, T>(c, r, nullptr, w1))) return st;
    for (int i = 1; i < c->opt.n_pre; ++i) {
      if ((st = ho_sweep<P, false, T, T, T>(c, r, w1, w2))) return st;
      T *t = w1;
      w1 = w2;
      w2 = t;
    }
  } else {
    HMG_CUDA(c, cudaMemsetAsync(w1, 0, sizeof(T) * TT, c->stream));
  }
  T *cb = static_cast<T *>(c->cb);
  {
    Prof pr(c, kCompResidual, 2);
    const bool zsweep = c->opt.n_pre == 1;   // w1 is one sweep from zero                       // line 3
    const double rkeep = zsweep ? 1.0 - h.factor_omega : 0.0;
    bool by_row = true;
    if constexpr (sizeof(T) == 4 && P > 1) {
      by_row = first_form(c, h.T < kHoFacetRows<P>);
      if (!by_row) {
        auto k = zsweep ? ho_residual_facets_kernel<P, true> : ho_residual_facets_kernel<P, false>;
        k<<<grid_for(g.nhf + g.nzf, kHoRowThreads), kHoRowThreads, 0, c->stream>>>(g, TT, HoPrec<T>::S(h), r, w1, w2, rkeep);
      }
    }
    if (by_row) {
      auto k = zsweep ? ho_residual_kernel<P, true, T> : ho_residual_kernel<P, false, T>;
      k<<<grid_for(TT, kHoRows<P>), kHoThreads<P, T>, 0, c->stream>>>(g, TT, HoPrec<T>::S(h), r, w1, w2, rkeep);
    }
    ho_restrict_kernel<P, T><<<grid_for(C, 64), 64, 0, c->stream>>>(g, C, w2, HoPrec<T>::gamma(h), cb);   // lines 4-5
    HMG_CUDA(c, cudaGetLastError());
  }
  T *dpi = nullptr;
  {
    Prof pv(c, kCompVcycle, vcycle_launches(c));
    if ((st = vcycle<T>(c, cb, &dpi))) return st;                                                 // line 6
  }
  {
    Prof pp(c, kCompProlong);
    ho_prolong_kernel<P, T><<<grid_for(TT, 256), 256, 0, c->stream>>>(g, TT, w1, dpi, w2);          // line 7
    HMG_CUDA(c, cudaGetLastError());
  }
  const int np = c->opt.n_post;                                                                    // line 8
  if (np == 0) {
    ho_convert_kernel<T, double><<<grid_for(TT, 256), 256, 0, c->stream>>>(w2, z, TT);
    HMG_CUDA(c, cudaGetLastError());
    return HMG_OK;
  }
  T *cur = w2, *nxt = w3;
  for (int i = 0; i < np - 1; ++i) {
    if ((st = ho_sweep<P, false, T, T, T>(c, r, cur, nxt))) return st;
    T *t = cur;
    cur = nxt;
    nxt = t;
  }
  return ho_sweep<P, false, T, T, double>(c, r, cur, z);
}

// ---- degree dispatch ------------------------------------------------------------------------------
static int bad_degree(Ctx *c) { return fail(c, HMG_ERR_INVALID_ARG, "the degree-p path takes p = 1, 2, 3"); }

int ho_assemble(Ctx *c) {
  if (c->sc.preset != 1) return fail(c, HMG_ERR_INVALID_ARG, "degree p >= 1 is built for the Helmholtz preset (preset 1)");
  switch (c->degree) {
    case 1: return ho_assemble_p<1>(c);
    case 2: return ho_assemble_p<2>(c);
    case 3: return ho_assemble_p<3>(c);
    default: return bad_degree(c);
  }
}

int ho_refactor_if_needed(Ctx *c) {
  if (c->opt.precision == HMG_PRECISION_MIXED && !c->ho.have_fp32) {   // switched to the FP32 preconditioner
    int st = HMG_OK;
    switch (c->degree) {
      case 1: st = ho_build_fp32<1>(c); break;
      case 2: st = ho_build_fp32<2>(c); break;
      case 3: st = ho_build_fp32<3>(c); break;
      default: return bad_degree(c);
    }
    if (st) return st;
  }
  if (c->ho.factor_omega == c->opt.omega) return HMG_OK;
  switch (c->degree) {
    case 1: return ho_build_factors<1>(c);
    case 2: return ho_build_factors<2>(c);
    case 3: return ho_build_factors<3>(c);
    default: return bad_degree(c);
  }
}

int ho_launch_spmv(Ctx *c, const double *x, double *y, int mode, const double *w, int slot0, int slot1) {
  switch (c->degree) {
    case 1: return ho_launch_spmv_p<1>(c, x, y, mode, w, slot0, slot1);
    case 2: return ho_launch_spmv_p<2>(c, x, y, mode, w, slot0, slot1);
    case 3: return ho_launch_spmv_p<3>(c, x, y, mode, w, slot0, slot1);
    default: return bad_degree(c);
  }
}

int ho_trace_rhs(Ctx *c, const double *Ru, const double *Rp, double *B) {
  switch (c->degree) {
    case 1: return ho_trace_rhs_p<1>(c, Ru, Rp, B);
    case 2: return ho_trace_rhs_p<2>(c, Ru, Rp, B);
    case 3: return ho_trace_rhs_p<3>(c, Ru, Rp, B);
    default: return bad_degree(c);
  }
}

int ho_reconstruct(Ctx *c, const double *lam, const double *Ru, const double *Rp, double *u, double *pi) {
  switch (c->degree) {
    case 1: return ho_reconstruct_p<1>(c, lam, Ru, Rp, u, pi);
    case 2: return ho_reconstruct_p<2>(c, lam, Ru, Rp, u, pi);
    case 3: return ho_reconstruct_p<3>(c, lam, Ru, Rp, u, pi);
    default: return bad_degree(c);
  }
}

int ho_line_smooth(Ctx *c, const double *b, double *lam, int nsweeps) {
  switch (c->degree) {
    case 1: return ho_line_smooth_p<1>(c, b, lam, nsweeps);
    case 2: return ho_line_smooth_p<2>(c, b, lam, nsweeps);
    case 3: return ho_line_smooth_p<3>(c, b, lam, nsweeps);
    default: return bad_degree(c);
  }
}

int ho_precond(Ctx *c, const double *r, double *z) {
  const bool mixed = c->opt.precision == HMG_PRECISION_MIXED;
  switch (c->degree) {
    case 1: return mixed ? ho_precond_p<1, float>(c, r, z) : ho_precond_p<1, double>(c, r, z);
    case 2: return mixed ? ho_precond_p<2, float>(c, r, z) : ho_precond_p<2, double>(c, r, z);
    case 3: return mixed ? ho_precond_p<3, float>(c, r, z) : ho_precond_p<3, double>(c, r, z);
    default: return bad_degree(c);
  }
}

}  // namespace hmg
