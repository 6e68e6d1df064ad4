// dense_lu.cu -- FP64 LU with partial pivoting of dense c x c matrices in device memory, over the
// whole GPU, with one right-hand side on either side carried through the elimination (A8: the
// reduced absorbing-chain solve of Sec. 4; Sec. 8: the robust value's policy evaluation).
//
// Right-looking, panels of kNb columns: lu_panel_kernel factors a panel (one CTA, the panel in
// shared memory), lu_rows_kernel applies its row swaps to the other columns and solves U12 = L11^-1
// A12 (a thread per column), lu_update_kernel subtracts L21 U12 from the trailing matrix (32 x 32
// tiles over the GPU).  Matrices of up to kSingle columns are one panel.  Factors and pivots are
// those of lu_factor (linalg.cuh): unit lower L, whole-row swaps, piv[k] = row swapped with row k,
// ties to the smallest row.
//
// A row vector y (solving x A = y) rides along as a row below the matrix that is never a pivot: its
// multipliers are z = y U^-1.  A column vector b (solving A x = b) rides along as a column right of
// it and becomes L^-1 P b.  One triangular solve each is left (upper_solve, lower_t_solve).
//
// Bound: the chain panel, rows, update of every kNb columns.  By GB300's FP64 pipe (about 2 FMA per
// clock and SM) the trailing updates' c^3 / 3 FMA take 1.1 ms over all SMs at c = 1,251 and the panels'
// c^2 kNb / 4 take 0.7 on one SM; the kernels' durations there (profiles/solve_launches.md) are
// panels 3.7 ms (23 us each, 35 the tallest: pivots and barriers of one CTA), updates 2.0 (13 us), rows
// 1.0 (6.4 us) and the two triangular solves 0.4, of a call's 7.55.  Before, one CTA eliminated
// column by column: 222 ms at c = 1,251, 0.80 ms at c = 97.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "afc_internal.h"
#include "dense_lu.cuh"
#include "linalg.cuh"

namespace afc {

namespace {

constexpr int kNb = 8;               // columns of a panel
constexpr int kSingle = 112;         // matrices up to this size are one panel
constexpr int kPanelThreads = 1024;
constexpr int kTile = 32;            // rows and columns of an update tile
constexpr int kPanelStatic = 4096;   // at least the panel kernel's static arrays

// Leading dimension of the panel in shared memory: odd, so that the elements of a row (one per
// column) fall into different banks when it is filled and written back.
__host__ __device__ inline int panel_ld(int rows) { return ((rows + 15) & ~15) + 1; }

__host__ inline size_t panel_bytes(int rows, int cols) {
  return sizeof(double) * (size_t)panel_ld(rows) * (size_t)cols;
}

// Panel kb .. kb + nb - 1 of problem blockIdx.x: rows kb .. c - 1 and the extra row; with_col: the
// extra column is eliminated with it (the last panel).  SMEM: the panel in shared memory, else in
// place (panels too tall for it).  L entries stay unscaled until they are written back.
template <bool SMEM>
__global__ void __launch_bounds__(kPanelThreads, 1)
lu_panel_kernel(LuBatch B, int c, int kb, int nb, int with_col) {
  extern __shared__ __align__(16) double panel[];
  __shared__ unsigned long long skey[32];
  __shared__ int sidx[32];
  __shared__ double sinv[kSingle];
  const uint32_t p = blockIdx.x;
  if (B.active && !B.active[p]) return;
  double *A = B.A + (size_t)p * B.a_stride;
  int32_t *piv = B.piv + (size_t)p * B.v_stride;
  double *row = B.row ? B.row + (size_t)p * B.v_stride : nullptr;
  double *col = B.col ? B.col + (size_t)p * B.v_stride : nullptr;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = c - kb, mr = m + (row ? 1 : 0), nc = nb + (with_col && col ? 1 : 0);
  const int ld = panel_ld(mr);
  // element (i, j) of the panel: i = m the extra row, j = nb the extra column
  auto global_at = [&](int i, int j) -> double * {
    if (i == m) return j == nb ? nullptr : row + kb + j;
    return j == nb ? col + kb + i : A + (size_t)(kb + i) * c + kb + j;
  };
  auto at = [&](int i, int j) -> double & {
    if constexpr (SMEM) return panel[(size_t)j * ld + i];
    else return *global_at(i, j);
  };
  if constexpr (SMEM) {
    for (int q = tid; q < mr * nc; q += kPanelThreads) {
      const int i = q / nc, j = q - i * nc;
      const double *g = global_at(i, j);
      panel[(size_t)j * ld + i] = g ? *g : 0.0;
    }
    __syncthreads();
  }
  // threads as row threads x column groups
  int rg = 32;
  while (rg < mr && rg < kPanelThreads) rg <<= 1;
  const int rt = tid & (rg - 1), cg = tid / rg, ncg = kPanelThreads / rg, nw = rg >> 5;
  unsigned long long key = 0ull;
  int idx = 0;
  if (cg == 0)
    for (int i = rt; i < m; i += rg) {
      const unsigned long long k = mag(at(i, 0));
      if (k > key) { key = k; idx = i; }
    }
  for (int k = 0; k < nb; ++k) {
    if (cg == 0) {
      warp_argmax(key, idx);
      if (lane == 0) { skey[warp] = key; sidx[warp] = idx; }
    }
    __syncthreads();
    key = lane < nw ? skey[lane] : 0ull;
    idx = lane < nw ? sidx[lane] : 0x7FFFFFFF;
    warp_argmax(key, idx);
    if (key == 0ull) {   // uniform over the CTA
      if (tid == 0) atomicOr(B.status, kErrSolve);
      for (int q = k + tid; q < nb; q += kPanelThreads) piv[kb + q] = kb + q;
      return;
    }
    const int pr = idx;
    for (int j = tid; j < nc; j += kPanelThreads) {
      const double a = at(pr, j);
      if (j == k) sinv[k] = 1.0 / a;
      if (pr != k) { at(pr, j) = at(k, j); at(k, j) = a; }
    }
    if (tid == 0) piv[kb + k] = kb + pr;
    __syncthreads();
    const double inv = sinv[k];
    key = 0ull;
    idx = 0;
    for (int i = k + 1 + rt; i < mr; i += rg) {
      if (k + 1 + cg >= nc) break;
      const double l = at(i, k) * inv;
      for (int j = k + 1 + cg; j < nc; j += ncg) {
        if (!SMEM && i == m && j == nb) continue;   // the corner is no element in place
        const double x = fma(-l, at(k, j), at(i, j));
        at(i, j) = x;
        if (j == k + 1 && i < m) {
          const unsigned long long kk = mag(x);
          if (kk > key) { key = kk; idx = i; }
        }
      }
    }
  }
  __syncthreads();
  if constexpr (SMEM) {
    for (int q = tid; q < mr * nc; q += kPanelThreads) {
      const int i = q / nc, j = q - i * nc;
      double *g = global_at(i, j);
      const double x = panel[(size_t)j * ld + i];
      if (g) *g = j < nb && i > j ? x * sinv[j] : x;
    }
  } else {
    for (int q = tid; q < mr * nb; q += kPanelThreads) {
      const int i = q / nb, j = q - i * nb;
      if (i > j) *global_at(i, j) *= sinv[j];
    }
  }
}

// The other columns (and the extra column unless the panel took it): the panel's row swaps, and
// right of the panel U12 = L11^-1 A12.  A thread per column; blockIdx.y = problem.
__global__ void __launch_bounds__(128)
lu_rows_kernel(LuBatch B, int c, int kb, int nb, int with_col) {
  __shared__ double L[kNb][kNb];
  __shared__ int32_t sp[kNb];
  const uint32_t p = blockIdx.y;
  if (B.active && !B.active[p]) return;
  double *A = B.A + (size_t)p * B.a_stride;
  const int32_t *piv = B.piv + (size_t)p * B.v_stride;
  double *col = B.col ? B.col + (size_t)p * B.v_stride : nullptr;
  const int ke = kb + nb;
  for (int q = (int)threadIdx.x; q < nb * nb; q += (int)blockDim.x)
    L[q / nb][q % nb] = A[(size_t)(kb + q / nb) * c + kb + q % nb];
  if ((int)threadIdx.x < nb) sp[threadIdx.x] = piv[kb + threadIdx.x];
  __syncthreads();
  const int q = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  const int j = q < kb ? q : q + nb;
  if (j > c || (j == c && (!col || with_col))) return;
  double *M = j == c ? col : A + j;
  const size_t st = j == c ? 1 : (size_t)c;
  double u[kNb];
#pragma unroll
  for (int r = 0; r < kNb; ++r) u[r] = r < nb ? M[(size_t)(kb + r) * st] : 0.0;
#pragma unroll
  for (int k = 0; k < kNb; ++k) {
    const int32_t pr = k < nb ? sp[k] : 0;
    if (k < nb && pr >= ke) {
      const double t = M[(size_t)pr * st];
      M[(size_t)pr * st] = u[k];
      u[k] = t;
    }
#pragma unroll
    for (int r = k + 1; r < kNb; ++r)
      if (k < nb && r == pr - kb) { const double t = u[k]; u[k] = u[r]; u[r] = t; }
  }
  if (j >= ke) {
#pragma unroll
    for (int r = 1; r < kNb; ++r)
      if (r < nb)
#pragma unroll
        for (int t = 0; t < r; ++t) u[r] = fma(-L[r][t], u[t], u[r]);
  }
#pragma unroll
  for (int r = 0; r < kNb; ++r)
    if (r < nb) M[(size_t)(kb + r) * st] = u[r];
}

// Trailing matrix (extra row and column included) -= L21 U12; blockIdx.z = problem.
__global__ void __launch_bounds__(256)
lu_update_kernel(LuBatch B, int c, int kb, int nb) {
  __shared__ double Ls[kTile][kNb + 1];
  __shared__ double Us[kNb][kTile];
  const uint32_t p = blockIdx.z;
  if (B.active && !B.active[p]) return;
  double *A = B.A + (size_t)p * B.a_stride;
  double *row = B.row ? B.row + (size_t)p * B.v_stride : nullptr;
  double *col = B.col ? B.col + (size_t)p * B.v_stride : nullptr;
  const int ke = kb + nb, i0 = ke + (int)blockIdx.y * kTile, j0 = ke + (int)blockIdx.x * kTile;
  const int ni = c + (row ? 1 : 0), nj = c + (col ? 1 : 0);
  const int tid = (int)threadIdx.x;
  {
    const int i = i0 + tid / kNb, k = tid % kNb;   // 256 = kTile * kNb
    Ls[tid / kNb][k] = (i < ni && k < nb) ? (i == c ? row[kb + k] : A[(size_t)i * c + kb + k]) : 0.0;
    const int k2 = tid / kTile, j = j0 + tid % kTile;
    Us[k2][tid % kTile] =
        (j < nj && k2 < nb) ? (j == c ? col[kb + k2] : A[(size_t)(kb + k2) * c + j]) : 0.0;
  }
  __syncthreads();
  const int tx = tid % kTile, ty = tid / kTile;    // a column, rows ty, ty + 8, ..
  const int j = j0 + tx;
  if (j >= nj) return;
#pragma unroll
  for (int a = 0; a < kTile / 8; ++a) {
    const int ii = ty + 8 * a, i = i0 + ii;
    if (i >= ni || (i == c && j == c)) continue;
    double *x = i == c ? row + j : j == c ? col + i : A + (size_t)i * c + j;
    double acc = *x;
#pragma unroll
    for (int k = 0; k < kNb; ++k) acc = fma(-Ls[ii][k], Us[k][tx], acc);
    *x = acc;
  }
}

}  // namespace

cudaError_t launch_lu(const LuBatch &B, int32_t c, int32_t count, int smem_optin,
                      cudaStream_t stream) {
  if (c <= 0 || count <= 0) return cudaSuccess;
  const size_t cap = (size_t)std::max(0, smem_optin - kPanelStatic);
  const bool single = c <= kSingle && panel_bytes(c + 1, c + 1) <= cap;
  for (int kb = 0; kb < c;) {
    const int nb = single ? c : std::min(kNb, c - kb), ke = kb + nb;
    const int last = ke >= c ? 1 : 0;
    const size_t bytes = panel_bytes(c - kb + 1, nb + last);
    if (bytes <= cap) {
      allow_shared(reinterpret_cast<const void *>(lu_panel_kernel<true>), kPanelStatic);
      lu_panel_kernel<true><<<count, kPanelThreads, bytes, stream>>>(B, c, kb, nb, last);
    } else {
      lu_panel_kernel<false><<<count, kPanelThreads, 0, stream>>>(B, c, kb, nb, last);
    }
    const int others = c - nb + (B.col && !last ? 1 : 0);
    if (others > 0)
      lu_rows_kernel<<<dim3((unsigned)((others + 127) / 128), (unsigned)count), 128, 0, stream>>>(
          B, c, kb, nb, last);
    if (!last) {
      const unsigned tj = (unsigned)((c - ke + (B.col ? 1 : 0) + kTile - 1) / kTile);
      const unsigned ti = (unsigned)((c - ke + (B.row ? 1 : 0) + kTile - 1) / kTile);
      lu_update_kernel<<<dim3(tj, ti, (unsigned)count), 256, 0, stream>>>(B, c, kb, nb);
    }
    kb = ke;
  }
  return cudaGetLastError();
}

}  // namespace afc
