// dense_lu.cuh -- the device-wide LU's batch description (dense_lu.cu) and the triangular solves
// that finish a system whose right-hand side went through the elimination; the solves run on one
// CTA of whole warps and all its threads must call them together.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace afc {

// Problem p's matrix at A + p a_stride (row-major c x c, factored in place), its vectors at
// p v_stride; row / col: right-hand sides (or null, see dense_lu.cu); active: problems with 0 are
// skipped (or null); status gets kErrSolve when a pivot column is zero.
struct LuBatch {
  double *A;
  size_t a_stride;
  int32_t *piv;
  size_t v_stride;
  double *row, *col;
  const uint32_t *active;
  uint32_t *status;
};

// Factors `count` c x c matrices; asynchronous on `stream`.
cudaError_t launch_lu(const LuBatch &B, int32_t c, int32_t count, int smem_optin,
                      cudaStream_t stream);

// Scratch of the solves: the diagonal block, scaled, in shared memory.
struct TriScratch {
  double d[32][33];
  double x[32], inv[32];
};

// U x = b in place (b: generic pointer).  Blocks of 32: the CTA stages the diagonal block divided
// by its diagonal, warp 0 solves it (one multiply-add per step: the diagonal is gone), the CTA
// subtracts the block's columns from the rows above.  FP64 bound (c^2 / 2 FMA on one SM).
__device__ inline void upper_solve(const double *LU, int32_t c, double *b, TriScratch &s) {
  const int tid = (int)threadIdx.x, lane = tid & 31, nt = (int)blockDim.x;
  for (int32_t kb = ((c - 1) / 32) * 32; kb >= 0; kb -= 32) {
    const int nb = min(32, c - kb);
    __syncthreads();   // b complete, the scratch free
    for (int q = tid; q < 32 * 32; q += nt) {
      const int i = q >> 5, j = q & 31;
      s.d[i][j] = (i < nb && j < nb && j >= i) ? LU[(size_t)(kb + i) * c + kb + j] : 0.0;
    }
    __syncthreads();
    if (tid < 32) s.inv[lane] = lane < nb ? 1.0 / s.d[lane][lane] : 0.0;
    __syncthreads();
    for (int q = tid; q < 32 * 32; q += nt) {
      const int i = q >> 5, j = q & 31;
      s.d[i][j] = j > i ? s.d[i][j] * s.inv[i] : 0.0;
    }
    __syncthreads();
    if (tid < 32) {
      double v = lane < nb ? b[kb + lane] * s.inv[lane] : 0.0;
      for (int i = nb - 1; i > 0; --i) {
        const double xi = __shfl_sync(0xFFFFFFFFu, v, i);
        v = fma(-s.d[lane][i], xi, v);   // 0 up to the diagonal
      }
      s.x[lane] = v;
      if (lane < nb) b[kb + lane] = v;
    }
    __syncthreads();
    for (int32_t i = tid; i < kb; i += nt) {
      const double *u = LU + (size_t)i * c + kb;
      double acc = b[i];
      if (nb == 32) {
#pragma unroll 8
        for (int t = 0; t < 32; ++t) acc = fma(-u[t], s.x[t], acc);
      } else {
        for (int t = 0; t < nb; ++t) acc = fma(-u[t], s.x[t], acc);
      }
      b[i] = acc;
    }
  }
  __syncthreads();
}

// L^T w = b in place, then the row swaps undone (x = P^T w); L unit lower.
__device__ inline void lower_t_solve(const double *LU, int32_t c, const int32_t *piv, double *b,
                                     TriScratch &s) {
  const int tid = (int)threadIdx.x, lane = tid & 31, nt = (int)blockDim.x;
  for (int32_t kb = ((c - 1) / 32) * 32; kb >= 0; kb -= 32) {
    const int nb = min(32, c - kb);
    __syncthreads();
    for (int q = tid; q < 32 * 32; q += nt) {
      const int i = q >> 5, j = q & 31;
      s.d[i][j] = (i < nb && j < i) ? LU[(size_t)(kb + i) * c + kb + j] : 0.0;
    }
    __syncthreads();
    if (tid < 32) {
      double v = lane < nb ? b[kb + lane] : 0.0;
      for (int i = nb - 1; i > 0; --i) {
        const double wi = __shfl_sync(0xFFFFFFFFu, v, i);
        v = fma(-s.d[i][lane], wi, v);   // 0 from the diagonal on
      }
      s.x[lane] = v;
      if (lane < nb) b[kb + lane] = v;
    }
    __syncthreads();
    for (int32_t i = tid; i < kb; i += nt) {
      double acc = b[i];
      if (nb == 32) {
#pragma unroll 8
        for (int t = 0; t < 32; ++t) acc = fma(-LU[(size_t)(kb + t) * c + i], s.x[t], acc);
      } else {
        for (int t = 0; t < nb; ++t) acc = fma(-LU[(size_t)(kb + t) * c + i], s.x[t], acc);
      }
      b[i] = acc;
    }
  }
  int moved = 0;   // usually no row moved (the matrices are close to diagonally dominant)
  for (int32_t k = tid; k < c; k += nt) moved |= piv[k] != k ? 1 : 0;
  moved = __syncthreads_or(moved);
  if (moved && tid == 0)
    for (int32_t k = c - 1; k >= 0; --k) {
      const int32_t p = piv[k];
      if (p != k) { const double t = b[k]; b[k] = b[p]; b[p] = t; }
    }
  __syncthreads();
}

}  // namespace afc
