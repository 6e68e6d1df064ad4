// robust.cu -- robust analysis on the estimated AMC.
//
// Device (Sec. 8 post-processing; uncertainty set of Sec. 5.1):
//   robust_inner_kernel  T_i(v) = inf over q_i in U_i of sum_j q_ij v_j + (1 - sum_j q_ij) v_bot,
//                        U_i the box [(Q0_ij - eps)_+, min(Q0_ij + eps, 1)] (on the row's
//                        support, or on every j) with sum_j q_ij <= 1 - r_min.  A warp per row
//                        solves the LP exactly: every entry starts at its lower bound, then the
//                        budget goes to the entries in ascending order of v_j - v_bot (ties by
//                        j) while that coefficient is negative, each up to its upper bound.  The
//                        order is the same for every row (robust_order_kernel).
//                        robust_inner_in_place_kernel does both in one launch for callers without
//                        room for the order
//   launch_robust_eval   A = I - Q*, its LU over the whole GPU (dense_lu.cu) with f and s in the
//                        elimination, V = A^-1 f and the change of V; the robust value comes from
//                        policy iteration on the host (inner problem at V, evaluate, until V stops
//                        changing)
//   star_kernel          the AFC of the scenario kernel: mu A = s from the last elimination
// Host (Sec. 9 robust experiment): the Wasserstein-1 distance between two node distributions
// under the base graph's hop metric.
//
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <functional>
#include <limits>
#include <queue>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "afc_internal.h"
#include "dense_lu.cuh"
#include "linalg.cuh"

namespace afc {

namespace {

// The transient row of the estimated kernel: Q0_ij = scale_i counts_ij with the assembly's
// row-scale rule.  Returns scale_i; the warp's lanes all get it.
__device__ double row_scale_warp(const uint32_t *row, int32_t n, uint32_t R, double alpha,
                                 double eta) {
  unsigned long long all = 0;
  for (int32_t j = threadIdx.x & 31; j < n; j += 32) all += row[j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
  const double q_sum = (1.0 - alpha) * (double)all / (double)R;
  const double r_i = alpha + (1.0 - alpha) * (double)row[n] / (double)R;
  double scale = (1.0 - alpha) / (double)R;
  if (r_i == 0.0 && q_sum > 0.0) scale *= (1.0 - eta) / q_sum;
  return scale;
}

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}

// v ordered like its value as an unsigned integer (NaN last)
__device__ __forceinline__ unsigned long long sortable(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return v != v ? ~0ull : (b >> 63) ? ~b : b | 0x8000000000000000ull;
}

// order[] = the columns with a negative coefficient cf_j = vsign v_j - vb in ascending (cf, j) and
// *nneg how many: every row of the inner problem spends its budget in this order, so it is made
// once per call (a warp per column counts the columns before it, in integer compares).
__device__ void order_columns(int32_t n, const double *v, double vb, double vsign, int32_t *order,
                              uint32_t warp, uint32_t nwarps) {
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t j = warp; j < (uint32_t)n; j += nwarps) {
    const double cj = vsign * v[j] - vb;
    if (!(cj < 0.0)) continue;
    const unsigned long long kj = sortable(cj);
    uint32_t before = 0;
    for (uint32_t i = lane; i < (uint32_t)n; i += 32) {
      const unsigned long long ki = sortable(vsign * v[i] - vb);
      before += (ki < kj || (ki == kj && i < j)) ? 1u : 0u;
    }
    before = __reduce_add_sync(0xFFFFFFFFu, before);
    if (lane == 0) order[before] = (int32_t)j;
  }
}

// How many columns order_columns placed: the columns with a negative coefficient.
__device__ __forceinline__ uint32_t count_negative(int32_t n, const double *v, double vb, double vsign) {
  uint32_t k = 0;
  for (int32_t j = threadIdx.x & 31; j < n; j += 32) k += vsign * v[j] - vb < 0.0 ? 1u : 0u;
  return __reduce_add_sync(0xFFFFFFFFu, k);
}

// Row i of the inner problem by one warp at the continuation value vsign * (v, v_bot) (vb = vsign
// v_bot, nneg = count_negative): the budget is handed out 32 columns of the common order at a time,
// by a prefix sum of their caps.  (Searching the next column for each row cost n per column: 550 us
// at n = 500.)  Every lane gets T_i.
__device__ double inner_row(uint32_t i, int32_t n, uint32_t R, double alpha, double eta,
                            const uint32_t *counts, double eps, double r_min, int support_only,
                            const double *v, double vb, double vsign, const int32_t *order,
                            uint32_t nneg, double *Qstar, uint32_t *status) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t *row = counts + (size_t)i * ((size_t)n + 1);
  const double scale = row_scale_warp(row, n, R, alpha, eta);
  double *qs = Qstar ? Qstar + (size_t)i * n : nullptr;
  // every entry at its lower bound
  double base = 0.0, low = 0.0;
  for (int32_t j = lane; j < n; j += 32) {
    const uint32_t k = row[j];
    double l = 0.0;
    if (k) {
      const double q = scale * (double)k;
      l = q > eps ? q - eps : 0.0;
      base += l * (vsign * v[j] - vb);
      low += l;
    }
    if (qs) qs[j] = l;
  }
  base = warp_sum_d(base);
  low = warp_sum_d(low);
  __syncwarp();   // the lower bounds written by every lane, before the budget is added
  double budget = (1.0 - r_min) - low;
  if (budget < -1e-12) {
    if (lane == 0) atomicOr(status, kErrInput);   // U_i is empty
    budget = 0.0;
  }
  // the budget to the most negative coefficients first, each entry up to its upper bound
  double acc = 0.0;
  for (uint32_t k0 = 0; k0 < nneg && budget > 0.0; k0 += 32) {
    const uint32_t k = k0 + lane;
    int32_t j = 0;
    double cap = 0.0;
    if (k < nneg) {
      j = order[k];
      const double q = scale * (double)row[j];
      if (q > 0.0) cap = fmin(q + eps, 1.0) - (q > eps ? q - eps : 0.0);
      else if (!support_only) cap = fmin(eps, 1.0);
      if (!(cap > 0.0)) cap = 0.0;
    }
    if (!__any_sync(0xFFFFFFFFu, cap > 0.0)) continue;
    double incl = cap;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    double before = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
    if (lane == 0) before = 0.0;
    const double d = fmin(cap, fmax(budget - before, 0.0));
    if (d > 0.0) {
      acc += d * (vsign * v[j] - vb);
      if (qs) qs[j] += d;
    }
    budget -= __shfl_sync(0xFFFFFFFFu, incl, 31);
  }
  return vsign * (vb + base + warp_sum_d(acc));
}

// The rows warp, warp + nwarps, ...
__device__ void inner_rows(int32_t n, uint32_t R, double alpha, double eta,
                           const uint32_t *counts, double eps, double r_min, int support_only,
                           const double *v, double v_bot, double vsign, const int32_t *order,
                           double *T, double *Qstar, uint32_t *status, uint32_t warp,
                           uint32_t nwarps) {
  if (warp >= (uint32_t)n) return;
  const double vb = vsign * v_bot;
  const uint32_t nneg = count_negative(n, v, vb, vsign);
  for (uint32_t i = warp; i < (uint32_t)n; i += nwarps) {
    const double t = inner_row(i, n, R, alpha, eta, counts, eps, r_min, support_only, v, vb, vsign,
                               order, nneg, Qstar, status);
    if ((threadIdx.x & 31u) == 0) T[i] = t;
  }
}

// Waits until every CTA of a cooperative launch has come this far (arrived: 0 at the launch; want:
// CTAs times the barriers so far).  False after about a second without them.
__device__ bool grid_barrier(uint32_t *arrived, uint32_t want) {
  __shared__ int met;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(arrived, 1u);
    int ok = 0;
    for (uint32_t k = 0; k < (1u << 24) && !ok; ++k) {
      ok = *reinterpret_cast<volatile uint32_t *>(arrived) >= want;
      if (!ok) __nanosleep(64);
    }
    met = ok;
    __threadfence();
  }
  __syncthreads();
  return met != 0;
}

constexpr uint32_t kKeptRows = 64;   // rows per warp of the kernel below

// The whole inner problem (vsign 1) without scratch of its own: the order of the columns, 4 n bytes,
// stands in T until every row is done, and the rows' values wait in registers (lane k of a warp
// keeps its rows k and k + 32).  One cooperative launch of at least n / (8 kKeptRows) CTAs of 8 warps.
// A call takes 54 us at n = 500 and 279 at n = 3,000 (with the order in an allocation of the call's
// own and two launches: 182 and 440).
__global__ void __launch_bounds__(256)
robust_inner_in_place_kernel(int32_t n, uint32_t R, double alpha, double eta, const uint32_t *counts,
                             double eps, double r_min, int support_only, const double *v, double vb,
                             double *T, double *Qstar, uint32_t *status, uint32_t *arrived) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  int32_t *order = reinterpret_cast<int32_t *>(T);
  order_columns(n, v, vb, 1.0, order, warp, nwarps);
  bool ok = grid_barrier(arrived, gridDim.x);
  double kept[2] = {0.0, 0.0};
  if (ok && warp < (uint32_t)n) {
    const uint32_t nneg = count_negative(n, v, vb, 1.0);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      for (uint32_t k = 0; k < 32; ++k) {
        const uint32_t i = warp + (32u * h + k) * nwarps;
        if (i >= (uint32_t)n) break;
        const double t = inner_row(i, n, R, alpha, eta, counts, eps, r_min, support_only, v, vb, 1.0,
                                   order, nneg, Qstar, status);
        if (lane == k) kept[h] = t;
      }
  }
  ok = grid_barrier(arrived, 2 * gridDim.x) && ok;   // every row has read the order
  if (!ok && threadIdx.x == 0) atomicOr(status, kErrPassLimit);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t i = warp + (32u * h + lane) * nwarps;
    if (ok && i < (uint32_t)n) T[i] = kept[h];
  }
}

__global__ void robust_order_kernel(int32_t n, const double *v, double v_bot, double vsign,
                                    int32_t *order) {
  order_columns(n, v, vsign * v_bot, vsign, order, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                (gridDim.x * blockDim.x) >> 5);
}

__global__ void robust_inner_kernel(int32_t n, uint32_t R, double alpha, double eta,
                                    const uint32_t *counts, double eps, double r_min,
                                    int support_only, const double *v, double v_bot, double vsign,
                                    const int32_t *order, double *T, double *Qstar,
                                    uint32_t *status) {
  inner_rows(n, R, alpha, eta, counts, eps, r_min, support_only, v, v_bot, vsign, order, T, Qstar,
             status, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
             (gridDim.x * blockDim.x) >> 5);
}

// A = I - Q*, and the right-hand sides the elimination carries: x = f (1 when null), mu = s
// (uniform when null).
__global__ void build_a_kernel(int32_t n, const double *Qstar, const double *f, const double *s,
                               double *A, double *x, double *mu) {
  const size_t nn = (size_t)n * n;
  const size_t k0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (size_t k = k0; k < nn; k += (size_t)gridDim.x * blockDim.x)
    A[k] = ((k / n) == (k % n) ? 1.0 : 0.0) - Qstar[k];
  for (size_t k = k0; k < (size_t)n; k += (size_t)gridDim.x * blockDim.x) {
    x[k] = f ? f[k] : 1.0;
    mu[k] = s ? s[k] : 1.0 / (double)n;
  }
}

// One CTA: V_new = U^-1 x (x = L^-1 P f from the elimination), diff = max |V_new - V| relative to
// max |V_new|, V <- V_new.
__device__ void eval_body(int32_t n, const double *A, double *V, double *x, double *diff,
                          TriScratch &tri, double *red) {
  upper_solve(A, n, x, tri);
  double m = 0.0, scale = 1.0;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
    m = fmax(m, fabs(x[i] - V[i]));
    scale = fmax(scale, fabs(x[i]));
  }
  m = block_max(m, red);
  scale = block_max(scale, red);
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) V[i] = x[i];
  if (threadIdx.x == 0) *diff = m / scale;
}

__global__ void __launch_bounds__(1024, 1)
eval_kernel(int32_t n, const double *A, double *V, double *x, double *diff) {
  __shared__ TriScratch tri;
  __shared__ double red[33];
  eval_body(n, A, V, x, diff, tri, red);
}

// The AFC of the scenario kernel from the last elimination (mu = s U^-1): L^T mu, out[0] = E_s[T]
// = sum mu, out[1] = b . f (f = 1 when null gives 1).
__global__ void __launch_bounds__(1024, 1)
star_kernel(int32_t n, const double *A, const int32_t *piv, const double *f, double *mu, double *b,
            double *out) {
  __shared__ TriScratch tri;
  __shared__ double red[33];
  lower_t_solve(A, n, piv, mu, tri);
  double t = 0.0, tf = 0.0;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
    t += mu[i];
    tf += mu[i] * (f ? f[i] : 1.0);
  }
  const double T = block_sum(t, red);
  const double TF = block_sum(tf, red);
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) b[i] = mu[i] / T;
  if (threadIdx.x == 0) { out[0] = T; out[1] = TF / T; }
}

// ---- batched robust problems (the envelopes): problem p's arrays at p times the stride ----

__global__ void order_batched_kernel(int32_t n, const EnvBatch B) {
  const uint32_t p = blockIdx.y;
  if (!B.active[p]) return;
  order_columns(n, B.V + p * B.vstride, 0.0, B.vsign[p], B.piv + p * B.vstride,
                (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5);
}

// inner problem of every active problem (blockIdx.y = problem)
__global__ void inner_batched_kernel(int32_t n, uint32_t R, double alpha, double eta,
                                     const uint32_t *counts, double eps, double r_min,
                                     int support_only, const EnvBatch B, uint32_t *status) {
  const uint32_t p = blockIdx.y;
  if (!B.active[p]) return;
  const size_t nn = (size_t)n * n;
  inner_rows(n, R, alpha, eta, counts, eps, r_min, support_only, B.V + p * B.vstride, 0.0,
             B.vsign[p], B.piv + p * B.vstride, B.T + p * B.vstride, B.Qs + p * nn, status,
             (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5);
}

// every active problem's A = I - Q* and right-hand sides: x = f_p, and T (the inner values are no
// longer needed) = s
__global__ void build_a_batched_kernel(int32_t n, const EnvBatch B, const double *s) {
  const uint32_t p = blockIdx.y;
  if (!B.active[p]) return;
  const size_t nn = (size_t)n * n;
  const double *Qs = B.Qs + p * nn;
  double *A = B.A + p * nn;
  const size_t k0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (size_t k = k0; k < nn; k += (size_t)gridDim.x * blockDim.x)
    A[k] = ((k / n) == (k % n) ? 1.0 : 0.0) - Qs[k];
  for (size_t k = k0; k < (size_t)n; k += (size_t)gridDim.x * blockDim.x) {
    B.x[p * B.vstride + k] = B.f[p * B.vstride + k];
    B.T[p * B.vstride + k] = s ? s[k] : 1.0 / (double)n;
  }
}

// one CTA per active problem: V <- U^-1 x, diff
__global__ void __launch_bounds__(1024, 1) eval_batched_kernel(int32_t n, const EnvBatch B) {
  __shared__ TriScratch tri;
  __shared__ double red[33];
  const uint32_t p = blockIdx.x;
  if (!B.active[p]) return;
  eval_body(n, B.A + p * (size_t)n * n, B.V + p * B.vstride, B.x + p * B.vstride, B.diff + p, tri,
            red);
}

// one CTA per active problem: the visits mu of its kernel (L^T mu from the last elimination),
// ratio[p] = mu_v / sum mu = b_v for the problem's node v
__global__ void __launch_bounds__(1024, 1)
star_batched_kernel(int32_t n, const EnvBatch B) {
  __shared__ TriScratch tri;
  __shared__ double red[33];
  const uint32_t p = blockIdx.x;
  if (!B.active[p]) return;
  double *mu = B.T + p * B.vstride;
  lower_t_solve(B.A + p * (size_t)n * n, n, B.piv + p * B.vstride, mu, tri);
  double t = 0.0;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) t += mu[i];
  const double T = block_sum(t, red);
  if (threadIdx.x == 0) B.ratio[p] = mu[B.node[p]] / T;
}

// f_p = e_v - lambda_p for every active problem
__global__ void env_reward_kernel(int32_t n, uint32_t P, const EnvBatch B) {
  const size_t total = (size_t)P * n;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < total;
       k += (size_t)gridDim.x * blockDim.x) {
    const uint32_t p = (uint32_t)(k / n);
    const int32_t j = (int32_t)(k % n);
    if (!B.active[p]) continue;
    B.f[p * B.vstride + j] = (j == B.node[p] ? 1.0 : 0.0) - B.lambda[p];
    B.V[p * B.vstride + j] = 0.0;
  }
}

}  // namespace

cudaError_t launch_env_reward(int32_t n, uint32_t P, const EnvBatch &B, cudaStream_t stream) {
  const size_t total = (size_t)P * n;
  const int grid = (int)std::max<size_t>(1, std::min<size_t>((total + 255) / 256, 4096));
  env_reward_kernel<<<grid, 256, 0, stream>>>(n, P, B);
  return cudaGetLastError();
}

cudaError_t launch_env_round(int32_t n, uint32_t R, double alpha, double eta,
                             const uint32_t *counts, double eps, double r_min, int support_only,
                             uint32_t P, const EnvBatch &B, const double *s, uint32_t *status,
                             int smem_optin, cudaStream_t stream) {
  const dim3 grid((unsigned)std::min<int64_t>(((int64_t)n + 7) / 8, 1024), P);
  order_batched_kernel<<<grid, 256, 0, stream>>>(n, B);
  inner_batched_kernel<<<grid, 256, 0, stream>>>(n, R, alpha, eta, counts, eps, r_min,
                                                 support_only, B, status);
  const dim3 agrid((unsigned)std::min<int64_t>(((int64_t)n * n + 1023) / 1024, 1024), P);
  build_a_batched_kernel<<<agrid, 256, 0, stream>>>(n, B, s);
  const LuBatch L{B.A, (size_t)n * n, B.piv, B.vstride, B.T, B.x, B.active, status};
  cudaError_t e = launch_lu(L, n, (int32_t)P, smem_optin, stream);
  if (e != cudaSuccess) return e;
  eval_batched_kernel<<<P, 1024, 0, stream>>>(n, B);
  return cudaGetLastError();
}

cudaError_t launch_env_ratio(int32_t n, uint32_t P, const EnvBatch &B, cudaStream_t stream) {
  star_batched_kernel<<<P, 1024, 0, stream>>>(n, B);
  return cudaGetLastError();
}

cudaError_t launch_robust_inner(int32_t n, uint32_t R, double alpha, double eta,
                                const uint32_t *counts, double eps, double r_min,
                                int support_only, const double *v, double v_bot, double vsign,
                                int32_t *order, double *T, double *Qstar, uint32_t *status,
                                cudaStream_t stream) {
  const int grid = (int)std::min<int64_t>(((int64_t)n + 7) / 8, 1024);
  robust_order_kernel<<<grid, 256, 0, stream>>>(n, v, v_bot, vsign, order);
  robust_inner_kernel<<<grid, 256, 0, stream>>>(n, R, alpha, eta, counts, eps, r_min,
                                                support_only, v, v_bot, vsign, order, T, Qstar,
                                                status);
  return cudaGetLastError();
}

cudaError_t launch_robust_inner_in_place(int32_t n, uint32_t R, double alpha, double eta,
                                         const uint32_t *counts, double eps, double r_min,
                                         int support_only, const double *v, double v_bot, double *T,
                                         double *Qstar, uint32_t *status, uint32_t *arrived,
                                         int num_sms, cudaStream_t stream) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, robust_inner_in_place_kernel, 256, 0);
  if (e != cudaSuccess) return e;
  const int64_t fit = (int64_t)std::max(1, per_sm) * std::max(1, num_sms);
  const int64_t grid = std::min<int64_t>(((int64_t)n + 7) / 8, fit);
  if ((int64_t)n > grid * 8 * kKeptRows) return cudaErrorInvalidConfiguration;   // counts beyond 280 GB
  void *args[] = {&n, &R, &alpha, &eta, &counts, &eps, &r_min, &support_only, &v, &v_bot, &T, &Qstar,
                  &status, &arrived};
  e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(robust_inner_in_place_kernel),
                                  dim3((unsigned)grid), dim3(256), args, 0, stream);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_robust_eval(int32_t n, const double *Qstar, double *A, int32_t *piv,
                               const double *f, const double *s, double *V, double *x, double *mu,
                               double *diff, uint32_t *status, int smem_optin, cudaStream_t stream) {
  const int grid = (int)std::min<int64_t>(((int64_t)n * n + 255) / 256, 4096);
  build_a_kernel<<<grid, 256, 0, stream>>>(n, Qstar, f, s, A, x, mu);
  const LuBatch B{A, 0, piv, 0, mu, x, nullptr, status};
  cudaError_t e = launch_lu(B, n, 1, smem_optin, stream);
  if (e != cudaSuccess) return e;
  eval_kernel<<<1, 1024, 0, stream>>>(n, A, V, x, diff);
  return cudaGetLastError();
}

cudaError_t launch_robust_star(int32_t n, const double *A, const int32_t *piv, const double *f,
                               double *mu, double *b, double *out, cudaStream_t stream) {
  star_kernel<<<1, 1024, 0, stream>>>(n, A, piv, f, mu, b, out);
  return cudaGetLastError();
}

namespace {

// Order of numpy's argmax: a larger value first (NaN above every number), then a smaller index.
__device__ __forceinline__ bool beats(double a, int32_t ia, double b, int32_t ib) {
  const bool na = isnan(a), nb = isnan(b);
  if (na != nb) return na;
  if (!na && a != b) return a > b;
  return ia < ib;
}

// arg[0] = argmax of d1, arg[1] = argmax of d2 (-1 for a NULL array or count 0).
__global__ void __launch_bounds__(256) argmax2_kernel(int32_t count, const double *d1,
                                                      const double *d2, int32_t *arg) {
  __shared__ double sv[256];
  __shared__ int32_t si[256];
  const int t = threadIdx.x;
  for (int w = 0; w < 2; ++w) {
    const double *d = w ? d2 : d1;
    if (!d) {
      if (t == 0) arg[w] = -1;
      continue;
    }
    double bv = 0.0;
    int32_t bi = -1;
    for (int32_t k = t; k < count; k += blockDim.x) {
      const double x = d[k];
      if (bi < 0 || beats(x, k, bv, bi)) {
        bv = x;
        bi = k;
      }
    }
    sv[t] = bv;
    si[t] = bi;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
      if (t < s && si[t + s] >= 0 && (si[t] < 0 || beats(sv[t + s], si[t + s], sv[t], si[t]))) {
        sv[t] = sv[t + s];
        si[t] = si[t + s];
      }
      __syncthreads();
    }
    if (t == 0) arg[w] = si[0];
    __syncthreads();
  }
}

// Sampled envelopes: lo[v] / hi[v] = the smallest / largest of b0[v] and rows[k][v].
__global__ void envelope_kernel(int32_t n, int32_t count, const double *rows, const double *b0,
                                double *lo, double *hi) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    double a = b0[v], z = a;
    for (int32_t k = 0; k < count; ++k) {
      const double x = rows[(size_t)k * (size_t)n + v];
      a = fmin(a, x);
      z = fmax(z, x);
    }
    if (lo) lo[v] = a;
    if (hi) hi[v] = z;
  }
}

}  // namespace

cudaError_t launch_robust_summary(int32_t n, int32_t count, const double *rows, const double *b0,
                                  const double *d1, const double *d2, int32_t *arg, double *lo,
                                  double *hi, cudaStream_t stream) {
  if (arg) argmax2_kernel<<<1, 256, 0, stream>>>(count, d1, d2, arg);
  if (lo || hi) {
    const int grid = std::max(1, std::min((n + 255) / 256, 1024));
    envelope_kernel<<<grid, 256, 0, stream>>>(n, count, rows, b0, lo, hi);
  }
  return cudaGetLastError();
}

// W1 on a graph metric is an uncapacitated transshipment problem on the graph itself (each
// unit of mass moved across an edge costs 1).  It is solved exactly by successive shortest
// paths: node potentials keep the reduced arc costs non-negative, each round runs a
// multi-source Dijkstra from every node with excess mass and stops at the first node with a
// deficit, then pushes as much as the path allows (the source's excess, the sink's deficit,
// the flow on any arc the path cancels).  Costs are integers, so distances and potentials are
// exact; the masses are doubles and are settled to within a relative 1e-14.
double w1_graph_host(int32_t n, const int32_t *rp, const int32_t *col, const int32_t *eid,
                     const double *x, const double *y) {
  const int32_t arcs = rp[n];
  // partner arc of every arc (the other direction of the same edge)
  std::vector<int32_t> rev(std::max<int32_t>(arcs, 1), -1);
  int32_t maxe = 0;
  for (int32_t a = 0; a < arcs; ++a) maxe = std::max(maxe, eid[a] + 1);
  std::vector<int32_t> seen((size_t)maxe, -1);
  for (int32_t a = 0; a < arcs; ++a) {
    const int32_t e = eid[a];
    if (seen[e] < 0) { seen[e] = a; } else { rev[a] = seen[e]; rev[seen[e]] = a; }
  }
  std::vector<double> ex(n), flow(std::max<int32_t>(arcs, 1), 0.0);
  double scale = 0.0;
  for (int32_t v = 0; v < n; ++v) {
    ex[v] = x[v] - y[v];
    scale = std::max(scale, std::fabs(ex[v]));
  }
  const double tol = 1e-14 * std::max(scale, 1e-300);
  std::vector<int64_t> pot(n, 0), dist(n);
  std::vector<int32_t> par(n);        // arc into the node on the shortest path (-1: a source)
  std::vector<int32_t> pnode(n);      // the node that arc leaves
  std::vector<uint8_t> cancel(n), done(n);
  using Item = std::pair<int64_t, int32_t>;
  const int64_t kInf = std::numeric_limits<int64_t>::max() / 4;
  double cost = 0.0;
  for (int32_t guard = 0; guard < 8 * n + 8 * arcs + 64; ++guard) {
    std::priority_queue<Item, std::vector<Item>, std::greater<Item>> pq;
    std::fill(dist.begin(), dist.end(), kInf);
    std::fill(done.begin(), done.end(), 0);
    for (int32_t v = 0; v < n; ++v)
      if (ex[v] > tol) { dist[v] = 0; par[v] = -1; pq.push({0, v}); }
    if (pq.empty()) break;
    int32_t t = -1;
    while (!pq.empty()) {
      const auto [d, u] = pq.top();
      pq.pop();
      if (done[u] || d != dist[u]) continue;
      done[u] = 1;
      if (ex[u] < -tol) { t = u; break; }
      for (int32_t a = rp[u]; a < rp[u + 1]; ++a) {
        const int32_t v = col[a];
        // cancelling flow on v -> u costs -1, a new unit on u -> v costs +1
        const bool can = rev[a] >= 0 && flow[rev[a]] > tol;
        const int64_t nd = d + (can ? -1 : 1) + pot[u] - pot[v];
        if (nd < dist[v]) {
          dist[v] = nd; par[v] = a; pnode[v] = u; cancel[v] = can ? 1 : 0;
          pq.push({nd, v});
        }
      }
    }
    if (t < 0) break;   // mass left without a reachable deficit (disconnected support)
    const int64_t dt = dist[t];
    for (int32_t v = 0; v < n; ++v) pot[v] += done[v] ? dist[v] : dt;
    // bottleneck along the path t <- ... <- s
    double delta = -ex[t];
    int32_t v = t;
    while (par[v] >= 0) {
      if (cancel[v]) delta = std::min(delta, flow[rev[par[v]]]);
      v = pnode[v];
    }
    delta = std::min(delta, ex[v]);
    const int32_t s = v;
    for (v = t; par[v] >= 0; v = pnode[v]) {
      const int32_t a = par[v];
      if (cancel[v]) { flow[rev[a]] -= delta; cost -= delta; }
      else { flow[a] += delta; cost += delta; }
    }
    ex[s] -= delta;
    ex[t] += delta;
  }
  return cost;
}

}  // namespace afc
