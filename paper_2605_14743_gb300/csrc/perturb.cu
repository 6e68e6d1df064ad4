// perturb.cu -- A9: row-wise perturbation sweep of the estimated kernel (Sec. 5.1 row-wise
// uncertainty, Sec. 5.4 first-order sensitivity, Sec. 5.5 ranking reversals), with the l1 row
// model or the multiplicative one of the robust experiment (Sec. 9), and KL(b' || b0) per
// perturbation for the sampled robust search (Remark on the robust optimisation viewpoint).
//
// One CTA handles one perturbation p at a time (persistent over p).  The perturbation is
// regenerated from Philox (counter (column, row, p, 1)), never stored as a matrix: every row i is
// moved on its support J_i (transient columns in C plus the absorbing column).  With
// D = sum_U s_i (q'_i - q_i) the perturbed reduced systems are (I - Q'_CC)^T mu'_C = y0 + D and
// (I - Q'_CC) t = 1, solved by defect correction (below); the ranking of the perturbed AFC b' is
// compared with the nominal one.
//
// What bounds it: GB300's FP64 pipe takes 16 cycles per warp instruction and SM (2 lanes a clock),
// 64 times an FP32 or integer one.  So FP64 is kept for what reaches a result and the rest runs in
// integers or FP32: a draw's shift is an exact 64-bit integer turned into a double by integer
// instructions, whether anything clips or reaches the floor is decided in FP32 with a margin (inside it
// in FP64), and an unclipped entry costs one FP64 multiply-add.  The rows' (N' 1)_i are screened in FP32; the ones that can be the
// maximum are computed in FP64.  Measured, before (8 FP64 operations per entry, a factorisation or
// two chains of triangular solves per round, (N' 1) by a thread per row) and now: c = 97, n = 1,000,
// 2,000 perturbations 13.4 -> 4.7 ms; c = 751, n = 3,000, 304 perturbations 30.8 -> 8.2 ms, its
// kernel with the FP64 pipe 47% and issue 31% active (16 warps per SM wait for loads and chains).
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "afc_device.cuh"
#include "afc_internal.h"
#include "linalg.cuh"

namespace afc {

// Two resident CTAs per SM: one perturbation's solves are barrier-bound, so two overlap their waits.
// 512 threads where the matrix fits shared memory (c up to 162: the rows' chains of dependent loads
// and reductions want warps; 64 registers), 256 beyond (every warp has its own column sums, and the
// blocked factorisation's tiles want 256).
constexpr int kPerturbCtasPerSm = 2;
constexpr int kThreadsOnChip = 512, kThreadsSlab = 256;
__host__ __device__ constexpr int sweep_threads(bool on_chip) { return on_chip ? kThreadsOnChip : kThreadsSlab; }
constexpr int kMaxK2 = 32;
constexpr int kMaxHist = 64;
constexpr int kSweepStatic = 8 * 1024;   // at least the sweep kernel's static arrays

// Leading dimension of the FP32 inverse: whole 128-byte lines, padded with zeros.
__host__ __device__ inline size_t inv_ld(int32_t c) { return ((size_t)(c > 0 ? c : 1) + 31) & ~size_t(31); }

size_t perturb_inverse_bytes(int32_t c) { return 2 * sizeof(float) * (size_t)(c > 0 ? c : 1) * inv_ld(c); }

__host__ __device__ inline size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

// One CTA's device slab (byte offsets): c-vectors, the perturbed C rows (FP64, c + 1 apart), the
// other rows (FP32) and the dense matrix of the factorisation fallback.  The fallback's FP32 copy
// takes the C rows' place: they are in the matrix by then, and the next perturbation writes them
// anew.  (With a place of its own a chain of 9,000 observed states needed 298 GB of slabs instead of
// 248, and one of 1,200 had room for one CTA per SM instead of two.)
struct SweepSlab {
  size_t A, piv, by, rv, x, xt, z, yp, vec, sf, qp, qf, total;
};
// Entries of a warp's draw buffer: the longest row, in whole warps (none below the register form).
__host__ __device__ inline size_t draw_ld(int32_t c) { return c + 1 <= 128 ? 0 : ((size_t)c + 32) & ~size_t(31); }
// The per-CTA vectors that live in shared memory when they fit: column sums of every warp, mu',
// t, two FP32 vectors of inv_ld floats and every warp's buffer of a row's draws.
__host__ __device__ inline size_t vec_bytes(int32_t c, int threads) {
  const size_t cc = (size_t)(c > 0 ? c : 1);
  return 8 * ((size_t)threads / 32 + 2) * cc + 2 * 4 * inv_ld(c) + 4 * ((size_t)threads / 32) * draw_ld(c);
}
__host__ __device__ inline SweepSlab sweep_slab(int32_t n, int32_t c) {
  const size_t cc = (size_t)(c > 0 ? c : 1), nn = (size_t)n;
  SweepSlab s{};
  size_t o = 0;
  s.piv = o; o = up256(o + 4 * cc);
  s.by = o;  o = up256(o + 8 * cc);
  s.rv = o;  o = up256(o + 8 * cc);
  s.x = o;   o = up256(o + 8 * cc);
  s.xt = o;  o = up256(o + 8 * cc);
  s.z = o;   o = up256(o + 8 * cc);
  s.yp = o;  o = up256(o + 8 * cc);
  s.vec = o; o = up256(o + vec_bytes(c, kThreadsOnChip));
  s.sf = o;  o = up256(o + 4 * nn);
  s.qp = o;  o = up256(o + 8 * cc * (cc + 1));
  s.qf = o;  o = up256(o + 4 * nn * (cc + 1));
  s.A = o;   o = up256(o + 8 * cc * cc);
  s.total = o;
  return s;
}

size_t perturb_slab_bytes(int32_t n, int32_t c) { return sweep_slab(n, c).total; }

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}

// ---- integer instructions in the place of FP64 ones ---------------------------------------
// The double of an integer below 2^53 in magnitude, exactly.
__device__ __forceinline__ double exact_double(long long d) {
  const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
  const int lz = __clzll((long long)a);   // >= 11
  const unsigned long long m = (a << ((lz - 11) & 63)) + ((unsigned long long)(uint32_t)(1085 - lz) << 52);
  const unsigned long long sign = (unsigned long long)d & 0x8000000000000000ull;
  return a ? __longlong_as_double((long long)(m | sign)) : 0.0;
}

// The same for any 64-bit integer, rounded towards zero.
__device__ __forceinline__ double trunc_double(long long d) {
  const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
  const int lz = __clzll((long long)a);
  const unsigned long long m = ((a << (lz & 63)) >> 11) + ((unsigned long long)(uint32_t)(1085 - lz) << 52);
  const unsigned long long sign = (unsigned long long)d & 0x8000000000000000ull;
  return a ? __longlong_as_double((long long)(m | sign)) : 0.0;
}

// x rounded towards zero to FP32; 0 below 2^-126.  |x| < 2^128.
__device__ __forceinline__ float trunc_f32(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t mag = hi & 0x7FFFFFFFu;
  const uint32_t bits = ((mag - 0x38000000u) << 3) | (lo >> 29);
  return mag < 0x38100000u ? 0.0f : __uint_as_float(bits | (hi & 0x80000000u));
}

// The double of a normal positive float, exactly.
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// 1 / x for positive x within the FP32 range: the FP32 reciprocal (error 2^-22) and one
// third-order step, y (1 + e + e^2) with e = 1 - x y.
__device__ __forceinline__ double recip(double x) {
  const double y = widen(1.0f / trunc_f32(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// floor(2^62 x) of 0 <= x <= 1.
constexpr double kTwoM62 = 1.0 / 4611686018427387904.0;
__device__ __forceinline__ long long fixed62(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int sh = (int)(b >> 52) - 1013;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  return (long long)(sh >= 0 ? m << (sh & 63) : (sh > -64 ? m >> (-sh & 63) : 0ull));
}

// Sum of 64-bit integers over the warp's lanes (modulo 2^64).
__device__ __forceinline__ long long warp_sum_ll(long long x) {
  const uint32_t a = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)x & 0xFFFFFFu);
  const uint32_t b = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(x >> 24) & 0xFFFFFFu);
  const int32_t h = __reduce_add_sync(0xFFFFFFFFu, (int32_t)(x >> 48));
  return (long long)a + ((long long)b << 24) + (long long)((unsigned long long)(long long)h << 48);
}

// ---- ranking ------------------------------------------------------------------------------
// Whether node u precedes node v: bu - bv > tau, or within the band and u < v.  Decided in FP32
// where the difference is clear of the band by more than the truncation; bu is called only
// otherwise.  uf, vf: the values truncated to FP32; ok: both below 2^126 in magnitude.
template <typename Exact>
__device__ __forceinline__ bool precedes(float uf, float vf, float tau_up, bool ok, int32_t u, int32_t v,
                                         double tau, const Exact &diff) {
  const float d = uf - vf;
  const float m = tau_up + 2e-6f * (fabsf(uf) + fabsf(vf)) + 1e-36f;
  if (ok && d > m) return true;
  if (ok && d < -m) return false;
  const double x = diff();
  return x > tau || (fabs(x) <= tau && u < v);
}

__device__ __forceinline__ bool f32_range(double x) {
  return ((uint32_t)__double2hiint(x) & 0x7FFFFFFFu) < 0x47D00000u;
}

// Nominal ranking: rank0[v] = #{u : u precedes v}; byrank0[a] = node of nominal rank a < k2.  A
// warp per node (a thread per node left all but n / 256 SMs idle: 0.8 ms at n = 3,000).
__global__ void __launch_bounds__(256)
nominal_rank_kernel(int32_t n, const double *b0, double tie_rel, int32_t k2, int32_t *rank0,
                    int32_t *byrank0) {
  __shared__ double red[33];
  double mx = 0.0;
  for (int32_t v = threadIdx.x; v < n; v += blockDim.x) mx = fmax(mx, b0[v]);
  mx = block_max(mx, red);
  const double tau = tie_rel * mx;
  const float tau_up = __double2float_ru(tau);
  const int32_t lane = (int32_t)(threadIdx.x & 31u);
  const int32_t nwarps = (int32_t)((gridDim.x * blockDim.x) >> 5);
  for (int32_t v = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); v < n; v += nwarps) {
    const double bv = b0[v];
    const float vf = trunc_f32(bv);
    const bool okv = f32_range(bv);
    int32_t r = 0;
    for (int32_t u = lane; u < n; u += 32) {
      if (u == v) continue;
      const double bu = b0[u];
      r += precedes(trunc_f32(bu), vf, tau_up, okv && f32_range(bu), u, v, tau,
                    [&] { return bu - bv; }) ? 1 : 0;
    }
    r = __reduce_add_sync(0xFFFFFFFFu, r);
    if (lane == 0) {
      rank0[v] = r;
      if (r < k2) atomicMax(&byrank0[r], v);
    }
  }
}

// One CTA per SM's worth of warps at most.
static int rank_grid(int32_t n) { return (int)std::min<int64_t>(((int64_t)n + 7) / 8, 1216); }

constexpr double kTwoM31 = 1.0 / 2147483648.0;   // 2^-31, exact

__device__ __forceinline__ int32_t draw(uint32_t j, uint32_t i, uint32_t p, uint32_t k0, uint32_t k1) {
  return (int32_t)(philox4x32_10(make_uint4(j, i, p, 1u), k0, k1).x - 0x80000000u);
}

// ---- the FP32 inverse of the nominal matrix -------------------------------------------------
// inv = (I - Q_CC)^-1 from the solve's FP64 factors, rounded to FP32, and its transpose; NR columns
// per CTA, blocked substitution with the columns in shared memory.  It only steers the defect
// correction, whose residuals and solutions are FP64; with it a correction is one coalesced
// product instead of two chains of 2 c / 32 dependent blocks.  Once per launch.
constexpr int kInvThreads = 256;
__host__ __device__ inline size_t inverse_smem(int32_t c, int nr) {
  return sizeof(float) * ((((size_t)c * nr + 31) & ~size_t(31)) + 256 * 33 + 2 * 32 * 33);
}

template <int NR>
__global__ void __launch_bounds__(kInvThreads)
inverse32_kernel(const double *lu, const int32_t *piv, int32_t c, size_t ld, float *inv, float *inv_t) {
  extern __shared__ __align__(16) float fsm[];
  float *X = fsm;                                                     // [c][NR]
  float *tile = X + (((size_t)c * NR + 31) & ~size_t(31));            // [256][33]
  float *diag = tile + 256 * 33;                                      // [2][32][33]
  __shared__ int32_t first;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t j0 = (int32_t)blockIdx.x * NR;
  for (int32_t q = tid; q < c * NR; q += kInvThreads) X[q] = 0.0f;
  if (tid == 0) first = c;
  __syncthreads();
  if (tid < NR && j0 + tid < c) {   // the unit vector through the row swaps
    int32_t pos = j0 + tid;
    for (int32_t k = 0; k < c; ++k) {
      const int32_t q = piv[k];
      if (pos == k) pos = q;
      else if (pos == q) pos = k;
    }
    X[pos * NR + tid] = 1.0f;
    atomicMin(&first, pos);
  }
  __syncthreads();
  // diagonal block kb into one of two buffers: the next block's is loaded during the update
  auto stage = [&](int32_t kb, bool lower, float *D) {
    const int nb = min(32, c - kb);
    for (int q = tid; q < 32 * 32; q += kInvThreads) {
      const int i = q >> 5, j = q & 31;
      D[i * 33 + j] = i < nb && j < nb && (lower ? j < i : j >= i)
                          ? trunc_f32(lu[(size_t)(kb + i) * c + kb + j]) : 0.0f;
    }
  };
  // rows [r0, r0 + 256) take their products with the block's NR columns off; a warp stages the
  // rows that its own lanes use
  auto update = [&](int32_t first, int32_t last, int32_t kb, int nb) {
    for (int32_t r0 = first; r0 < last; r0 += kInvThreads) {
      float *mine = tile + warp * 32 * 33;
#pragma unroll 8
      for (int q = 0; q < 32; ++q) {
        const int32_t row = r0 + warp * 32 + q;
        mine[q * 33 + lane] = row < last && lane < nb ? trunc_f32(lu[(size_t)row * c + kb + lane]) : 0.0f;
      }
      __syncwarp();
      const int32_t row = r0 + tid;
      if (row < last) {
        float acc[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = X[row * NR + r];
        for (int t = 0; t < nb; ++t) {
          const float a = mine[lane * 33 + t];
#pragma unroll
          for (int r = 0; r < NR; ++r) acc[r] = fmaf(-a, X[(kb + t) * NR + r], acc[r]);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) X[row * NR + r] = acc[r];
      }
      __syncwarp();
    }
  };
  int buf = 0;
  const int32_t kb0 = first / 32 * 32;   // the columns are zero above
  stage(kb0, true, diag);
  for (int32_t kb = kb0; kb < c; kb += 32) {                          // L, unit lower
    const int nb = min(32, c - kb);
    const float *D = diag + buf * 32 * 33;
    __syncthreads();
    if (warp < NR) {
      float v = lane < nb ? X[(kb + lane) * NR + warp] : 0.0f;
      for (int i = 0; i + 1 < nb; ++i) v = fmaf(-D[lane * 33 + i], __shfl_sync(0xFFFFFFFFu, v, i), v);
      if (lane < nb) X[(kb + lane) * NR + warp] = v;
    }
    __syncthreads();
    buf ^= 1;
    if (kb + 32 < c) stage(kb + 32, true, diag + buf * 32 * 33);
    else stage(kb, false, diag + buf * 32 * 33);   // the last block again, for U
    update(kb + nb, c, kb, nb);
  }
  for (int32_t kb = ((c - 1) / 32) * 32; kb >= 0; kb -= 32) {         // U
    const int nb = min(32, c - kb);
    const float *D = diag + buf * 32 * 33;
    __syncthreads();
    if (warp < NR) {
      const float d = lane < nb ? 1.0f / D[lane * 33 + lane] : 0.0f;
      float v = lane < nb ? X[(kb + lane) * NR + warp] : 0.0f;
      for (int i = nb - 1; i > 0; --i) {
        const float x = __shfl_sync(0xFFFFFFFFu, v * d, i);
        if (lane < i) v = fmaf(-D[lane * 33 + i], x, v);
      }
      if (lane < nb) X[(kb + lane) * NR + warp] = v * d;
    }
    __syncthreads();
    buf ^= 1;
    if (kb > 0) stage(kb - 32, false, diag + buf * 32 * 33);
    update(0, kb, kb, nb);
  }
  __syncthreads();
  for (int32_t q = tid; q < c * NR; q += kInvThreads) {
    const int32_t i = q / NR, r = q % NR;
    if (j0 + r < c) {
      inv[(size_t)i * ld + j0 + r] = X[q];
      inv_t[(size_t)(j0 + r) * ld + i] = X[q];
    }
  }
}

// FP64 iterative refinement with FP32 factors: x <- x + F^-1 (b - op(A) x) until the update
// is below 1e-15 of x (op(A) = A^T when TRANS); b = NULL means all ones.  Since every admissible
// kernel has ||N||_inf <= 1 / r_min, I - Q' is well conditioned and each round gains about
// seven digits.  Returns false when 12 rounds do not get there.
template <bool TRANS>
__device__ bool refine(const double *A, const float *Af, const int32_t *piv, int32_t c,
                       const double *b, double *x, double *r, LinScratch ls, double *red) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int it = 0; it < 12; ++it) {
    if (TRANS) {
      for (int32_t j = threadIdx.x; j < c; j += blockDim.x) {
        double acc = b ? b[j] : 1.0;
        for (int32_t i = 0; i < c; ++i) acc = fma(-A[(size_t)i * c + j], x[i], acc);
        r[j] = acc;
      }
    } else {
      for (int32_t i = warp; i < c; i += nw) {
        double acc = 0.0;
        for (int32_t j = lane; j < c; j += 32) acc = fma(A[(size_t)i * c + j], x[j], acc);
        acc = warp_sum(acc);
        if (lane == 0) r[i] = (b ? b[i] : 1.0) - acc;
      }
    }
    __syncthreads();
    if (TRANS) lu_solve_transposed_blocked_t(Af, c, c, piv, r);
    else lu_solve_blocked_t(Af, c, c, piv, r);
    double dm = 0.0, xm = 0.0;
    for (int32_t k = threadIdx.x; k < c; k += blockDim.x) {
      x[k] += r[k];
      dm = fmax(dm, fabs(r[k]));
      xm = fmax(xm, fabs(x[k]));
    }
    dm = block_max(dm, red);
    xm = block_max(xm, red);
    if (dm <= 1e-15 * xm) return true;
  }
  return false;
}

// ---- the nominal solution's own defects -------------------------------------------------------
// y0 = s_C + s_U Q_UC and the defects rho = y0 - mu0_C (I - Q_CC), rho_t = 1 - (I - Q_CC) t0 of the
// solve's solutions, summed in pairs of doubles: added to the right-hand sides below, they take the
// solve's rounding out of every perturbed solution (1e-15 of it otherwise).  Once per launch.
struct Pair { double h, l; };
__device__ __forceinline__ Pair pair_add(Pair a, double x) {   // Knuth's exact sum
  const double s = a.h + x, b = s - a.h;
  return Pair{s, a.l + ((a.h - (s - b)) + (x - b))};
}
__device__ __forceinline__ Pair pair_fma(Pair a, double x, double y) {
  const double p = x * y;
  a = pair_add(a, p);
  a.l += fma(x, y, -p);
  return a;
}
constexpr int kDefectChunks = 128;

// part [chunks][2][c]: column sums of a chunk of rows, those outside C and those of C.  One CTA per
// chunk, a row at a time (its columns are distinct), from the sparse rows the solve left.
__global__ void __launch_bounds__(256)
nominal_defect_kernel(ChainDev C, const int32_t *nzptr, const int32_t *nzcol, const double *nzval,
                      const double *mu0, Pair *part) {
  const int32_t n = C.n, c = C.c;
  const int32_t per = (n + (int32_t)gridDim.x - 1) / (int32_t)gridDim.x;
  const int32_t i0 = (int32_t)blockIdx.x * per, i1 = min(n, i0 + per);
  Pair *u = part + (size_t)blockIdx.x * 2 * c, *a = u + c;
  const double unif = 1.0 / (double)n;
  for (int32_t k = (int32_t)threadIdx.x; k < 2 * c; k += (int32_t)blockDim.x) u[k] = Pair{0.0, 0.0};
  __syncthreads();
  for (int32_t i = i0; i < i1; ++i) {
    const int32_t e0 = nzptr[i], len = nzptr[i + 1] - 1 - e0;
    const bool in_c = C.c_index[i] >= 0;
    const double w = in_c ? mu0[i] : C.s ? C.s[i] : unif;
    Pair *to = in_c ? a : u;
    for (int32_t k = (int32_t)threadIdx.x; k < len; k += (int32_t)blockDim.x) {
      const int32_t pj = nzcol[e0 + k];
      to[pj] = pair_fma(to[pj], w, nzval[e0 + k]);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ Pair warp_pair_sum(Pair r) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double h = __shfl_xor_sync(0xFFFFFFFFu, r.h, o), l = __shfl_xor_sync(0xFFFFFFFFu, r.l, o);
    r = pair_add(r, h);
    r.l += l;
  }
  return r;
}

// A warp per observed state: its column's parts, and its row's defect rho_t.
__global__ void __launch_bounds__(256)
nominal_finish_kernel(ChainDev C, const double *mu0, const Pair *part, int chunks,
                      const int32_t *nzptr, const int32_t *nzcol, const double *nzval,
                      const double *t0, double *y0, double *rho, double *rho_t) {
  const int32_t c = C.c, lane = (int32_t)(threadIdx.x & 31u);
  const int32_t step = (int32_t)((gridDim.x * blockDim.x) >> 5);
  for (int32_t b = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); b < c; b += step) {
    const int32_t i = C.c_list[b], e0 = nzptr[i], len = nzptr[i + 1] - 1 - e0;
    Pair u{0.0, 0.0}, a{0.0, 0.0}, r{0.0, 0.0};
    for (int k = lane; k < chunks; k += 32) {
      const Pair pu = part[(size_t)k * 2 * c + b], pa = part[((size_t)k * 2 + 1) * c + b];
      u = pair_add(u, pu.h);
      u.l += pu.l;
      a = pair_add(a, pa.h);
      a.l += pa.l;
    }
    for (int32_t k = lane; k < len; k += 32) r = pair_fma(r, nzval[e0 + k], t0[nzcol[e0 + k]]);
    u = warp_pair_sum(u);
    a = warp_pair_sum(a);
    r = pair_add(pair_add(warp_pair_sum(r), 1.0), -t0[b]);
    if (lane == 0) {
      u = pair_add(u, C.s ? C.s[i] : 1.0 / (double)C.n);
      y0[b] = u.h + u.l;
      u = pair_add(pair_add(u, a.h), -mu0[i]);
      rho[b] = u.h + (u.l + a.l);
      rho_t[b] = r.h + r.l;
    }
  }
}

// ---- the perturbed rows ---------------------------------------------------------------------
struct RowArgs {
  const int32_t *nzcol, *c_list;
  const double *nzval;
  int32_t c;
  uint32_t n, p, k0, k1;
  int32_t model;
  double radius, r_min, rel;
  float radius_f, floor_f;       // of the FP32 tests (floor_f: r_min and a margin)
  float screen;                  // margin of the (N' 1) screen, in units of the largest t
  bool always_general;           // the radius is beyond what they cover
};

enum RowMode {
  kRowU,     // row outside C: column sums, FP32 copy
  kRowC,     // row of C: column sums, FP64 copy, sum_j (q'_ij - q_ij) t_j
  kRowDot    // sum_j q'_ij t_j in FP64
};

// Moves row i (entries e0 .. e0 + supp - 1 of the sparse rows, absorption last) by one warp and
// adds w (q' - q) to the columns' sums at acc (own: this warp's own array, else shared by the CTA);
// w_more (q' - q) goes to x_more where more is set.  kRowC returns sum_j (q'_ij - q_ij) t_j, kRowDot
// sum_j q'_ij t_j.  T = 4: a lane holds its entries in registers (rows of up to 128); T = 0: any
// length, the draws wait in the warp's buffer zb.  (Unrolled register forms of 256 and 416 entries
// missed the instruction cache: a third of their stalls.)
//
// l1 model: with d_j = z_j supp - sum_k z_k (z as integers, exact) the shift (z_j - mean)
// l1_radius / ||z - mean||_1 is d_j coef with coef = l1_radius / sum_k |d_k|.  The shifts sum to 0
// and the nominal row to 1, so the row sums to 1 plus what clipping at 0 adds (tot); with the factor
// g = 1 / tot, and (1 - r_min) / (1 - q'_abs) more where the absorption falls below r_min,
//   q' - q = d (coef g) + q (g - 1), and -q where clipped,
// which is one multiply-add for a row that neither clips nor reaches r_min (g = 1) and two for the
// others.  What clips is decided in FP32, in FP64 where that is too close; what clipping adds is
// summed in 64-bit integers.  (Chains estimated from few realizations clip in most rows: entries of
// 0.0004 against shifts of up to 0.0004.)
template <int T, int MODE>
__device__ __forceinline__ double move_row(const RowArgs &R, int32_t i, int32_t e0, int32_t supp,
                                           double w, double *acc, bool own, bool more, double w_more,
                                           double *x_more, float *outf, double *outd,
                                           const double *t, int32_t *zb) {
  constexpr int kUnroll = T > 0 ? T : 2;
  constexpr int TT = T > 0 ? T : 1;
  const int32_t lane = (int32_t)(threadIdx.x & 31u), c = R.c;
  const int nt = T > 0 ? T : (supp + 31) >> 5;
  const int32_t *cols = R.nzcol + e0;
  const double *vals = R.nzval + e0;
  // the lane's entries: column (c: absorption or none), value and shift; T = 0 reads them again
  int32_t col[TT], zi[TT];
  double val[TT], dd[TT];
  long long isum = 0;
  if constexpr (T > 0) {
#pragma unroll
    for (int s = 0; s < T; ++s) {
      const int32_t k = lane + 32 * s;
      col[s] = k < supp ? cols[k] : c;
      val[s] = k < supp ? vals[k] : 0.0;
    }
  }
#pragma unroll (kUnroll)
  for (int s = 0; s < nt; ++s) {
    const int32_t k = lane + 32 * s;
    int32_t z = 0;
    if (k < supp) {
      int32_t pj;
      if constexpr (T > 0) pj = col[s];
      else pj = cols[k];
      if (R.model == 0 || pj < c)
        z = draw(pj < c ? (uint32_t)R.c_list[pj] : R.n, (uint32_t)i, R.p, R.k0, R.k1);
    }
    if (T == 0) zb[k] = z;
    if constexpr (T > 0) zi[s] = z;
    isum += z;
  }
  auto z_of = [&](int s) {
    if constexpr (T > 0) return zi[s];
    else return zb[lane + 32 * s];
  };
  auto col_of = [&](int s) {
    if constexpr (T > 0) return col[s];
    else return lane + 32 * s < supp ? cols[lane + 32 * s] : c;
  };
  auto val_of = [&](int s) {
    if constexpr (T > 0) return val[s];
    else return lane + 32 * s < supp ? vals[lane + 32 * s] : 0.0;
  };
  auto add = [&](int32_t pj, double wt, double d) {
    if (own) acc[pj] = fma(wt, d, acc[pj]);
    else atomicAdd(&acc[pj], wt * d);
  };
  double dot = 0.0;
  if (R.model == 1) {
    // multiplicative: q' = clamp(q (1 + rel z), 0, 1) on the transient entries, scaled to
    // 1 - r_min when above it; the absorption is the remainder
    auto value = [&](int s) {
      return fmin(fmax(val_of(s) * (1.0 + R.rel * (exact_double(z_of(s)) * kTwoM31)), 0.0), 1.0);
    };
    double ts = 0.0;
#pragma unroll (kUnroll)
    for (int s = 0; s < nt; ++s)
      if (col_of(s) < c) ts += value(s);
    ts = warp_sum(ts);
    const double g = ts > 1.0 - R.r_min ? (1.0 - R.r_min) / ts : 1.0;
#pragma unroll (kUnroll)
    for (int s = 0; s < nt; ++s) {
      const int32_t k = lane + 32 * s, pj = col_of(s);
      if (pj >= c) continue;
      const double v = value(s);
      if (MODE == kRowDot) { dot = fma(v, t[pj], dot); continue; }
      const double d = fma(v, g, -val_of(s));
      if (MODE == kRowU) outf[k] = trunc_f32(v) * trunc_f32(g);
      else outd[k] = v * g;
      if (MODE == kRowC) dot = fma(d, t[pj], dot);
      add(pj, w, d);
      if (more) atomicAdd(&x_more[pj], w_more * d);
    }
    return MODE == kRowDot ? g * warp_sum(dot) : MODE == kRowC ? warp_sum(dot) : 0.0;
  }
  const long long S = warp_sum_ll(isum);
  auto shift = [&](int s) { return (long long)z_of(s) * (long long)supp - S; };
  long long dab = 0;
#pragma unroll (kUnroll)
  for (int s = 0; s < nt; ++s) {
    const long long d = lane + 32 * s < supp ? shift(s) : 0;
    dab += d < 0 ? -d : d;
    if constexpr (T > 0) dd[s] = exact_double(d);
  }
  auto d_of = [&](int s) {
    if constexpr (T > 0) return dd[s];
    else return lane + 32 * s < supp ? exact_double(shift(s)) : 0.0;
  };
  dab = warp_sum_ll(dab);
  const double rec = dab > 0 ? recip(trunc_double(dab)) : 0.0;
  const float coef_f = R.radius_f * trunc_f32(rec);
  // v = q + d coef in FP32, off by at most 5e-7 of the shift and 2e-7 of q.  An entry that clips has
  // a shift of at least q, so 1e-5 q covers it; an absorption in [0, r_min) has a shift of at most
  // q + r_min, so the floor's margin is 1e-6 q on top of 1e-4 r_min (a margin in r_min alone misses
  // rows whose q is more than 240 r_min).  neg_bits: the entries that clip (those of the first 32
  // per lane)
  bool general = R.always_general, close = R.always_general || nt > 32;
  uint32_t neg_bits = 0;
#pragma unroll (kUnroll)
  for (int s = 0; s < nt; ++s) {
    const int32_t k = lane + 32 * s;
    const float q0 = trunc_f32(val_of(s));
    const float v = fmaf(trunc_f32(d_of(s)), coef_f, q0), band = 4e-6f * q0;
    if (k < supp) {
      general |= v < (k < supp - 1 ? 1e-5f * q0 : fmaxf(1e-5f * q0, fmaf(1e-6f, q0, R.floor_f)));
      if (v < -band) neg_bits |= 1u << (s & 31);
      close |= !(fabsf(v) > band);
    }
  }
  general = __any_sync(0xFFFFFFFFu, general) != 0;
  const double coef = R.radius * rec;
  if (MODE == kRowU && !general) {
    const double wc = w * coef;
#pragma unroll (kUnroll)
    for (int s = 0; s < nt; ++s) {
      const int32_t k = lane + 32 * s, pj = col_of(s);
      if (pj >= c) continue;
      const double d = d_of(s);
      outf[k] = fmaf(trunc_f32(d), coef_f, trunc_f32(val_of(s)));
      add(pj, wc, d);
      if (more) atomicAdd(&x_more[pj], (w_more * coef) * d);
    }
    return 0.0;
  }
  double g = 1.0;
  auto is_neg = [&](int s) {   // in FP64
    return lane + 32 * s < supp && __double2hiint(fma(d_of(s), coef, val_of(s))) < 0;
  };
  if (general) {
    if (__any_sync(0xFFFFFFFFu, close)) {
      neg_bits = 0;
      for (int s = 0; s < min(nt, 32); ++s) {
        bool neg = false;
        if constexpr (T > 0) {
#pragma unroll
          for (int q = 0; q < T; ++q)
            if (q == s) neg = is_neg(q);
        } else {
          neg = is_neg(s);
        }
        if (neg) neg_bits |= 1u << s;
      }
    }
    auto neg_of = [&](int s) { return s < 32 ? ((neg_bits >> s) & 1u) != 0u : is_neg(s); };
    long long dneg = 0, qneg = 0;
    bool any = false;
#pragma unroll (kUnroll)
    for (int s = 0; s < nt; ++s)
      if (neg_of(s)) {
        dneg += shift(s);
        qneg += fixed62(val_of(s));
        any = true;
      }
    if (__any_sync(0xFFFFFFFFu, any)) {
      dneg = warp_sum_ll(dneg);
      qneg = warp_sum_ll(qneg);
      const double tot = 1.0 - fma(trunc_double(dneg), coef, trunc_double(qneg) * kTwoM62);
      g = R.always_general ? 1.0 / tot : recip(tot);
    }
    // the absorbing entry, the row's last
    const int sl = (supp - 1) >> 5;
    double dl = 0.0, vl = 0.0;
    if constexpr (T > 0) {
#pragma unroll
      for (int s = 0; s < T; ++s)
        if (s == sl) { dl = dd[s]; vl = val[s]; }
    } else {
      dl = d_of(sl);
      vl = val_of(sl);
    }
    const double ra = __shfl_sync(0xFFFFFFFFu, fmax(fma(dl, coef, vl), 0.0), (supp - 1) & 31) * g;
    if (ra < R.r_min && ra < 1.0) g *= (1.0 - R.r_min) / (1.0 - ra);
  }
  const double cg = coef * g, g1 = g - 1.0;
  const double wcg = w * cg, wg1 = w * g1;
  const float gf = trunc_f32(g);
#pragma unroll (kUnroll)
  for (int s = 0; s < nt; ++s) {
    const int32_t k = lane + 32 * s, pj = col_of(s);
    if (pj >= c) continue;
    const bool neg = s < 32 ? general && ((neg_bits >> (s & 31)) & 1u) != 0u : general && is_neg(s);
    const double q = val_of(s), d = d_of(s);
    if (MODE == kRowU) {
      const float v = fmaf(trunc_f32(d), coef_f, trunc_f32(q));
      outf[k] = neg ? 0.0f : fmaxf(R.always_general ? trunc_f32(fma(d, cg, q * g)) : v * gf, 0.0f);
      const double a = neg ? 0.0 : wcg, b = neg ? -w : wg1;
      if (own) acc[pj] = fma(d, a, fma(q, b, acc[pj]));
      else atomicAdd(&acc[pj], fma(d, a, q * b));
      if (more) atomicAdd(&x_more[pj], w_more * (neg ? -q : fma(d, cg, q * g1)));
    } else {
      const double dq = neg ? -q : fma(d, cg, q * g1);
      const double v = neg ? 0.0 : q + dq;
      if (MODE == kRowDot) { dot = fma(v, t[pj], dot); continue; }
      outd[k] = v;
      dot = fma(dq, t[pj], dot);
      add(pj, w, dq);
    }
  }
  return MODE == kRowU ? 0.0 : warp_sum(dot);
}

template <int MODE>
__device__ __forceinline__ double move_row_any(const RowArgs &R, int32_t i, int32_t e0, int32_t supp,
                                               double w, double *acc, bool own, bool more,
                                               double w_more, double *x_more, float *outf,
                                               double *outd, const double *t, int32_t *zb) {
  return supp <= 128
      ? move_row<4, MODE>(R, i, e0, supp, w, acc, own, more, w_more, x_more, outf, outd, t, zb)
      : move_row<0, MODE>(R, i, e0, supp, w, acc, own, more, w_more, x_more, outf, outd, t, zb);
}

// ---- defect correction ------------------------------------------------------------------------
// Everything one perturbation's solves read and write; vectors in shared memory or the slab.
struct SweepCtx {
  int32_t c;
  size_t ld;
  const int32_t *c_list, *nzptr, *nzcol;
  const double *nzval;
  const float *inv, *inv_t;      // FP32 inverse of the nominal matrix and its transpose
  double *acc;                   // column sums: one array per warp (own) or one
  bool own;
  double *mu, *t;                // the solutions; the changes from the nominal ones before that
  const double *x, *xt;          // their right-hand sides
  float *rm, *rt;                // FP32 residuals [ld], zero beyond c
  const double *qp;              // perturbed C rows, c + 1 apart
  float *red;                    // [(THREADS / 32)][2]
};

// acc += x^T Q'_CC, and rt = xt - t + Q'_CC t (LIN: acc += x^T Q_CC only, the nominal rows).  A warp
// per row, four rows' partial dot products reduced together (6 additions instead of 20).
template <int THREADS, bool LIN>
__device__ __forceinline__ void defect_rows(const SweepCtx &X, const double *x) {
  const int32_t lane = (int32_t)(threadIdx.x & 31u), warp = (int32_t)(threadIdx.x >> 5), c = X.c;
  double *acc = X.own ? X.acc + (size_t)warp * c : X.acc;
  constexpr int32_t NW = THREADS / 32;
  struct Chunk { double q[4]; int32_t pj[4]; };
  for (int32_t a0 = warp; a0 < c; a0 += 4 * NW) {
    // the four rows' extents first, then each row's first 128 entries while the one before is used
    int32_t e0[4], len[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int32_t i = a0 + g * NW < c ? X.c_list[a0 + g * NW] : -1;
      e0[g] = i >= 0 ? X.nzptr[i] : 0;
      len[g] = i >= 0 ? X.nzptr[i + 1] - 1 - e0[g] : 0;
    }
    auto load = [&](int g, int32_t k0) {
      const double *q = LIN ? X.nzval + e0[g] : X.qp + (size_t)(a0 + g * NW) * (c + 1);
      Chunk ch;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int32_t k = k0 + 32 * u;
        ch.pj[u] = k < len[g] ? X.nzcol[e0[g] + k] : -1;
        ch.q[u] = k < len[g] ? q[k] : 0.0;
      }
      return ch;
    };
    double part[4];
    Chunk next = load(0, lane);
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      Chunk ch = next;
      if (g < 3) next = load(g + 1, lane);
      part[g] = 0.0;
      const double xa = a0 + g * NW < c ? x[a0 + g * NW] : 0.0;
      for (int32_t k0 = lane;;) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (ch.pj[u] >= 0) {
            const int32_t pj = ch.pj[u];
            if (X.own) acc[pj] = fma(xa, ch.q[u], acc[pj]);
            else atomicAdd(&acc[pj], xa * ch.q[u]);
            if (!LIN) part[g] = fma(ch.q[u], X.t[pj], part[g]);
          }
        k0 += 128;
        if (k0 - lane >= len[g]) break;
        ch = load(g, k0);
      }
      __syncwarp();   // the next row's columns may be other lanes'
    }
    if (!LIN) {
      const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
      double k0 = h16 ? part[2] : part[0], k1 = h16 ? part[3] : part[1];
      k0 += __shfl_xor_sync(0xFFFFFFFFu, h16 ? part[0] : part[2], 16);
      k1 += __shfl_xor_sync(0xFFFFFFFFu, h16 ? part[1] : part[3], 16);
      double v = h8 ? k1 : k0;
      v += __shfl_xor_sync(0xFFFFFFFFu, h8 ? k0 : k1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      const int32_t a = a0 + (lane >> 3) * NW;
      if ((lane & 7) == 0 && a < c) X.rt[a] = trunc_f32(X.xt[a] - X.t[a] + v);
    }
  }
}

// Sum of column k's partial sums, cleared for the next use.
template <int THREADS>
__device__ __forceinline__ double take_column(const SweepCtx &X, int32_t k) {
  double s = 0.0;
  const int32_t arrays = X.own ? (THREADS / 32) : 1;
  for (int32_t w = 0; w < arrays; ++w) {
    s += X.acc[(size_t)w * X.c + k];
    X.acc[(size_t)w * X.c + k] = 0.0;
  }
  return s;
}

// x += rm M^-1 and (BOTH) t += M^-1 rt with the FP32 inverse; m: largest |correction| of each.  A
// warp per row of the inverse, four rows at a time.
template <int THREADS, bool BOTH>
__device__ __forceinline__ void correct(const SweepCtx &X, double *x, float m[2]) {
  const int32_t lane = (int32_t)(threadIdx.x & 31u), warp = (int32_t)(threadIdx.x >> 5), c = X.c;
  float mx[2] = {0.0f, 0.0f};
  for (int32_t k0 = warp; k0 < c; k0 += 4 * (THREADS / 32)) {
    float sm[4] = {0.0f, 0.0f, 0.0f, 0.0f}, st[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int32_t j = 4 * lane; j < (int32_t)X.ld; j += 128) {
      const float4 a = *reinterpret_cast<const float4 *>(X.rm + j);
      float4 b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (BOTH) b = *reinterpret_cast<const float4 *>(X.rt + j);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const size_t k = (size_t)min(k0 + g * (THREADS / 32), c - 1);
        const float4 f = *reinterpret_cast<const float4 *>(X.inv_t + k * X.ld + j);
        sm[g] = fmaf(f.x, a.x, fmaf(f.y, a.y, fmaf(f.z, a.z, fmaf(f.w, a.w, sm[g]))));
        if (BOTH) {
          const float4 h = *reinterpret_cast<const float4 *>(X.inv + k * X.ld + j);
          st[g] = fmaf(h.x, b.x, fmaf(h.y, b.y, fmaf(h.z, b.z, fmaf(h.w, b.w, st[g]))));
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        sm[g] += __shfl_xor_sync(0xFFFFFFFFu, sm[g], o);
        if (BOTH) st[g] += __shfl_xor_sync(0xFFFFFFFFu, st[g], o);
      }
    float dm = sm[0], dt = st[0];
#pragma unroll
    for (int g = 1; g < 4; ++g)
      if (lane == g) { dm = sm[g]; dt = st[g]; }
    const int32_t k = k0 + lane * (THREADS / 32);
    if (lane < 4 && k < c) {
      x[k] += (double)dm;
      mx[0] = fmaxf(mx[0], fabsf(dm));
      if (dm != dm) mx[0] = __int_as_float(0x7F800000);   // fmaxf drops NaN
      if (BOTH) {
        X.t[k] += (double)dt;
        mx[1] = fmaxf(mx[1], fabsf(dt));
        if (dt != dt) mx[1] = __int_as_float(0x7F800000);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {   // non-negative floats order like their bits
    const uint32_t b = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx[q]));
    if (lane == 0) X.red[warp * 2 + q] = __uint_as_float(b);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    m[q] = 0.0f;
    for (int w = 0; w < (THREADS / 32); ++w) m[q] = fmaxf(m[q], X.red[w * 2 + q]);
  }
  __syncthreads();
}

// One unknown's progress: converged when a correction, or what the contraction leaves after it, is
// below 1e-17 of the solution's scale; from the third round on a correction that shrinks by less than
// 5x has come down to the defects' rounding (below 1e-15: converged too) or stalls.  The rounding
// grows with the change: at l1 moves of 0.5 it is reached before 1e-17, and without that rule every
// such perturbation was factored (c = 200, 304 perturbations: 4.9 ms a call, 1.66 with it; c = 1,900,
// 32: 285 and 28 ms).  In FP32, like the corrections themselves: every thread keeps the account, and
// in FP64 it took 3% of a sweep's time at c = 97 (4.88 -> 4.72 ms, 2,000 perturbations) and 10% at
// c = 914.  The scale is finite, so an infinite or NaN correction never converges.
struct Progress {
  float scale, prev = 0.0f;
  bool done = false, stalled = false;
  __device__ __forceinline__ void step(int it, float dm) {
    if (done) return;
    if (dm <= 1e-17f * scale || (it > 0 && dm < 0.2f * prev && dm * dm <= 1e-17f * scale * prev)) done = true;
    else if (it >= 2 && !(dm < 0.2f * prev)) {
      done = dm <= 1e-15f * scale;
      stalled = !done;
    }
    prev = dm;
  }
};

// The changes e = mu' - mu and h = t' - t of the solutions on C: e (I - Q'_CC) = x and
// (I - Q'_CC) h = xt together, by e <- e + (defect of e) M^-1 with M the nominal matrix, from 0; then
// mu = mu0 + e, t = t0 + h.  Solving for the changes keeps the defects' rounding at the changes'
// size.  The defects are FP64 over the perturbed C rows, summed in a fixed order where every warp
// has its own column sums; M^-1 is in FP32, which costs the contraction nothing: the error shrinks
// by the spectral radius of M^-1 (Q' - Q)_CC a round (about 0.004 for l1 moves of 0.05 on a chain
// whose rows absorb 10%).  False when it does not settle (the caller then factors I - Q'_CC).  acc
// is zero before and after.
template <int THREADS>
__device__ inline bool defect_solve(const SweepCtx &X, const double *mu0, const double *t0,
                                    float mu_scale, float t_scale) {
  for (int32_t k = threadIdx.x; k < X.c; k += THREADS) {
    X.mu[k] = 0.0;
    X.t[k] = 0.0;
    X.rm[k] = trunc_f32(X.x[k]);
    X.rt[k] = trunc_f32(X.xt[k]);
  }
  __syncthreads();
  Progress pm{mu_scale}, pt{t_scale};
  for (int it = 0; it < 40; ++it) {
    float m[2];
    correct<THREADS, true>(X, X.mu, m);
    pm.step(it, m[0]);
    pt.step(it, m[1]);
    if (pm.done && pt.done) {
      for (int32_t k = threadIdx.x; k < X.c; k += THREADS) {
        X.mu[k] += mu0[X.c_list[k]];
        X.t[k] += t0[k];
      }
      __syncthreads();
      return true;
    }
    if (pm.stalled || pt.stalled) return false;
    defect_rows<THREADS, false>(X, X.mu);
    __syncthreads();
    for (int32_t k = threadIdx.x; k < X.c; k += THREADS)
      X.rm[k] = trunc_f32(X.x[k] - X.mu[k] + take_column<THREADS>(X, k));
    __syncthreads();
  }
  return false;
}

// z (I - Q_CC) = x on the nominal rows (the first-order prediction), to 1e-17 of scale; rm is
// overwritten.  Two to three rounds: only the inverse's rounding is corrected.
template <int THREADS>
__device__ inline bool nominal_solve(const SweepCtx &X, double *z, float scale) {
  for (int32_t k = threadIdx.x; k < X.c; k += THREADS) {
    z[k] = 0.0;
    X.rm[k] = trunc_f32(X.x[k]);
  }
  __syncthreads();
  Progress pz{scale};
  for (int it = 0; it < 12; ++it) {
    float m[2];
    correct<THREADS, false>(X, z, m);
    pz.step(it, m[0]);
    if (pz.done) return true;
    if (pz.stalled) return false;
    defect_rows<THREADS, true>(X, z);
    __syncthreads();
    for (int32_t k = threadIdx.x; k < X.c; k += THREADS)
      X.rm[k] = trunc_f32(X.x[k] - z[k] + take_column<THREADS>(X, k));
    __syncthreads();
  }
  return false;
}

__device__ __forceinline__ void atomic_max_pos(double *addr, double v) {
  atomicMax(reinterpret_cast<unsigned long long *>(addr), (unsigned long long)__double_as_longlong(v));
}

// ON_CHIP: the factorisation's matrix in shared memory (small c); vec_smem: the vectors there.
// inv null: always factor (the shortest chains, and columns too long for the inverse's kernel).
template <bool ON_CHIP>
__global__ void __launch_bounds__(sweep_threads(ON_CHIP), kPerturbCtasPerSm)
perturb_kernel(ChainDev C, afc_perturb_params pp, const double *mu0, const double *b0,
               const double *lu0, const int32_t *piv0, const int32_t *nzptr, const int32_t *nzcol,
               const double *nzval, const int32_t *byrank0, const double *y0, const double *t0,
               const double *rho, const double *rho_t, const float *inv, const float *inv_t, uint64_t *counters, uint64_t *pair_flips,
               uint64_t *shift_hist, double *maxima, double *b_out, unsigned char *slabs,
               size_t slab_bytes, int vec_smem, uint32_t vec_off,
               unsigned long long *solve_stats, uint32_t *status) {
  constexpr int THREADS = sweep_threads(ON_CHIP);
  constexpr bool on_chip = ON_CHIP;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sval[33];
  __shared__ int32_t sidx[32];
  __shared__ double sb[2];
  __shared__ int32_t sflag[1];
  __shared__ double red[33];
  __shared__ float fred[(THREADS / 32) * 2];
  __shared__ int32_t rk[kMaxK2];
  __shared__ uint32_t loc_pair[kMaxK2 * kMaxK2];
  __shared__ uint32_t loc_hist[kMaxHist];
  __shared__ uint32_t loc_cnt[3];
  LinScratch ls{sval, sidx, sb, sflag};
  const int32_t n = C.n, c = C.c;
  const double s_unif = 1.0 / (double)n;   // the uniform initial law, divided once
  const int32_t k2 = min(pp.k2, min(kMaxK2, n));
  const int32_t kk = min(pp.top_k, n);
  const int32_t H = min(pp.hist_bins, kMaxHist);
  unsigned char *slab = slabs + (size_t)blockIdx.x * slab_bytes;
  const SweepSlab L = sweep_slab(n, c);
  double *A = reinterpret_cast<double *>(on_chip ? smem : slab + L.A);
  int32_t *piv = reinterpret_cast<int32_t *>(slab + L.piv);
  double *by = reinterpret_cast<double *>(slab + L.by), *rv = reinterpret_cast<double *>(slab + L.rv);
  double *x = reinterpret_cast<double *>(slab + L.x), *z = reinterpret_cast<double *>(slab + L.z);
  double *yp = reinterpret_cast<double *>(slab + L.yp), *xt = reinterpret_cast<double *>(slab + L.xt);
  float *sf = reinterpret_cast<float *>(slab + L.sf), *qf = reinterpret_cast<float *>(slab + L.qf);
  double *qp = reinterpret_cast<double *>(slab + L.qp);
  const int32_t warp = (int32_t)(threadIdx.x >> 5), lane = (int32_t)(threadIdx.x & 31u);
  constexpr int32_t nw = (THREADS / 32);
  unsigned char *vec = vec_smem ? smem + vec_off : slab + L.vec;
  SweepCtx X;
  X.c = c;
  X.ld = inv_ld(c);
  X.c_list = C.c_list; X.nzptr = nzptr; X.nzcol = nzcol; X.nzval = nzval;
  X.inv = inv; X.inv_t = inv_t;
  X.rm = reinterpret_cast<float *>(vec);
  X.rt = X.rm + X.ld;
  int32_t *zb = reinterpret_cast<int32_t *>(X.rt + X.ld) + (size_t)warp * draw_ld(c);
  X.mu = reinterpret_cast<double *>(X.rt + X.ld + (THREADS / 32) * draw_ld(c));
  X.t = X.mu + c;
  X.acc = X.t + c;
  X.own = vec_smem != 0;
  X.x = x; X.xt = xt;
  X.qp = qp;
  X.red = fred;
  // the factorisation's tiles take the place of the column sums
  unsigned char *tile = vec_smem ? reinterpret_cast<unsigned char *>(X.acc) : smem;
  double *my_acc = X.own ? X.acc + (size_t)warp * c : X.acc;
  for (int32_t k = threadIdx.x; k < kMaxK2 * kMaxK2; k += blockDim.x) loc_pair[k] = 0;
  for (int32_t k = threadIdx.x; k < kMaxHist; k += blockDim.x) loc_hist[k] = 0;
  if (threadIdx.x < 3) loc_cnt[threadIdx.x] = 0;
  for (int32_t k = threadIdx.x; k < 2 * (int32_t)X.ld; k += blockDim.x) X.rm[k] = 0.0f;
  // nominal E[T], and the scale of the solutions
  double part = 0.0, pmx = 0.0;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) { part += mu0[i]; pmx = fmax(pmx, mu0[i]); }
  const double T0 = block_sum(part, red);
  const double invT0 = 1.0 / T0;
  const float mu0_max = fminf((float)block_max(pmx, red), 1e30f);   // finite: see Progress
  pmx = 0.0;
  for (int32_t k = threadIdx.x; k < c; k += blockDim.x) pmx = fmax(pmx, t0[k]);
  const float t0_max = fminf((float)block_max(pmx, red), 1e30f);
  double loc_db = 0.0, loc_lin = 0.0, loc_t = 0.0;
  RowArgs R{nzcol, C.c_list, nzval, c, (uint32_t)n, 0u, (uint32_t)pp.seed, (uint32_t)(pp.seed >> 32),
            pp.model, pp.l1_radius, pp.r_min, pp.rel_radius, 0.0f, 0.0f, 0.0f, !(pp.l1_radius <= 1e6)};
  R.radius_f = R.always_general ? 0.0f : trunc_f32(pp.l1_radius);
  R.floor_f = trunc_f32(pp.r_min) * 1.0001f;
  R.screen = R.always_general ? 4e-7f : 1.2e-6f * fminf(R.radius_f, 2.0f) + 4e-7f;
  // the multiplicative moves of the robust search (50% an entry) and l1 moves of more than three
  // quarters of a row rarely contract 5x a round; on chip the factorisation is the cheaper try for them
  const bool try_defect = inv != nullptr && !(on_chip && (pp.model == 1 || pp.l1_radius > 0.75));
  uint32_t loc_defect = 0, loc_factored = 0;
  const uint32_t p_end = pp.p_begin + pp.p_count;
  for (uint32_t p = pp.p_begin + blockIdx.x; p < p_end; p += gridDim.x) {
    R.p = p;
    // (1) every row moved, a warp per row: the C rows (kept in FP64), then the others (FP32 copy
    // for the screening below); x = sum_i mu_i (q'_i - q_i), yp = y0 + sum_U s_i (q'_i - q_i)
    // (mu_i = s_i outside C, so one sum serves both), xt_i = sum_j (q'_ij - q_ij) t_j
    const int32_t sums = (X.own ? nw : 1) * c;
    for (int32_t k = threadIdx.x; k < sums; k += blockDim.x) X.acc[k] = 0.0;
    __syncthreads();
    for (int32_t a = warp; a < c; a += nw) {
      const int32_t i = C.c_list[a], e0 = nzptr[i];
      const double h = move_row_any<kRowC>(R, i, e0, nzptr[i + 1] - e0, mu0[i], my_acc, X.own, false,
                                           0.0, nullptr, nullptr, qp + (size_t)a * (c + 1), t0, zb);
      if (lane == 0) xt[a] = h + rho_t[a];
      __syncwarp();
    }
    __syncthreads();
    for (int32_t k = threadIdx.x; k < c; k += blockDim.x) x[k] = take_column<THREADS>(X, k);
    __syncthreads();
    for (int32_t i = warp; i < n; i += nw) {
      if (C.c_index[i] >= 0) continue;
      const int32_t e0 = nzptr[i];
      const double si = C.s ? C.s[i] : s_unif;
      const double mi = mu0[i];
      const bool more = __double_as_longlong(mi) != __double_as_longlong(si);   // never after a solve
      move_row_any<kRowU>(R, i, e0, nzptr[i + 1] - e0, si, my_acc, X.own, more, mi - si, x, qf + e0,
                          nullptr, nullptr, zb);
      __syncwarp();
    }
    __syncthreads();
    for (int32_t k = threadIdx.x; k < c; k += blockDim.x) {
      const double d = take_column<THREADS>(X, k);
      x[k] += d;
      yp[k] = y0[k] + d;
    }
    __syncthreads();
    // (2) first-order z = x N0, mu'_C, (N' 1)_C
    bool ok = true;
    if (c > 0) {
      if (inv == nullptr || !nominal_solve<THREADS>(X, z, mu0_max)) {
        for (int32_t k = threadIdx.x; k < sums; k += blockDim.x) X.acc[k] = 0.0;
        for (int32_t k = threadIdx.x; k < c; k += blockDim.x) z[k] = x[k];
        __syncthreads();
        lu_solve_transposed_blocked_t(lu0, c, c, piv0, z);
      }
      for (int32_t k = threadIdx.x; k < c; k += blockDim.x) x[k] += rho[k];
      __syncthreads();
      if (try_defect && defect_solve<THREADS>(X, mu0, t0, mu0_max, t0_max)) {
        ++loc_defect;
      } else {
        ++loc_factored;
        // I - Q'_CC from the perturbed C rows
        for (size_t k = threadIdx.x; k < (size_t)c * c; k += blockDim.x)
          A[k] = (k / c == k % c) ? 1.0 : 0.0;
        for (int32_t k = threadIdx.x; k < c; k += blockDim.x) {
          X.mu[k] = yp[k];
          by[k] = yp[k];
          X.t[k] = 1.0;
        }
        __syncthreads();
        for (int32_t a = warp; a < c; a += nw) {
          const int32_t i = C.c_list[a], e0 = nzptr[i], len = nzptr[i + 1] - 1 - e0;
          for (int32_t k = lane; k < len; k += 32)
            A[(size_t)a * c + nzcol[e0 + k]] -= qp[(size_t)a * (c + 1) + k];
        }
        __syncthreads();
        if constexpr (on_chip) {
          ok = lu_factor(A, c, c, piv, ls);
          if (ok) {
            lu_solve_transposed(A, c, c, piv, X.mu, ls);
            lu_solve(A, c, c, piv, X.t, ls);
          }
        } else {
          // blocked LU of an FP32 copy, then FP64 iterative refinement against the FP64 matrix; if
          // the refinement stalls, the FP64 blocked LU of A itself
          const size_t cc = (size_t)c * c;
          float *af = reinterpret_cast<float *>(qp);   // the C rows are in A by now
          for (size_t k = threadIdx.x; k < cc; k += blockDim.x) af[k] = (float)A[k];
          __syncthreads();
          bool mixed = lu_factor_blocked_t<float>(af, c, c, piv, ls, reinterpret_cast<float *>(tile));
          if (mixed) {
            lu_solve_transposed_blocked_t(af, c, c, piv, X.mu);
            mixed = refine<true>(A, af, piv, c, by, X.mu, rv, ls, red);
          }
          if (mixed) {
            lu_solve_blocked_t(af, c, c, piv, X.t);
            mixed = refine<false>(A, af, piv, c, nullptr, X.t, rv, ls, red);
          }
          if (!mixed) {
            for (int32_t k = threadIdx.x; k < c; k += blockDim.x) { X.mu[k] = by[k]; X.t[k] = 1.0; }
            __syncthreads();
            ok = lu_factor_blocked(A, c, c, piv, ls, reinterpret_cast<double *>(tile));
            if (ok) {
              lu_solve_transposed(A, c, c, piv, X.mu, ls);
              lu_solve(A, c, c, piv, X.t, ls);
            }
          }
        }
      }
    }
    if (!ok) {
      if (threadIdx.x == 0) atomicOr(status, kErrSolve);
      continue;
    }
    // (3) E'[T], max b', z . 1
    double pT = 0.0, pY = 0.0, pm = 0.0;
    float tm = 0.0f;   // the largest (N' 1)_i on C, truncated
    for (int32_t v = threadIdx.x; v < n; v += blockDim.x) {
      const int32_t pv = C.c_index[v];
      pT += pv >= 0 ? X.mu[pv] : (C.s ? C.s[v] : s_unif);
    }
    for (int32_t k = threadIdx.x; k < c; k += blockDim.x) {
      pY += z[k];
      X.rt[k] = trunc_f32(X.t[k]);
      tm = fmaxf(tm, X.rt[k]);
      loc_t = fmax(loc_t, X.t[k]);
    }
    const double T = block_sum(pT, red);
    const double Y1 = block_sum(pY, red) * invT0;
    const double invT = 1.0 / T;
    for (int32_t v = threadIdx.x; v < n; v += blockDim.x) {
      const int32_t pv = C.c_index[v];
      const double bv = (pv >= 0 ? X.mu[pv] : (C.s ? C.s[v] : s_unif)) * invT;
      const double bn = b0[v];
      double lin = fma(-bn, Y1, bn);
      if (pv >= 0) lin = fma(z[pv], invT0, lin);
      pm = fmax(pm, bv);
      loc_db = fmax(loc_db, fabs(bv - bn));
      loc_lin = fmax(loc_lin, fabs(bv - lin));
      if (b_out) b_out[(size_t)(p - pp.p_begin) * n + v] = bv;
    }
    if (pp.kl_out) {   // KL(b' || b0), the discrepancy the robust search maximises
      double kl = 0.0;
      for (int32_t v = threadIdx.x; v < n; v += blockDim.x) {
        const int32_t pv = C.c_index[v];
        const double bv = (pv >= 0 ? X.mu[pv] : (C.s ? C.s[v] : s_unif)) * invT;
        if (bv > 0.0) kl += bv * log(bv / b0[v]);
      }
      kl = block_sum(kl, red);
      if (threadIdx.x == 0) pp.kl_out[p - pp.p_begin] = kl;
    }
    const double bmax = block_max(pm, red);
    const double tau = pp.tie_rel * bmax;
    // (4) the largest (N' 1)_i outside C: S_i = sum_j q'_ij t_j of every row in FP32, then in FP64 the
    // rows that can hold the maximum over all rows.  With t at most tm, the FP32 S_i is off by
    //   tm (5e-7 sum_j |shift_j| + 2e-7) for the entries (move_row's bounds; the shifts of the entries
    // kept sum to at most 2 after the row's scaling, whatever the radius) and, all terms being
    // positive, by S_i (4e-7 + 2^-24 (c / 32 + 7)) for t, the scaling and the additions, S_i <= tm.
    // Two rows' errors count, and a row below tm - 1 is below the rows of C.
    float best = 0.0f;
    for (int32_t i0 = warp; i0 < n; i0 += 4 * nw) {
      float part[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int32_t i = i0 + g * nw;
        part[g] = 0.0f;
        if (i < n && C.c_index[i] < 0) {
          const int32_t e0 = nzptr[i], len = nzptr[i + 1] - 1 - e0;
          for (int32_t k0 = lane; k0 < len; k0 += 128) {
            float q[4];
            int32_t pj[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const bool in = k0 + 32 * u < len;
              pj[u] = in ? nzcol[e0 + k0 + 32 * u] : 0;
              q[u] = in ? qf[e0 + k0 + 32 * u] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) part[g] = fmaf(q[u], X.rt[pj[u]], part[g]);
          }
        }
      }
      const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
      float r0 = h16 ? part[2] : part[0], r1 = h16 ? part[3] : part[1];
      r0 += __shfl_xor_sync(0xFFFFFFFFu, h16 ? part[0] : part[2], 16);
      r1 += __shfl_xor_sync(0xFFFFFFFFu, h16 ? part[1] : part[3], 16);
      float s = h8 ? r1 : r0;
      s += __shfl_xor_sync(0xFFFFFFFFu, h8 ? r0 : r1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
      const int32_t i = i0 + (lane >> 3) * nw;
      if ((lane & 7) == 0 && i < n) sf[i] = s;
      best = fmaxf(best, s);
    }
#pragma unroll
    for (int o = 16; o > 4; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    tm = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(tm)));   // not negative
    if (lane == 0) { fred[2 * warp] = best; fred[2 * warp + 1] = tm; }
    __syncthreads();
    for (int32_t w = 0; w < nw; ++w) {
      best = fmaxf(best, fred[2 * w]);
      tm = fmaxf(tm, fred[2 * w + 1]);
    }
    const float least = fmaxf(best, tm - 1.0f) - tm * (2e-6f + R.screen + 2.5e-7f * (float)(c / 32 + 1));
    for (int32_t i = warp; i < n; i += nw) {
      if (C.c_index[i] >= 0 || !(sf[i] >= least)) continue;
      const int32_t e0 = nzptr[i];
      loc_t = fmax(loc_t, 1.0 + move_row_any<kRowDot>(R, i, e0, nzptr[i + 1] - e0, 0.0, nullptr, false, false,
                                                      0.0, nullptr, nullptr, nullptr, X.t, zb));
    }
    // (5) ranks of the nominal top-k2 nodes under b'
    const float tau_up = __double2float_ru(tau), invTf = trunc_f32(invT);
    for (int32_t a = warp; a < k2; a += nw) {
      const int32_t v = byrank0[a];
      const int32_t pv = C.c_index[v];
      const double mv = pv >= 0 ? X.mu[pv] : (C.s ? C.s[v] : s_unif);
      const float vf = trunc_f32(mv) * invTf;
      int32_t r = 0;
      for (int32_t u = lane; u < n; u += 32) {
        if (u == v) continue;
        const int32_t pu = C.c_index[u];
        const double m = pu >= 0 ? X.mu[pu] : (C.s ? C.s[u] : s_unif);
        r += precedes(trunc_f32(m) * invTf, vf, tau_up, true, u, v, tau,
                      [&] { return m * invT - mv * invT; }) ? 1 : 0;
      }
      r = __reduce_add_sync(0xFFFFFFFFu, r);
      if (lane == 0) rk[a] = r;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      bool set_changed = false, order_changed = false;
      for (int32_t a = 0; a < kk && a < k2; ++a) {
        if (rk[a] >= kk) set_changed = true;
        if (rk[a] != a) order_changed = true;
      }
      if (k2 > 0 && rk[0] != 0) loc_cnt[0]++;
      if (set_changed) loc_cnt[1]++;
      if (order_changed) loc_cnt[2]++;
      for (int32_t a = 0; a < k2; ++a) {
        int32_t sh = abs(rk[a] - a);
        if (sh > H - 1) sh = H - 1;
        loc_hist[sh]++;
      }
    }
    for (int32_t q = threadIdx.x; q < k2 * k2; q += blockDim.x) {
      const int32_t a = q / k2, b = q % k2;
      if (a < b && rk[a] > rk[b]) loc_pair[a * kMaxK2 + b]++;
    }
    __syncthreads();
  }
  // flush
  loc_db = block_max(loc_db, red);
  loc_lin = block_max(loc_lin, red);
  loc_t = block_max(loc_t, red);
  if (threadIdx.x == 0 && solve_stats && !on_chip) {
    if (loc_defect) atomicAdd(&solve_stats[0], (unsigned long long)loc_defect);
    if (loc_factored) atomicAdd(&solve_stats[1], (unsigned long long)loc_factored);
  }
  if (threadIdx.x == 0) {
    atomic_max_pos(&maxima[0], loc_db);
    atomic_max_pos(&maxima[1], loc_lin);
    atomic_max_pos(&maxima[2], loc_t);
    for (int k = 0; k < 3; ++k)
      if (loc_cnt[k]) atomicAdd(reinterpret_cast<unsigned long long *>(&counters[k]), (unsigned long long)loc_cnt[k]);
  }
  for (int32_t q = threadIdx.x; q < k2 * k2; q += blockDim.x) {
    const int32_t a = q / k2, b = q % k2;
    const uint32_t v = loc_pair[a * kMaxK2 + b];
    if (v) atomicAdd(reinterpret_cast<unsigned long long *>(&pair_flips[a * pp.k2 + b]), (unsigned long long)v);
  }
  for (int32_t h = threadIdx.x; h < H; h += blockDim.x)
    if (loc_hist[h]) atomicAdd(reinterpret_cast<unsigned long long *>(&shift_hist[h]), (unsigned long long)loc_hist[h]);
}

// Position of every node in the order (rank, id) -- rank counts of a tie-band ranking need
// not be distinct, the band is not transitive -- and topk[pos] = v for positions below k.
__global__ void rank_order_kernel(int32_t n, const int32_t *rank, int32_t k, int32_t *topk) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const int32_t rv = rank[v];
    int32_t pos = 0;
    for (int32_t u = 0; u < n; ++u) {
      const int32_t ru = rank[u];
      pos += (ru < rv || (ru == rv && u < v)) ? 1 : 0;
    }
    if (pos < k) topk[pos] = v;
  }
}

cudaError_t launch_rank(int32_t n, const double *b, double tie_rel, int32_t k, int32_t *rank,
                        int32_t *topk, cudaStream_t stream) {
  const int grid = (n + 255) / 256;
  nominal_rank_kernel<<<rank_grid(n), 256, 0, stream>>>(n, b, tie_rel, 0, rank, nullptr);
  if (topk && k > 0) rank_order_kernel<<<grid, 256, 0, stream>>>(n, rank, k, topk);
  return cudaGetLastError();
}

bool perturb_on_chip(int32_t c, int smem_optin) {
  const size_t cc = (size_t)(c > 0 ? c : 1);
  return (int64_t)up256(8 * cc * cc + 28 * cc + 64) + 16 * 1024 <= (int64_t)smem_optin;
}

cudaError_t launch_perturb(const ChainDev &C, const afc_perturb_params &pp, const double *mu0,
                           const double *b0, const double *lu0, const int32_t *piv0,
                           uint64_t *counters, uint64_t *pair_flips, uint64_t *shift_hist,
                           double *maxima, double *b_out, unsigned char *ws, const SolveWs &L,
                           uint32_t *status_dev, int num_sms, cudaStream_t stream) {
  if (pp.p_count == 0) return cudaSuccess;
  const int32_t n = C.n, c = C.c;
  const int32_t *nzptr = reinterpret_cast<const int32_t *>(ws + L.off_nzptr);
  const int32_t *nzcol = reinterpret_cast<const int32_t *>(ws + L.off_nzcol);
  const double *nzval = reinterpret_cast<const double *>(ws + L.off_nzval);
  const double *t0 = reinterpret_cast<const double *>(ws + L.off_t);   // the solve's N 1 on C
  double *y0 = reinterpret_cast<double *>(ws + L.off_y);
  int32_t *rank0 = reinterpret_cast<int32_t *>(ws + L.off_flags);
  int32_t *byrank0 = reinterpret_cast<int32_t *>(ws + L.off_tmp);
  cudaMemsetAsync(byrank0, 0, sizeof(int32_t) * kMaxK2, stream);
  nominal_rank_kernel<<<rank_grid(n), 256, 0, stream>>>(n, b0, pp.tie_rel, min(pp.k2, kMaxK2),
                                                        rank0, byrank0);
  double *rho = reinterpret_cast<double *>(ws + L.off_tmp + 512), *rho_t = rho + c;   // 4 n + 4 c there
  if (c > 0) {
    const int chunks = (int)std::max<size_t>(
        1, std::min({(size_t)n, (size_t)kDefectChunks, (L.total - L.off_slab) / (2 * sizeof(Pair) * (size_t)c)}));
    Pair *part = reinterpret_cast<Pair *>(ws + L.off_slab);
    nominal_defect_kernel<<<chunks, 256, 0, stream>>>(C, nzptr, nzcol, nzval, mu0, part);
    nominal_finish_kernel<<<std::min((c + 7) / 8, 608), 256, 0, stream>>>(C, mu0, part, chunks, nzptr,
                                                                         nzcol, nzval, t0, y0, rho, rho_t);
  }
  int max_optin = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  float *inv = nullptr, *inv_t = nullptr;
  const int nr = inverse_smem(c, 8) <= (size_t)max_optin - 1024 ? 8 : 2;   // c up to 5,900 / 23,700
  // The shortest chains are factored: the factorisation costs less than the rounds of the
  // corrections and the inverse before them, with wider moves (more rounds) up to a larger size.
  // Factored / corrected, us for 304 perturbations: radius 0.05 c = 8 134 / 218, 16 189 / 265, 20 244 /
  // 262; 0.25 c = 20 265 / 335; 0.5 c = 24 337 / 465.  Where both take about the same time the
  // corrections stay: their results are closer to 64 bits (error 4.3e-16 against 5.3e-16 at c = 16).
  const int32_t direct = pp.model == 0 && pp.l1_radius > 0.1 ? 24 : 16;
  if (c > direct && inverse_smem(c, nr) <= (size_t)max_optin - 1024) {
    inv = reinterpret_cast<float *>(ws + L.off_inv);
    inv_t = inv + (size_t)c * inv_ld(c);
    cudaMemsetAsync(inv, 0, perturb_inverse_bytes(c), stream);
    auto kernel = nr == 8 ? inverse32_kernel<8> : inverse32_kernel<2>;
    allow_shared(reinterpret_cast<const void *>(kernel), 1024);
    kernel<<<(c + nr - 1) / nr, kInvThreads, inverse_smem(c, nr), stream>>>(lu0, piv0, c, inv_ld(c),
                                                                           inv, inv_t);
  }
  // shared memory: the factorisation's matrix (small c), then the vectors while they fit; the
  // factorisation's tiles (large c) take the place of the column sums
  const int on_chip = perturb_on_chip(c, max_optin) ? 1 : 0;
  const size_t tiles = on_chip ? 0 : sizeof(double) * (size_t)lu_blocked_smem_doubles();
  const int threads = sweep_threads(on_chip != 0);
  const size_t sums = 8 * (size_t)(threads / 32) * (size_t)(c > 0 ? c : 1);
  const size_t mat = on_chip ? up256(8 * (size_t)(c > 0 ? c : 1) * (size_t)(c > 0 ? c : 1)) : 0;
  const size_t vec = vec_bytes(c, threads) - sums + std::max(sums, tiles);
  const int vec_smem = mat + vec + kSweepStatic <= (size_t)max_optin ? 1 : 0;
  const size_t dyn = vec_smem ? mat + vec : std::max(mat, tiles);
  auto kernel = on_chip ? perturb_kernel<true> : perturb_kernel<false>;
  allow_shared(reinterpret_cast<const void *>(kernel), kSweepStatic);
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, dyn);
  if (e != cudaSuccess) return e;
  const size_t slab_bytes = perturb_slab_bytes(n, c);
  size_t fit = (L.total - L.off_slab) / slab_bytes;
  fit = std::min(fit, (size_t)num_sms * (size_t)std::max(1, std::min(per_sm, kPerturbCtasPerSm)));
  fit = std::min(fit, (size_t)pp.p_count);
  if (fit == 0) return cudaErrorMemoryAllocation;
  kernel<<<(int)fit, threads, dyn, stream>>>(
      C, pp, mu0, b0, lu0, piv0, nzptr, nzcol, nzval, byrank0, y0, t0, rho, rho_t, inv, inv_t, counters,
      pair_flips, shift_hist, maxima, b_out, ws + L.off_slab, slab_bytes, vec_smem,
      (uint32_t)mat, reinterpret_cast<unsigned long long *>(pp.solve_stats), status_dev);
  return cudaGetLastError();
}

}  // namespace afc
