// Predictor calibration (Algorithm 1, its two least-squares fits; Section 3.2: linear regressors that are
// trained in closed form; Appendix A: the regularizer rate is 1e-3):
//
//   W = argmin_W || X W^T (+ b) - Y ||^2 + rate * trace(X^T X) / n_in * ||W||^2
//
// over the calibration tokens, X = [in0 ; in1] (16-bit rows, n features), Y the layer's keys or values (d features).
//
// Device pipeline (every step a kernel of this library):
//   1. fit_gram_kernel: the normal equations as ONE product [X ; Y]^T X on the tensor cores, straight from the
//      token-major rows (16-bit products are exact, accumulation is fp32).
//   2. Column sums (only with an intercept), the trace and the ridge term; the (n + d) x n product goes to double
//      precision with the centring correction  - s_i s_j / T  and the ridge on the diagonal.
//   3. fit_solve_kernel: G = L L^T (n x n) and, in the same pass, the forward solve of the d rows below it
//      (Z = C^T L^-T is what a Cholesky factorisation does to rows appended under the matrix); a second launch
//      of it, the other way round, solves W L = Z.  Everything in double precision.
//   4. W is rounded to the cache's 16-bit type as [d_kv][n_in] (a linear layer's weight); the
//      intercept is b = mean(Y) - mean(X) W^T.
#pragma once

#include "common.cuh"
#include "gemm_pred.cuh"

namespace aquakv {

constexpr int kFitNB = 64;                     // tile side of the factorisation and of the back substitution
constexpr int kFitLd = kFitNB + 4;             // doubles per row of a tile in shared memory: rows start 4 doubles (8 banks)
                                               // apart, so the fragments of the fp64 products read without conflicts

// ---------------------------------------------------------------------------------------------
// Normal equations: P[s][i][j] = sum over the tokens of k-slice s of F_i F_j, F = [X ; Y] (i < n + d), j < n; of the
// tiles above the diagonal of X^T X nothing is written.
//
// A CTA pair forms a 256 x 256 tile with tcgen05.mma.cta_group::2.  The tokens are the summation index and the rows
// are stored feature-contiguous, so both operands are MN-major: a TMA box of 64 features x 64 tokens is 64 rows of
// 128 swizzled bytes, 8 tokens (one swizzle atom) 1024 bytes apart, the next 64 features 8192 bytes apart.  (A
// K-major product needs token-contiguous copies of X and Y first: 63 us per matrix of 32768 x 1024.)
// A key fit has 26 such tiles and a value fit 68 for 74 CTA pairs, so the tokens are cut into `slices` work units per
// tile (the partial sums are added in double by fit_prepare_kernel, in slice order); unit u works on slice
// u / n_tiles, so the pairs that run together read the same tokens.
// 32768 tokens, d_kv 1024, bf16: 85 us (key fit) and 197 us (value fit), bound by the tensor cores; before, with the
// copies and a 128 x 256 tile per CTA, 5 x 63 us + 4 x 82 us.
// ---------------------------------------------------------------------------------------------
constexpr int kGramStages = 6;
constexpr int kGramBoxBytes = 64 * 64 * 2;                       // 64 tokens x 64 features
constexpr int kGramStageBytes = 4 * kGramBoxBytes;               // this CTA's 128 A features and its half of the 256 B features

struct GramSmemTail {
  uint64_t full[kGramStages];
  uint64_t empty[kGramStages];
  uint64_t acc_full[kAccStages];
  uint64_t acc_empty[kAccStages];
  uint32_t tmem_base;
  int abort_flag;
};
constexpr size_t kGramSmemBytes = 1024 + size_t(kGramStages) * kGramStageBytes + sizeof(GramSmemTail);

struct GramArgs {
  int n, d;          // features of X and of Y; the first d of X come from map x0, the next d (if any) from x1
  int nk;            // k-blocks of 64 tokens (tokens past the last are zero-filled by TMA)
  int slices;
  float* P;          // [slices][n + d][n]
  int* status;
};

// Tiles of 256 x 256 that are needed: rows of X down to the diagonal, all of Y's rows.
__host__ __device__ inline int gram_tiles(int n, int d) { return (n / 256) * (n / 256 + 1) / 2 + (d / 256) * (n / 256); }
__device__ __forceinline__ void gram_tile(int t, int n, int& mi, int& nj) {
  const int nb = n / 256;
  for (mi = 0;; ++mi) {
    const int w = mi < nb ? mi + 1 : nb;
    if (t < w) break;
    t -= w;
  }
  nj = t;
}

// Shared-memory descriptor of an MN-major operand: 64 features (128 bytes, swizzled) x 8 tokens per atom, the
// atoms of the next 8 tokens 1024 bytes and of the next 64 features one box further on.
__device__ __forceinline__ uint64_t umma_smem_desc_mn128(uint32_t smem_addr) {
  uint64_t desc = 0;
  desc |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);
  desc |= static_cast<uint64_t>(kGramBoxBytes >> 4) << 16;
  desc |= static_cast<uint64_t>(1024 >> 4) << 32;
  desc |= static_cast<uint64_t>(1) << 46;
  desc |= static_cast<uint64_t>(2) << 61;
  return desc;
}

template <bool kBf16>
__global__ void __launch_bounds__(kGemmThreads, 1)
fit_gram_kernel(const __grid_constant__ CUtensorMap tmX0, const __grid_constant__ CUtensorMap tmX1,
                const __grid_constant__ CUtensorMap tmY, const GramArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_align<1024>(smem_raw);
  GramSmemTail* tail = reinterpret_cast<GramSmemTail*>(smem + size_t(kGramStages) * kGramStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int n_tiles = gram_tiles(a.n, a.d), n_units = n_tiles * a.slices;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGramStages; ++s) {
      mbar_init(&tail->full[s], 1);
      mbar_init(&tail->empty[s], 1);
    }
    for (int s = 0; s < kAccStages; ++s) {
      mbar_init(&tail->acc_full[s], 1);
      mbar_init(&tail->acc_empty[s], 8);     // four epilogue warps of each CTA (used in the leader only)
    }
    tail->abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&tail->tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after_sync();
  const uint32_t tmem_base = tail->tmem_base;
  volatile int* abort_flag = &tail->abort_flag;
  pdl_sync();

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&tmX0);
      tma_prefetch_desc(&tmX1);
      tma_prefetch_desc(&tmY);
      int stage = 0, issued = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int u = pair; ok && u < n_units; u += n_pairs) {
        int mi, nj;
        gram_tile(u % n_tiles, a.n, mi, nj);
        const int s = u / n_tiles;
        const int kb0 = int((long long)a.nk * s / a.slices), kb1 = int((long long)a.nk * (s + 1) / a.slices);
        const int fa = mi * 256 + int(rank) * 128, fb = nj * 256 + int(rank) * 128;      // first features of this CTA
        const CUtensorMap* ma = fa >= a.n ? &tmY : (fa >= a.d ? &tmX1 : &tmX0);
        const CUtensorMap* mb = fb >= a.d ? &tmX1 : &tmX0;
        const int xa = fa >= a.n ? fa - a.n : fa % a.d, xb = fb % a.d;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_bounded(&tail->empty[stage], phase ^ 1u, abort_flag, a.status)) {
            ok = false;
            break;
          }
          uint8_t* dst = smem + size_t(stage) * kGramStageBytes;
          if (rank == 0) mbar_arrive_expect_tx(&tail->full[stage], 2 * kGramStageBytes);
          tma_load_2d_pair(dst, ma, &tail->full[stage], xa, kb * kBK);
          tma_load_2d_pair(dst + kGramBoxBytes, ma, &tail->full[stage], xa + 64, kb * kBK);
          tma_load_2d_pair(dst + 2 * kGramBoxBytes, mb, &tail->full[stage], xb, kb * kBK);
          tma_load_2d_pair(dst + 3 * kGramBoxBytes, mb, &tail->full[stage], xb + 64, kb * kBK);
          ++issued;
          if (++stage == kGramStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && rank == 0) {
        // let the copies in flight land before the shared memory is released
        int s = stage;
        uint32_t pb = phase;
        const int pending = issued < kGramStages ? issued : kGramStages;
        for (int i = 0; i < pending; ++i) {
          if (s == 0) { s = kGramStages; pb ^= 1u; }
          --s;
          const unsigned long long t0 = global_timer_ns();
          while (!mbar_try_wait(&tail->full[s], pb) && global_timer_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = umma_idesc_f16(2 * kBM, kBN, kBf16) | (1u << 15) | (1u << 16);   // both operands MN-major
      int stage = 0, it = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int u = pair; ok && u < n_units; u += n_pairs, ++it) {
        const int s = u / n_tiles;
        const int kb0 = int((long long)a.nk * s / a.slices), kb1 = int((long long)a.nk * (s + 1) / a.slices);
        const int acc = it & 1;
        if (!mbar_wait_bounded(&tail->acc_empty[acc], ((it >> 1) & 1u) ^ 1u, abort_flag, a.status)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t tmem_d = tmem_base + uint32_t(acc * kBN);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_bounded(&tail->full[stage], phase, abort_flag, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint32_t a_addr = smem_u32(smem + size_t(stage) * kGramStageBytes), b_addr = a_addr + 2 * kGramBoxBytes;
#pragma unroll
          for (int k = 0; k < kBK / kUmmaK; ++k)      // 16 tokens = two 8-token atoms
            umma_f16_pair(tmem_d, umma_smem_desc_mn128(a_addr + k * 2048), umma_smem_desc_mn128(b_addr + k * 2048), idesc,
                          (kb > kb0 || k > 0) ? 1u : 0u);
          umma_commit_pair(&tail->empty[stage]);
          if (++stage == kGramStages) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair(&tail->acc_full[acc]);
      }
    }
  } else {
    const int quarter = warp & 3;
    int it = 0;
    for (int u = pair; u < n_units; u += n_pairs, ++it) {
      int mi, nj;
      gram_tile(u % n_tiles, a.n, mi, nj);
      const int acc = it & 1;
      if (!mbar_wait_bounded(&tail->acc_full[acc], (it >> 1) & 1u, abort_flag, a.status)) break;
      tc_fence_after_sync();
      const int row = mi * 256 + int(rank) * 128 + quarter * 32 + lane;
      const uint32_t taddr = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(acc * kBN);
      float* out = a.P + ((long long)(u / n_tiles) * (a.n + a.d) + row) * a.n + nj * 256;
#pragma unroll 1
      for (int c = 0; c < kBN / 32; ++c) {
        float v[32];
        tmem_ld_32x32b_x32(taddr + uint32_t(c * 32), v);
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4*>(out + c * 32 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_leader(&tail->acc_empty[acc]);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();          // neither CTA leaves while its peer may still signal its barriers
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

template <bool kBf16>
__device__ __forceinline__ float fit_to_float(uint16_t b) {
  if constexpr (kBf16) return __uint_as_float(uint32_t(b) << 16);
  else return __half2float(__ushort_as_half(b));
}

// sums[c] += sum over this block's tokens of in[t][c].  Grid (ceil(T / 256), ncols/32), block (32, 8).
template <bool kBf16>
__global__ void fit_colsum_kernel(const uint16_t* __restrict__ in, long long ld_in, long long T,
                                  double* __restrict__ sums) {
  __shared__ double part[8][32];
  pdl_sync();
  const int c = blockIdx.y * 32 + threadIdx.x;
  const long long t0 = (long long)blockIdx.x * 256;
  double s = 0.0;
  for (int r = threadIdx.y; r < 256; r += 8) {
    const long long t = t0 + r;
    if (t < T) s += double(fit_to_float<kBf16>(in[t * ld_in + c]));
  }
  part[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0) {
    for (int r = 1; r < 8; ++r) s += part[r][threadIdx.x];
    atomicAdd(&sums[c], s);
  }
}

// ridge = rate * trace(centred G) / n.  One block of 256 threads.  sx == nullptr: no centring.
__global__ void fit_ridge_kernel(const float* __restrict__ P, int slices, int n, int d, double T, const double* __restrict__ sx,
                                 double rate, double* __restrict__ ridge) {
  __shared__ double part[256];
  pdl_sync();
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) {
    double g = 0.0;
    for (int k = 0; k < slices; ++k) g += double(P[(size_t(k) * (n + d) + i) * n + i]);
    if (sx != nullptr) g -= sx[i] * sx[i] / T;
    s += g;
  }
  part[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *ridge = rate * part[0] / double(n);
}

// M[i][j] = sum over the slices of P - s_i s_j / T + (i == j) ridge  for the lower triangle of the first n rows and
// all of the d rows below.  sx holds the sums of [X ; Y]; nullptr: no centring.  Grid (n / 256, n + d), 256 threads.
__global__ void fit_prepare_kernel(const float* __restrict__ P, int slices, int n, int d, double T,
                                   const double* __restrict__ sx, const double* __restrict__ ridge,
                                   double* __restrict__ M) {
  pdl_sync();
  const int i = blockIdx.y, j = blockIdx.x * 256 + threadIdx.x;
  if (i < n && j > i) return;
  double g = 0.0;
  for (int k = 0; k < slices; ++k) g += double(P[(size_t(k) * (n + d) + i) * n + j]);
  if (sx != nullptr) g -= sx[i] * sx[j] / T;
  if (i == j) g += *ridge;
  M[size_t(i) * n + j] = g;
}

// ---------------------------------------------------------------------------------------------
// Factorisation with the forward solve, and the back substitution: one persistent launch each.
//
// M is (n + d) x n row-major, cut into 64 x 64 tiles.  Forward (kBack = false), in place, tile (i, j) becomes
//   i == j:  the Cholesky factor of  M_jj - sum_{k<j} L_jk L_jk^T
//   i >  j:  (M_ij - sum_{k<j} L_ik L_jk^T) L_jj^-T          (rows i >= n / 64: the forward solve)
// Back (kBack = true), rows i >= n / 64 only, columns from the last:  W_ij = (Z_ij - sum_{k>j} W_ik L_kj) L_jj^-1.
//
// Tasks are numbered column by column and handed out in that order by a counter; a finished tile raises its flag in
// global memory and a task waits only for tiles of smaller number, which running CTAs already hold, so the schedule
// cannot dead-lock however many CTAs are resident; every wait is bounded.  The products run as warp-level fp64 m8n8k4
// matrix instructions (61 of the SM's 64 FMA per clock) from double-buffered shared-memory tiles.
//
// What bounds it: the chain diagonal tile -> tile below it -> next diagonal tile, n / 64 times; the arithmetic
// (n^3 / 3 + n^2 d) would take 0.2 ms of the 2048-feature fit.  A step of the chain, by time stamps: flag and tiles 1.8 us, last
// product 2.4, diagonal tile 10, store and flag 1.1, its tile to the one below 1.3, triangular solve 1.6, store and flag 0.7.
// d = 1024, n = 1024 and 2048: forward 0.29 and 0.59 ms, back 0.12 and 0.29 (ncu, serialised; with one pivot at a time and solves of a column
// at a time both fits took 1.36 forward and 0.57 back; with a launch per step of 32 columns 8.4 in all).
// ---------------------------------------------------------------------------------------------
constexpr int kFitThreads = 256;
constexpr int kFitTile = kFitNB * kFitLd;                                  // doubles of a tile in shared memory
struct FitCholSmem {
  double2 col[2][kFitNB];                                                  // a step's two columns
  double pivot[kFitNB], scale[kFitNB];
};
struct FitSolveSmem {
  double t[2][2][kFitTile];                                                // [buffer][row tile, column tile]
  FitCholSmem chol;
  int ready;
  int task;
  int abort_flag;
};

__device__ __forceinline__ void fit_cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void fit_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void fit_cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// A 64 x 64 tile of M (leading dimension ld) into shared memory, by the whole CTA.
__device__ __forceinline__ void fit_load_tile(double* dst, const double* src, long long ld) {
#pragma unroll
  for (int it = 0; it < kFitNB * 32 / kFitThreads; ++it) {
    const int e = it * kFitThreads + threadIdx.x, r = e >> 5, c = (e & 31) * 2;
    fit_cp_async16(dst + r * kFitLd + c, src + r * ld + c);
  }
}

// D (8 x 8) += A (8 x 4) B (4 x 8) in double: A element (lane / 4, lane % 4), B element (lane % 4, lane / 4),
// D elements (lane / 4, 2 (lane % 4)) and the one right of it.
__device__ __forceinline__ void dmma_8x8x4(double& d0, double& d1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(d0), "+d"(d1)
               : "d"(a), "d"(b));
}

__device__ __forceinline__ int fit_flag(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Called by one thread: waits until both flags are up; false after kWaitLimitNs or when the CTA has aborted.
__device__ __forceinline__ bool fit_wait(const int* f0, const int* f1, volatile int* abort_flag, int* status) {
  if (fit_flag(f0) && fit_flag(f1)) return true;
  const unsigned long long t0 = global_timer_ns();
  uint32_t spins = 0;
  while (!(fit_flag(f0) && fit_flag(f1))) {
    __nanosleep(32);
    if ((++spins & 0xFFu) == 0 && (*abort_flag || global_timer_ns() - t0 > kWaitLimitNs)) {
      *abort_flag = 1;
      atomicExch(status, kStatusTimeout);
      return false;
    }
  }
  return true;
}

// Cholesky factor of the 64 x 64 tile in shared memory (lower triangle), in place, its 16 x 16 diagonal blocks replaced
// by their inverses (all that the solves need of them).  Thread (ty, tx) of 16 x 16 owns rows ty + 16 u and columns tx + 16 v in registers.
// Two pivots a step: with the columns c0, c1 of the pair as they stand, m = p10 / p00, y = c1 - m c0 (what the first pivot's
// elimination leaves of c1) and det = p00 p11 - p10^2 (p00 times the second pivot),
//   a[r][c] -= c0[r] (c0[c] / p00) + y[r] (y[c] (p00 / det)),
// the two steps of an elimination one pivot at a time with reciprocals that do not wait for one another.  det carries the
// rounding error of p10^2 along (Kahan's difference of two products), so that it is exactly zero for a feature given twice, p00 = p10 = p11.  Columns stay
// unscaled until the end: L = (c0, y) / sqrt(pivot).  Blocks above the diagonal are left out.
// What bounds it is the chain of a step, columns to shared memory, barrier, reciprocals, update, and its double-precision
// instructions, of which an SM issues two warps' worth a clock at best.  Both reciprocals are one call, the odd lanes with the other argument
// (two calls: 2 % of a calibration of 32768 tokens, d_kv 1024).  One pivot at a time, with the scaling by a double-precision rsqrt in the
// chain, took 16.2 us a tile, this 10.
// A pivot that is not positive sets *status (the matrix was not positive definite) and counts as 1.
__device__ __forceinline__ void fit_chol_tile(double* t, FitCholSmem& cs, int* status) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  double a[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) a[u][v] = t[(ty + 16 * u) * kFitLd + tx + 16 * v];
#pragma unroll
  for (int v0 = 0; v0 < 4; ++v0) {
#pragma unroll 1
    for (int h = 0; h < 8; ++h) {
      const int p = 16 * v0 + 2 * h;
      double2* cb = cs.col[h & 1];
      if ((tx >> 1) == h) {
#pragma unroll
        for (int u = v0; u < 4; ++u) reinterpret_cast<double*>(cb + ty + 16 * u)[tx & 1] = a[u][v0];
      }
      __syncthreads();
      double p00 = cb[p].x;
      const double p10 = cb[p + 1].x, p11 = cb[p + 1].y;
      if (!(p00 > 0.0)) {
        if (threadIdx.x == 0) atomicExch(status, kStatusNumeric);
        p00 = 1.0;
      }
      const double pp = p10 * p10;
      double det = fma(p00, p11, -pp) - fma(p10, p10, -pp);
      if (!(det > 0.0)) {
        if (threadIdx.x == 0) atomicExch(status, kStatusNumeric);
        det = p00;
      }
      const double rr = __drcp_rn(threadIdx.x & 1 ? det : p00);
      const double r0 = __shfl_sync(0xffffffffu, rr, 0), rd = __shfl_sync(0xffffffffu, rr, 1);
      if (threadIdx.x == 0) {
        cs.pivot[p] = p00;
        cs.pivot[p + 1] = det * r0;
      }
      const double m = p10 * r0, r1 = p00 * rd;
      double c0[4], y[4];
#pragma unroll
      for (int u = v0; u < 4; ++u) {
        const double2 c = cb[ty + 16 * u];
        c0[u] = c.x;
        y[u] = fma(-m, c.x, c.y);
      }
      if (tx == 2 * h + 1) {
#pragma unroll
        for (int u = v0; u < 4; ++u) a[u][v0] = y[u];
      }
#pragma unroll
      for (int v = v0; v < 4; ++v) {
        const double2 c = cb[tx + 16 * v];
        const double w0 = c.x * r0, w1 = fma(-m, c.x, c.y) * r1;
        if (v > v0 || (tx >> 1) > h) {
#pragma unroll
          for (int u = v; u < 4; ++u) a[u][v] = fma(-y[u], w1, fma(-c0[u], w0, a[u][v]));
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < kFitNB) cs.scale[threadIdx.x] = rsqrt(cs.pivot[threadIdx.x]);
  __syncthreads();
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const double sc = cs.scale[tx + 16 * v];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u > v || (u == v && ty > tx)) t[(ty + 16 * u) * kFitLd + tx + 16 * v] = a[u][v] * sc;
  }
  __syncthreads();
  // inverses of the diagonal blocks: thread (block, column) solves L x = e_column (L's diagonal is 1 / scale)
  double x[16];
  const int blk = threadIdx.x >> 4, c = threadIdx.x & 15;
  if (threadIdx.x < kFitNB) {
    const double* lb = t + (16 * blk) * kFitLd + 16 * blk;
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = r == c ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      x[k] *= cs.scale[16 * blk + k];
#pragma unroll
      for (int r = k + 1; r < 16; ++r) x[r] = fma(-lb[r * kFitLd + k], x[k], x[r]);
    }
  }
  __syncthreads();
  if (threadIdx.x < kFitNB) {
#pragma unroll
    for (int r = 0; r < 16; ++r) t[(16 * blk + r) * kFitLd + 16 * blk + c] = x[r];
  }
  __syncthreads();
}

// X op(L) = T for eight rows of a 64 x 64 tile: op(L) = L^T or, kBack, L.  `l`: a tile that fit_chol_tile left, in shared
// memory.  x enters holding T and leaves holding X as accumulators of the fp64 products: x[c][e] of a lane is row lane / 4,
// column 8 c + 2 (lane % 4) + e.  Sixteen columns at a time: the block's columns times the inverse of L's diagonal block, then
// their products with L's blocks beside it off the columns still to come.  An accumulator's element e is an A fragment of the
// columns 2 k + e, so the rows never leave the warp's registers.  (A column at a time, four lanes a row: 6.1 us a tile,
// this 1.6.)
template <bool kBack>
__device__ __forceinline__ void fit_trsm_rows(double (&x)[8][2], const double* l, int lane) {
  const int g = lane >> 2, k2 = (lane & 3) * 2;
  // element (k, n) of the B fragment for input columns 8 ct + 2 k + e and output columns 8 co + n
  auto bfrag = [&](int ct, int co, int e) {
    return kBack ? l[(8 * ct + k2 + e) * kFitLd + 8 * co + g] : l[(8 * co + g) * kFitLd + 8 * ct + k2 + e];
  };
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int b = kBack ? 6 - 2 * s : 2 * s;          // first of the block's two column tiles
    double y[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
    for (int o = 0; o < 2; ++o)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (kBack ? i < o : i > o) continue;          // the inverse is lower triangular
#pragma unroll
        for (int e = 0; e < 2; ++e) dmma_8x8x4(y[o][0], y[o][1], x[b + i][e], bfrag(b + i, b + o, e));
      }
#pragma unroll
    for (int o = 0; o < 2; ++o)
#pragma unroll
      for (int e = 0; e < 2; ++e) x[b + o][e] = y[o][e];
#pragma unroll
    for (int ct = 0; ct < 2; ++ct)
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int co = 0; co < 8; ++co)
          if (kBack ? co < b : co > b + 1) dmma_8x8x4(x[co][0], x[co][1], -y[ct][e], bfrag(b + ct, co, e));
  }
}

// flags: [(n + d) / 64][n / 64] finished tiles, then the task counter; all zero at launch.
template <bool kBack>
__global__ void __launch_bounds__(kFitThreads, 1)
fit_solve_kernel(double* __restrict__ M, int n, int d, int* __restrict__ flags, int* __restrict__ status) {
  extern __shared__ __align__(16) uint8_t fit_smem_raw[];
  FitSolveSmem* sm = reinterpret_cast<FitSolveSmem*>(fit_smem_raw);
  const int nc = n / kFitNB, nr = (n + d) / kFitNB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, j4 = lane & 3;
  const int row = warp * 8 + g;                                 // this lane's row of the accumulators: a warp owns 8 x 64
  if (threadIdx.x == 0) sm->abort_flag = 0;
  volatile int* abort_flag = &sm->abort_flag;
  pdl_sync();
  int* next_task = flags + nr * nc;
  int col = 0, first = 0;                                       // forward: number of column `col`'s diagonal task
  for (;;) {
    if (threadIdx.x == 0) sm->task = atomicAdd(next_task, 1);
    __syncthreads();
    const int task = sm->task;
    int i, j;
    if constexpr (kBack) {
      if (task >= (nr - nc) * nc) break;
      j = nc - 1 - task / (nr - nc);
      i = nc + task % (nr - nc);
    } else {
      while (col < nc && task >= first + nr - col) first += nr - col++;
      if (col >= nc) break;
      j = col;
      i = col + task - first;
    }
    double* Mij = M + ((long long)i * kFitNB) * n + j * kFitNB;
    double acc[8][2];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const double2 v = *reinterpret_cast<const double2*>(Mij + (long long)row * n + nt * 8 + 2 * j4);
      acc[nt][0] = v.x;
      acc[nt][1] = v.y;
    }
    // left-looking update with the tile pairs of step s = 0, 1, ..; the next pair is fetched while one is multiplied
    // (if it exists by then)
    const int steps = kBack ? nc - 1 - j : j;
    auto ktile = [&](int s) { return kBack ? nc - 1 - s : s; };
    auto flag_a = [&](int s) { return flags + i * nc + ktile(s); };
    auto flag_b = [&](int s) { return kBack ? flag_a(s) : flags + j * nc + ktile(s); };     // back: L is complete
    int fetched = 0;
    auto fetch = [&](int s) {
      const int k = ktile(s);
      fit_load_tile(sm->t[s & 1][0], M + ((long long)i * kFitNB) * n + k * kFitNB, n);
      if constexpr (kBack) fit_load_tile(sm->t[s & 1][1], M + ((long long)k * kFitNB) * n + j * kFitNB, n);
      else if (i != j) fit_load_tile(sm->t[s & 1][1], M + ((long long)j * kFitNB) * n + k * kFitNB, n);
      fit_cp_commit();
      fetched = s + 1;
    };
    bool stop = false;
    for (int s = 0; s < steps; ++s) {
      if (fetched <= s) {                  // not there yet: wait for it
        if (threadIdx.x == 0) fit_wait(flag_a(s), flag_b(s), abort_flag, status);
        __syncthreads();
        if (*abort_flag) { stop = true; break; }
        fetch(s);
      }
      fit_cp_wait_all();
      if (threadIdx.x == 0) sm->ready = s + 1 < steps && fit_flag(flag_a(s + 1)) && fit_flag(flag_b(s + 1));
      __syncthreads();
      if (sm->ready) fetch(s + 1);
      const double* ta = sm->t[s & 1][0];
      const double* tb = !kBack && i == j ? ta : sm->t[s & 1][1];
#pragma unroll 4
      for (int kk = 0; kk < kFitNB / 4; ++kk) {
        const double av = -ta[row * kFitLd + kk * 4 + j4];
        double bv[8];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
          bv[nt] = kBack ? tb[(kk * 4 + j4) * kFitLd + nt * 8 + g] : tb[(nt * 8 + g) * kFitLd + kk * 4 + j4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) dmma_8x8x4(acc[nt][0], acc[nt][1], av, bv[nt]);
      }
      __syncthreads();                     // buffer s & 1 may be overwritten, sm->ready read by all
    }
    if (stop) break;
    if (!kBack && i == j) {
      double* tt = sm->t[0][0];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
        *reinterpret_cast<double2*>(tt + row * kFitLd + nt * 8 + 2 * j4) = make_double2(acc[nt][0], acc[nt][1]);
      __syncthreads();
      fit_chol_tile(tt, sm->chol, status);
      for (int e = threadIdx.x; e < kFitNB * kFitNB / 2; e += kFitThreads) {
        const int r = e >> 5, c = (e & 31) * 2;
        *reinterpret_cast<double2*>(Mij + (long long)r * n + c) = *reinterpret_cast<const double2*>(tt + r * kFitLd + c);
      }
    } else {
      if (!kBack && threadIdx.x == 0) fit_wait(flags + j * nc + j, flags + j * nc + j, abort_flag, status);
      __syncthreads();
      if (*abort_flag) break;
      fit_load_tile(sm->t[1][1], M + ((long long)j * kFitNB) * n + j * kFitNB, n);
      fit_cp_commit();
      fit_cp_wait_all();
      __syncthreads();
      fit_trsm_rows<kBack>(acc, sm->t[1][1], lane);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
        *reinterpret_cast<double2*>(Mij + (long long)row * n + nt * 8 + 2 * j4) = make_double2(acc[nt][0], acc[nt][1]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {                // one releasing thread: the barrier ordered the CTA's stores before its fence
      __threadfence();
      asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(flags + i * nc + j), "r"(1) : "memory");
    }
  }
}

// W16 = round16(W) and, optionally, W32 = float(W), element by element ([d][n]).
template <bool kBf16>
__global__ void fit_store_kernel(const double* __restrict__ W, long long count, uint16_t* __restrict__ W16, float* __restrict__ W32) {
  pdl_sync();
  for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < count; o += (long long)gridDim.x * blockDim.x) {
    const double v = W[o];
    // one rounding, from the double
    uint16_t b;
    if constexpr (kBf16) {
      // round the double's mantissa to bf16's 8 significant bits, ties to even, on its bit pattern
      unsigned long long u = (unsigned long long)__double_as_longlong(v);
      const unsigned long long lsb = (u >> 45) & 1ull;
      u = (u + ((1ull << 44) - 1ull) + lsb) & ~((1ull << 45) - 1ull);
      b = uint16_t(__float_as_uint(float(__longlong_as_double((long long)u))) >> 16);
    } else {
      b = __half_as_ushort(__double2half(v));
    }
    W16[o] = b;
    if (W32 != nullptr) W32[o] = float(v);
  }
}

// bias[c] = (sum of Y_c - sum_r (sum of X_r) W[c][r]) / T.  One warp per output feature; block of 128 threads.
__global__ void fit_bias_kernel(const double* __restrict__ W, int n, int d, const double* __restrict__ sx, double T,
                                float* __restrict__ bias) {
  pdl_sync();
  const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= d) return;
  double s = 0.0;
  for (int r = lane; r < n; r += 32) s += sx[r] * W[size_t(c) * n + r];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) bias[c] = float((sx[n + c] - s) / T);
}

}  // namespace aquakv
