// Backbone vector quantizer with the four-dimensional grid (Section 4.1 "Alternative quantizers": besides
// the p = 2 grids the paper runs one 2-bit grid with d = 4, n = 256, for which it had no fast GPU kernel;
// its d is the grid dimension).  The steps are those of the p = 2 quantizer (Section 2; the residual / add-back
// steps of Algorithm 2 and Algorithm 3) with consecutive 4-tuples in place of pairs: root-mean-square
// group scale stored as fp16, normalisation with the rounded scale, random signs, Hadamard rotation in
// blocks of h values, nearest of the 256 grid points (lowest index on a tie), one byte per tuple.
//
// One warp per row, the whole row in registers as in the rotated kernels of uniform.cuh: v[c][i] is value
// 256 c + 8 lane + i, so a lane holds the tuples 64 c + 2 lane and 64 c + 2 lane + 1 of every chunk and
// writes their codes as one 16-bit store.
//
// Search.  The hypercube [-4, 4)^4 is cut into 32^4 cells of side 1/4.  A table built on the device when
// the context is created (grid4_table_kernel) lists, for every cell, every point that can be the nearest
// one somewhere in the cell: of the points whose smallest squared distance to the (slightly inflated) cell is at
// most the smallest of the largest ones, those that no other point beats everywhere in the cell (the difference of two
// squared distances is linear, so its largest value over the cell is a sum of four).  Evaluating the list in
// ascending index order with a strict "<" gives the result of the exhaustive search.  An entry is 16 bytes: up to 15
// indices, the last one repeated as padding, and their count (3.3 on average for a Gaussian-optimal grid and 7.8 for
// the longest of a warp's 32 lists; 4.9 and 11.7 without the second criterion); 255 as the count marks a cell with
// more candidates.  A tuple in such a cell or outside the hypercube (6e-5 of the coordinates of a normalised row; also
// every non-finite value) is searched exhaustively by the whole warp: by its own lane alone it held the warp for 256
// dependent look-ups, and one row in fifteen has such a tuple.
//
// What bounds it: the look-ups of candidates at random indices in shared memory (about eleven passes of the
// shared-memory pipe each; ncu: that pipe 65 % busy, issue slots 39 %) and the latency of the chain around them at four warps per scheduler.  9472 rows of 1024,
// with predictor: 77 us (171 us with the lists of the first criterion alone and the exhaustive search per lane).
#pragma once

#include "uniform.cuh"

namespace aquakv {

struct Grid4Args {
  UniformArgs u;              // X, P, codes, scales, hat, T, d, log_g as for the uniform backbone
  const float4* grid;         // [256] grid points
  const uint4* table;         // [32^4] candidate lists of the cells (grid4_table_kernel); encode only
  const uint32_t* signmask;   // [32]: lane's word, bit 8 c + i set where the sign of value 256 c + 8 lane + i is -1
  int log_h;                  // 6 .. 10
};

struct Grid4Smem {
  float4 g[256];
};

constexpr int kGrid4Cells = 32;             // per dimension
constexpr float kGrid4Lo = -4.0f;           // the table covers [-4, 4)^4
constexpr float kGrid4InvW = 4.0f;          // 1 / cell width
constexpr unsigned kGrid4Overflow = 255u;   // count byte of a cell with more than 15 candidates

__device__ __forceinline__ void grid4_load(Grid4Smem& sm, const float4* grid) {
  for (int k = threadIdx.x; k < 256; k += blockDim.x) sm.g[k] = grid[k];
  __syncthreads();
}

__device__ __forceinline__ ulonglong2 lds128(uint32_t addr) {
  ulonglong2 v;
  asm("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(addr));
  return v;
}

// Half the squared distance of the tuple (y01, y23) to the point at a shared address, less the tuple's own half square
// (which all points share): the same instruction sequence wherever a candidate is evaluated.  The order of the
// roundings decides near ties, so it is part of the result.  (Half the point's square is recomputed: a look-up of its own
// would load the shared-memory pipe, which is what bounds the search.  Packed differences instead, five instructions for nine: no faster, 417 us
// against 416 for 8192 tokens there and back.)
__device__ __forceinline__ float grid4_score(uint32_t addr, f32x2_t y01, f32x2_t y23) {
  const ulonglong2 g = lds128(addr);
  float g0, g1, g2, g3, y0, y1, y2, y3;
  unpack2(g.x, g0, g1);
  unpack2(g.y, g2, g3);
  unpack2(y01, y0, y1);
  unpack2(y23, y2, y3);
  float s = 0.5f * fmaf(g3, g3, fmaf(g2, g2, fmaf(g1, g1, g0 * g0)));
  s = fmaf(-y0, g0, s);
  s = fmaf(-y1, g1, s);
  s = fmaf(-y2, g2, s);
  return fmaf(-y3, g3, s);
}

// Candidate lists of all cells: one thread per cell, distances in double.
__global__ void __launch_bounds__(256) grid4_table_kernel(const float4* __restrict__ grid, uint4* __restrict__ table) {
  __shared__ float4 g[256];
  for (int k = threadIdx.x; k < 256; k += blockDim.x) g[k] = grid[k];
  __syncthreads();
  constexpr int C = kGrid4Cells;
  const long long n_cells = (long long)C * C * C * C;
  for (long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x; cell < n_cells;
       cell += (long long)gridDim.x * blockDim.x) {
    int idx[4] = {int(cell / (C * C * C)), int(cell / (C * C) % C), int(cell / C % C), int(cell % C)};
    double lo[4], hi[4];
    for (int k = 0; k < 4; ++k) {
      // inflated by 1e-5: the kernel finds the cell of a value with one fp32 rounding
      lo[k] = double(kGrid4Lo) + double(idx[k]) / double(kGrid4InvW) - 1e-5;
      hi[k] = double(kGrid4Lo) + double(idx[k] + 1) / double(kGrid4InvW) + 1e-5;
    }
    auto bounds = [&](int p, double& dmin, double& dmax) {
      const double c[4] = {double(g[p].x), double(g[p].y), double(g[p].z), double(g[p].w)};
      dmin = dmax = 0.0;
      for (int k = 0; k < 4; ++k) {
        const double below = lo[k] - c[k], above = c[k] - hi[k];
        const double out = below > 0.0 ? below : (above > 0.0 ? above : 0.0);
        const double far = fmax(fabs(c[k] - lo[k]), fabs(c[k] - hi[k]));
        dmin += out * out;
        dmax += far * far;
      }
    };
    double U = 1.0e300;
    int nearest = 0;
    for (int p = 0; p < 256; ++p) {
      double dmin, dmax;
      bounds(p, dmin, dmax);
      if (dmax < U) {
        U = dmax;
        nearest = p;
      }
    }
    // Two evaluations of grid4_score in single precision are off by at most 16 roundings of its terms, so the distances
    // they compare by 32 units of 2^-24 of half a point's square plus its largest product with a tuple of the cell:
    // a point is left out only if it loses by more (twice that, at least 1e-5).
    auto slack = [&](int p) {
      const double c[4] = {double(g[p].x), double(g[p].y), double(g[p].z), double(g[p].w)};
      double terms = 0.0;
      for (int k = 0; k < 4; ++k) terms += 0.5 * c[k] * c[k] + fabs(c[k]) * fmax(fabs(lo[k]), fabs(hi[k]));
      return 1e-5 + 4e-6 * terms;
    };
    const double limit = U * (1.0 + 1e-4) + 1e-6, slack_u = slack(nearest);
    // candidates by distance, then without those that another one beats everywhere in the cell
    constexpr int kMost = 96;
    unsigned char cand[kMost];
    int m = 0;
    for (int p = 0; p < 256 && m <= kMost; ++p) {
      double dmin, dmax;
      bounds(p, dmin, dmax);
      if (dmin <= limit + fmax(slack(p), slack_u)) {
        if (m < kMost) cand[m] = (unsigned char)p;
        ++m;
      }
    }
    unsigned w[4] = {0u, 0u, 0u, 0u};
    int n = 0, last = 0;
    for (int i = 0; i < (m <= kMost ? m : 0); ++i) {
      const float4 gi = g[cand[i]];
      const double a[4] = {double(gi.x), double(gi.y), double(gi.z), double(gi.w)};
      const double slack_i = slack(cand[i]);
      bool beaten = false;
      for (int j = 0; j < m && !beaten; ++j) {
        const float4 gj = g[cand[j]];
        const double b[4] = {double(gj.x), double(gj.y), double(gj.z), double(gj.w)};
        // max over the cell of |y - g_j|^2 - |y - g_i|^2 = sum_k 2 y_k (a_k - b_k) + b_k^2 - a_k^2
        double most = 0.0;
        for (int k = 0; k < 4; ++k) most += fmax(2.0 * lo[k] * (a[k] - b[k]), 2.0 * hi[k] * (a[k] - b[k])) + b[k] * b[k] - a[k] * a[k];
        beaten = most < -fmax(slack_i, slack(cand[j]));
      }
      if (!beaten) {
        if (n < 15) w[n >> 2] |= unsigned(cand[i]) << (8 * (n & 3));
        last = cand[i];
        ++n;
      }
    }
    if (n > 15 || n == 0) {
      w[3] = (w[3] & 0x00ffffffu) | (kGrid4Overflow << 24);
    } else {
      for (int i = n; i < 15; ++i) w[i >> 2] |= unsigned(last) << (8 * (i & 3));
      w[3] |= unsigned(n) << 24;
    }
    table[cell] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Candidate list of a tuple.  Rounding y * 4 + 15.5 to a whole number gives floor(4 y) + 16, the cell's number along an
// axis, which is below 32 in all four exactly inside the hypercube (not for NaN).
__device__ __forceinline__ uint4 grid4_entry(const uint4* __restrict__ table, f32x2_t y01, f32x2_t y23) {
  constexpr float kOff = -kGrid4Lo * kGrid4InvW - 0.5f;
  constexpr unsigned C = kGrid4Cells, M = kSearchMagicBits;
  const f32x2_t w2 = pack2(kGrid4InvW, kGrid4InvW), off2 = pack2(kOff, kOff), m2 = pack2(kSearchMagic, kSearchMagic);
  float a, b, c, d;
  unpack2(add2(fma2(y01, w2, off2), m2), a, b);
  unpack2(add2(fma2(y23, w2, off2), m2), c, d);
  const unsigned ua = __float_as_uint(a), ub = __float_as_uint(b), uc = __float_as_uint(c), ud = __float_as_uint(d);
  const bool inside = max(max(ua - M, ub - M), max(uc - M, ud - M)) < C;
  const unsigned cell = ((ua * C + ub) * C + uc) * C + ud - M * (C * C * C + C * C + C + 1u);
  uint4 e = make_uint4(0u, 0u, 0u, kGrid4Overflow << 24);
  if (inside) e = __ldg(table + cell);
  return e;
}

// Shared address of the nearest point of a tuple: the candidates of its cell in ascending order, strict "<" keeps the
// lowest index; the exhaustive loop for what the table does not cover.
__device__ __forceinline__ uint32_t grid4_nearest(uint32_t grid, const uint4& entry, f32x2_t y01, f32x2_t y23) {
  const unsigned n = entry.w >> 24;
  const bool listed = n != kGrid4Overflow;
  const unsigned n_max = __reduce_max_sync(0xffffffffu, listed ? n : 0u);
  uint32_t at = grid + (entry.x & 0xffu) * 16u;
  float best = grid4_score(at, y01, y23);
#pragma unroll
  for (int w = 0; w < 8; ++w) {            // two candidates at a time
    if (w < 2 || unsigned(2 * w) < n_max) {         // the same for the whole warp; shorter lists repeat their last index
      const unsigned word = w < 2 ? entry.x : (w < 4 ? entry.y : (w < 6 ? entry.z : entry.w));
#pragma unroll
      for (int j = (w == 0 ? 1 : 0); j < (w == 7 ? 1 : 2); ++j) {
        const uint32_t a = grid + ((word >> (8 * (2 * (w & 1) + j))) & 0xffu) * 16u;
        const float t = grid4_score(a, y01, y23);
        if (t < best) at = a;
        best = fminf(t, best);
      }
    }
  }
  // what the table does not cover: the warp searches all points for one such lane after the other, eight points a lane
  for (unsigned todo = __ballot_sync(0xffffffffu, !listed); todo != 0u; todo &= todo - 1u) {
    const int src = __ffs(todo) - 1, lane = threadIdx.x & 31;
    float y0, y1, y2, y3;
    unpack2(y01, y0, y1);
    unpack2(y23, y2, y3);
    const f32x2_t s01 = pack2(__shfl_sync(0xffffffffu, y0, src), __shfl_sync(0xffffffffu, y1, src));
    const f32x2_t s23 = pack2(__shfl_sync(0xffffffffu, y2, src), __shfl_sync(0xffffffffu, y3, src));
    float b = 3.0e38f;
    int k = lane;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float t = grid4_score(grid + 16u * (32 * i + lane), s01, s23);
      if (t < b) {
        b = t;
        k = 32 * i + lane;
      }
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {           // the smallest distance, the lowest index of equal ones
      const float ob = __shfl_xor_sync(0xffffffffu, b, off);
      const int ok = __shfl_xor_sync(0xffffffffu, k, off);
      if (ob < b || (ob == b && ok < k)) {
        b = ob;
        k = ok;
      }
    }
    if (lane == src) at = grid + 16u * unsigned(k);
  }
  return at;
}

template <bool kBf16, int NCH>
__global__ void __launch_bounds__(kUniformWarps * 32, 4)
grid4_encode_rows_kernel(const Grid4Args ga) {
  __shared__ Grid4Smem sm;
  grid4_load(sm, ga.grid);
  const UniformArgs& a = ga.u;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * kUniformWarps + (threadIdx.x >> 5);
  const long long n_warps = (long long)gridDim.x * kUniformWarps;
  const int lanes_per_group = a.log_g >= 8 ? 32 : 1 << (a.log_g - 3);
  const int chunks_per_group = a.log_g > 8 ? 1 << (a.log_g - 8) : 1;
  const int n_groups = a.d >> a.log_g;
  const uint32_t sbits = ga.signmask[lane], grid = smem_u32(sm.g);
  const float rs = rsqrtf(float(1 << ga.log_h));
  const float inv_g = 1.0f / float(1 << a.log_g);
  pdl_sync();
  for (long long t = warp; t < a.T; t += n_warps) {
    f32x2_t v[NCH][4];
    {
      // the prediction is read again for the reconstruction: holding it through the search would cost 32 registers
      f32x2_t pred[NCH][4];
      row_load_pred<NCH, false>(a, t, lane, pred);
      row_residual<kBf16, NCH>(a, t, lane, pred, v);
    }
    // group scale: root mean square of the residual, rounded to fp16; the rounded value normalises
    float ss[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      ss[c] = 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float lo, hi;
        unpack2(v[c][k], lo, hi);
        ss[c] = fmaf(hi, hi, fmaf(lo, lo, ss[c]));
      }
    }
    for (int off = 1; off < lanes_per_group; off <<= 1) {
#pragma unroll
      for (int c = 0; c < NCH; ++c) ss[c] += __shfl_xor_sync(0xffffffffu, ss[c], off);
    }
    float f[NCH];                          // scale
#pragma unroll
    for (int c0 = 0; c0 < NCH; ++c0) {
      float sum = 0.0f;                    // a group of several chunks: the sum over its chunks
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        if ((c & ~(chunks_per_group - 1)) == (c0 & ~(chunks_per_group - 1))) sum += ss[c];
      const __half s16 = __float2half_rn(fminf(sqrtf(sum * inv_g), 65504.0f));
      const float sf = __half2float(s16);
      f[c0] = sf;
      if ((lane & (lanes_per_group - 1)) == 0 && (c0 & (chunks_per_group - 1)) == 0)
        a.scales[t * n_groups + ((256 * c0 + 8 * lane) >> a.log_g)] = __half_as_ushort(s16);
      const float inv = sf > 0.0f ? __fdiv_rn(1.0f, sf) : 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) v[c0][k] = mul2(v[c0][k], row_signed(inv, sbits, c0, k));
    }
    row_hadamard<NCH>(v, ga.log_h, lane);
    const f32x2_t rs2 = pack2(rs, rs);
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[c][k] = mul2(v[c][k], rs2);
    // nearest grid point of every 4-tuple, two chunks at a time (their candidate lists take 16 registers)
    constexpr int CH = NCH < 2 ? NCH : 2;
#pragma unroll
    for (int c0 = 0; c0 < NCH; c0 += CH) {
      uint4 entry[CH][2];
#pragma unroll
      for (int c = 0; c < CH; ++c)
#pragma unroll
        for (int u = 0; u < 2; ++u) entry[c][u] = grid4_entry(ga.table, v[c0 + c][2 * u], v[c0 + c][2 * u + 1]);
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        uint32_t at[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) at[u] = grid4_nearest(grid, entry[c][u], v[c0 + c][2 * u], v[c0 + c][2 * u + 1]);
        *reinterpret_cast<uint16_t*>(a.codes + t * (long long)(a.d / 4) + 64 * (c0 + c) + 2 * lane) =
            uint16_t(((at[0] - grid) >> 4) | (((at[1] - grid) >> 4) << 8));
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const ulonglong2 g = lds128(at[u]);
          v[c0 + c][2 * u] = g.x;
          v[c0 + c][2 * u + 1] = g.y;
        }
      }
    }
    if (a.hat != nullptr) {
      f32x2_t pred[NCH][4];
      row_load_pred<NCH>(a, t, lane, pred);
      row_rotate_back<kBf16, NCH>(a, t, lane, ga.log_h, sbits, rs, v, f, pred);
    }
  }
}

template <bool kBf16, int NCH>
__global__ void __launch_bounds__(kUniformWarps * 32, 4)
grid4_decode_rows_kernel(const Grid4Args ga) {
  __shared__ Grid4Smem sm;
  grid4_load(sm, ga.grid);
  const UniformArgs& a = ga.u;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * kUniformWarps + (threadIdx.x >> 5);
  const long long n_warps = (long long)gridDim.x * kUniformWarps;
  const int n_groups = a.d >> a.log_g;
  const uint32_t sbits = ga.signmask[lane], grid = smem_u32(sm.g);
  const float rs = rsqrtf(float(1 << ga.log_h));
  pdl_sync();
  for (long long t = warp; t < a.T; t += n_warps) {
    f32x2_t y[NCH][4], pred[NCH][4];
    float f[NCH];
    row_load_pred<NCH>(a, t, lane, pred);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const uint32_t two = *reinterpret_cast<const uint16_t*>(a.codes + t * (long long)(a.d / 4) + 64 * c + 2 * lane);
      f[c] = __half2float(__ushort_as_half(a.scales[t * n_groups + ((256 * c + 8 * lane) >> a.log_g)]));
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const ulonglong2 g = lds128(grid + ((two >> (8 * u)) & 0xffu) * 16u);
        y[c][2 * u] = g.x;
        y[c][2 * u + 1] = g.y;
      }
    }
    row_rotate_back<kBf16, NCH>(a, t, lane, ga.log_h, sbits, rs, y, f, pred);
  }
}

}  // namespace aquakv
