// Row routines of the planar quantizer for d_kv = 256 and 512 (any supported Hadamard block and scale group): the steps of
// codec.cuh with ONE warp per token row.
//
// v[c][k] of a lane holds values 256 c + 8 lane + 2 k and the next (the layout of a team of d_kv / 256 warps with the
// chunks in one warp), so index bits 0-2 select a register, 3-7 the lane and bit 8 the chunk: the butterfly between chunks is a
// register operation, and the sums of squares of a group of two chunks meet in one lane.  Stages, sums and roundings are
// those of the teams, in their order: the results are the same bit for bit.
//
// A team of two warps met at a named barrier for every exchange (four a row, each with a trip through shared memory) and did
// the scale, the control flow and the reports twice; one warp has two chunks to interleave instead.  For the layer kernel (layer_kernel.cuh: kChunkRowWarps has the times of both):
// the stand-alone row kernels, whose calls of a thousand rows need every warp they can get, keep the teams.
#pragma once

#include "rowwarp.cuh"

namespace aquakv {

// Butterflies over index bits 0 .. log_h - 1, ascending, of a row of NCH chunks.
template <int NCH>
__device__ __forceinline__ void row_hadamard(f32x2_t (&v)[NCH][4], int log_h, int lane) {
#pragma unroll
  for (int c = 0; c < NCH; ++c) fwht_packed<8>(v[c], log_h, lane);
#pragma unroll
  for (int k = 8; k < 10; ++k) {
    const int m = 1 << (k - 8);
    if (m < NCH && k < log_h) {
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        if ((c & m) == 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const f32x2_t a = v[c][i], b = v[c | m][i];
            v[c][i] = add2(a, b);
            v[c | m][i] = sub2(a, b);
          }
        }
    }
  }
}

// (f, f) with the signs of pair (c, k) of the row: bit 8 c + 2 k and the next of `bits`.
__device__ __forceinline__ f32x2_t row_signed(float f, uint32_t bits, int c, int k) {
  const int s = 31 - 8 * c - 2 * k;
  return pack2(__uint_as_float(__float_as_uint(f) ^ ((bits << s) & 0x80000000u)),
               __uint_as_float(__float_as_uint(f) ^ ((bits << (s - 1)) & 0x80000000u)));
}

struct ChunkRowCtx {
  SearchCtx search;        // encoder
  uint32_t signs;          // bit 8 c + i set <=> value 256 c + 8 lane + i is multiplied by -1
  float inv_g;             // 1 / scale group
  float rs;                // 1 / sqrt(Hadamard block)
  int log_h, log_g;
  int lane;
};
__device__ __forceinline__ void chunk_ctx_init(ChunkRowCtx& rc, int log_h, int log_g, int lane) {
  rc.lane = lane;
  rc.log_h = log_h;
  rc.log_g = log_g;
  rc.inv_g = __int_as_float((127 - log_g) << 23);                       // 2^-log_g, exact
  rc.rs = __int_as_float((127 - (log_h >> 1)) << 23) * ((log_h & 1) ? 0.70710678118654752f : 1.0f);
}

// hat = round16(pred + scale * sign * rs * H(v)) for the row's grid points v; pr: the prediction (zeros without one).
template <int NC, bool kBf16>
__device__ __forceinline__ void chunk_finish_row(const ChunkRowCtx& rc, f32x2_t (&v)[NC][4], const float (&sf)[NC],
                                                 const f32x2_t (&pr)[NC][4], uint16_t* __restrict__ hat_row) {
  row_hadamard<NC>(v, rc.log_h, rc.lane);
  const f32x2_t rs2 = pack2(rc.rs, rc.rs);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[c][k] = fma2(mul2(v[c][k], rs2), row_signed(sf[c], rc.signs, c, k), pr[c][k]);
    hat_store8(hat_row + (c * 256 + rc.lane * 8), make_uint4(store16x2p<kBf16>(v[c][0]), store16x2p<kBf16>(v[c][1]),
                                                             store16x2p<kBf16>(v[c][2]), store16x2p<kBf16>(v[c][3])));
  }
}

// The lane's prediction values, zeros without a predictor.  The rows must be 32-byte aligned.
template <int NC>
__device__ __forceinline__ void chunk_load_pred(const float* __restrict__ pred_row, int lane, f32x2_t (&pr)[NC][4]) {
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if (pred_row != nullptr) {
      wr_load_pred8(pred_row + (c * 256 + lane * 8), pr[c]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) pr[c][k] = pack2(0.0f, 0.0f);
    }
  }
}

// One token row of Q and of the reconstruction; arguments as encode_row of codec.cuh.  The prediction is read twice.
template <int NC, int NPTS, bool kBf16>
__device__ __forceinline__ void chunk_encode_row(const ChunkRowCtx& rc, const RowSmem<NPTS>* __restrict__ rsm,
                                                 const uint16_t* __restrict__ x_row, const float* __restrict__ pred_row,
                                                 uint8_t* __restrict__ codes_row, uint16_t* __restrict__ scales_row,
                                                 uint16_t* __restrict__ hat_row) {
  constexpr int BITS = NPTS == 16 ? 4 : (NPTS == 64 ? 6 : 8);
  const int lane = rc.lane;
  f32x2_t v[NC][4];
  {
    uint4 raw[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) raw[c] = __ldcs(reinterpret_cast<const uint4*>(x_row + c * 256 + lane * 8));   // read once
    f32x2_t pr[NC][4];
    if (pred_row != nullptr) chunk_load_pred<NC>(pred_row, lane, pr);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const uint32_t w[4] = {raw[c].x, raw[c].y, raw[c].z, raw[c].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[c][k] = load16x2<kBf16>(w[k]);
        if (pred_row != nullptr) v[c][k] = sub2(v[c][k], pr[c][k]);
      }
    }
  }
  // sums of squares of the chunks, sign flip
  float ss[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    f32x2_t acc = mul2(v[c][0], v[c][0]);
#pragma unroll
    for (int k = 1; k < 4; ++k) acc = fma2(v[c][k], v[c][k], acc);
    float lo, hi;
    unpack2(acc, lo, hi);
    ss[c] = lo + hi;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      unpack2(v[c][k], lo, hi);
      v[c][k] = pack2(apply_sign(lo, rc.signs, 8 * c + 2 * k), apply_sign(hi, rc.signs, 8 * c + 2 * k + 1));
    }
  }
#pragma unroll
  for (int b = 3; b < 8; ++b)
    if (b < rc.log_g) {
#pragma unroll
      for (int c = 0; c < NC; ++c) ss[c] += __shfl_xor_sync(0xffffffffu, ss[c], 1 << (b - 3));
    }
  row_hadamard<NC>(v, rc.log_h, lane);
  // group scale: root mean square, stored as fp16; normalise with the rounded value
  float sf[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    float tot = ss[c];
    int cpg = 1;                               // chunks of a group
    if (NC > 1 && rc.log_g > 8) {
      cpg = 1 << (rc.log_g - 8);
      tot = 0.0f;
#pragma unroll
      for (int c2 = 0; c2 < NC; ++c2)
        if (c2 / cpg == c / cpg) tot += ss[c2];
    }
    const __half s16 = __float2half_rn(fminf(sqrtf(tot * rc.inv_g), 65504.0f));
    sf[c] = __half2float(s16);
    if (rc.log_g >= 8) {                       // one lane per group writes the scale
      if (lane == 0 && c % cpg == 0) scales_row[c / cpg] = __half_as_ushort(s16);
    } else {
      const int lpg = 1 << (rc.log_g - 3);     // lanes per group
      if (lane % lpg == 0) scales_row[c * (256 >> rc.log_g) + lane / lpg] = __half_as_ushort(s16);
    }
    const float inv = (sf[c] > 0.0f ? __frcp_rn(sf[c]) : 0.0f) * rc.rs;
    const f32x2_t inv2 = pack2(inv, inv);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[c][k] = mul2(v[c][k], inv2);
  }
  // nearest grid point per pair: all table entries of a chunk first, then the candidates
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    uint32_t entry[4], at[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) entry[k] = search_entry(v[c][k], rc.search);
    const uint32_t emax = merge_entries<NPTS>(merge_entries<NPTS>(entry[0], entry[1]), merge_entries<NPTS>(entry[2], entry[3]));
#pragma unroll
    for (int k = 0; k < 4; ++k) at[k] = nearest_of_candidates<NPTS>(v[c][k], entry[k], rc.search.grid);
    if (__any_sync(0xffffffffu, entry_special<NPTS>(emax))) {     // a pair in a cell with more candidates (rare for n <= 64)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (entry_special<NPTS>(entry[k])) at[k] = nearest_special<NPTS>(v[c][k], entry[k], rsm);
    }
    uint32_t word = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      word |= ((at[k] - rc.search.grid) >> 3) << (k * BITS);
      v[c][k] = lds64(at[k]);
    }
    store_code_word<BITS>(codes_row, c, lane, word);
  }
  if (hat_row != nullptr) {      // uniform over the warp
    f32x2_t pr[NC][4];
    chunk_load_pred<NC>(pred_row, lane, pr);           // the rotation hides it
    chunk_finish_row<NC, kBf16>(rc, v, sf, pr, hat_row);
  }
}

// One token row of Algorithm 3 given the prediction.
template <int NC, int NPTS, bool kBf16>
__device__ __forceinline__ void chunk_decode_row(const ChunkRowCtx& rc, const f32x2_t* __restrict__ grid_s,
                                                 const uint8_t* __restrict__ codes_row, const uint16_t* __restrict__ scales_row,
                                                 const float* __restrict__ pred_row, uint16_t* __restrict__ hat_row) {
  constexpr int BITS = NPTS == 16 ? 4 : (NPTS == 64 ? 6 : 8);
  f32x2_t pr[NC][4], v[NC][4];
  float sf[NC];
  uint32_t word[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    word[c] = load_code_word<BITS>(codes_row, c, rc.lane);
    sf[c] = __half2float(__ushort_as_half(scales_row[(c * 256 + rc.lane * 8) >> rc.log_g]));
  }
  chunk_load_pred<NC>(pred_row, rc.lane, pr);
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) v[c][k] = grid_s[(word[c] >> (k * BITS)) & (NPTS - 1)];
  chunk_finish_row<NC, kBf16>(rc, v, sf, pr, hat_row);
}

}  // namespace aquakv
