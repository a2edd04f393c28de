// Alternative backbone quantizer (Section 4.1 "Alternative quantizers": the Quanto-style
// one, plain rounding to the nearest level after dividing by the group's largest magnitude, groups of 64
// values inside a token; Section 3.2: any quantizer Q can sit under the predictors) for the residual / add-back steps of
// Algorithm 2 and Algorithm 3.
//
// For b bits per value the levels are the 2^b signed integers -2^(b-1) .. 2^(b-1)-1 times the group
// scale; scale = absmax / 2^(b-1), stored as fp16 (clamped to 65504), and the ROUNDED scale normalises;
// a value goes to the nearest level, the lower one on an exact tie, saturating at the ends; a group of
// zeros has scale 0 and level 0.  The code of a value is level + 2^(b-1); codes are packed LSB-first in
// value order.  No rotation, no sign flips.
//
// Rotated variant (the appendix' additional results for Section 4.1: a backbone that puts a randomized
// Hadamard transform in front of ordinary scalar quantization, one group per row): had_block = h > 1
// multiplies the residual by the role's random signs, rotates every block of h values by the orthonormal
// Hadamard matrix, quantizes the ROTATED values as above (absmax after the rotation), and the inverse
// rotates level * scale back and applies the signs again (template argument kRot).
//
// One warp per row, the whole row in registers as packed pairs: v[c][k] holds values 256 c + 8 lane + 2 k and the next
// (16-byte accesses), so index bits 0-2 are register bits, bits 3-7 the lane's bits and bits 8-9 register bits again.  A
// group of g <= 256 values is g/8 neighbouring lanes, so its absmax is log2(g/8) shuffle steps; a larger one spans
// chunks.  A Hadamard block of h = 2^k values is one butterfly per index bit below k, on two values per instruction.
// The lane's 8 codes of a chunk are b contiguous bytes of the row's code stream.
//
// The kernels are bound by instruction issue, then by their memory traffic, so the loops over chunks are unrolled for the
// row width (address arithmetic was a third of the instructions) and the arithmetic is packed: 747 instead of 1273
// warp instructions to encode a row of 1024 values at b = 4, 9472 rows in 16.8 instead of 21.9 us (with predictor).
#pragma once

#include "codec.cuh"
#include "rowchunk.cuh"

namespace aquakv {

struct UniformArgs {
  const uint16_t* X;        // encode: target rows (16-bit) [T, ldX]
  long long ldX;
  const float* P;           // prediction rows (fp32) or nullptr [T, ldP]
  long long ldP;
  uint8_t* codes;           // [T, d * b / 8]
  uint16_t* scales;         // [T, d / g] fp16 bits
  uint16_t* hat;            // reconstruction rows or nullptr (encode) [T, ldHat]
  long long ldHat;
  int T;
  int d;                    // 256, 512 or 1024
  int log_g;                // 5 .. 10
};

constexpr int kUniformWarps = 4;

template <int BITS>
__device__ __forceinline__ void uniform_store_codes(uint8_t* dst, uint32_t word) {
  if constexpr (BITS == 2) {
    *reinterpret_cast<uint16_t*>(dst) = uint16_t(word);
  } else if constexpr (BITS == 4) {
    *reinterpret_cast<uint32_t*>(dst) = word;
  } else {
    dst[0] = uint8_t(word);
    dst[1] = uint8_t(word >> 8);
    dst[2] = uint8_t(word >> 16);
  }
}
template <int BITS>
__device__ __forceinline__ uint32_t uniform_load_codes(const uint8_t* src) {
  if constexpr (BITS == 2) return *reinterpret_cast<const uint16_t*>(src);
  else if constexpr (BITS == 4) return *reinterpret_cast<const uint32_t*>(src);
  else return uint32_t(src[0]) | (uint32_t(src[1]) << 8) | (uint32_t(src[2]) << 16);
}

__device__ __forceinline__ f32x2_t add2_ru(f32x2_t a, f32x2_t b) {      // rounded up
  f32x2_t r;
  asm("add.rp.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Levels (as floats, in place of the values) and packed codes of a lane's eight values: the nearest level, the lower one
// on a tie, is ceil(r / sf - 0.5).  The quotient r * (1 / sf) is within 2e-6 of it, so with 2^-17 taken off the
// rounding up gives the level or the one below, and the sign of r - (level + 1/2) sf, which one FMA gives exactly,
// decides.  The rounding up is an addition of 1.5 * 2^23 + 2^(b-1), which also leaves the code in the low mantissa
// bits: no division and no conversion (both took the special-function pipe: 128 of its instructions a row of 1024).
template <int BITS>
__device__ __forceinline__ uint32_t uniform_levels(f32x2_t (&r)[4], float sf) {
  constexpr int HALF = 1 << (BITS - 1);
  constexpr float M = 12582912.0f + HALF;
  const float inv = sf > 0.0f ? __frcp_rn(sf) : 0.0f;
  const float den = sf > 0.0f ? sf : __int_as_float(0x7f800000);      // a zero scale leaves every value at level 0
  const f32x2_t inv2 = pack2(inv, inv), den2 = pack2(den, den), m2 = pack2(M, M);
  const f32x2_t off2 = pack2(-0.5f - 7.62939453125e-6f, -0.5f - 7.62939453125e-6f), half2 = pack2(0.5f, 0.5f);
  uint32_t word = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const f32x2_t t2 = add2_ru(fma2(r[k], inv2, off2), m2);
    float t[2], over[2];
    unpack2(t2, t[0], t[1]);
    unpack2(fma2(sub2(sub2(m2, t2), half2), den2, r[k]), over[0], over[1]);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (over[e] > 0.0f) t[e] += 1.0f;
      t[e] = fminf(fmaxf(t[e], M - HALF), M + (HALF - 1));
      word |= (__float_as_uint(t[e]) & uint32_t((1 << BITS) - 1)) << (BITS * (2 * k + e));
    }
    r[k] = sub2(pack2(t[0], t[1]), m2);
  }
  return word;
}

// Levels (as floats) of a lane's eight codes.
template <int BITS>
__device__ __forceinline__ void uniform_code_levels(uint32_t word, f32x2_t (&q)[4]) {
  constexpr float M = 12582912.0f + (1 << (BITS - 1));
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t a = (word >> (BITS * 2 * k)) & uint32_t((1 << BITS) - 1), b = (word >> (BITS * (2 * k + 1))) & uint32_t((1 << BITS) - 1);
    q[k] = sub2(pack2(__uint_as_float(a | 0x4B400000u), __uint_as_float(b | 0x4B400000u)), pack2(M, M));
  }
}

struct UniformRotArgs {
  UniformArgs u;              // plain variant: the rest is not read
  const uint32_t* signmask;   // [32]: lane's word, bit 8 c + i set where the sign of value 256 c + 8 lane + i is -1
  int log_h;                  // 6 .. 10
};

// The lane's values of row t of the prediction (zeros without one).  kStream: its last read (evict-first); otherwise it
// stays cached for a second one.
template <int NCH, bool kStream = true>
__device__ __forceinline__ void row_load_pred(const UniformArgs& a, long long t, int lane, f32x2_t (&pred)[NCH][4]) {
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    if (a.P != nullptr) {
      const float4* p = reinterpret_cast<const float4*>(a.P + t * a.ldP + 256 * c + 8 * lane);
      const float4 lo = kStream ? __ldcs(p) : p[0], hi = kStream ? __ldcs(p + 1) : p[1];
      pred[c][0] = pack2(lo.x, lo.y);
      pred[c][1] = pack2(lo.z, lo.w);
      pred[c][2] = pack2(hi.x, hi.y);
      pred[c][3] = pack2(hi.z, hi.w);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) pred[c][k] = pack2(0.0f, 0.0f);
    }
  }
}

// v = x - pred for row t.
template <bool kBf16, int NCH>
__device__ __forceinline__ void row_residual(const UniformArgs& a, long long t, int lane, const f32x2_t (&pred)[NCH][4],
                                             f32x2_t (&v)[NCH][4]) {
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    const uint4 raw = __ldcs(reinterpret_cast<const uint4*>(a.X + t * a.ldX + 256 * c + 8 * lane));
    v[c][0] = sub2(load16x2<kBf16>(raw.x), pred[c][0]);
    v[c][1] = sub2(load16x2<kBf16>(raw.y), pred[c][1]);
    v[c][2] = sub2(load16x2<kBf16>(raw.z), pred[c][2]);
    v[c][3] = sub2(load16x2<kBf16>(raw.w), pred[c][3]);
  }
}

template <bool kBf16>
__device__ __forceinline__ void row_store_pair4(uint16_t* dst, const f32x2_t (&h)[4]) {
  __stcs(reinterpret_cast<uint4*>(dst), make_uint4(store16x2p<kBf16>(h[0]), store16x2p<kBf16>(h[1]), store16x2p<kBf16>(h[2]),
                                                   store16x2p<kBf16>(h[3])));
}

// hat = round16(pred + f[c] * signs . (rs * H(y))) for the row's values y before the inverse rotation.  rs = 1 / sqrt(h)
// is a rounding of its own, after the rotation in both directions: on the signs before it, which saves a multiplication,
// it moves last bits wherever it is no power of two (h = 128, 512), and with them codes.
template <bool kBf16, int NCH>
__device__ __forceinline__ void row_rotate_back(const UniformArgs& a, long long t, int lane, int log_h, uint32_t sbits, float rs,
                                                f32x2_t (&y)[NCH][4], const float (&f)[NCH], const f32x2_t (&pred)[NCH][4]) {
  row_hadamard<NCH>(y, log_h, lane);
  const f32x2_t rs2 = pack2(rs, rs);
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
#pragma unroll
    for (int k = 0; k < 4; ++k) y[c][k] = fma2(mul2(y[c][k], rs2), row_signed(f[c], sbits, c, k), pred[c][k]);
    row_store_pair4<kBf16>(a.hat + t * a.ldHat + 256 * c + 8 * lane, y[c]);
  }
}

// codes, scales = Q(x - pred);  hat = round16(pred + Q^-1(codes, scales)).  kRot: with the rotation.
template <int BITS, bool kBf16, int NCH, bool kRot>
__global__ void __launch_bounds__(kUniformWarps * 32, 4)
uniform_encode_rows_kernel(const UniformRotArgs ra) {
  constexpr int HALF = 1 << (BITS - 1);
  const UniformArgs& a = ra.u;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * kUniformWarps + (threadIdx.x >> 5);
  const long long n_warps = (long long)gridDim.x * kUniformWarps;
  const int lanes_per_group = a.log_g >= 8 ? 32 : 1 << (a.log_g - 3);
  const int chunks_per_group = a.log_g > 8 ? 1 << (a.log_g - 8) : 1;
  const int n_groups = (256 * NCH) >> a.log_g;
  const uint32_t sbits = kRot ? ra.signmask[lane] : 0u;
  const float rs = kRot ? rsqrtf(float(1 << ra.log_h)) : 1.0f;
  pdl_sync();
  for (long long t = warp; t < a.T; t += n_warps) {
    f32x2_t v[NCH][4], pred[NCH][4];
    row_load_pred<NCH>(a, t, lane, pred);
    row_residual<kBf16, NCH>(a, t, lane, pred, v);
    if constexpr (kRot) {
#pragma unroll
      for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[c][k] = mul2(v[c][k], row_signed(1.0f, sbits, c, k));
      row_hadamard<NCH>(v, ra.log_h, lane);
      const f32x2_t rs2 = pack2(rs, rs);
#pragma unroll
      for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[c][k] = mul2(v[c][k], rs2);
    }
    // group absmax
    float m[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      m[c] = 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float lo, hi;
        unpack2(v[c][k], lo, hi);
        m[c] = fmaxf(m[c], fmaxf(fabsf(lo), fabsf(hi)));
      }
    }
    for (int off = 1; off < lanes_per_group; off <<= 1) {
#pragma unroll
      for (int c = 0; c < NCH; ++c) m[c] = fmaxf(m[c], __shfl_xor_sync(0xffffffffu, m[c], off));
    }
    // a group of several chunks: the maximum over its chunks (mg is a second array: m is read in full)
    float mg[NCH];
#pragma unroll
    for (int c0 = 0; c0 < NCH; ++c0) {
      mg[c0] = 0.0f;
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        if ((c & ~(chunks_per_group - 1)) == (c0 & ~(chunks_per_group - 1))) mg[c0] = fmaxf(mg[c0], m[c]);
    }
    uint8_t* codes = a.codes + t * (long long)(32 * NCH * BITS) + lane * BITS;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const __half s16 = __float2half_rn(fminf(mg[c] * (1.0f / HALF), 65504.0f));
      const float sf = __half2float(s16);
      if ((lane & (lanes_per_group - 1)) == 0 && (c & (chunks_per_group - 1)) == 0)
        a.scales[t * n_groups + ((256 * c + 8 * lane) >> a.log_g)] = __half_as_ushort(s16);
      uniform_store_codes<BITS>(codes + 32 * c * BITS, uniform_levels<BITS>(v[c], sf));
      const f32x2_t sf2 = pack2(sf, sf);
      if constexpr (kRot) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[c][k] = mul2(v[c][k], sf2);            // a block may span groups
      } else if (a.hat != nullptr) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[c][k] = fma2(v[c][k], sf2, pred[c][k]);
        row_store_pair4<kBf16>(a.hat + t * a.ldHat + 256 * c + 8 * lane, v[c]);
      }
    }
    if constexpr (kRot) {
      float f[NCH];
#pragma unroll
      for (int c = 0; c < NCH; ++c) f[c] = 1.0f;
      if (a.hat != nullptr) row_rotate_back<kBf16, NCH>(a, t, lane, ra.log_h, sbits, rs, v, f, pred);
    }
  }
}

// hat = round16(pred + Q^-1(codes, scales)).
template <int BITS, bool kBf16, int NCH, bool kRot>
__global__ void __launch_bounds__(kUniformWarps * 32, 4)
uniform_decode_rows_kernel(const UniformRotArgs ra) {
  const UniformArgs& a = ra.u;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * kUniformWarps + (threadIdx.x >> 5);
  const long long n_warps = (long long)gridDim.x * kUniformWarps;
  const int n_groups = (256 * NCH) >> a.log_g;
  const uint32_t sbits = kRot ? ra.signmask[lane] : 0u;
  const float rs = kRot ? rsqrtf(float(1 << ra.log_h)) : 1.0f;
  pdl_sync();
  for (long long t = warp; t < a.T; t += n_warps) {
    f32x2_t y[NCH][4], pred[NCH][4];
    row_load_pred<NCH>(a, t, lane, pred);
    const uint8_t* codes = a.codes + t * (long long)(32 * NCH * BITS) + lane * BITS;
    uint32_t word[NCH];
    float sf[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      word[c] = uniform_load_codes<BITS>(codes + 32 * c * BITS);
      sf[c] = __half2float(__ushort_as_half(a.scales[t * n_groups + ((256 * c + 8 * lane) >> a.log_g)]));
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      uniform_code_levels<BITS>(word[c], y[c]);
      const f32x2_t sf2 = pack2(sf[c], sf[c]);
      if constexpr (kRot) {
#pragma unroll
        for (int k = 0; k < 4; ++k) y[c][k] = mul2(y[c][k], sf2);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) y[c][k] = fma2(y[c][k], sf2, pred[c][k]);
        row_store_pair4<kBf16>(a.hat + t * a.ldHat + 256 * c + 8 * lane, y[c]);
      }
    }
    if constexpr (kRot) {
      float f[NCH];
#pragma unroll
      for (int c = 0; c < NCH; ++c) f[c] = 1.0f;
      row_rotate_back<kBf16, NCH>(a, t, lane, ra.log_h, sbits, rs, y, f, pred);
    }
  }
}

}  // namespace aquakv
