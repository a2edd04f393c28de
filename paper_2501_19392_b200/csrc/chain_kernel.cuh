// Algorithm 4's loop over layers for SMALL calls (a decode step of a batch of sequences, a short
// prompt): Algorithm 2 (encode) or Algorithm 3 (decode) for every layer in ONE persistent launch.
//
// Why a second kernel.  The per-layer kernel (layer_kernel.cuh) is built for tens of thousands of
// tokens: a 128 x 256 tcgen05 tile per CTA pair, a wave of token blocks per job.  With 64 tokens one
// layer is a chain of four dependent steps (key prediction -> key rows -> value prediction -> value
// rows) in which four CTA pairs stream 6 MB of adapter weights while 140 SMs wait, and every layer
// pays a launch, a prologue and six tensor-map encodings.  The bound of such a call is the weight
// stream (6 d^2 bytes per layer) and the latency of the hand-offs, not arithmetic.  So here
//   - a warp owns 32 features x 128 input features of a layer's weights and holds them in registers
//     (64 of its 128): it loads them as soon as its rows of the layer before are done, while it would
//     otherwise wait for the other CTAs' rows, and multiplies one 16-token tile after the other with them.  The
//     products are warp-level m16n8k16 tensor-core products whose operand fragments come straight from 16-byte
//     global loads (the order of the summation index inside a 32-element chunk is free as long as both operands
//     use the same one).  So a token tile costs an SM 64 KB of activations on the critical path instead of
//     320 KB of weights and activations (units of 16 x 64 x 128, both operands loaded after the wait).  The tcgen05 path needs M >= 64 rows per instruction and an operand round
//     trip through shared memory, which a 16-row unit bound by its load latency does not repay;
//   - the slices of one output tile (8 or 16, of 128 input features) run on the warps of one CTA
//     at the same time and are added through shared memory in ascending slice order (then the bias),
//     so the result does not depend on timing and the fp32 prediction is written once; the CTAs that
//     cover all features once form a group, and the groups of a team share the token tiles;
//   - the key chain (K^_l needs only K^_{l-1}) runs on one team of CTAs, the value chain
//     (V^_l needs V^_{l-1} and K^_l) on another, one layer behind where it must be, so a layer costs
//     the key chain's two hand-offs, not four;
//   - the data themselves say when they are there: a prediction is an 8-byte word of the value and the number of
//     its layer, and the reconstructions that later products read lie in buffers of their own, one per layer,
//     preset to a word (two NaNs of one pattern) that no reconstruction contains.  A reader polls the words it needs,
//     with loads of word size that bypass L1, so no order between words is assumed.  (A counter per tile and stage, behind a
//     fence, cost 1.0-1.6 thousand cycles for the fence and about as much again between the counter's arrival
//     and the data's, four times a layer.)  Every wait is bounded, all CTAs are resident (at most one per SM), and a
//     stage only waits on earlier stages, so the schedule cannot dead-lock;
//   - a warp that has loaded its weights asks L2 for those of the next layer, and a row team for its next row's input;
//   - the decoder rotates a row's codes back before the layer's prediction stage, while the rows of the
//     layer before are on their way; what follows the prediction is one FMA per value.
// The row work itself is that of codec.cuh / rowwarp.cuh, unchanged.
//
// The partial sums are added in a different order than the per-layer kernel's single accumulation,
// so reconstructions can differ from that kernel's in the last bit of the 16-bit type; a cache
// written by the chain encoder is reproduced bit for bit by the chain decoder.
#pragma once

#include "attn.cuh"
#include "codec.cuh"
#include "common.cuh"
#include "layer_kernel.cuh"
#include "rowwarp.cuh"

namespace aquakv {

constexpr int kChainMaxLayers = 128;
constexpr int kChainWarps = 16;
constexpr int kChainThreads = kChainWarps * 32;
constexpr int kChainMT = 16;       // tokens of a unit (MMA M)
constexpr int kChainNT = 32;       // output features of a unit
constexpr int kChainKS = 128;      // input features of a unit
constexpr int kChainMB = 2;        // token tiles between two CTA barriers
constexpr int kChainRedLd = 40;    // floats between the rows of a partial product in shared memory (8-byte accesses of a
                                   // quarter-warp's four rows fall on different banks)

struct ChainLayer {
  const uint16_t* K;       // encode targets [T, ldX] (encode only)
  const uint16_t* V;
  const uint16_t* Wk;      // [d][d]; nullptr: the layer has no predictor
  const uint16_t* Wv;      // [d][2d]
  const float* bk;         // optional biases
  const float* bv;
  uint8_t* Kcodes;         // written by encode, read by decode
  uint16_t* Kscales;
  uint8_t* Vcodes;
  uint16_t* Vscales;
  uint16_t* Khat;          // this layer's reconstruction [T, ldHat] for the caller, or nullptr
  uint16_t* Vhat;
  uint16_t* Kpass;         // the same [T, d] for the products that read it, preset to kChainEmpty; nullptr: none does
  uint16_t* Vpass;
  long long ldHat;
};

struct ChainArgs {
  int T, L;
  long long ldX;
  const uint16_t* Khat_init;   // reconstruction of the layer before the first one (needed iff layer 0 has a predictor)
  const uint16_t* Vhat_init;
  long long ldInit;
  unsigned long long* Pk;      // key predictions   [T][d]: fp32 value in the low half, layer in the high half (preset to ones)
  unsigned long long* Pv;      // value predictions [T][d]
  int n_ctas_k;                // CTAs of the key team (the rest run the value chain)
  const uint32_t* signmask_k;
  const uint32_t* signmask_v;
  const float4* grid4;
  SearchDev search;
  int log_h, log_g;
  int* status;
  ChainLayer layer[kChainMaxLayers];
};

// A warp's weights: features n0 .. n0+31, input features kw .. kw+127, as the B fragments of eight k-steps.
struct ChainWeights {
  uint4 b[kChainKS / 32][kChainNT / 8];
};
__device__ __forceinline__ void chain_load_weights(ChainWeights& w, const uint16_t* __restrict__ W, long long ldW, int n0, int kw,
                                                   int lane) {
  const uint16_t* pw = W + (long long)(n0 + (lane >> 2)) * ldW + kw + (lane & 3) * 8;
#pragma unroll
  for (int c = 0; c < kChainKS / 32; ++c) {
#pragma unroll
    for (int nt = 0; nt < kChainNT / 8; ++nt) w.b[c][nt] = __ldg(reinterpret_cast<const uint4*>(pw + (long long)nt * 8 * ldW + c * 32));
  }
}

constexpr uint32_t kChainEmpty = 0xffffffffu;

// A bounded wait's bookkeeping: true while the caller may go on polling.
struct ChainPoll {
  volatile int* abort_flag;
  int* status;
  unsigned long long t0 = 0;
  uint32_t spins = 0;
  __device__ __forceinline__ ChainPoll(volatile int* f, int* s) : abort_flag(f), status(s) {}
  __device__ __forceinline__ bool again() {
    if (t0 == 0) t0 = global_timer_ns();
    __nanosleep(20);
    if ((++spins & 0xFFu) == 0) {
      if (*abort_flag) return false;
      if (global_timer_ns() - t0 > kWaitLimitNs) {
        *abort_flag = 1;
        atomicExch(status, kStatusTimeout);
        return false;
      }
    }
    return true;
  }
};
__device__ __forceinline__ uint4 ld_relaxed4(const void* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_relaxed1(const void* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A prediction row that other SMs are writing.  A wait that runs out leaves what was read: the abort flag ends the
// call at the next layer and no warp of a row's team is left alone at a barrier.
struct ChainPred {
  const unsigned long long* row;     // nullptr: the layer has no predictor
  uint32_t layer;
  volatile int* abort_flag;
  int* status;
  __device__ __forceinline__ ChainPred operator+(int i) const { return ChainPred{row + i, layer, abort_flag, status}; }
  __device__ __forceinline__ bool operator!=(decltype(nullptr)) const { return row != nullptr; }
};
// Called by whole warps.
__device__ __forceinline__ void chain_pred8(const ChainPred& p, float (&f)[8]) {
  ChainPoll poll(p.abort_flag, p.status);
  bool there;
  do {
    there = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      unsigned long long w0, w1;
      asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p.row + 2 * i) : "memory");
      f[2 * i] = __uint_as_float(uint32_t(w0));
      f[2 * i + 1] = __uint_as_float(uint32_t(w1));
      there = there && uint32_t(w0 >> 32) == p.layer && uint32_t(w1 >> 32) == p.layer;
    }
    there = __all_sync(0xffffffffu, there);
  } while (!there && __any_sync(0xffffffffu, poll.again()));
}
__device__ __forceinline__ void pred_load8(const ChainPred& p, float4& a, float4& b) {
  float f[8];
  chain_pred8(p, f);
  a = make_float4(f[0], f[1], f[2], f[3]);
  b = make_float4(f[4], f[5], f[6], f[7]);
}
__device__ __forceinline__ void wr_load_pred8(const ChainPred& p, f32x2_t (&out)[4]) {
  float f[8];
  chain_pred8(p, f);
#pragma unroll
  for (int i = 0; i < 4; ++i) out[i] = pack2(f[2 * i], f[2 * i + 1]);
}
// The words that this lane has polled before: plain loads, which may overlap one another (polled again, each chunk of a
// row cost the encoder a trip to L2 of its own: 256 tokens 22.5 -> 21.2 us per layer).
struct ChainSettledPred {
  const unsigned long long* row;
  __device__ __forceinline__ ChainSettledPred operator+(int i) const { return ChainSettledPred{row + i}; }
  __device__ __forceinline__ bool operator!=(decltype(nullptr)) const { return row != nullptr; }
};
template <> struct SettledPred<ChainPred> { typedef ChainSettledPred type; };
__device__ __forceinline__ ChainSettledPred pred_settled(const ChainPred& p) { return ChainSettledPred{p.row}; }
__device__ __forceinline__ void wr_load_pred8(const ChainSettledPred& p, f32x2_t (&out)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2*>(p.row + 2 * i));
    out[i] = pack2(__uint_as_float(uint32_t(w.x)), __uint_as_float(uint32_t(w.y)));
  }
}

// A reconstruction row: the caller's and the one later products read.
struct ChainHat {
  uint16_t* out;
  uint16_t* pass;
  __device__ __forceinline__ ChainHat operator+(int i) const {
    return ChainHat{out != nullptr ? out + i : nullptr, pass != nullptr ? pass + i : nullptr};
  }
  __device__ __forceinline__ bool operator!=(decltype(nullptr)) const { return out != nullptr || pass != nullptr; }
};
__device__ __forceinline__ void hat_store8(const ChainHat& h, const uint4& v) {
  if (h.pass != nullptr) {
    auto full = [](uint32_t w) { return w == kChainEmpty ? 0x7fff7fffu : w; };      // two NaNs stay two NaNs
    asm volatile("st.relaxed.gpu.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(h.pass), "r"(full(v.x)), "r"(full(v.y)),
                 "r"(full(v.z)), "r"(full(v.w))
                 : "memory");
  }
  if (h.out != nullptr) __stcs(reinterpret_cast<uint4*>(h.out), v);
}

// One unit: the 16 x 32 fp32 partial product  A[row0 .. row0+15][k-slice] . W[n0 .. n0+31][k-slice]^T,
// left in `red` (rows of kChainRedLd floats, shared memory) for the CTA's reduction over the slices.
// fresh: A is written during this kernel (a preset buffer); otherwise it is the caller's and complete.  first: the first
// tile after the rows' stage, for which the warp may have to wait.
template <bool kBf16>
__device__ __forceinline__ void chain_gemm_unit(const uint16_t* __restrict__ A, long long ldA, int ka, bool fresh, bool first, const ChainWeights& w,
                                                int row0, int T, volatile int* abort_flag, int* status,
                                                float* __restrict__ red, int lane) {
  const int g = lane >> 2, j = lane & 3;
  if (fresh && first) {
    // one word of each half of a row's slice until the rows are there: polling whole rows would load L2
    const int rp = row0 + (lane & 15) < T ? row0 + (lane & 15) : T - 1;
    const uint16_t* pp = A + (long long)rp * ldA + ka + (lane >> 4) * 64;
    ChainPoll poll(abort_flag, status);
    while (!__all_sync(0xffffffffu, ld_relaxed1(pp) != kChainEmpty) && __any_sync(0xffffffffu, poll.again())) {
    }
  }
  const int ra = row0 + g < T ? row0 + g : T - 1, rb = row0 + g + 8 < T ? row0 + g + 8 : T - 1;
  const uint16_t* pa = A + (long long)ra * ldA + ka + j * 8;
  const uint16_t* pb = A + (long long)rb * ldA + ka + j * 8;
  constexpr int NC = kChainKS / 32;
  uint4 alo[NC], ahi[NC];
  ChainPoll poll(abort_flag, status);
  for (;;) {
    uint32_t most = 0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      alo[c] = ld_relaxed4(pa + c * 32);
      ahi[c] = ld_relaxed4(pb + c * 32);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      most = max(most, max(max(alo[c].x, alo[c].y), max(alo[c].z, alo[c].w)));
      most = max(most, max(max(ahi[c].x, ahi[c].y), max(ahi[c].z, ahi[c].w)));
    }
    if (!fresh || __all_sync(0xffffffffu, most != kChainEmpty) || !__any_sync(0xffffffffu, poll.again())) break;
  }
  float acc[kChainNT / 8][4];
#pragma unroll
  for (int nt = 0; nt < kChainNT / 8; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.0f;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
#pragma unroll
    for (int nt = 0; nt < kChainNT / 8; ++nt) {
      const uint4 b = w.b[c][nt];
      mma_16x8x16<kBf16>(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3], alo[c].x, ahi[c].x, alo[c].y, ahi[c].y, b.x, b.y);
      mma_16x8x16<kBf16>(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3], alo[c].z, ahi[c].z, alo[c].w, ahi[c].w, b.z, b.w);
    }
  }
#pragma unroll
  for (int nt = 0; nt < kChainNT / 8; ++nt) {
    *reinterpret_cast<float2*>(red + g * kChainRedLd + nt * 8 + 2 * j) = make_float2(acc[nt][0], acc[nt][1]);
    *reinterpret_cast<float2*>(red + (g + 8) * kChainRedLd + nt * 8 + 2 * j) = make_float2(acc[nt][2], acc[nt][3]);
  }
}

template <int D, int NPTS, bool kEncode, bool kWarpRows>
struct ChainSmem {
  typename LayerTables<kEncode, NPTS>::type tables;
  LayerRowScratch<D, kChainWarps, kWarpRows> scratch;
  float red[kChainWarps][kChainMB][kChainMT * kChainRedLd];     // partial products per warp
  // decoder with row teams: the rotated-back codes and the scales of a team's first row of a layer
  ulonglong2 ahead[kEncode || kWarpRows ? 1 : kChainWarps][2][32];
  float ahead_scale[kEncode || kWarpRows ? 1 : kChainWarps][32];
  ChainLayer layer[kChainMaxLayers];     // ChainArgs::layer: read from the constant bank, every layer's pointers missed its cache
  int abort_flag;
};

// kWarpRows (D = 1024 with Hadamard block = scale group = 1024 only, checked on the host): the
// one-warp-per-row routines, which keep more rows in flight; otherwise the team routines (D / 256 warps per
// row, any supported block / group), whose rows finish sooner.  A layer of a small call is a chain of
// dependent steps, so the host picks the team routines while every row still gets a team at once and the warp routines beyond
// (run_chain's launch_chain_dnb has the times of both).
template <bool kEncode, int D, int NPTS, bool kBf16, bool kWarpRows>
__global__ void __launch_bounds__(kChainThreads, 1) chain_kernel(const __grid_constant__ ChainArgs a) {
  static_assert(!kWarpRows || D == 1024, "one warp per row needs d_kv = 1024");
  constexpr bool WR = kWarpRows;
  constexpr int TEAM = WR ? 1 : RowTeam<D>::TEAM;
  constexpr int BITS = NPTS == 16 ? 4 : (NPTS == 64 ? 6 : 8);
  constexpr int CODE_BYTES = D / 2 * BITS / 8;
  constexpr int NTILES = D / kChainNT;               // feature tiles of a row
  extern __shared__ __align__(16) uint8_t chain_smem_raw[];
  using Smem = ChainSmem<D, NPTS, kEncode, kWarpRows>;
  Smem* sm = reinterpret_cast<Smem*>(smem_align<int(alignof(Smem))>(chain_smem_raw));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if constexpr (kEncode) {
    row_smem_fill<NPTS>(&sm->tables, a.search.table, a.grid4);
  } else {
    for (int i = threadIdx.x; i < NPTS; i += blockDim.x) {
      const float4 g = a.grid4[i];
      sm->tables.grid[i] = pack2(g.x, g.y);
    }
  }
  if (threadIdx.x == 0) sm->abort_flag = 0;
  for (int i = threadIdx.x; i < a.L * int(sizeof(ChainLayer) / 4); i += blockDim.x)
    reinterpret_cast<uint32_t*>(sm->layer)[i] = reinterpret_cast<const uint32_t*>(a.layer)[i];
  __syncthreads();
  pdl_sync();
  volatile int* abort_flag = &sm->abort_flag;

  const bool is_v = int(blockIdx.x) >= a.n_ctas_k;
  const int team_ctas = is_v ? int(gridDim.x) - a.n_ctas_k : a.n_ctas_k;
  const int n_warps = team_ctas * kChainWarps;
  const int n_mt = (a.T + kChainMT - 1) / kChainMT;
  const int n_in = is_v ? 2 : 1;
  const int n_slices = n_in * D / kChainKS;
  unsigned long long* P = is_v ? a.Pv : a.Pk;
  const int log_h = WR ? 10 : a.log_h, log_g = WR ? 10 : a.log_g;
  const int n_groups = D >> log_g;

  // row contexts
  RowCtx rck;
  WarpRowCtx wrc;
  if constexpr (WR) {
    wrc.lane = lane;
    if constexpr (kEncode) wrc.search = search_ctx<NPTS>(&sm->tables, a.search.inv_w);
    wrc.signs = (is_v ? a.signmask_v : a.signmask_k)[lane];
    rck.member = 0;
    rck.barrier = 0;
  } else {
    row_ctx_init(rck, is_v ? a.signmask_v : a.signmask_k, a.search.inv_w, log_h, log_g, lane, warp % TEAM,
                 RowTeam<D>::NV, 1 + warp / TEAM);
  }

  const int cta = int(blockIdx.x) - (is_v ? a.n_ctas_k : 0);
  const int tiles_per_cta = kChainWarps / n_slices;                 // feature tiles of a CTA: 1 .. 8
  const int set = NTILES / tiles_per_cta;                           // CTAs of a group (they cover all features once)
  const int n_groups_mt = team_ctas >= set ? team_ctas / set : 1;   // groups: token tile mt belongs to group mt mod n_groups_mt
  const int n_sets = n_groups_mt * set;
  // consecutive rows go to different CTAs, so that a stage of few rows has an SM per row
  const int team = (warp / TEAM) * team_ctas + cta, n_teams = n_warps / TEAM;
  // the part of decoding row r of layer l that needs no prediction
  auto load_codes = [&](int l, int r, uint32_t (&words)[1], float (&sf)[1]) {
    if constexpr (!kEncode && !WR) {
      const ChainLayer& ly = sm->layer[l];
      decode_row_load_codes<D, NPTS>(rck, (is_v ? ly.Vcodes : ly.Kcodes) + (long long)r * CODE_BYTES,
                                     (is_v ? ly.Vscales : ly.Kscales) + (long long)r * n_groups, words, sf);
    }
  };
  auto rotate_codes = [&](uint32_t word, f32x2_t (&wp)[4]) {
    if constexpr (!kEncode && !WR) {
#pragma unroll
      for (int k = 0; k < 4; ++k) wp[k] = sm->tables.grid[(word >> (k * BITS)) & (NPTS - 1)];
      team_rotate_back<D>(rck, &sm->scratch.team[warp / TEAM], wp);
    }
  };
  for (int l = 0; l < a.L; ++l) {
    const ChainLayer& ly = sm->layer[l];
    const bool has_pred = ly.Wk != nullptr;
    const uint16_t* W = is_v ? ly.Wv : ly.Wk;
    const long long ldW = (long long)n_in * D;
    // this warp's part of a group: feature tile `nt` and slice `ks`
    const int wi = warp / n_slices, ks = warp % n_slices;
    ChainWeights wreg;
    auto load_weights = [&](int s) {
      const int nt = (s % set) * tiles_per_cta + wi;
      chain_load_weights(wreg, W, ldW, nt * kChainNT, ks * kChainKS, lane);
      // the next layer's weights depend on nothing: towards L2
      const uint16_t* Wn = l + 1 < a.L ? (is_v ? sm->layer[l + 1].Wv : sm->layer[l + 1].Wk) : nullptr;
      if (Wn != nullptr) {
        const uint16_t* pw = Wn + (long long)(nt * kChainNT + lane) * ldW + ks * kChainKS;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pw));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pw + 64));
      }
    };
    uint32_t words[1] = {0u};
    float sf[1] = {0.0f};
    if (!kEncode && !WR && team < a.T) load_codes(l, team, words, sf);
    if (has_pred && cta < n_sets) load_weights(cta);
    // The same row's input of the next layer: towards L2.  (Here, where the reconstructions of the layer before are still on
    // their way: a prefetch from a page that the SM has not touched held up the loads behind it for 1500 cycles.)
    if (l + 1 < a.L && team < a.T) {
      const ChainLayer& nx = sm->layer[l + 1];
      if constexpr (kEncode) {
        const uint16_t* x_row = (is_v ? nx.V : nx.K) + (long long)team * a.ldX;
        if (lane * 64 < D / TEAM) asm volatile("prefetch.global.L2 [%0];" ::"l"(x_row + rck.member * (D / TEAM) + lane * 64));
      } else {
        const uint8_t* c_row = (is_v ? nx.Vcodes : nx.Kcodes) + (long long)team * CODE_BYTES;
        if (lane * 128 < CODE_BYTES / TEAM)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(c_row + rck.member * (CODE_BYTES / TEAM) + lane * 128));
        if (lane == 31 && rck.member == 0)
          asm volatile("prefetch.global.L2 [%0];" ::"l"((is_v ? nx.Vscales : nx.Kscales) + (long long)team * n_groups));
      }
    }
    if constexpr (!kEncode && !WR) {
      if (team < a.T) {
        f32x2_t wp[4];
        rotate_codes(words[0], wp);
#pragma unroll
        for (int i = 0; i < 2; ++i) sm->ahead[warp][i][lane] = make_ulonglong2(wp[2 * i], wp[2 * i + 1]);
        sm->ahead_scale[warp][lane] = sf[0];
      }
    }
    // the warps of a CTA enter a layer together (its prediction stage uses CTA-wide barriers), and a
    // wait that expired anywhere in the CTA ends the kernel for all of them here
    if (__syncthreads_or(*abort_flag)) break;
    // ------------------------------------------------------------------------------------------
    // predictions of this layer: the n_slices slices of an output tile (16 tokens x 32 features) run on
    // n_slices warps of ONE CTA and are added through shared memory in ascending slice order
    // ------------------------------------------------------------------------------------------
    if (has_pred) {
      const float* bias = is_v ? ly.bv : ly.bk;
      const uint16_t* prev = is_v ? (l == 0 ? a.Vhat_init : sm->layer[l - 1].Vpass) : (l == 0 ? a.Khat_init : sm->layer[l - 1].Kpass);
      const bool from_k = is_v && ks * kChainKS >= D;           // this slice reads the layer's fresh K^
      const uint16_t* A = from_k ? ly.Kpass : prev;
      const bool fresh = from_k || l > 0;
      const long long ldA = fresh ? D : a.ldInit;
      const int ka = from_k ? ks * kChainKS - D : ks * kChainKS;
      bool stop = false;
      for (int s = cta; !stop && s < n_sets; s += team_ctas) {      // once, unless the team is smaller than a group
        if (s != cta) load_weights(s);
        const int col0 = (s % set) * tiles_per_cta * kChainNT;
        for (int mt0 = s / set; mt0 < n_mt; mt0 += kChainMB * n_groups_mt) {
#pragma unroll 1
          for (int b = 0; b < kChainMB; ++b) {
            const int mt = mt0 + b * n_groups_mt;
            if (mt >= n_mt) break;
            // The rows of the previous layer are also the last readers of the prediction tile that this pass
            // overwrites: together the slices have seen every part of their reconstructions, which were formed from it.
            chain_gemm_unit<kBf16>(A, ldA, ka, fresh, b == 0, wreg, mt * kChainMT, a.T, abort_flag, a.status, sm->red[warp][b], lane);
          }
          if (__syncthreads_or(*abort_flag)) { stop = true; break; }
          // two neighbouring features per thread and step
          constexpr int PAIRS = kChainMT * kChainNT / 2;
          for (int o = threadIdx.x; o < kChainMB * tiles_per_cta * PAIRS; o += kChainThreads) {
            const int b = o / (tiles_per_cta * PAIRS), ti = o / PAIRS % tiles_per_cta, r = o % PAIRS / (kChainNT / 2),
                      cc = o % (kChainNT / 2) * 2;
            const int row = (mt0 + b * n_groups_mt) * kChainMT + r, col = col0 + ti * kChainNT + cc;
            if (row >= a.T) continue;
            const float* src = &sm->red[ti * n_slices][b][r * kChainRedLd + cc];
            constexpr int STEP = kChainMB * kChainMT * kChainRedLd;
            float2 sum = *reinterpret_cast<const float2*>(src);
            for (int sl = 1; sl < n_slices; ++sl) {
              const float2 v = *reinterpret_cast<const float2*>(src + sl * STEP);
              sum.x += v.x;
              sum.y += v.y;
            }
            if (bias != nullptr) {
              sum.x += __ldg(bias + col);
              sum.y += __ldg(bias + col + 1);
            }
            asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(P + (long long)row * D + col),
                         "l"((unsigned long long)(uint32_t(l)) << 32 | __float_as_uint(sum.x)),
                         "l"((unsigned long long)(uint32_t(l)) << 32 | __float_as_uint(sum.y))
                         : "memory");
          }
          __syncthreads();      // before the next partial products
        }
      }
      if (stop) break;
    }
    // ------------------------------------------------------------------------------------------
    // rows of this layer (TEAM warps per row)
    // ------------------------------------------------------------------------------------------
    for (int r = team; r < a.T; r += n_teams) {
      const ChainPred pred_row{has_pred ? P + (long long)r * D : nullptr, uint32_t(l), abort_flag, a.status};
      uint8_t* codes_row = (is_v ? ly.Vcodes : ly.Kcodes) + (long long)r * CODE_BYTES;
      uint16_t* out = is_v ? ly.Vhat : ly.Khat;
      uint16_t* pass = is_v ? ly.Vpass : ly.Kpass;
      const ChainHat hat_row{out != nullptr ? out + (long long)r * ly.ldHat : nullptr, pass != nullptr ? pass + (long long)r * D : nullptr};
      uint16_t* scales_row = (is_v ? ly.Vscales : ly.Kscales) + (long long)r * n_groups;
      if constexpr (WR) {
        unsigned long long* xbuf = sm->scratch.xbuf[warp];
        if constexpr (kEncode) {
          wr_encode_row<NPTS, kBf16, ChainPred, ChainHat>(wrc, &sm->tables, xbuf, (is_v ? ly.V : ly.K) + (long long)r * a.ldX, pred_row, codes_row,
                                     scales_row, hat_row);
        } else {
          if (hat_row != nullptr)
            wr_decode_row<NPTS, kBf16, false, false, ChainPred, ChainHat>(wrc, sm->tables.grid, xbuf, codes_row, scales_row, pred_row, hat_row);
        }
      } else {
        TeamSmem<D>* ts = &sm->scratch.team[warp / TEAM];
        if constexpr (kEncode) {
          encode_row<D, NPTS, kBf16, ChainPred, ChainHat>(rck, &sm->tables, ts, (is_v ? ly.V : ly.K) + (long long)r * a.ldX, pred_row, codes_row,
                                     scales_row, hat_row);
        } else {
          f32x2_t wp[4];
          float scale;
          if (r == team) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const ulonglong2 w2 = sm->ahead[warp][i][lane];
              wp[2 * i] = w2.x;
              wp[2 * i + 1] = w2.y;
            }
            scale = sm->ahead_scale[warp][lane];
          } else {
            load_codes(l, r, words, sf);
            rotate_codes(words[0], wp);
            scale = sf[0];
          }
          if (hat_row != nullptr) {
            float4 pq[2];
            if (has_pred) pred_load8(pred_row + (rck.member * 256 + lane * 8), pq[0], pq[1]);
            else pq[0] = pq[1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            team_add_pred(rck, wp, scale, pq);
            hat_store8(hat_row + (rck.member * 256 + lane * 8), make_uint4(store16x2p<kBf16>(wp[0]), store16x2p<kBf16>(wp[1]),
                                                                           store16x2p<kBf16>(wp[2]), store16x2p<kBf16>(wp[3])));
          }
        }
      }
    }
  }
}

}  // namespace aquakv
