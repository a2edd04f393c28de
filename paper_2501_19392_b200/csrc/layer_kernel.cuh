// One persistent kernel per layer call for Algorithm 2 (encode) and Algorithm 3 (decode) with
// predictors: the predictor GEMMs (the two predictions of Algorithm 2 / Algorithm 3) run on
// the tensor cores while, on the same SMs, other warps run the row work of the quantizer
// (Section 2 "Vector Quantization") and of the reconstruction on tokens whose prediction is
// already complete.  The fp32 prediction is handed from the GEMM warps to the row warps through a
// small ring of buffers that stays resident in L2; completion is tracked with counters in global
// memory.
//
// Work layout.  A token block is 128 tokens; a GEMM tile is one token block x 256 output features,
// so NTN = d_kv/256 CTAs share a token block.  CTAs run as pairs (clusters of two): pair p owns
// feature tile n = p % NTN and the two token-block slots ml = 2 * (p / NTN) + rank, and computes
// both tiles with one tcgen05.mma.cta_group::2 of M = 256: each CTA loads its own 128 token rows
// and HALF of the 256 weight rows, so a k-block costs 32 KB of L2 traffic per CTA instead of 48 KB
// (the GEMM is bound by L2 bandwidth, not by the tensor pipe).  Every "wave" covers
// gridDim.x / NTN token blocks.  For each wave a CTA computes
// its key-phase tile and its value-phase tile, and runs the row work of 128/NTN rows of its token
// block for both phases.  Jobs are ordered  K0, K1, V0, K2, V1, ..., so that the value-phase GEMM of
// a wave (which reads the reconstructed keys of that wave) is issued one job after its key rows.
//
// In the short last wave of a launch of one layer a tile may be 128 or 64 features wide (wave_log_split): more pairs then share a
// token block, and a pair's slots and feature tile are others than in a full wave.
//
// Dependencies (all counted per job j and token-block slot ml):
//   gemm_done[j][ml]  -- feature tiles of job j written to the ring (row warps wait for kTileWeight * NTN: a whole tile counts
//                        kTileWeight, a narrow one its part of it)
//   rows_done[j][ml]  -- CTAs whose row teams have finished job j on token block ml (target: the CTAs that have rows of the block,
//                        NTN in a full wave; the value-phase TMA producer waits for the key rows of its wave; the GEMM epilogue waits for
//                        job j - ring size before it overwrites that ring slot)
// The encoder's last value rows are reported with the key rows of the next job, still before any job that waits for them.
// Every job waits only on jobs with a smaller index (or the same index of the other role), so the
// schedule cannot dead-lock as long as all CTAs are resident, which the launch guarantees by using at
// most one CTA per SM.  Every wait is bounded; on expiry the CTA records AQUAKV_ERR_TIMEOUT and
// all its roles leave their loops.
//
// Warp roles: warp 0 = TMA producer, warp 1 = tensor-memory owner + MMA issuer, warps 2..5 =
// GEMM epilogue (tensor memory -> fp32 rows in the ring), then the row warps and, in the decoder
// instantiation that also attends (the attention read of Algorithm 4), four attention warps: as soon as the value
// rows of the CTA's token block are reconstructed they read the block's keys and values back from
// L2, form the single-query attention partials of the CTA's share of the KV heads for every sequence
// the block overlaps, and release the block's rows (attn_done), so that decoded rows which the
// caller does not ask for live only in a ring of three waves that never needs to reach DRAM.
#pragma once

#include "attn.cuh"
#include "codec.cuh"
#include "common.cuh"
#include "gemm_pred.cuh"
#include "rowchunk.cuh"
#include "rowwarp.cuh"

namespace aquakv {

// Operand stages of 32 KB per CTA: four, except three for the encoder with one warp per row (kWarpRows),
// whose row work is the longer side and whose shared memory is better spent on more row warps
// (measured: 3 and 4 stages alike).
constexpr int kLayerStagesMax = 4;
template <bool kEncode, bool kWarpRows> constexpr int kLayerStagesT = (kEncode && kWarpRows) ? 3 : 4;

// Row warps of a CTA.  With d_kv = 1024 and the Hadamard block and scale group spanning the whole row
// (kFull) a single warp owns a row (rowwarp.cuh); otherwise teams of d_kv/256 warps share a row
// (codec.cuh): 24 warps at 64 registers, or, for d_kv <= 512, one warp of rowchunk.cuh.  The register file is split over the SM's four schedulers, so
// the budget per thread follows from the warps per scheduler: 4 -> 128, 5 -> 96, 6 -> 80 registers.
//   encoder: its row work is the longer side of the kernel and gains from every resident warp, even at
//            80 registers (12 / 14 / 16 / 18 / 20 row warps measured: 1.35 / 1.28 / 1.28 / 1.33 / 1.37 ms per
//            131072 tokens, 361 / 347 / 350 / 356 / 365 us per 32768);
//   decoder: the GEMM is the longer side; 10 row warps keep the CTA at 16 warps and 128 registers, which
//            lets a row issue its prediction loads before the look-ups and the rotation (8 / 10 / 12 row
//            warps: 0.75 / 0.77 / 0.87 ms per 131072 tokens).
constexpr int kWrEncodeWarps = 16;
constexpr int kWrDecodeWarps = 10;
constexpr int kWrAttnDecodeWarps = 6;  // beside four attention warps: again 16 warps and 128 registers, which the
                                       // attention warps need as much as the row warps (4 / 5 / 6 / 7 row warps:
                                       // 2.54 / 2.41 / 2.23 / 2.94 ms per 8 x 32768 tokens)
static_assert(kWrAttnDecodeWarps <= kWrDecodeWarps, "the decoder's shared memory is sized for kWrDecodeWarps row warps");
enum RowKind { kRowTeams, kRowWarp, kRowChunks };
// One warp per row for d_kv <= 512 (rowchunk.cuh), row warps by what their registers hold (without spills but for 16 bytes of the
// d_kv 256 encoder with blocks shorter than the row).  us for 60000 tokens:
//   d_kv 512, Hadamard block and group = the row, encoder: teams 292; 10 / 12 / 14 / 16 warps 257 / 279 / 264 / 299;
//   d_kv 512, encoder with blocks of 64: teams 264, 10 / 14 warps 282 / 286, so the teams stay;
//   d_kv 512, decoder: teams 184; 10 / 12 / 14 / 16 warps 178 / 175 / 157 / 167 (blocks of 64: 168; 163 / 159 / 147 / 155);
//   d_kv 256: 24 / 18 / 16 warps 136 / 128 / 129 to encode and 98 / 88 / 91 to decode, 20000 tokens 63 / - / 59 and 44 / - / 41.
template <bool kEncode, int D> constexpr int kChunkRowWarps = D == 256 ? 16 : (kEncode ? 10 : 14);
template <bool kEncode, int D, bool kFull, int kAttnHD = 0>
struct LayerGeom {
  static constexpr bool WR = D == 1024 && kFull;
  static constexpr bool CR = D == 256 || (D == 512 && (!kEncode || kFull));
  static constexpr int ROW_WARPS = WR ? (kEncode ? kWrEncodeWarps : (kAttnHD > 0 ? kWrAttnDecodeWarps : kWrDecodeWarps))
                                      : (CR ? kChunkRowWarps<kEncode, D> : 24);
  static constexpr int TEAM = WR || CR ? 1 : RowTeam<D>::TEAM;
  static constexpr int KIND = WR ? kRowWarp : (CR ? kRowChunks : kRowTeams);
  static constexpr int TEAMS = ROW_WARPS / TEAM;          // rows a CTA works on at a time
  static constexpr int THREADS = 32 * (6 + ROW_WARPS);
  // With at most 16 warps per CTA (four per scheduler) a thread may use 128 registers: the row
  // routines then load ahead (next row's input, the prediction before the rotation).
  static constexpr bool AHEAD = WR && 6 + ROW_WARPS + (kAttnHD > 0 ? 4 : 0) <= 16;
};
constexpr int kAttnWarps = 4;
constexpr int kAttnSubTokens = 128;  // tokens of a token block that one attention warp covers (one partial slot each)
template <bool kEncode, int D, bool kFull, int kAttnHD>
constexpr int layer_threads() {
  return LayerGeom<kEncode, D, kFull, kAttnHD>::THREADS + (kAttnHD > 0 ? 32 * kAttnWarps : 0);
}

constexpr int kLayerRing = 3;       // prediction buffers
static_assert(kLayerRing >= 2, "a job reported with the next one must be out before the job that takes its buffer");
// Slots of the row warps' hand-offs.  A warp that waits for job g + s while another of its CTA has not finished job g must not meet
// that job's slot.  The predictions of a job wait for the CTA's rows of kLayerRing jobs before where those lie in the same token
// block; in a short last wave they lie in another block or nowhere, and the epilogue then looks kLayerRing jobs further back.  With the job of
// the last wave itself in between s is at most 2 kLayerRing + 1 (played through for 1 to 5 waves and 1 to 4 layers on 8 to 148 CTAs: 5).
constexpr int kJobRing = 8;
static_assert(2 * kLayerRing + 1 < kJobRing && (kJobRing & (kJobRing - 1)) == 0, "slots of two jobs would meet");

struct LayerSmemTail {
  uint64_t full[kLayerStagesMax];
  uint64_t empty[kLayerStagesMax];
  uint64_t acc_full[kAccStages];
  uint64_t acc_empty[kAccStages];
  uint32_t tmem_base;
  int abort_flag;
  // hand-offs of the row warps, by job modulo kJobRing; jobs count from 1 through the layers of the launch
  int poller[kJobRing];      // the latest job that a warp of this CTA polls the GEMM's counter for
  int ready[kJobRing];       // the latest job whose predictions are there
  int arrived[kJobRing];     // reports of row teams
};

// Grid only (decode needs no search table).
template <int NPTS>
struct GridSmem {
  f32x2_t grid[NPTS];
};
template <bool kEncode, int NPTS> struct LayerTables { typedef RowSmem<NPTS> type; };
template <int NPTS> struct LayerTables<false, NPTS> { typedef GridSmem<NPTS> type; };

template <int D, int ROW_WARPS, int kKind> struct LayerRowScratch { TeamSmem<D> team[ROW_WARPS / RowTeam<D>::TEAM]; };
template <int D, int ROW_WARPS> struct LayerRowScratch<D, ROW_WARPS, kRowWarp> { unsigned long long xbuf[ROW_WARPS][kWrItems]; };
template <int D, int ROW_WARPS> struct LayerRowScratch<D, ROW_WARPS, kRowChunks> {};

template <bool kEncode, int D, int NPTS, bool kFull>
struct LayerRowSmem {
  typename LayerTables<kEncode, NPTS>::type tables;
  LayerRowScratch<D, LayerGeom<kEncode, D, kFull>::ROW_WARPS, LayerGeom<kEncode, D, kFull>::KIND> scratch;
};

// The GEMM epilogue stages each 32-row x 32-column fp32 piece of a tile in shared memory (128-byte
// swizzle) and hands it to a TMA store.  With one warp per row: one 4 KB buffer per epilogue warp
// (two measured 2-3 % slower in the decoder and no faster in the encoder, where the space goes to
// the row warps).  With row teams: two, which the short calls of that path gain from, or one for the
// encoder with the 256-point grid, whose 2 KB grid would otherwise not fit.
template <bool kEncode, int NPTS, bool kWarpRows>
constexpr int kEpiBufs = (kWarpRows || (kEncode && NPTS > 64)) ? 1 : 2;
template <bool kEncode, int NPTS, bool kWarpRows>
constexpr int kEpiBytes = 4 * kEpiBufs<kEncode, NPTS, kWarpRows> * kEpiPieceBytes;

template <bool kEncode, int D, int NPTS, bool kFull>
constexpr size_t layer_smem_bytes() {
  constexpr bool WR = LayerGeom<kEncode, D, kFull>::WR;
  return 1024 + size_t(kLayerStagesT<kEncode, WR>) * kPairStageBytes + kEpiBytes<kEncode, NPTS, WR> + sizeof(LayerSmemTail) +
         sizeof(LayerRowSmem<kEncode, D, NPTS, kFull>);
}

__device__ __forceinline__ void tma_store_2d_hint(const CUtensorMap* map, const void* smem_src, int32_t x, int32_t y,
                                                  uint64_t policy) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3}], [%1], %4;" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(smem_src)), "r"(x), "r"(y), "l"(policy)
               : "memory");
}
struct LayerArgs {
  int T;                  // tokens
  int n_mblocks;          // ceil(T / 128)
  int mw;                 // token blocks per wave (gridDim.x / NTN)
  int n_waves;
  int last_log_split;     // wave_log_split of the last wave (launches of one layer)
  int nb;                 // prediction buffers in the ring
  const float* bk;        // optional biases [d_kv]
  const float* bv;
  float* P;               // ring: [nb][mw * 128][d_kv] fp32
  int* gemm_done;         // [2 * n_waves][mw], zero at launch
  int* rows_done;         // [2 * n_waves][mw], zero at launch
  int khat_ring;          // 0: K^ rows are indexed by token; r > 0: ring of r waves (rows of mw*128)
  // encode inputs
  const uint16_t* K;
  const uint16_t* V;
  long long ldX;
  // compressed cache (written by encode, read by decode)
  uint8_t* Kcodes;
  uint16_t* Kscales;
  uint8_t* Vcodes;
  uint16_t* Vscales;
  // reconstructions
  uint16_t* Khat;         // output rows (khat_ring == 0) or the ring
  long long ldKhat;
  uint16_t* Vhat;         // output rows or nullptr (encode only)
  long long ldVhat;
  const uint32_t* signmask_k;
  const uint32_t* signmask_v;
  const float4* grid4;
  SearchDev search;
  int log_h, log_g;
  int* status;
  // single-query attention over the decoded rows (decoder instantiations with kAttnHD > 0)
  int vhat_ring;            // like khat_ring, for V^ (both rings or neither)
  const uint16_t* q;        // [batch][n_q_heads][head_dim]
  int ctx;                  // tokens per sequence: token t belongs to sequence t / ctx
  int n_q_heads, n_kv_heads;
  int n_splits;             // partial slots per sequence: slot s of sequence b = sub-block (of kAttnSubTokens tokens) b*ctx/kAttnSubTokens + s
  float scale_log2;         // softmax scale * log2(e)
  float* part_ml;           // [batch][n_splits][n_q_heads][2]
  float* part_o;            // [batch][n_splits][n_q_heads][head_dim]
  int* attn_done;           // [n_waves][mw], zero at launch: attention warps that are done with the block
};

// The layers of one launch.  A launch of several layers (Algorithm 2 / 3 inside Algorithm 4's loop over
// layers) runs them back to back without a barrier in between: every role walks the layers on its own,
// the prediction ring and its counters continue across the layer boundary, and a layer's first jobs start
// while the previous layer's last wave is still being finished (a layer's wave w needs only wave w of the
// layer before it).  All layers share T, the wave geometry and the ring.
struct LayerMaps {
  CUtensorMap kprev, vprev, khat, wk, wv, p;
};
constexpr int kLayerBatchMax = 24;      // 24 x (arguments + six tensor maps) stays inside the 32 KB of kernel parameters
template <int kBatch>
struct LayerBatch {
  int n_layers;
  LayerArgs layer[kBatch];
  LayerMaps maps[kBatch];
};
// A launch of one layer has room for the maps of narrow tiles: weight boxes of kNarrowBox rows.
constexpr int kNarrowBox = 32;
template <>
struct LayerBatch<1> {
  int n_layers;
  LayerArgs layer[1];
  LayerMaps maps[1];
  CUtensorMap wk_narrow, wv_narrow;
};
static_assert(sizeof(LayerBatch<kLayerBatchMax>) <= 32764, "kernel parameters are limited to 32764 bytes");

__device__ __forceinline__ void layer_job(int j, int n_waves, int& phase, int& wave) {
  if (j == 0) { phase = 0; wave = 0; }
  else if (j == 2 * n_waves - 1) { phase = 1; wave = n_waves - 1; }
  else if (j & 1) { phase = 0; wave = (j + 1) >> 1; }
  else { phase = 1; wave = (j >> 1) - 1; }
}
// log2 of the number of tiles that a 256-feature tile is cut into in the last wave of a call, the only one that may be short.
// A short wave leaves CTA pairs without a tile, while those that have one take the k-blocks and the pieces of the epilogue
// (0.5 - 0.7 us per 32 features) one after the other: narrower tiles shorten both.  As many as there are pairs for, up to four (64 features:
// below that the token rows are most of what a k-block loads).  us with whole and with narrow tiles: 1000 tokens of
// d_kv 1024 encoded 49.7 / 42.7 and decoded 34.5 / 29.7, 2000 54.8 / 50.7 and 39.2 / 37.2, 5000 (the second wave is short) 86.4 / 83.6
// and 57.0 / 54.6.  Launches of several layers keep whole tiles: no room for the maps of narrow ones.
constexpr int kTileWeight = 4;
inline int wave_log_split(int blocks, int pairs, int ntn) {
  int ls = 0;
  while (ls < 2 && ((blocks + 1) / 2 * ntn << (ls + 1)) <= pairs) ++ls;
  return ls;
}
__device__ __forceinline__ int layer_key_job(int wave) { return wave == 0 ? 0 : 2 * wave - 1; }
__device__ __forceinline__ int layer_value_job(int wave, int n_waves) {
  return wave == n_waves - 1 ? 2 * n_waves - 1 : 2 * wave + 2;
}
// Value job j is followed by the key rows of a full wave, in which every CTA has rows.
__device__ __forceinline__ bool later_report(int j, int n_jobs) { return j >= 2 && j < n_jobs - 4; }

// Row work of a wave is spread evenly over ALL CTAs: CTA slot s takes rows [s*rpc, (s+1)*rpc) of
// the wave, rpc = the power of two >= rows / CTAs.  For a full wave this is rpc = 128 / NTN rows of
// the CTA's own token block; in the short last wave it keeps every SM busy instead of a few.
struct WaveRows {
  int tokens;      // rows of the wave
  int blocks;      // token blocks of the wave
  int rpc;         // rows per CTA slot (power of two, <= 128 / NTN)
};
__device__ __forceinline__ WaveRows wave_rows(int wave, int T, int mw, int n_ctas) {
  WaveRows w;
  const long long left = (long long)T - (long long)wave * mw * kBM;
  w.tokens = left < (long long)mw * kBM ? int(left) : mw * kBM;
  w.blocks = (w.tokens + kBM - 1) / kBM;
  const int need = (w.tokens + n_ctas - 1) / n_ctas;
  int rpc = 1;
  while (rpc < need) rpc <<= 1;
  w.rpc = rpc;
  return w;
}

// Number of CTAs that report on token block `block` of that wave.
__device__ __forceinline__ int wave_block_ctas(const WaveRows& w, int block, int n_ctas) {
  const int per_block = kBM / w.rpc;
  const int hi = (block + 1) * per_block < n_ctas ? (block + 1) * per_block : n_ctas;
  const int n = hi - block * per_block;
  return n > 0 ? n : 0;
}

// Longest pause (ns; nanosleep takes up to twice that) between two polls of a counter.  A call of one wave is a chain of
// four steps, and each waits for the one before, so what a poll comes late is lost (with pauses of 2 us 10 of the 38 us of 1024
// tokens encoded at d_kv 512); with more waves there is other work in the meantime.  With one row warp polling per CTA, us at pauses of
// 2048 / 512 / 256 for every poller: 5000 tokens decoded (two waves) 62 / 57 / 56.5, four sequences of 6017 tokens through four layers of a
// cache policy (six) 836 / 822 / 819; 2048 / 512: 32768 encoded (eight) 388 / 390, 131072 decoded (29) 895 / 891, 32 x 32768 decoded and
// attended (33 a chunk) 8420 / 8224.  2048 for the TMA producer and the epilogue alone: 387, 906, 8234.
__device__ __forceinline__ uint32_t poll_pause(int n_waves) { return n_waves > 1 ? 512u : 128u; }

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Spins until *ctr >= target.  Returns false after limit_ns or if the CTA already aborted.  The pause between two polls
// doubles up to max_pause: see poll_pause.
__device__ __forceinline__ bool counter_wait_bounded(const int* ctr, int target, volatile int* abort_flag,
                                                     int* status, uint32_t max_pause, unsigned long long limit_ns = kWaitLimitNs) {
  if (ld_acquire(ctr) >= target) return true;
  const unsigned long long t0 = global_timer_ns();
  uint32_t spins = 0;
  uint32_t pause = 64;
  while (ld_acquire(ctr) < target) {
    __nanosleep(pause);
    if (pause < max_pause) pause <<= 1;
    if ((++spins & 0x3Fu) == 0) {
      if (*abort_flag) return false;
      if (global_timer_ns() - t0 > limit_ns) {
        *abort_flag = 1;
        atomicExch(status, kStatusTimeout);
        return false;
      }
    }
  }
  return true;
}

__device__ __forceinline__ int ld_acquire_cta(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

// The row warps' wait for the predictions of job `job` (one lane of each team calls it): the first team of the CTA that
// comes polls the counter in global memory, the others look at shared memory.  (Every team polling for itself: up to 24
// pollers in each of 148 CTAs held up the very counters that they waited for.)
__device__ __forceinline__ bool row_wait(LayerSmemTail* tail, int job, const int* ctr, int target, int* status, uint32_t max_pause,
                                         unsigned long long limit_ns = kWaitLimitNs) {
  const int slot = job & (kJobRing - 1);
  if (ld_acquire_cta(&tail->ready[slot]) >= job) return true;
  volatile int* abort_flag = &tail->abort_flag;
  if (atomicMax(&tail->poller[slot], job) < job) {
    if (!counter_wait_bounded(ctr, target, abort_flag, status, max_pause, limit_ns)) return false;
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(&tail->ready[slot])), "r"(job) : "memory");
    return true;
  }
  const unsigned long long t0 = global_timer_ns();
  uint32_t spins = 0;
  while (ld_acquire_cta(&tail->ready[slot]) < job) {
    __nanosleep(64);
    if ((++spins & 0xFu) == 0) {
      if (*abort_flag) return false;
      if (global_timer_ns() - t0 > 2 * limit_ns) {           // the polling warp has given up before
        *abort_flag = 1;
        atomicExch(status, kStatusTimeout);
        return false;
      }
    }
  }
  return true;
}

// The failure paths of the three kinds of wait, one warp each, every one for something that never comes: a barrier that nothing
// arrives on, a counter that nothing raises, and (a row warp behind another that polls) a word in shared memory that
// nobody writes.  Each must give up after its limit, raise its abort flag and say so; only then *status reads kStatusTimeout.
// The loops end on %globaltimer alone.
__global__ void __launch_bounds__(96) bounded_wait_selftest_kernel(int* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  __shared__ LayerSmemTail tail[2];          // of the poller and of the warp behind one
  __shared__ int bar_abort, told[3], gave_up[3];
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    bar_abort = 0;
    for (int i = 0; i < 2; ++i) {
      tail[i].abort_flag = 0;
      for (int k = 0; k < kJobRing; ++k) tail[i].poller[k] = tail[i].ready[k] = 0;
    }
    tail[1].poller[1] = 1;
    for (int i = 0; i < 3; ++i) told[i] = gave_up[i] = 0;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    if (warp == 0) gave_up[0] = !mbar_wait_bounded(&bar, 0u, &bar_abort, &told[0], limit_ns);
    else gave_up[warp] = !row_wait(&tail[warp - 1], 1, status, 1, &told[warp], 512u, limit_ns);      // a status word is never above 0
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    bool all = bar_abort != 0 && tail[0].abort_flag != 0 && tail[1].abort_flag != 0;
    for (int i = 0; i < 3; ++i) all = all && gave_up[i] && told[i] == kStatusTimeout;
    if (all) atomicExch(status, kStatusTimeout);
  }
}

// A row team's report on job `job`; true for the last of the CTA's `teams`, which reports for all of them (its fence then
// covers the rows of the teams that it has synchronised with here).
__device__ __forceinline__ bool row_arrive(LayerSmemTail* tail, int job, int teams) {
  int old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.s32 %0, [%1], 1;" : "=r"(old) : "r"(smem_u32(&tail->arrived[job & (kJobRing - 1)])) : "memory");
  return (old + 1) % teams == 0;
}

__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_all() {
  asm volatile("fence.proxy.async;" ::: "memory");
}

// kFull: the Hadamard block and the scale group both span the whole row (the paper's setting for
// d_kv = 1024, Section 4.1); their logarithms are then compile-time constants of the row code.
// kAttnHD: 0, or the head dimension (64 / 128) of the attention the decoder also computes.
template <bool kEncode, int D, int NPTS, bool kBf16, bool kFull, int kAttnHD = 0, int kBatch = 1>
__global__ void __launch_bounds__((layer_threads<kEncode, D, kFull, kAttnHD>()), 1)
layer_kernel(const __grid_constant__ LayerBatch<kBatch> B) {
  using G = LayerGeom<kEncode, D, kFull, kAttnHD>;
  const LayerArgs& a = B.layer[0];         // what all layers of the launch share: geometry, tables, status word
  const int n_layers = kBatch == 1 ? 1 : B.n_layers;
  constexpr int NTN = D / kBN;             // feature tiles per token block = CTAs per token block
  constexpr int NKD = D / kBK;             // k-blocks per d_kv input features
  constexpr int BITS = NPTS == 16 ? 4 : (NPTS == 64 ? 6 : 8);
  constexpr int CODE_BYTES = D / 2 * BITS / 8;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_align<1024>(smem_raw);
  uint8_t* epi_smem = smem + size_t(kLayerStagesT<kEncode, G::WR>) * kPairStageBytes;      // 1024-byte aligned
  LayerRowSmem<kEncode, D, NPTS, kFull>* rsm = reinterpret_cast<LayerRowSmem<kEncode, D, NPTS, kFull>*>(
      epi_smem + kEpiBytes<kEncode, NPTS, G::WR>);                                        // 1024-byte aligned
  LayerSmemTail* tail = reinterpret_cast<LayerSmemTail*>(rsm + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();          // 0 = leader of the pair (issues the MMAs)
  const int pair = blockIdx.x >> 1;
  const int ml = 2 * (pair / NTN) + int(rank);      // token block and feature tile of this CTA in a full wave
  const int n_blk = pair % NTN;
  // The GEMM tile of this pair in a wave: token-block slots 2 * (pair / tiles), + 1 and feature tile pair % tiles of `width`
  // features, tiles = NTN << log_split.
  struct Tile {
    int log_split, width, ml, n;
    bool active;        // the pair's first token block exists
  };
  constexpr int LOG_NTN = NTN == 4 ? 2 : (NTN == 2 ? 1 : 0);
  auto wave_tile = [&](int wave) {
    Tile t;
    t.log_split = kBatch == 1 && wave == a.n_waves - 1 ? a.last_log_split : 0;
    t.width = kBN >> t.log_split;
    const int log_tiles = LOG_NTN + t.log_split, slot = (pair >> log_tiles) * 2;
    t.n = pair & ((1 << log_tiles) - 1);
    t.ml = slot + int(rank);
    t.active = wave * a.mw + slot < a.n_mblocks && slot < a.mw;
    return t;
  };
  const int n_jobs = 2 * a.n_waves;
  const uint32_t max_pause = poll_pause(a.n_waves);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kLayerStagesT<kEncode, G::WR>; ++s) {
      mbar_init(&tail->full[s], 1);
      mbar_init(&tail->empty[s], 1);
    }
    for (int s = 0; s < kAccStages; ++s) {
      mbar_init(&tail->acc_full[s], 1);
      mbar_init(&tail->acc_empty[s], 8);     // 4 epilogue warps of each CTA (used in the leader only)
    }
    tail->abort_flag = 0;
    for (int i = 0; i < kJobRing; ++i) tail->poller[i] = tail->ready[i] = tail->arrived[i] = 0;
    mbar_fence_init();
  }
  if constexpr (kEncode) {
    row_smem_fill<NPTS>(&rsm->tables, a.search.table, a.grid4);
  } else {
    for (int i = threadIdx.x; i < NPTS; i += blockDim.x) {
      const float4 g = a.grid4[i];
      rsm->tables.grid[i] = pack2(g.x, g.y);
    }
  }
  if (warp == 1) {
    tmem_alloc_pair(&tail->tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();          // the peer's barriers are initialised before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = tail->tmem_base;
  volatile int* abort_flag = &tail->abort_flag;
  pdl_sync();

  if (warp == 0) {
    // ------------------------------- TMA producer --------------------------------------------
    if (lane == 0) {
      const uint64_t pol_stream = l2_policy_evict_first(), pol_keep = l2_policy_evict_last();
      int stage = 0;
      uint32_t phase_bit = 0;
      bool ok = true;
      int issued = 0;
      for (int l = 0; ok && l < n_layers; ++l) {
      const LayerArgs& a = B.layer[l];
      const LayerMaps& tm = B.maps[l];
      tma_prefetch_desc(&tm.kprev);
      tma_prefetch_desc(&tm.vprev);
      tma_prefetch_desc(&tm.khat);
      tma_prefetch_desc(&tm.wk);
      tma_prefetch_desc(&tm.wv);
      for (int j = 0; ok && j < n_jobs; ++j) {
        int ph, wave;
        layer_job(j, a.n_waves, ph, wave);
        const Tile tile = wave_tile(wave);
        if (!tile.active) continue;
        const int ml = tile.ml, m = wave * a.mw + ml;
        const int nk = ph == 0 ? NKD : 2 * NKD;
        const int w_row = tile.n * tile.width + int(rank) * (tile.width / 2);     // this CTA's half of the weight rows
        const uint32_t stage_tx = 2u * uint32_t(kABytes + (kPairBBytes >> tile.log_split));
        const int khat_row = a.khat_ring ? ((wave % a.khat_ring) * a.mw + ml) * kBM : m * kBM;
        auto load_weights = [&](uint8_t* dst, const CUtensorMap* whole, int which, int x) {
          if constexpr (kBatch == 1) {
            if (tile.log_split > 0) {
              const CUtensorMap* narrow = which == 0 ? &B.wk_narrow : &B.wv_narrow;
              for (int r = 0; r < tile.width / 2; r += kNarrowBox)
                tma_load_2d_pair_hint(dst + r * (kBK * 2), narrow, &tail->full[stage], x, w_row + r, pol_keep);
              return;
            }
          }
          tma_load_2d_pair_hint(dst, whole, &tail->full[stage], x, w_row, pol_keep);
        };
        for (int kb = 0; kb < nk; ++kb) {
          if (l > 0 && kb == 0 && m < a.n_mblocks) {
            // the previous layer of this launch wrote this job's first input (its reconstructed keys for
            // the key phase, values for the value phase): its row warps must be done with this token block
            const LayerArgs& pa = B.layer[l - 1];
            const int pj = ph == 0 ? layer_key_job(wave) : layer_value_job(wave, a.n_waves);
            const int target = wave_block_ctas(wave_rows(wave, a.T, a.mw, gridDim.x), ml, gridDim.x);
            if (!counter_wait_bounded(pa.rows_done + pj * a.mw + ml, target, abort_flag, a.status, max_pause)) {
              ok = false;
              break;
            }
            fence_proxy_async_all();
          }
          if (ph == 1 && kb == NKD && m < a.n_mblocks) {
            // the remaining k-blocks read this wave's reconstructed keys, written by row warps
            const int target = wave_block_ctas(wave_rows(wave, a.T, a.mw, gridDim.x), ml, gridDim.x);
            if (!counter_wait_bounded(a.rows_done + layer_key_job(wave) * a.mw + ml, target, abort_flag,
                                      a.status, max_pause)) {
              ok = false;
              break;
            }
            fence_proxy_async_all();
          }
          if (!mbar_wait_bounded(&tail->empty[stage], phase_bit ^ 1u, abort_flag, a.status)) {
            ok = false;
            break;
          }
          uint8_t* a_dst = smem + size_t(stage) * kPairStageBytes;
          uint8_t* b_dst = a_dst + kABytes;
          // the leader's barrier collects the bytes of both CTAs
          if (rank == 0) mbar_arrive_expect_tx(&tail->full[stage], stage_tx);
          // token rows stream through L2 once; the adapter tiles are read again by every wave
          if (ph == 0) {
            tma_load_2d_pair_hint(a_dst, &tm.kprev, &tail->full[stage], kb * kBK, m * kBM, pol_stream);
            load_weights(b_dst, &tm.wk, 0, kb * kBK);
          } else {
            if (kb < NKD) {
              tma_load_2d_pair_hint(a_dst, &tm.vprev, &tail->full[stage], kb * kBK, m * kBM, pol_stream);
            } else {
              tma_load_2d_pair_hint(a_dst, &tm.khat, &tail->full[stage], (kb - NKD) * kBK, khat_row, pol_stream);
            }
            load_weights(b_dst, &tm.wv, 1, kb * kBK);
          }
          ++issued;
          if (++stage == kLayerStagesT<kEncode, G::WR>) { stage = 0; phase_bit ^= 1u; }
        }
      }
      }   // layers
      if (!ok && rank == 0) {
        // let the copies in flight land before the shared memory is released
        int s = stage;
        uint32_t pb = phase_bit;
        const int pending = issued < kLayerStagesT<kEncode, G::WR> ? issued : kLayerStagesT<kEncode, G::WR>;
        for (int i = 0; i < pending; ++i) {
          if (s == 0) { s = kLayerStagesT<kEncode, G::WR>; pb ^= 1u; }
          --s;
          const unsigned long long t0 = global_timer_ns();
          while (!mbar_try_wait(&tail->full[s], pb) && global_timer_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------- MMA issuer ----------------------------------------------
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t phase_bit = 0;
      bool ok = true;
      int it = 0;
      for (int l = 0; ok && l < n_layers; ++l)
      for (int j = 0; ok && j < n_jobs; ++j) {
        int ph, wave;
        layer_job(j, a.n_waves, ph, wave);
        const Tile tile = wave_tile(wave);
        if (!tile.active) continue;
        const uint32_t idesc = umma_idesc_f16(2 * kBM, tile.width, kBf16);
        const int nk = ph == 0 ? NKD : 2 * NKD;
        const int acc = it & 1;
        const uint32_t acc_phase = (it >> 1) & 1u;
        ++it;
        if (!mbar_wait_bounded(&tail->acc_empty[acc], acc_phase ^ 1u, abort_flag, a.status)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t tmem_d = tmem_base + uint32_t(acc * kBN);
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait_bounded(&tail->full[stage], phase_bit, abort_flag, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint32_t a_addr = smem_u32(smem + size_t(stage) * kPairStageBytes);
          const uint32_t b_addr = a_addr + kABytes;
#pragma unroll
          for (int k = 0; k < kBK / kUmmaK; ++k) {
            const uint64_t da = umma_smem_desc_k128(a_addr + k * kUmmaK * 2);
            const uint64_t db = umma_smem_desc_k128(b_addr + k * kUmmaK * 2);
            umma_f16_pair(tmem_d, da, db, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          }
          umma_commit_pair(&tail->empty[stage]);   // frees the stage in both CTAs
          if (++stage == kLayerStagesT<kEncode, G::WR>) { stage = 0; phase_bit ^= 1u; }
        }
        if (ok) umma_commit_pair(&tail->acc_full[acc]);
      }
    }
  } else if (warp < 6) {
    // ------------------------------- GEMM epilogue (4 warps) ---------------------------------
    const int quarter = warp & 3;   // tensor-memory lanes [32*quarter, 32*quarter+32)
    int it = 0;
    bool stop = false;
    for (int l = 0; !stop && l < n_layers; ++l) {
    const LayerArgs& a = B.layer[l];
    const LayerMaps& tm = B.maps[l];
    for (int j = 0; j < n_jobs; ++j) {
      int ph, wave;
      layer_job(j, a.n_waves, ph, wave);
      const Tile tile = wave_tile(wave);
      if (!tile.active) continue;
      const int ml = tile.ml, x0 = tile.n * tile.width, n_pieces = tile.width / 32;
      const int acc = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1u;
      ++it;
      bool ok = true;
      // the ring slot of this job was last used nb jobs earlier (counted through the layers of the launch):
      // that job's row work must be over
      const int gj = l * n_jobs + j;
      // ... the latest such job in whose wave this token block exists (the short last wave may not have it:
      // nobody then read or reports on this block's part of the slot)
      int go = gj - a.nb, ph_old = 0, wave_old = 0;
      while (go >= 0) {
        layer_job(go % n_jobs, a.n_waves, ph_old, wave_old);
        if (ml < wave_rows(wave_old, a.T, a.mw, gridDim.x).blocks) break;
        go -= a.nb;
      }
      if (go >= 0) {
        const int lo = go / n_jobs, jo = go % n_jobs;
        const int target = wave_block_ctas(wave_rows(wave_old, a.T, a.mw, gridDim.x), ml, gridDim.x);
        // one thread polls for the four warps; a failed wait has set the abort flag
        if (warp == 2 && lane == 0)
          counter_wait_bounded(B.layer[lo].rows_done + jo * a.mw + ml, target, abort_flag, a.status, max_pause);
        named_barrier(1, 128);
        ok = *abort_flag == 0;
      }
      if (ok) ok = mbar_wait_bounded(&tail->acc_full[acc], acc_phase, abort_flag, a.status);
      if (ok) {
        tc_fence_after_sync();
        const uint32_t taddr = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(acc * kBN);
        // ring row of this warp's 32 tokens; rows past the last token are written too (never read)
        const int ring_row = (gj % a.nb) * a.mw * kBM + ml * kBM + quarter * 32;
        const float* bias = ph == 0 ? a.bk : a.bv;
        constexpr int EB = kEpiBufs<kEncode, NPTS, G::WR>;
        const uint64_t pol_keep = l2_policy_evict_last();
        uint8_t* my_epi = epi_smem + (warp - 2) * EB * kEpiPieceBytes;
#pragma unroll 1
        for (int c = 0; c < n_pieces; ++c) {
          float v[32];
          tmem_ld_32x32b_x32(taddr + uint32_t(c * 32), v);
          if (bias != nullptr) {
            const float* b = bias + x0 + c * 32;
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __fadd_rn(v[i], __ldg(b + i));
          }
          uint8_t* buf = my_epi + (c & (EB - 1)) * kEpiPieceBytes;
          if (c >= EB) {                 // the store that last read this buffer must be done with it
            if (lane == 0) {
              if constexpr (EB == 2) bulk_wait_read_1(); else bulk_wait_read_0();
            }
            __syncwarp();
          }
          // lane = row of the piece; 16-byte chunk q of row r sits at chunk position q ^ (r % 8)
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<float4*>(buf + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d_hint(&tm.p, buf, x0 + c * 32, ring_row, pol_keep);   // read back soon by the row warps
            bulk_commit();
          }
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_leader(&tail->acc_empty[acc]);   // the leader's MMA issuer waits for both CTAs
          bulk_wait_all();               // the tile's rows are written
          fence_proxy_async_all();
        }
        __syncwarp();
      }
      // release by one thread after the barrier: its fence also covers the stores of the threads it
      // has synchronised with, and only that thread waits for them to become visible
      named_barrier(1, 128);
      if (*abort_flag) { stop = true; break; }
      if (warp == 2 && lane == 0) {
        __threadfence();
        atomicAdd(a.gemm_done + j * a.mw + ml, kTileWeight >> tile.log_split);
      }
    }
    }   // layers
  } else if (warp < 6 + G::ROW_WARPS) {
    // ------------------------------- row warps (TEAM warps per row; TEAMS rows at a time) ------
    constexpr int TEAM = G::TEAM, TEAMS = G::TEAMS;
    const int rw = warp - 6;
    const int team = rw / TEAM;
    constexpr int LOG_D = D == 1024 ? 10 : (D == 512 ? 9 : 8);
    const int log_h = kFull ? LOG_D : a.log_h, log_g = kFull ? LOG_D : a.log_g;
    // one context per warp; the sign bits are switched between key and value jobs
    RowCtx rck;
    WarpRowCtx wrc;
    ChunkRowCtx crc;
    uint32_t signs_k, signs_v;
    if constexpr (G::CR) {
      chunk_ctx_init(crc, log_h, log_g, lane);
      if constexpr (kEncode) crc.search = search_ctx<NPTS>(&rsm->tables, a.search.inv_w);
      signs_k = a.signmask_k[lane];
      signs_v = a.signmask_v[lane];
      rck.member = 0;
      rck.barrier = 0;
    } else if constexpr (G::WR) {
      wrc.lane = lane;
      if constexpr (kEncode) wrc.search = search_ctx<NPTS>(&rsm->tables, a.search.inv_w);
      wrc.signs = 0u;
      signs_k = a.signmask_k[lane];
      signs_v = a.signmask_v[lane];
      rck.member = 0;
      rck.barrier = 0;
    } else {
      row_ctx_init(rck, a.signmask_k, a.search.inv_w, log_h, log_g, lane, rw % TEAM, RowTeam<D>::NV, 3 + team);
      signs_k = a.signmask_k[lane] >> (rck.member * RowTeam<D>::NV);
      signs_v = a.signmask_v[lane] >> (rck.member * RowTeam<D>::NV);
    }
    const int n_groups = D >> log_g;
    bool stop = false;
    for (int l = 0; !stop && l < n_layers; ++l) {
    const LayerArgs& a = B.layer[l];
    for (int j = 0; j < n_jobs; ++j) {
      int ph, wave;
      layer_job(j, a.n_waves, ph, wave);
      const int gj = l * n_jobs + j;
      const WaveRows wr = wave_rows(wave, a.T, a.mw, gridDim.x);
      if (wr.tokens <= 0) continue;
      if constexpr (G::CR) crc.signs = ph == 0 ? signs_k : signs_v;
      else if constexpr (G::WR) wrc.signs = ph == 0 ? signs_k : signs_v;
      else row_ctx_set_signs(rck, ph == 0 ? signs_k : signs_v);
      const int slot_row = (ml * NTN + n_blk) * wr.rpc;      // first row (within the wave) of this CTA's slice
      const int rb = slot_row / kBM;                         // token block (within the wave) the slice lies in
      if (rb >= wr.blocks) continue;                         // nothing assigned, nobody waits for this CTA
      const int r_begin = slot_row % kBM;
      const int m = wave * a.mw + rb;
      const long long rows_left = (long long)a.T - (long long)m * kBM;
      const int r_end = rows_left < r_begin + wr.rpc ? int(rows_left) : r_begin + wr.rpc;
      if constexpr (kEncode) {
        // pull this job's input rows towards L2 while the prediction is still being produced
        const uint16_t* xin = ph == 0 ? a.K : a.V;
        for (int r = r_begin + (team + j) % TEAMS; r < r_end; r += TEAMS) {
          const long long g = (long long)m * kBM + r;
          if (lane < D / 256 / TEAM * 4)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(xin + g * a.ldX + rck.member * (D / TEAM) + lane * 64));
        }
      }
      bool ok = true;
      if constexpr (kAttnHD > 0) {
        // this layer's rows overwrite the reconstructions of two layers earlier (the caller alternates
        // two buffer pairs), which that layer's attention warps may, in principle, still be reading
        if (l >= 2) {
          if (lane == 0)
            ok = counter_wait_bounded(B.layer[l - 2].attn_done + wave * a.mw + rb, NTN * kAttnWarps, abort_flag, a.status, max_pause);
          ok = __shfl_sync(0xffffffffu, ok, 0);
        }
        // the key rows of this wave reuse the ring rows of wave - ring depth: the attention warps must
        // be done with them (they trail the rows by about one job, so this rarely waits)
        if (ok && ph == 0 && a.khat_ring > 0 && wave >= a.khat_ring) {
          if (lane == 0)
            ok = counter_wait_bounded(a.attn_done + (wave - a.khat_ring) * a.mw + rb, NTN * kAttnWarps, abort_flag,
                                      a.status, max_pause);
          ok = __shfl_sync(0xffffffffu, ok, 0);
        }
      }
      if (!ok) {
        // fall through to the report below with the abort flag set
      } else if (TEAM > 1) {
        // one thread polls for the team; all its warps must take the same path, so they agree
        // through the abort flag (set by a failed wait) between two barriers
        if (rck.member == 0 && lane == 0)
          row_wait(tail, gj + 1, a.gemm_done + j * a.mw + rb, kTileWeight * NTN, a.status, max_pause);
        team_barrier<D>(rck.barrier);
        ok = *abort_flag == 0;
        team_barrier<D>(rck.barrier);
      } else {
        if (lane == 0) ok = row_wait(tail, gj + 1, a.gemm_done + j * a.mw + rb, kTileWeight * NTN, a.status, max_pause);
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
      if (ok) {
        const float* pbuf = a.P + (size_t(gj % a.nb) * a.mw * kBM + size_t(rb) * kBM) * D;
        const size_t khat_base = a.khat_ring ? size_t((wave % a.khat_ring) * a.mw + rb) * kBM
                                             : size_t(m) * kBM;
        [[maybe_unused]] uint4 xraw[4];
        [[maybe_unused]] bool first_row = true;
        for (int r = r_begin + (team + j) % TEAMS; r < r_end; r += TEAMS) {   // rotated per job for balance
          const long long g = (long long)m * kBM + r;
          const float* pred_row = pbuf + size_t(r) * D;
          uint16_t* hat_row;
          if (ph == 0) hat_row = a.Khat + (khat_base + r) * a.ldKhat;
          else if (a.vhat_ring) hat_row = a.Vhat + (khat_base + r) * a.ldVhat;     // same ring geometry as K^
          else hat_row = a.Vhat != nullptr ? a.Vhat + g * a.ldVhat : nullptr;
          uint8_t* codes_row = (ph == 0 ? a.Kcodes : a.Vcodes) + g * CODE_BYTES;
          uint16_t* scales_row = (ph == 0 ? a.Kscales : a.Vscales) + g * n_groups;
          if constexpr (G::CR) {
            if constexpr (kEncode)
              chunk_encode_row<D / 256, NPTS, kBf16>(crc, &rsm->tables, (ph == 0 ? a.K : a.V) + g * a.ldX, pred_row, codes_row,
                                                     scales_row, hat_row);
            else
              chunk_decode_row<D / 256, NPTS, kBf16>(crc, rsm->tables.grid, codes_row, scales_row, pred_row, hat_row);
          } else if constexpr (G::WR) {
            unsigned long long* xbuf = rsm->scratch.xbuf[rw];
            if constexpr (kEncode) {
              const uint16_t* x_row = (ph == 0 ? a.K : a.V) + g * a.ldX;
              if constexpr (G::AHEAD) {
                if (first_row) wr_load_x_row(x_row, lane, xraw);
                first_row = false;
                const uint16_t* x_next = r + TEAMS < r_end ? x_row + TEAMS * a.ldX : nullptr;
                wr_encode_row_x<NPTS, kBf16, true>(wrc, &rsm->tables, xbuf, xraw, x_next, pred_row, codes_row, scales_row,
                                                   hat_row);
              } else {
                wr_encode_row<NPTS, kBf16>(wrc, &rsm->tables, xbuf, x_row, pred_row, codes_row, scales_row, hat_row);
              }
            } else {
              wr_decode_row<NPTS, kBf16, false, G::AHEAD>(wrc, rsm->tables.grid, xbuf, codes_row, scales_row, pred_row,
                                                          hat_row);
            }
          } else {
            TeamSmem<D>* ts = &rsm->scratch.team[team];
            if constexpr (kEncode) {
              const uint16_t* x_row = (ph == 0 ? a.K : a.V) + g * a.ldX;
              encode_row<D, NPTS, kBf16>(rck, &rsm->tables, ts, x_row, pred_row, codes_row,
                                         scales_row, hat_row);
            } else {
              decode_row<D, NPTS, kBf16>(rck, rsm->tables.grid, ts, codes_row, scales_row,
                                         pred_row, hat_row);
            }
          }
          // The row's prediction has been read for the last time: drop its lines from L2 without
          // writing them back (the ring is scratch; only whole, 128-byte aligned lines are dropped).
          // Not where the report of the rows does not release: see there.
          if (kEncode ? hat_row != nullptr : (ph == 0 || l + 1 < n_layers || j + kLayerRing >= n_jobs)) {
            __syncwarp();
            if constexpr (G::WR || G::CR) {
              const float* mine = pred_row + lane * 32;             // the row's lines, one per lane
              if (lane < D / 32 && (reinterpret_cast<uintptr_t>(mine) & 127) == 0)
                asm volatile("discard.global.L2 [%0], 128;" ::"l"(mine) : "memory");
            } else {
              const float* mine = pred_row + rck.member * 256 + lane * 8;
              if ((lane & 3) == 0 && (reinterpret_cast<uintptr_t>(mine) & 127) == 0)
                asm volatile("discard.global.L2 [%0], 128;" ::"l"(mine) : "memory");
            }
          }
        }
      }
      if (TEAM > 1) team_barrier<D>(rck.barrier); else __syncwarp();
      if (*abort_flag) { stop = true; break; }
      if (rck.member == 0 && lane == 0 && row_arrive(tail, gj + 1, TEAMS)) {   // one releasing thread per CTA (see the epilogue)
        // Key rows, and the value rows of all layers but the last, are read back by TMA loads of other CTAs; with attention all rows
        // are read by the attention warps of other CTAs: these reports release.  For the value rows of the last layer the
        // counter only lets an epilogue take the ring slot again.  It must then find the slot's predictions read (they
        // have been: the rows' stores depend on them) and the discards of its lines, which count as writes, in order before its TMA
        // stores.  The decoder leaves those discards out; the encoder reports such rows with the key rows of the
        // next job, whose release covers them (later_report), and else releases where the slot is taken again.
        // Measured against reports without a release and discards all the same (which was a race), us: 32768 tokens of d_kv 1024
        // encoded 387 / 386, 60000 684 / 685, 200000 2200 / 2245, 60000 of d_kv 512 272 / 275; 131072 of d_kv 1024 decoded 890 / 881, 60000 of d_kv 512
        // 177 / 175.  A release of its own for every report costs 1 to 2 %, encoded rows without discards 1 to 1.5 % from 30000 tokens on (but 60000 and
        // fewer gain by the later report), decoded rows reported later 4 to 5 %; a fourth buffer would halve what the long encodes lose, but
        // the decoder loses by it and the workspace grows.
        if (ph == 0 || l + 1 < n_layers) {
          fence_acq_rel_gpu();
          fence_proxy_async_all();
          if (kEncode && ph == 0 && l + 1 == n_layers && later_report(j - 1, n_jobs))
            atomicAdd(a.rows_done + (j - 1) * a.mw + rb, 1);       // both are full waves: the same token block
          atomicAdd(a.rows_done + j * a.mw + rb, 1);
        } else if (kAttnHD > 0) {
          fence_acq_rel_gpu();
          atomicAdd(a.rows_done + j * a.mw + rb, 1);
        } else if (!(kEncode && later_report(j, n_jobs))) {
          if (kEncode && j + kLayerRing < n_jobs) {
            fence_acq_rel_gpu();
            fence_proxy_async_all();
          }
          atomicAdd(a.rows_done + j * a.mw + rb, 1);
        }
      }
    }
    }   // layers
  } else {
    // ------------------------------- attention warps ------------------------------------------------
    if constexpr (kAttnHD > 0) {
      // A warp takes one KV head, 64 of its output dimensions (with head_dim 128 two warps share a head)
      // and one sub-block of kAttnSubTokens tokens of the token block; every (sub-block, sequence) has
      // its own partial slot.  (Eight warps on 64-token sub-blocks measured slower than four on whole
      // blocks: the kernel then runs at 80 registers and the row warps spill.)
      constexpr int WPH = kAttnHD / 64;                // warps per head and sub-block
      constexpr int NSUB = kBM / kAttnSubTokens;       // sub-blocks of a token block
      constexpr int HPAR = kAttnWarps / (WPH * NSUB);  // heads in flight per CTA
      const int aw = warp - 6 - G::ROW_WARPS;
      const int half = aw % WPH;
      const int sub = (aw / WPH) % NSUB;
      const int hpc = a.n_kv_heads / NTN;              // KV heads of a token block that this CTA attends over
      const int rep = a.n_q_heads / a.n_kv_heads;
      bool stop = false;
      for (int l = 0; !stop && l < n_layers; ++l) {
      const LayerArgs& a = B.layer[l];
      for (int wave = 0; wave < a.n_waves; ++wave) {
        const WaveRows wr = wave_rows(wave, a.T, a.mw, gridDim.x);
        if (ml >= wr.blocks) continue;                  // this CTA's block does not exist in the (last) wave
        bool ok = true;
        if (lane == 0)
          ok = counter_wait_bounded(a.rows_done + layer_value_job(wave, a.n_waves) * a.mw + ml,
                                    wave_block_ctas(wr, ml, gridDim.x), abort_flag, a.status, max_pause);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) { stop = true; break; }
        const long long blk = (long long)wave * a.mw + ml;       // token block of the call
        const long long sblk = blk * NSUB + sub;                 // this warp's sub-block of the call
        const long long tok0 = sblk * kAttnSubTokens;
        const long long tok1 = tok0 + kAttnSubTokens < a.T ? tok0 + kAttnSubTokens : a.T;
        const long long ring_row0 =
            a.khat_ring ? ((long long)(wave % a.khat_ring) * a.mw + ml) * kBM + sub * kAttnSubTokens : tok0;
        for (int h = n_blk * hpc + aw / (WPH * NSUB); h < (n_blk + 1) * hpc; h += HPAR) {
          long long t = tok0;
          while (t < tok1) {                            // one segment per sequence the sub-block overlaps
            const long long b = t / a.ctx;
            const long long seg_end = (b + 1) * a.ctx < tok1 ? (b + 1) * a.ctx : tok1;
            const long long row = ring_row0 + (t - tok0);
            const long long split = sblk - (b * a.ctx) / kAttnSubTokens;
            const long long pidx = (b * a.n_splits + split) * a.n_q_heads + (long long)h * rep;
            attn_segment_warp<kAttnHD, kBf16>(a.Khat + row * a.ldKhat + h * kAttnHD,
                                              a.Vhat + row * a.ldVhat + h * kAttnHD + half * 64, a.ldKhat, a.ldVhat,
                                              int(seg_end - t), a.q + (b * a.n_q_heads + (long long)h * rep) * kAttnHD,
                                              rep, a.scale_log2, half == 0 ? a.part_ml + pidx * 2 : nullptr,
                                              a.part_o + pidx * kAttnHD + half * 64, lane);
            t = seg_end;
          }
        }
        __syncwarp();
        if (lane == 0) {
          __threadfence();
          atomicAdd(a.attn_done + wave * a.mw + ml, 1);
        }
      }
      }   // layers
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

}  // namespace aquakv
