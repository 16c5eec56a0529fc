// Integer GEMM of b-bit codes held as E4M3 digit planes, on 5th-generation tensor cores (sm_103a).
//
//   acc[t, o] = sum_i (q_x[t, i] - z[t]) q_w[o, i],   y[t, o] = acc * s_x[t] * s_w[o]    (Sec. 3, Eq. 5)
//
// Codes of more than 4 bits do not fit one FP8 operand exactly, so each code is split into base-16
// digits, q = d0 + 16 d1 (|d| <= 16), one E4M3 byte per digit (d * 2^-9, exact).  With DX activation
// and DW weight digit planes the product splits by digit weight:
//   sum_i q_x q_w = sum_{g} 16^g P_g,   P_g = sum_{a + b = g} sum_i d_a(x) d_b(w),
// and every P_g is accumulated by tcgen05.mma kind::f8f6f4 in its own fp32 tensor-memory accumulator:
// its terms are products of digits (|d_x d_w| <= 16 * 8), so |P_g| * 2^18 stays below 2^24 and the
// accumulation is exact for d_in up to 2^16 (checked on the host).  The epilogue turns each P_g into
// an integer and adds them in int32; asymmetric activations then subtract z[t] times the weight row's
// code sum (the zero-point correction), and the product is scaled by the two steps in fp32.
//
// Tiles: 256 tokens (MMA M) x NB output channels per CTA pair (tcgen05.mma.cta_group::2): each CTA holds 128
// token rows and NB / 2 channel rows, every digit plane of both, so a channel row loaded once serves 256
// tokens.  A stage is KS codes of every plane (128, or 256 with one plane on either side): at the widest NB
// 64 KB or 48 KB a CTA, for 1024 cycles of MMAs, i.e. 48-64 B per cycle from L2; one CTA with a 128 x 128
// tile needed 64-96 and was held by that.  Persistent pairs, tiles in bands (tile_coords):
//   warps 0, 2   TMA producers of the token and the channel planes (one thread each)
//   warps 1, 3   even CTA: MMA issuers; odd CTA: forward its stages' readiness to the even CTA
//   warps 4..11  epilogue: two warps per TMEM lane quadrant, half of the tile's channels each
// The accumulators (one of NB columns per digit weight) are double-buffered where they fit twice in tensor
// memory.  Where they don't, the epilogue adds them up into registers first (int32, NB / 2 a thread) and
// gives tensor memory back before it scales and stores, so the next tile's MMAs wait for the loads only.
// Measured (8-bit asymmetric activations x 4-bit weights, 2048 x 4096 -> 6144; 8 x 8 bits, 1000 x 14336
// -> 4096): 230 and 185 us with one CTA per 128 x 128 tile and scalar stores, now 63 and 118 us; with one MMA
// issuer instead of two (and whole tiles) the second took 154 us, with two 130.
// Outputs that TMA cannot store (d_out % 4) go through the staging buffer too and out by a row's 32 channels a store: 121 x 192
// -> 10354 at 4 x 4 bits 32 us with each lane storing its own row, 23 now (10356: 19); up to 32 tokens, two warps of a pair
// that wait for each chunk's rows, 32 x 1024 -> 10354 21.5 and 23.7, so there each lane stores its own.
// Where whole tiles leave the last wave short, the last one to two waves are cut into equal ranges of (tile, stage) steps,
// one per pair (the stream part below): 8 x 8 bits, 1000 x 14336 -> 4096, 128 tiles on 76 pairs, 129.6 -> 117.5 us.
// Every wait is bounded.
#include <atomic>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "gemm_pair.cuh"
#include "per_device.h"

namespace cat {
namespace {

constexpr int BM = 128;                              // token rows per CTA (256 per pair)
constexpr int KB = 128;                              // codes (bytes) of one 128-byte swizzle atom
constexpr int kThreads = 384;
constexpr int kEpiWarp0 = 4, kEpiWarps = 8;
constexpr uint32_t kAtomA = BM * KB;                 // 16 KiB: one plane's atom of the token rows
constexpr uint32_t kEpiStage = 32 * 32 * 4;          // y staging buffer of an epilogue warp
constexpr int kMaxStages = 8;

// Token rows of a load: a CTA's tile, or as many as there are in whole swizzle atoms (the others keep what the shared
// memory held: their sums are not stored).  128-row boxes over a handful of rows were slow, by how much depending on
// where they lay in memory: one token, 4096 -> 14336 at 8 x 8 bits 75 to 89 us, with boxes of 8 rows 52, as from 16
// tokens on.
__host__ __device__ constexpr int token_rows(int64_t n) { return n >= BM ? BM : (int)((n + 7) / 8 * 8); }

struct DpBars {
  uint64_t full[kMaxStages], ready[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2], mma_done;
  uint32_t fwd_word[kMaxStages];                     // even CTA: targets of the odd CTA's st.async per stage
  uint32_t tmem_addr;
  int abort;
};

// DX, DW digit planes; NB channels per pair tile.
template <int DX, int DW, int NB>
struct DpGemmCfg {
  // accumulators: one per digit weight; with one plane on either side one per atom of a stage, so that the
  // two MMA issuers always have their own
  static constexpr int G = DX + DW == 2 ? 2 : DX + DW - 1;
  static constexpr int SHIFT = DX + DW == 2 ? 0 : 4;               // accumulator g stands for (1 << SHIFT g)
  static constexpr int NACC = 2 * G * NB <= 512 ? 2 : 1;           // copies of them in tensor memory
  static constexpr int AT = DX + DW == 2 ? 2 : 1;                  // atoms of codes per stage
  static constexpr int KS = AT * KB;                               // codes per stage
  static constexpr uint32_t ATOM_B = (uint32_t)(NB / 2) * KB;
  static constexpr uint32_t A_BYTES = (uint32_t)(DX * AT) * kAtomA, B_BYTES = (uint32_t)(DW * AT) * ATOM_B;
  static constexpr uint32_t STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t EPI_OFF_MAX = 192 * 1024;
  static constexpr int S = (int)(EPI_OFF_MAX / STAGE) < kMaxStages ? (int)(EPI_OFF_MAX / STAGE) : kMaxStages;
  static constexpr uint32_t EPI_OFF = S * STAGE;
  static constexpr uint32_t BAR_OFF = EPI_OFF + kEpiWarps * kEpiStage;
  static constexpr size_t SMEM = BAR_OFF + 512 + 1024;
  static constexpr uint32_t TMEM_COLS = NACC * G * NB <= 128 ? 128 : (NACC * G * NB <= 256 ? 256 : 512);
  static constexpr int CHUNKS = NB / 32;                           // 32-column chunks of the tile
  static constexpr int CH = (CHUNKS + 1) / 2;                      // a quadrant's first epilogue warp takes these, the second the rest
  static_assert(S >= 3 && SMEM <= 227 * 1024, "shared memory");
  static_assert(sizeof(DpBars) <= 512 && STAGE % 1024 == 0 && ATOM_B % 1024 == 0 && G * NB <= 512, "layout");
  static_assert(NB % 32 == 0, "pair MMAs have N in steps of 32");
};

// Bound of the pipeline waits (ns); kWaitLimitNs unless a test shortens it (cat_set_wait_limit_ns).
__device__ uint64_t g_dp_wait_limit = kWaitLimitNs;

// ---- the stream part: the last tiles as equal ranges of stages ---------------------------------
// Tiles [0, num_full) are whole, num_full / pairs per pair.  The others go in columns of `lanes` tiles (all token tiles of
// some channels, or single tiles): the steps (column, stage) are cut into one contiguous range per group of `lanes`
// pairs, and each pair of a group walks one tile of the column, so that a group reads its channel rows once, at the same time
// (1000 x 14336 -> 4096 at 8 x 8 bits with single tiles instead: 126.1 against 117.5 us).  A tile cut between groups is finished by the pair with its
// first step (its
// owner, whose range ends in it); the other pairs begin with their part of it, so the parts are on their way early: each
// epilogue warp sums its accumulators to int32, stores them to the pair's slice of device scratch and sets the
// pair's flag for that warp; the owner's same warp waits for it (bounded; the launch is cooperative, so all pairs are
// resident, and only owners wait) and adds.  Integer sums: exact in any order.  Flags hold the launch's number on its
// slot of scratch, counted on the device (the last warp to start moves it on), so nothing has to be reset, also after
// a launch that gave up, and graph replays count as launches.
// A launch takes every SM and is cooperative (all its CTAs are resident at once), so of two the later one begins when
// the earlier one ends; slots are handed out in turn all the same, for the edges of the two.  42 MB.
constexpr int kStreamSlots = 2;
constexpr int kStreamCtas = 160;
constexpr int kStreamWarpInt4 = 4 * 8 * 32;   // a warp's part: up to four chunks of 32 columns x 32 rows
__device__ int4 g_dp_part[kStreamSlots][kStreamCtas][kEpiWarps][kStreamWarpInt4];
__device__ uint32_t g_dp_flag[kStreamSlots][kStreamCtas][kEpiWarps];
__device__ uint32_t g_dp_epoch[kStreamSlots][2];   // launches so far; epilogue warps started

__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A pair's work: whole tiles, then its range of the stream part, tile by tile.
struct DpWork {
  int tile, k0, k1;                                // stages [k0, k1) of the tile
};
template <bool STREAM>
struct DpWalk {                                    // (not STREAM: whole tiles only)
  int next_full, num_full, pairs, num_k;
  int lanes, lane, group, groups, steps, g, g1;    // g: next step of the stream part
  __device__ DpWalk(int pair, int pairs_, int num_full_, int num_tiles, int num_k_, int lanes_)
      : next_full(pair), num_full(num_full_), pairs(pairs_), num_k(num_k_) {
    if constexpr (STREAM) {
      lanes = lanes_;
      lane = pair % lanes;
      group = pair / lanes;
      groups = pairs / lanes;
      steps = (num_tiles - num_full) / lanes * num_k;
      g = group < groups ? begin(group) : 0;
      g1 = group < groups ? begin(group + 1) : 0;
    }
  }
  __device__ int begin(int q) const { return (int)((int64_t)q * steps / groups); }
  __device__ bool next(DpWork* w) {
    if (next_full < num_full) {
      *w = {next_full, 0, num_k};
      next_full += pairs;
      return true;
    }
    if constexpr (STREAM) {
      if (g >= g1) return false;
      const int k0 = g % num_k, k1 = min(num_k, k0 + g1 - g);
      *w = {num_full + g / num_k * lanes + lane, k0, k1};
      g += k1 - k0;
      return true;
    }
    return false;
  }
};

__device__ __forceinline__ void tma_load_3d(void* smem_dst, const CUtensorMap* map, int32_t x, int32_t y, int32_t z,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// A staged 32 x 32 chunk to y without TMA: `rows` x `cols` of it, a row at a time.
__device__ __forceinline__ void plain_store(const uint8_t* buf, float* y, int d_out, int rows, int cols) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll 1
  for (int r0 = 0; r0 < rows; r0 += 8) {               // eight rows' loads in flight (rows past the end: whatever is there)
    float u[8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
      u[r] = *reinterpret_cast<const float*>(buf + (r0 + r) * 128 + (((lane >> 2) ^ r) << 4) + (lane & 3) * 4);
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (lane < cols && r0 + r < rows) y[(int64_t)(r0 + r) * d_out + lane] = u[r];
  }
}

// PLAIN: y without TMA (d_out % 4).  A kernel of its own: beside the TMA stores, inline or called, the plain ones cost the
// accumulators registers (1000 x 4096 -> 6144 at 8 x 4 bits 37.4 -> 38.0 us).
template <int DX, int DW, int NB, bool STREAM, bool PLAIN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    dp_gemm_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                   const __grid_constant__ CUtensorMap tmY, const float* __restrict__ sx, const int32_t* __restrict__ zx,
                   const float* __restrict__ sw, const int32_t* __restrict__ w_rowsum, int n, int d_in, int d_out,
                   float* __restrict__ y, int32_t* __restrict__ acc_out, int num_full,
                   int stream_lanes, int stream_slot, uint32_t* __restrict__ status) {
  using C = DpGemmCfg<DX, DW, NB>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  DpBars* bars = reinterpret_cast<DpBars*>(smem + C::BAR_OFF);
  volatile int* abort_flag = &bars->abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();               // 0: the pair's MMA issuer
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  const int num_m = (n + 2 * BM - 1) / (2 * BM), num_n = (d_out + NB - 1) / NB;
  const int num_tiles = num_m * num_n;
  const int num_k = (d_in + C::KS - 1) / C::KS;

  if (tid == 0) {
    for (int s = 0; s < C::S; ++s) {
      mbar_init(&bars->full[s], 2);                   // the two producers (+ 4 bytes from the odd CTA)
      mbar_init(&bars->ready[s], 2);
      mbar_init(&bars->empty[s], 2);                  // both MMA issuers' multicast commits
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->acc_full[b], 2);
      mbar_init(&bars->acc_empty[b], 2 * kEpiWarps);  // the epilogue warps of both CTAs (even CTA)
    }
    mbar_init(&bars->mma_done, 2);
    bars->abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  pdl_wait_then_release();                            // nothing global or in tensor memory before this
  const uint64_t lim = g_dp_wait_limit;
  if (warp == 0) tmem_alloc_pair(&bars->tmem_addr, C::TMEM_COLS);
  tc_fence_before();
  cluster_sync();                                     // both CTAs' barriers are initialized before any remote arrive
  tc_fence_after();
  const uint32_t tmem = bars->tmem_addr;

  if (warp == 0 || warp == 2) {
    // ------------------------------------------------------------------ TMA producers (warp 0: tokens, warp 2: channels)
    if (lane == 0) {
      const bool is_a = warp == 0;
      const CUtensorMap* map = is_a ? &tmX : &tmW;
      const uint32_t a_bytes = (uint32_t)(DX * C::AT * token_rows(n)) * KB;
      prefetch_tensormap(map);
      uint32_t it = 0;
      bool ok = true;
      DpWalk<STREAM> walk(pair, num_pairs, num_full, num_tiles, num_k, stream_lanes);
      for (DpWork w; ok && walk.next(&w);) {
        int m, nn;
        tile_coords(w.tile, num_m, num_n, &m, &nn);
        const int row = is_a ? m * 2 * BM + (int)rank * BM : nn * NB + (int)rank * (NB / 2);
        for (int ks = STREAM ? w.k0 : 0; ks < (STREAM ? w.k1 : num_k); ++ks, ++it) {
          const uint32_t s = it % C::S, use = it / C::S;
          if (use > 0 && !(ok = mbar_wait_bounded(&bars->empty[s], (use - 1) & 1, abort_flag, __LINE__, lim))) break;
          uint8_t* dst = smem + s * C::STAGE + (is_a ? 0u : C::A_BYTES);
          uint64_t* fb = rank == 0 ? &bars->full[s] : &bars->ready[s];
          mbar_arrive_expect_tx(fb, (is_a ? a_bytes : C::B_BYTES) + (is_a && rank == 0 ? 4u : 0u));
          const int planes = is_a ? DX : DW;
          const uint32_t atom = is_a ? kAtomA : C::ATOM_B;
          for (int p = 0; p < planes; ++p)
#pragma unroll
            for (int at = 0; at < C::AT; ++at)
              tma_load_3d(dst + (p * C::AT + at) * atom, map, ks * C::KS + at * KB, row, p, fb);
        }
      }
      // the copies in flight land before the CTA exits (they have, unless a wait gave up)
      volatile int no_abort = 0;
      for (uint32_t j = it > (uint32_t)C::S ? it - C::S : 0; j < it; ++j)
        mbar_wait_bounded(rank == 0 ? &bars->full[j % C::S] : &bars->ready[j % C::S], (j / C::S) & 1, &no_abort);
    }
  } else if ((warp == 1 || warp == 3) && rank == 1) {
    // ------------------------------------------------------------------ odd CTA: forward stage readiness
    // Each forwarder takes the stages of one parity, so that every barrier's phases are waited for in order
    // by one thread, whatever the number of stages.
    if (lane == 0) {
      const uint32_t grp = warp == 1 ? 0u : 1u;
      uint32_t it = 0;
      bool ok = true;
      DpWalk<STREAM> walk(pair, num_pairs, num_full, num_tiles, num_k, stream_lanes);
      for (DpWork w; ok && walk.next(&w);)
        for (int ks = STREAM ? w.k0 : 0; ks < (STREAM ? w.k1 : num_k); ++ks, ++it) {
          const uint32_t s = it % C::S;
          if ((s & 1u) != grp) continue;
          if (!(ok = mbar_wait_bounded(&bars->ready[s], (it / C::S) & 1, abort_flag, __LINE__, lim))) break;
          tc_fence_after();
          st_async_signal(&bars->fwd_word[s], &bars->full[s], 0);
        }
    }
  } else if (warp == 1 || warp == 3) {
    // ------------------------------------------------------------------ MMA issuers (even CTA)
    // Two threads, each with accumulators of its own: a thread's wait for a stage returns only once its
    // earlier MMAs have been handed on, and meanwhile the other's keep the tensor core busy.  Digit weights
    // go to issuer g & 1 (equal work: weight 1 has two products where there are three); with one plane on
    // either side each issuer takes one atom of the stage.
    if (lane == 0) {
      constexpr uint32_t kIdesc = idesc_e4m3_f32(2 * BM, NB);
      const int me = warp == 1 ? 0 : 1;
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      DpWalk<STREAM> walk(pair, num_pairs, num_full, num_tiles, num_k, stream_lanes);
      for (DpWork w; ok && walk.next(&w); ++tcount) {
        const uint32_t ab = tcount % C::NACC, use = tcount / C::NACC;
        if (use > 0 && !(ok = mbar_wait_bounded(&bars->acc_empty[ab], (use - 1) & 1, abort_flag, __LINE__, lim))) break;
        tc_fence_after();
        const uint32_t acc = tmem + ab * C::G * NB;
        for (int ks = STREAM ? w.k0 : 0; ks < (STREAM ? w.k1 : num_k); ++ks, ++it) {
          const uint32_t s = it % C::S;
          if (!(ok = mbar_wait_bounded(&bars->full[s], (it / C::S) & 1, abort_flag, __LINE__, lim))) break;
          tc_fence_after();
          const uint32_t abase = smem_u32(smem + s * C::STAGE), bbase = abase + C::A_BYTES;
#pragma unroll
          for (int a = 0; a < DX; ++a)
#pragma unroll
            for (int b = 0; b < DW; ++b)
#pragma unroll
              for (int at = 0; at < C::AT; ++at) {
                const int g = DX + DW == 2 ? at : a + b;
                if ((g & 1) != me) continue;
                // the pair (a, b) is the first one of its weight when a = 0 or b is the last plane
                const bool first = a == 0 || b == DW - 1;
#pragma unroll
                for (int kk = 0; kk < KB / 32; ++kk) {    // K = 32 codes per MMA: +32 B within an atom
                  const uint64_t da = sdesc_kmajor_sw128(abase + (uint32_t)(a * C::AT + at) * kAtomA) + 2 * kk;
                  const uint64_t db = sdesc_kmajor_sw128(bbase + (uint32_t)(b * C::AT + at) * C::ATOM_B) + 2 * kk;
                  mma_pair_ss(acc + g * NB, da, db, kIdesc, (ks != (STREAM ? w.k0 : 0) || kk != 0 || !first) ? 1u : 0u);
                }
              }
          mma_commit_pair(&bars->empty[s]);
        }
        if (ok) mma_commit_pair(&bars->acc_full[ab]);
      }
      mma_commit_pair(&bars->mma_done);                // all MMAs complete before TMEM is released
      volatile int no_abort = 0;
      mbar_wait_bounded(&bars->mma_done, 0, &no_abort);
    }
  } else if (warp >= kEpiWarp0) {
    // ------------------------------------------------------------------ epilogue: token row = TMEM lane
    const int quad = warp & 3, half = (warp - kEpiWarp0) >> 2;
    uint8_t* buf = smem + C::EPI_OFF + (warp - kEpiWarp0) * kEpiStage;
    const int ew = warp - kEpiWarp0;
    [[maybe_unused]] uint32_t mark = 0;                // this launch's number on its slot
    if constexpr (STREAM) {
      if (lane == 0) {
        uint32_t* epoch = g_dp_epoch[stream_slot];
        const uint32_t e = ld_acquire_gpu(&epoch[0]);
        mark = e + 1u;
        __threadfence();
        if (atomicAdd(&epoch[1], 1u) == gridDim.x * kEpiWarps - 1u) {   // every warp has read the number
          epoch[1] = 0u;
          __threadfence();
          epoch[0] = e + 1u;
        }
      }
      mark = __shfl_sync(0xFFFFFFFFu, mark, 0);
    }
    uint32_t tcount = 0;
    DpWalk<STREAM> walk(pair, num_pairs, num_full, num_tiles, num_k, stream_lanes);
    bool ok = true;
    for (DpWork w; ok && walk.next(&w); ++tcount) {
      const uint32_t ab = tcount % C::NACC;
      const bool is_part = STREAM && w.k0 > 0, is_owner = STREAM && w.k0 == 0 && w.k1 < num_k;
      int m, nn;
      tile_coords(w.tile, num_m, num_n, &m, &nn);
      const int row0 = m * 2 * BM + (int)rank * BM + quad * 32, t = row0 + lane;
      const int col0 = nn * NB + half * C::CH * 32, chunks = half == 0 ? C::CH : C::CHUNKS - C::CH;
      const float sxt = t < n ? sx[t] : 0.f;
      const uint32_t zt = (t < n && zx) ? (uint32_t)zx[t] : 0u;
      if (!mbar_wait_bounded(&bars->acc_full[ab], (tcount / C::NACC) & 1, abort_flag, __LINE__, lim)) break;
      __syncwarp();
      tc_fence_after();
      const uint32_t tcol = tmem + ((uint32_t)(quad * 32) << 16) + ab * C::G * NB + half * C::CH * 32;
      auto gather = [&](int c, uint32_t (&acc)[32]) {  // chunk c: sum over the digit weights, int32
#pragma unroll
        for (int g = 0; g < C::G; ++g) {
          uint32_t r[32];
          __syncwarp();
          CAT_TMEM_LD32(tcol + g * NB + c * 32, r);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const uint32_t v = (uint32_t)__float2int_rn(__uint_as_float(r[j]) * kAccScale) << (C::SHIFT * g);
            acc[j] = g == 0 ? v : acc[j] + v;
          }
        }
      };
      auto release = [&] {                             // the accumulators are read: the MMAs may have them back
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(&bars->acc_empty[ab], 0);
      };
      auto put_part = [&](int c, const uint32_t (&acc)[32]) {
        int4* dst = g_dp_part[stream_slot][blockIdx.x][ew] + c * 8 * 32 + lane;
#pragma unroll
        for (int q = 0; q < 8; ++q)
          __stcg(dst + q * 32, make_int4((int)acc[4 * q], (int)acc[4 * q + 1], (int)acc[4 * q + 2], (int)acc[4 * q + 3]));
      };
      auto set_flag = [&] {
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicExch(&g_dp_flag[stream_slot][blockIdx.x][ew], mark);
      };
      // the owner: the groups after this one whose ranges begin before the tile ends
      auto parts = [&](auto&& f) {
        const int tile_end = ((w.tile - num_full) / walk.lanes + 1) * num_k;
        for (int q = walk.group + 1; q < walk.groups && walk.begin(q) < tile_end; ++q)
          if (walk.begin(q) < walk.begin(q + 1)) f(2 * (q * walk.lanes + walk.lane) + (int)rank);
      };
      auto wait_parts = [&] {
        bool got = true;
        parts([&](int cta) {
          const uint32_t* flag = &g_dp_flag[stream_slot][cta][ew];
          if (got && lane == 0 && ld_acquire_gpu(flag) != mark) {
            const uint64_t t0 = globaltimer_ns();
            for (uint32_t i = 1; got && ld_acquire_gpu(flag) != mark; ++i) {
              __nanosleep(64);
              if ((i & 63u) == 0u && (*abort_flag || globaltimer_ns() - t0 > lim)) {
                if (*abort_flag == 0) *abort_flag = __LINE__;
                got = false;
              }
            }
          }
          got = __shfl_sync(0xFFFFFFFFu, (int)got, 0);
        });
        __threadfence();                               // the parts' stores are seen by every lane, not by the polling one alone
        return got;
      };
      auto add_parts = [&](int c, uint32_t (&acc)[32]) {
        parts([&](int cta) {
          const int4* src = g_dp_part[stream_slot][cta][ew] + c * 8 * 32 + lane;
          constexpr int B = 2;                         // loads in flight: the registers left beside the accumulators
#pragma unroll
          for (int i0 = 0; i0 < 8; i0 += B) {
            int4 v[B];
#pragma unroll
            for (int i = 0; i < B; ++i) v[i] = __ldcg(src + (i0 + i) * 32);
#pragma unroll
            for (int i = 0; i < B; ++i) {
              acc[4 * (i0 + i)] += (uint32_t)v[i].x;
              acc[4 * (i0 + i) + 1] += (uint32_t)v[i].y;
              acc[4 * (i0 + i) + 2] += (uint32_t)v[i].z;
              acc[4 * (i0 + i) + 3] += (uint32_t)v[i].w;
            }
          }
        });
      };
      auto finish = [&](int c, uint32_t (&acc)[32]) {
        const int o0 = col0 + c * 32;
        if (o0 >= d_out || row0 >= n) return;          // warp-uniform: nothing of this chunk is in range
        const bool in = o0 + lane < d_out;             // the chunk's 32 channel steps and code sums, one per lane
        const float swl = in ? __ldg(sw + o0 + lane) : 0.f;
        if (zx) {
          // zero points: the result fits int32, so the difference may be taken modulo 2^32
          const uint32_t rsl = in ? (uint32_t)__ldg(w_rowsum + o0 + lane) : 0u;
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] -= zt * __shfl_sync(0xFFFFFFFFu, rsl, j);
        }
        if (acc_out && t < n) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (o0 + j < d_out) acc_out[(int64_t)t * d_out + o0 + j] = (int32_t)acc[j];
        }
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = (float)(int32_t)acc[j] * sxt * __shfl_sync(0xFFFFFFFFu, swl, j);
        if constexpr (PLAIN) {
          if (n <= 32) {                               // one warp's rows: every lane its own
            if (t < n) {
              float* yrow = y + (int64_t)t * d_out;
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (o0 + j < d_out) yrow[o0 + j] = v[j];
            }
            return;
          }
        } else {
          if (lane == 0) bulk_wait_read_all();         // the store before has read the buffer
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q)                    // row `lane`, 16-byte chunk q at q ^ (lane % 8)
          *reinterpret_cast<float4*>(buf + lane * 128 + ((q ^ (lane & 7)) << 4)) =
              make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        if constexpr (!PLAIN) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tmY, buf, o0, row0);
            bulk_commit();
          }
        } else {
          plain_store(buf, y + (int64_t)row0 * d_out + o0, d_out, min(32, n - row0), min(32, d_out - o0));
        }
      };
      if constexpr (C::NACC == 2) {                    // the other copy takes the next tile meanwhile
        static_assert(!STREAM || C::NACC == 1, "the stream part is for the widest tiles");
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          uint32_t acc[32];
          gather(c, acc);
          if (c == chunks - 1) release();
          finish(c, acc);
        }
      } else {
        uint32_t acc[C::CH][32];
#pragma unroll
        for (int c = 0; c < C::CH; ++c)
          if (c < chunks) gather(c, acc[c]);
        release();
        if constexpr (STREAM) {
          if (is_part) {
#pragma unroll
            for (int c = 0; c < C::CH; ++c)
              if (c < chunks) put_part(c, acc[c]);
            set_flag();
            continue;
          }
          if (is_owner) {
            if (!(ok = wait_parts())) break;
#pragma unroll
            for (int c = 0; c < C::CH; ++c)
              if (c < chunks) add_parts(c, acc[c]);
          }
        }
#pragma unroll
        for (int c = 0; c < C::CH; ++c)
          if (c < chunks) finish(c, acc[c]);
      }
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
  }

  tc_fence_before();
  cluster_sync();                                     // the pair's MMAs and both epilogues are done with TMEM
  if (bars->abort && tid == 0) report(status, timeout_bits(kWhereGemmDp, bars->abort));
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, C::TMEM_COLS);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// Tensor map of D digit planes [D][rows][d_in] bytes: box 128 codes x box_rows rows x 1 plane, 128B swizzle;
// rows past the end read as zero.
bool plane_map(CUtensorMap* map, const uint8_t* planes, int64_t rows, int64_t d_in, int D, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  memset(map, 0, sizeof(*map));
  cuuint64_t dims[3] = {(cuuint64_t)d_in, (cuuint64_t)rows, (cuuint64_t)D};
  cuuint64_t strides[2] = {(cuuint64_t)d_in, (cuuint64_t)(rows * d_in)};
  cuuint32_t box[3] = {(cuuint32_t)KB, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(planes), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// y [n][d_out] float32, box 32 x 32, 128-byte swizzle (the epilogue's staging layout).
bool output_map(CUtensorMap* map, float* y, int64_t n, int64_t d_out) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)d_out, (cuuint64_t)n};
  cuuint64_t strides[1] = {(cuuint64_t)d_out * sizeof(float)};
  cuuint32_t box[2] = {32, 32};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, y, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

int num_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
  return sms;
}

// Whole tiles of a launch with a stream part: all but the last one to two waves (tiles >= pairs).
int64_t stream_full(int64_t tiles, int64_t pairs) { return (tiles / pairs - 1) * pairs; }
// Tiles of a column of the stream part: all token tiles, where they are one band (tile_coords), whole columns remain
// and few pairs are left over; else single tiles.
int stream_lanes(int64_t n, int64_t tiles, int64_t pairs) {
  const int64_t num_m = (n + 2 * BM - 1) / (2 * BM);
  const bool fits = num_m <= kBandM && stream_full(tiles, pairs) % num_m == 0 && 16 * (pairs % num_m) <= pairs;
  return fits ? (int)num_m : 1;
}

struct DpCall {
  const uint8_t* x_planes;
  const float* sx;
  const int32_t* zx;
  const uint8_t* w_planes;
  const float* sw;
  const int32_t* w_rowsum;
  int64_t n, d_in, d_out;
  float* y;
  int32_t* acc_out;
  uint32_t* status;
  cudaStream_t stream;
};

// Whether a cooperative launch of `pairs` CTA pairs, all that the device has, fits on it (checked once per device).
template <int DX, int DW, int NB>
bool stream_launch_ok(int64_t pairs) {
  using C = DpGemmCfg<DX, DW, NB>;
  static PerDevice<bool> asked;
  return asked.get([&] {
    auto fits = [&](auto kernel) {
      cudaLaunchConfig_t cfg;
      memset(&cfg, 0, sizeof(cfg));
      cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
      cfg.blockDim = dim3(kThreads, 1, 1);
      cfg.dynamicSmemBytes = C::SMEM;
      int clusters = 0;
      return allow_smem(kernel, C::SMEM) == cudaSuccess &&
             cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters >= pairs;
    };
    int dev = 0, coop = 0;
    const bool ok = 2 * pairs <= kStreamCtas && cudaGetDevice(&dev) == cudaSuccess &&
                    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
                    fits(dp_gemm_kernel<DX, DW, NB, true, false>) && fits(dp_gemm_kernel<DX, DW, NB, true, true>);
    cudaGetLastError();
    return ok;
  });
}

// One turn for every kind of this kernel: they share the slots.
int next_stream_slot() {
  static std::atomic<unsigned> next{0};
  return (int)(next.fetch_add(1, std::memory_order_relaxed) % kStreamSlots);
}

template <int DX, int DW, int NB, bool STREAM, bool PLAIN>
cudaError_t launch_as(const DpCall& c, const CUtensorMap& my) {
  using C = DpGemmCfg<DX, DW, NB>;
  static_assert(C::CH * 8 * 32 <= kStreamWarpInt4, "a warp's part");
  CUtensorMap mx, mw;
  if (!plane_map(&mx, c.x_planes, c.n, c.d_in, DX, token_rows(c.n)) || !plane_map(&mw, c.w_planes, c.d_out, c.d_in, DW, NB / 2))
    return cudaErrorInvalidValue;
  static PerDevice<cudaError_t> allowed;
  const cudaError_t attr = allowed.get([] { return allow_smem(dp_gemm_kernel<DX, DW, NB, STREAM, PLAIN>, C::SMEM); });
  if (attr != cudaSuccess) return attr;
  const int64_t tiles = ((c.n + 2 * BM - 1) / (2 * BM)) * ((c.d_out + NB - 1) / NB);
  if (tiles > 0x3FFFFFFF) return cudaErrorInvalidValue;
  const int64_t pairs = num_sms() / 2;
  const int64_t num_full = STREAM ? stream_full(tiles, pairs) : tiles;
  const int lanes = STREAM ? stream_lanes(c.n, tiles, pairs) : 1;
  const int slot = STREAM ? next_stream_slot() : 0;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)(2 * (STREAM || tiles > pairs ? pairs : tiles)), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = c.stream;
  cudaLaunchAttribute attrs[2];
  attrs[0] = pdl_attr();
  attrs[1].id = cudaLaunchAttributeCooperative;   // owners wait for their tiles' other parts
  attrs[1].val.cooperative = 1;
  cfg.attrs = attrs;
  cfg.numAttrs = STREAM ? 2 : 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, dp_gemm_kernel<DX, DW, NB, STREAM, PLAIN>, mx, mw, my, c.sx, c.zx, c.sw, c.w_rowsum, (int)c.n,
                            (int)c.d_in, (int)c.d_out, c.y, c.acc_out, (int)num_full, lanes, slot, c.status);
}

template <int DX, int DW, int NB, bool STREAM = false>
cudaError_t launch_nb(const DpCall& c) {
  CUtensorMap my;
  memset(&my, 0, sizeof(my));
  const bool tma = c.d_out % 4 == 0 && output_map(&my, c.y, c.n, c.d_out);
  return tma ? launch_as<DX, DW, NB, STREAM, false>(c, my) : launch_as<DX, DW, NB, STREAM, true>(c, my);
}

// The cycles a launch with NB-wide tiles should take: whole waves of tiles, each its stages (the MMAs of a
// stage plus the ~200 cycles its barrier wait idles the tensor core, or the stage's loads at ~55 B per cycle
// and SM) and an epilogue of ~8 cycles per column and accumulator.  With a stream part (from one whole wave on) the
// stages spread evenly over the pairs of whole groups, for one epilogue and the exchange of the parts more.
constexpr double kStreamExchange = 16000.0;   // measured 13 to 20 thousand, the loss of L2 sharing included
template <int DX, int DW, int NB>
double tile_model(int64_t n, int64_t d_in, int64_t d_out, int64_t pairs, bool stream = false) {
  using C = DpGemmCfg<DX, DW, NB>;
  const int64_t tiles = ((n + 2 * BM - 1) / (2 * BM)) * ((d_out + NB - 1) / NB);
  const double mma = (double)DX * DW * (C::KS / 32) * (NB / 2) + 200.0, load = C::STAGE / 55.0;
  const int64_t num_k = (d_in + C::KS - 1) / C::KS;
  const double stage = mma > load ? mma : load, epi = 8.0 * C::G * NB / C::NACC;
  if (!stream) return (double)((tiles + pairs - 1) / pairs) * (num_k * stage + epi);
  if (tiles <= pairs || tiles % pairs == 0) return 1e30;
  const int64_t full = stream_full(tiles, pairs), lanes = stream_lanes(n, tiles, pairs);
  const double waves = (double)(full / pairs) + (double)(tiles - full) / (double)(pairs / lanes * lanes);
  return waves * num_k * stage + (waves + 1.0) * epi + kStreamExchange;
}

// Wide tiles load the token planes less often and have more MMA work behind each wait; narrow ones spread
// a small call over more pairs, and the widths between fill the last wave (2048 tokens -> 6144 channels: 192
// tiles of 256 are 2.53 waves, 224 of 224 are 2.95, of seven eighths the work: 71.4 -> 65.3 us at 8 x 4 bits).
template <int DX, int DW>
cudaError_t launch_dx_dw(const DpCall& c) {
  constexpr int WIDE = DX + DW == 4 ? 128 : 256;         // G accumulators of WIDE columns fit tensor memory
  constexpr int MID1 = WIDE - 32, MID2 = WIDE == 256 ? 192 : WIDE / 2;   // 224 and 192; 96
  const int64_t pairs = num_sms() / 2;
  const double cost[4] = {tile_model<DX, DW, WIDE>(c.n, c.d_in, c.d_out, pairs),
                          tile_model<DX, DW, MID1>(c.n, c.d_in, c.d_out, pairs),
                          tile_model<DX, DW, MID2>(c.n, c.d_in, c.d_out, pairs),
                          tile_model<DX, DW, WIDE / 2>(c.n, c.d_in, c.d_out, pairs)};
  int best = 0;
  for (int i = 1; i < 4; ++i)
    if (cost[i] < cost[best]) best = i;
  // The stream part where the model sees 3.5 % in it (what it is wrong by); 96-wide tiles take a tenth longer than
  // modelled.  8 x 8 bits: 1000 x 14336 -> 4096 (1.68 waves) 129.6 -> 117.5 us, 2048 x 4096 -> 6144 (5.05, then 96 wide)
  // 125.7 -> 112.9, 3000 x 4096 -> 4096 126.1 -> 113.0, 512 x 8192 -> 8192 80.0 -> 75.9; below the line 4096 x 4096 -> 4096
  // (6.74 waves) 144.7 -> 147.6, at 8 x 4 bits 5000 x 4096 -> 6144 (6.3) 151.0 -> 155.9, and tiles for less than a wave,
  // where nothing hides the exchange, 256 x 8192 -> 8192 43.5 -> 52.3.
  const double whole = cost[best] * ((best == 1 && MID1 == 96) ? 1.1 : 1.0);
  if (tile_model<DX, DW, WIDE>(c.n, c.d_in, c.d_out, pairs, true) < 0.965 * whole &&
      stream_launch_ok<DX, DW, WIDE>(pairs))
    return launch_nb<DX, DW, WIDE, true>(c);
  switch (best) {
    case 0: return launch_nb<DX, DW, WIDE>(c);
    case 1: return launch_nb<DX, DW, MID1>(c);
    case 2: return launch_nb<DX, DW, MID2>(c);
    default: return launch_nb<DX, DW, WIDE / 2>(c);
  }
}

}  // namespace

cudaError_t set_dp_wait_limit(uint64_t ns) { return cudaMemcpyToSymbol(g_dp_wait_limit, &ns, sizeof(ns)); }

// x_planes [DX][n][d_in], w_planes [DW][d_out][d_in] digit bytes; zx / w_rowsum both given for
// asymmetric activations (else both NULL).
cudaError_t launch_dp_gemm(const uint8_t* x_planes, int DX, const float* sx, const int32_t* zx, const uint8_t* w_planes,
                           int DW, const float* sw, const int32_t* w_rowsum, int64_t n, int64_t d_in, int64_t d_out,
                           float* y, int32_t* acc_out, uint32_t* status, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const DpCall c = {x_planes, sx, zx, w_planes, sw, w_rowsum, n, d_in, d_out, y, acc_out, status, stream};
  if (DX == 1 && DW == 1) return launch_dx_dw<1, 1>(c);
  if (DX == 2 && DW == 1) return launch_dx_dw<2, 1>(c);
  if (DX == 1 && DW == 2) return launch_dx_dw<1, 2>(c);
  if (DX == 2 && DW == 2) return launch_dx_dw<2, 2>(c);
  return cudaErrorInvalidValue;
}

}  // namespace cat
