// Policy-indexed chunk-causal attention (Eq. 4, Section 3.2) for a batch of
// denoising nodes on sm_103a.
//
// For node n, head h and query u of the node's own chunk:
//   O[u] = sum_v softmax_v(scale * q_u . k_v + M(u, v)) v_v,
// where M is 0 on every key of the node's own slot (bidirectional inside the
// chunk) and of its visible context slots, and -inf everywhere else.  Keys
// outside those slots are never read, so the mask costs nothing except on the
// zero pad rows of each slot's last tile, which get -inf explicitly.
//
// One CTA computes one work unit: (node, head, a pair of 128-query tiles Q0,
// Q1) and streams every key tile of every slot the node reads; each K/V tile
// in shared memory serves both query tiles.
//   warp 0     TMA producer: Q0/Q1 once, then K and V tiles of the slot list
//              into rings of shared-memory stages (128B swizzle);
//   warps 1, 3 MMA issuers, warp 1 for query tile 0 and warp 3 for query
//              tile 1 (each whole warp runs its loop, one elected lane
//              issues); warp 1 also owns TMEM;
//   warps 4-11 softmax, all eight warps on one query tile at a time (Q0 then
//              Q1 of every key tile): two threads per query row, 64 keys
//              each; S from TMEM, fp32 online softmax in the log2 domain with
//              a lazy rescale of O, P written back over S as bf16; then the
//              epilogue (O / l to bf16 global, optional LSE).
// TMEM columns (d = 128): S0 [0,128), S1 [128,256), O0 [256,384), O1 [384,512).
// Each issuer's order per key tile i is PV_b,i then S_b,i+1, so the softmax of
// either query tile has the other tile's PV and S (two 128x128x128 MMAs) to
// hide behind.  A tcgen05.mma costs its issuing warp nearly as long as the
// tensor pipe takes to run it (about 60 of 64 cycles while the softmax warps
// share the SM), so one issuer for both tiles left the pipe idle whenever it
// waited on a barrier; two issuers on different sub-partitions each have half
// the MMAs to issue.  A commit that completes S_b of tile i also implies PV_b
// of tile i-1 is complete (one issuer per tile, MMAs of a thread execute in
// issue order), so the rescale of O_b needs no extra barrier.
//
// Head dimension 64 halves the MMAs of a key tile (1024 tensor cycles instead
// of 2048) but not its softmax, so the loop above, whose period is two
// softmaxes one after the other plus the hand-overs, ran as slowly as at 128
// (2300 cycles a key tile, tensor pipe 40% busy, MUFU 42%, no unit near its
// limit).  There:
//   - warps 4-7 own query tile 0 and warps 8-11 query tile 1, a thread per row
//     with all 128 keys: two independent softmax chains, in opposite phase
//     because of the buffer rotation below, so that one's exponentials run
//     while the other waits for loads and barriers (in phase they contend for
//     the MUFU and then idle together: 2700 cycles);
//   - O needs 64 columns a tile, so three S buffers fit: S columns [0,384) by
//     step n = (key tile, query tile) mod 3, O0 [384,448), O1 [448,512).  The
//     S of a step are issued one and a half key tiles before their softmax,
//     right behind the PV that reads the buffer they overwrite;
//   - both issuers together need all the issue slots they can get: an MMA run
//     is issued under one election (an election per MMA held a single issuer
//     at 1450 cycles a step), the even steps' PV by warp 1, the odd ones' by
//     warp 3, and the V stages are freed by their commits.
// 2 nodes x 16 heads x 2160 tokens over 10800 keys: 217 -> 176 us (880 -> 1085
// TFLOP/s).  What bounds it now is the chain of one step: S wait 190 cycles,
// TMEM load 200, max and vote 230, exponentials 780, P store and hand-over 150.
// A unit may be split into n_split contiguous key ranges (when there are too
// few units to fill the GPU's waves): each split CTA writes its normalised
// partial O with its row max and sum to the workspace and bumps the unit's
// arrival counter; the last to arrive merges the partials (the usual
// log-sum-exp combination) and writes the output, then resets the counter.
// Where all splits fit on the GPU at once a unit's ranges are a cluster of two
// to eight CTAs instead, which merge through distributed shared memory (16 key
// tiles, 12 heads: 21.5 us through the workspace, 14.8 us so).
// All waits are bounded (1 s by default): on expiry the CTA records
// SVA_ERR_DEVICE_TIMEOUT in the status word, drains its own copies and MMAs,
// frees TMEM and exits.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace sva {
namespace {

using namespace ptx;

template <int D>
struct AttnCfg {
  static_assert(D == 64 || D == 128, "head_dim");
  static constexpr int kBoxBytes = kTile * 64 * 2;   // one 128-row x 64-column bf16 box
  static constexpr int kBoxes = D / 64;
  static constexpr int kTileBytes = kBoxBytes * kBoxes;
  static constexpr int kKStages = (D == 128) ? 3 : 4;
  static constexpr int kVStages = (D == 128) ? 2 : 6;
  static constexpr int kOffQ0 = 0;
  static constexpr int kOffQ1 = kTileBytes;
  static constexpr int kOffK = 2 * kTileBytes;
  static constexpr int kOffV = kOffK + kKStages * kTileBytes;
  static constexpr int kSmemBytes = kOffV + kVStages * kTileBytes + 1024;  // + alignment slack
  static constexpr uint32_t kTmemCols = 512;
  // Head dimension 64: each softmax warpgroup owns one query tile (a thread
  // per row), three S buffers.  See the note above the kernel.
  static constexpr bool kOwnTile = D == 64;
  static constexpr int kStepBars = kOwnTile ? 6 : 2;        // S (and P) barriers
  static constexpr int kTilesPerWarp = kOwnTile ? 1 : 2;    // query tiles a softmax warp works on
  static constexpr int kRowThreads = kOwnTile ? 1 : 2;      // threads per query row
  static constexpr int kChunks = 4 / kRowThreads;           // 32-key chunks of a row per thread
};

// TMEM columns.  D = 128: one S buffer per query tile and the two O
// accumulators fill the 512 columns.  D = 64: O takes 64 columns a tile, which
// leaves room for a third S buffer; the steps (key tile, query tile) take the
// three in turn.
template <int D>
__device__ __forceinline__ uint32_t col_s(int buf) {
  return (uint32_t)buf * 128u;
}
template <int D>
__device__ __forceinline__ uint32_t col_o(int b) {
  return D == 128 ? (b ? 384u : 256u) : (b ? 448u : 384u);
}

// 12 warps: warpgroup 0 = TMA producer (warp 0), MMA issuers (warps 1 and
// 3), warp 2 (the block-sparse mask gather in the prologue, then idle);
// warpgroups 1 and 2 = softmax.  The launch gives every thread kLaunchRegs
// registers; warpgroup 0 then gives registers back (setmaxnreg.dec to
// kRegsLow) and the softmax warpgroups take them (setmaxnreg.inc to
// kRegsHigh).  The split must fit the launch's pool: 4*32*kRegsLow +
// 8*32*kRegsHigh <= 384*kLaunchRegs, checked at launch.  At D = 64 a softmax
// thread holds 128 scores and spills below 216 (88 + 208 was 3% slower).
constexpr int kThreads = 384;
constexpr int kLaunchRegs = 168;
template <int D>
struct AttnRegs {
  static constexpr int kLow = D == 128 ? 88 : 72;
  static constexpr int kHigh = D == 128 ? 208 : 216;
  static constexpr int kPool = 4 * 32 * kLow + 8 * 32 * kHigh;
  static_assert(kPool <= kThreads * kLaunchRegs, "register split");
};
// Lazy rescale of O: a row's running max m is only moved (and O, l scaled)
// when a tile's max exceeds it by more than this many log2 units, so P =
// 2^(x - m) <= 2^64 between rescales.  Then l <= 2^(64 + 16) for up to 2^16
// keys and |O| <= 2^86 for |V| <= 2^6, far below the fp32 and bf16 limit of
// 2^128, while bf16 keeps P's relative precision at any magnitude.  With
// x10 outliers in q and k a row's max keeps jumping by more than 2^8 long
// into the key sequence, and each jump cost the warp a TMEM round trip of O
// on the softmax's critical path (stress14b: 2^64 instead of 2^8 is 1.8%
// faster).
constexpr float kRescaleThreshold = 64.0f;

template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ uint64_t f2u(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ void u2f(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}

// (a0, a1) * bb + cc, two lanes in one instruction
__device__ __forceinline__ void ffma2(float& o0, float& o1, float a0, float a1, uint64_t bb,
                                      uint64_t cc) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2u(a0, a1)), "l"(bb), "l"(cc));
  u2f(r, o0, o1);
}

__device__ __forceinline__ uint64_t fadd2(uint64_t a, float b0, float b1) {
  uint64_t r;
  asm("add.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(f2u(b0, b1)));
  return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 r = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&r);
}

struct Bars {
  uint64_t q_full;
  // S and P of a query tile's steps.  D = 128: one each per query tile.  D =
  // 64: three per query tile taken in turn, so that each barrier has one
  // waiter, which waits for every phase (the S of a query tile run up to two
  // key tiles ahead of its softmax, and its P up to two ahead of the issuer).
  uint64_t s_full[6];
  uint64_t p_full[6];
  uint64_t o_final;
  uint64_t drain;
  uint64_t k_full[4];
  uint64_t k_empty[4];
  uint64_t v_full[6];
  uint64_t v_empty[6];
};

// Block-sparse launches: a role's walk over the key tiles that either query
// tile of the unit may attend (bitmaps in the kernel's tile order).  The
// current word's remaining bits stay in a register, so a step reads shared
// memory only when it moves to the next word.  start() takes a set bit (or
// n_all); the first next() returns it, each later one the following tile of
// the walk, or n_all past the last.
template <int W>
struct TileWalk {
  const uint32_t (*tm)[W];
  int n_all, w;
  uint32_t u;
  __device__ __forceinline__ void start(const uint32_t (*tm_)[W], int from, int n_all_) {
    tm = tm_;
    n_all = n_all_;
    w = from >> 5;
    u = from < n_all ? (tm[0][w] | tm[1][w]) & (~0u << (from & 31)) : 0u;
  }
  __device__ __forceinline__ int next() {
    const int words = (n_all + 31) >> 5;
    while (u == 0u) {
      if (++w >= words) return n_all;
      u = tm[0][w] | tm[1][w];
    }
    const int k = (w << 5) + __ffs(u) - 1;
    u &= u - 1u;
    return k;
  }
};

// The lowest n bits (none for n <= 0, all 32 for n >= 32).
__device__ __forceinline__ uint32_t first_bits(int n) {
  return n >= 32 ? ~0u : (n <= 0 ? 0u : (1u << n) - 1u);
}

// -inf where a key's bit is clear: bit e of w[c] belongs to s[c][e].
template <int NC>
__device__ __forceinline__ void hide_keys(uint32_t (&s)[NC][32], const uint32_t (&w)[NC]) {
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (!((w[c] >> e) & 1u)) s[c][e] = 0xFF800000u;
}

template <int NC>
__device__ __forceinline__ float max_score(const uint32_t (&s)[NC][32]) {
  float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int e = 0; e < 32; e += 8) {
      const int k = (c & 1) * 2 + (e >> 4);
      mx[k] = max3(mx[k], __uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1]));
      mx[k] = max3(mx[k], __uint_as_float(s[c][e + 2]), __uint_as_float(s[c][e + 3]));
      mx[k] = max3(mx[k], __uint_as_float(s[c][e + 4]), __uint_as_float(s[c][e + 5]));
      mx[k] = max3(mx[k], __uint_as_float(s[c][e + 6]), __uint_as_float(s[c][e + 7]));
    }
  return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}

// The same over the visible ones (bit e of w[c] belongs to s[c][e]).
template <int NC>
__device__ __forceinline__ float max_visible(const uint32_t (&s)[NC][32], const uint32_t (&w)[NC]) {
  float mx = -INFINITY;
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if ((w[c] >> e) & 1u) mx = fmaxf(mx, __uint_as_float(s[c][e]));
  return mx;
}

// Masks of one tile, for a whole warp (instances without token masks, where
// few tiles hold masked keys).  w: this thread's visible keys; m_part:
// the maximum of its unmasked scores, replaced by the maximum that the running
// max m (log2 units, sl2 per unit of score) has to be compared with.  A warp
// whose rows all see every key of the tile is left alone.  Otherwise the
// hidden scores become -inf, and the maximum over the rest is only taken when
// some row's unmasked maximum exceeds its m by the rescale threshold: below
// that m does not move whatever the mask hides, so any smaller value (-inf)
// has the same effect.  (Selecting and taking the maximum for every tile that
// could hold a masked key took 2.2 times a dense tile.)
template <int NC>
__device__ __forceinline__ void mask_tile(uint32_t (&s)[NC][32], const uint32_t (&w)[NC],
                                          float& m_part, float m, float sl2) {
  uint32_t all = w[0];
#pragma unroll
  for (int c = 1; c < NC; ++c) all &= w[c];
  if (!__any_sync(0xffffffffu, all != ~0u)) return;
  hide_keys(s, w);
  m_part = __any_sync(0xffffffffu, m_part * sl2 > m + kRescaleThreshold) ? max_score(s) : -INFINITY;
}

__device__ __forceinline__ void record_timeout(const AttnParams& p, volatile int* abort_flag) {
  *abort_flag = 1;
  atomicCAS(p.status, kStatusOk, kStatusTimeout);
}

// Instances: kSparse = a bitmap of key tiles is walked: those of the caller's
// tile mask (all without one) that the token masks leave anything of, where
// the launch scanned them; kToken = token masks, of the own chunk or the
// history or both, are applied (only with kSparse); kCluster = every unit is
// split over the CTAs of one cluster, which merge through their shared memory.
// Each extra feature costs the per-tile loop, so a launch takes the leanest
// instance that covers it.
template <int D, bool kSparse, bool kToken, bool kCluster>
__global__ void __launch_bounds__(kThreads, 1) attend_kernel(const __grid_constant__ AttnParams p) {
  using C = AttnCfg<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  __shared__ Bars bars;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_flag;
  __shared__ int last_split;
  __shared__ float range_lost;  // kCluster: not 0 once a key range of the unit has timed out

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  pdl_launch_dependents();

  // Work unit, head-major so the CTAs that share a head's K/V run together.
  // The first n_full units run unsplit (one CTA each, the full waves); the
  // others are split n_split ways, the splits of a unit adjacent.
  // kCluster: one cluster of n_split CTAs per unit (n_full = 0).
  int ns = 1, split = 0, unit = (int)blockIdx.x;  // key ranges of the unit, this CTA's
  if (kCluster || unit >= p.n_full) {
    ns = p.n_split;
    const uint32_t rem = blockIdx.x - (uint32_t)p.n_full, u = rem / (uint32_t)ns;
    split = (int)(rem - u * (uint32_t)ns);
    unit = p.n_full + (int)u;
  }
  const int sunit = unit - p.n_full;     // index among the split units
  // Or, where frame causality makes the pairs of a node uneven, pair-major with
  // the longest walks first, so that the short ones fill the gaps at the end.
  const uint32_t by = (uint32_t)(p.qp_major ? p.H * p.n_nodes : p.n_qp);
  const uint32_t major = (uint32_t)unit / by, minor = (uint32_t)unit - major * by;
  const int qp = p.qp_major ? p.n_qp - 1 - (int)major : (int)minor;
  const uint32_t rest = p.qp_major ? minor : major;
  const int h = (int)(rest / (uint32_t)p.n_nodes);
  const int ni = (int)rest - h * p.n_nodes;
  const AttnNode& nd = p.nodes[ni];
  const int n_all = nd.n_kv * p.nt_slot;  // key tiles of the node
  const int qt0 = 2 * qp;
  const bool has_q1 = qt0 + 1 < p.n_qt;
  // Under frame causality the own chunk's key tiles past the frame of the
  // pair's last query row hold no key that either query tile may see: the
  // node's key tiles [gap_lo, gap_hi) are skipped.
  int gap_lo = n_all, gap_hi = n_all;
  if (nd.frame_causal) {
    const int last_row = min((qt0 + (has_q1 ? 2 : 1)) * kTile, p.T) - 1;
    const int frame_end = (last_row / p.frame_tokens + 1) * p.frame_tokens;
    gap_lo = min((frame_end + kTile - 1) / kTile, p.nt_slot);
    gap_hi = p.nt_slot;
  }
  // the key tile after kt in this CTA's walk (dense instances)
  auto next_kt = [gap_lo, gap_hi](int kt) { return kt + 1 == gap_lo ? gap_hi : kt + 1; };
  // Key tiles of this CTA: a contiguous range of the node's tiles that are
  // not skipped, or under a block-sparse mask a contiguous range of the
  // tiles either query tile may attend (set in the prologue below).
  constexpr bool sparse = kSparse;  // a launch with a block-sparse tile mask
  const int n_eff = n_all - (gap_hi - gap_lo);
  int t_begin = 0, n_tiles = n_eff;
  if (ns > 1) {
    t_begin = split * n_eff / ns;
    n_tiles = (split + 1) * n_eff / ns - t_begin;
  }
  if (t_begin >= gap_lo) t_begin += gap_hi - gap_lo;
  // per query tile, bit i = kernel key tile i (block-sparse instances only)
  __shared__ uint32_t tmask[2][kSparse ? kMaskWords : 1];
  __shared__ int sp_first, sp_count;

  uint8_t* sQ0 = smem + C::kOffQ0;
  uint8_t* sQ1 = smem + C::kOffQ1;
  uint8_t* sK = smem + C::kOffK;
  uint8_t* sV = smem + C::kOffV;
  auto load_q = [&]() {
    mbar_arrive_expect_tx(&bars.q_full, (has_q1 ? 2 : 1) * C::kTileBytes);
#pragma unroll
    for (int b = 0; b < C::kBoxes; ++b) {
      tma_load_4d(sQ0 + b * C::kBoxBytes, &p.tmap_q, &bars.q_full, b * 64, h, qt0 * kTile, nd.q_index);
      if (has_q1)
        tma_load_4d(sQ1 + b * C::kBoxBytes, &p.tmap_q, &bars.q_full, b * 64, h, (qt0 + 1) * kTile,
                    nd.q_index);
    }
  };
  if (threadIdx.x == 0) {
    prefetch_tmap(&p.tmap_q);
    prefetch_tmap(&p.tmap_kv);
    abort_flag = 0;
    if constexpr (kCluster) range_lost = 0.0f;
    mbar_init(&bars.q_full, 1);
    mbar_init(&bars.o_final, 2);  // one commit per MMA issuer
    mbar_init(&bars.drain, 2);
    for (int b = 0; b < C::kStepBars; ++b) {
      mbar_init(&bars.s_full[b], 1);
      mbar_init(&bars.p_full[b], 128 * C::kRowThreads);
    }
    for (int s = 0; s < C::kKStages; ++s) {
      mbar_init(&bars.k_full[s], 1);
      mbar_init(&bars.k_empty[s], C::kOwnTile && has_q1 ? 2 : 1);  // D = 64: one per query tile
    }
    for (int s = 0; s < C::kVStages; ++s) {
      mbar_init(&bars.v_full[s], 1);
      mbar_init(&bars.v_empty[s], C::kOwnTile && has_q1 ? 2 : 1);
    }
    fence_mbar_init();
    if constexpr (!sparse) {
      // Q and the first K tile are on their way while the CTA sets up the
      // rest: they used to follow the set-up, 600 cycles later.
      fence_proxy_async_smem();
      pdl_wait();
      load_q();
      if (n_tiles > 0) {
        const int st = t_begin / p.nt_slot;
        const int row_k = (nd.slot[st] * 2 * p.H + h) * p.Tpad + (t_begin - st * p.nt_slot) * kTile;
        const uint64_t keep = l2_policy_evict_last();
        mbar_arrive_expect_tx(&bars.k_full[0], C::kTileBytes);
#pragma unroll
        for (int b = 0; b < C::kBoxes; ++b)
          tma_load_2d_hint(sK + b * C::kBoxBytes, &p.tmap_kv, &bars.k_full[0], b * 64, row_k, keep);
      }
    }
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base_sh, C::kTmemCols);
    tmem_relinquish();
  }
  pdl_wait();  // everything above is this CTA's own; what follows reads and writes global memory
  if constexpr (sparse) if (warp == 2) {
    // Gather the caller's mask rows of the two query tiles into the kernel's
    // key tile order (slot list without hidden context slots), then take
    // this split's share of the union's set bits.  Without a tile mask every
    // key tile is kept that the token masks leave something of.
    const int words = (n_all + 31) >> 5;  // <= kMaskWords, checked on the host
    const uint32_t* row0 =
        p.tile_mask ? p.tile_mask + ((size_t)nd.q_index * p.n_qt + qt0) * p.mask_words : nullptr;
    const uint32_t* row1 = row0 ? row0 + p.mask_words : nullptr;
    const uint8_t* any0 =
        p.any_tile ? p.any_tile + ((size_t)nd.q_index * p.n_qt + qt0) * p.any_stride : nullptr;
    const uint8_t* any1 = any0 ? any0 + p.any_stride : nullptr;
    int total = 0;
    for (int w = 0; w < words; ++w) {
      const int i = (w << 5) + lane;
      bool b0 = false, b1 = false;
      if (i < n_all && (i < gap_lo || i >= gap_hi)) {
        const int s = i / p.nt_slot;
        const int k = nd.src[s] * p.nt_slot + (i - s * p.nt_slot);
        b0 = row0 ? ((row0[k >> 5] >> (k & 31)) & 1u) != 0u : true;
        if (has_q1) b1 = row1 ? ((row1[k >> 5] >> (k & 31)) & 1u) != 0u : true;
        if (any0) {
          b0 = b0 && any0[k] != 0;
          b1 = b1 && any1[k] != 0;
        }
      }
      const uint32_t m0 = __ballot_sync(0xffffffffu, b0);
      const uint32_t m1 = __ballot_sync(0xffffffffu, b1);
      if (lane == 0) {
        tmask[0][w] = m0;
        tmask[1][w] = m1;
      }
      total += __popc(m0 | m1);
    }
    if (lane == 0) {
      const int lo = (int)((long long)split * total / ns);
      const int hi = (int)((long long)(split + 1) * total / ns);
      int first = n_all, seen = 0;
      for (int w = 0; hi > lo && w < words; ++w) {
        uint32_t u = tmask[0][w] | tmask[1][w];
        const int cnt = __popc(u);
        if (seen + cnt > lo) {
          for (int r = lo - seen; r > 0; --r) u &= u - 1;  // drop the bits before the lo-th
          first = (w << 5) + __ffs(u) - 1;
          break;
        }
        seen += cnt;
      }
      sp_first = first;
      sp_count = hi - lo;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if constexpr (sparse) {
    t_begin = sp_first;
    n_tiles = sp_count;
  }
  const uint32_t tbase = tmem_base_sh;
  const uint64_t tmo = p.timeout_ns;

  int k_issued = 0, v_issued = 0;  // producer: tiles whose K / V copies were started

  if (warp < 4) {
    regs_dec<AttnRegs<D>::kLow>();
    if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      if constexpr (sparse) load_q();
      const uint64_t keep = l2_policy_evict_last();
      TileWalk<kSparse ? kMaskWords : 1> walk;
      if constexpr (sparse) walk.start(tmask, t_begin, n_all);
      int i = sparse ? walk.next() : t_begin;  // key tile of the node
      for (int j = 0; j < n_tiles; ++j, i = sparse ? walk.next() : next_kt(i)) {
        const int ks = j % C::kKStages;
        const int vs = j % C::kVStages;
        const int slot = nd.slot[i / p.nt_slot];
        const int t = i - (i / p.nt_slot) * p.nt_slot;
        const int row_k = ((slot * 2 + 0) * p.H + h) * p.Tpad + t * kTile;
        const int row_v = row_k + p.H * p.Tpad;
        if (sparse || j > 0) {  // a dense walk's first K tile is on its way already
          if (!mbar_wait(&bars.k_empty[ks], ((uint32_t)(j / C::kKStages) & 1u) ^ 1u, &abort_flag,
                         tmo)) {
            record_timeout(p, &abort_flag);
            break;
          }
          mbar_arrive_expect_tx(&bars.k_full[ks], C::kTileBytes);
#pragma unroll
          for (int b = 0; b < C::kBoxes; ++b)
            tma_load_2d_hint(sK + ks * C::kTileBytes + b * C::kBoxBytes, &p.tmap_kv,
                             &bars.k_full[ks], b * 64, row_k, keep);
        }
        k_issued = j + 1;
        if (!mbar_wait(&bars.v_empty[vs], ((uint32_t)(j / C::kVStages) & 1u) ^ 1u, &abort_flag,
                       tmo)) {
          record_timeout(p, &abort_flag);
          break;
        }
        // fault_mode 1 (test hook): withhold the V copy of the second tile,
        // so the MMA issuer's bounded wait on it expires.
        if (!(p.fault_mode == 1 && j == 1)) {
          mbar_arrive_expect_tx(&bars.v_full[vs], C::kTileBytes);
#pragma unroll
          for (int b = 0; b < C::kBoxes; ++b)
            tma_load_2d_hint(sV + vs * C::kTileBytes + b * C::kBoxBytes, &p.tmap_kv,
                             &bars.v_full[vs], b * 64, row_v, keep);
        }
        v_issued = j + 1;
      }
    }
  } else if (warp == 1 || warp == 3) {
    // ------------------------------------------------------------ MMA issuers
    // The whole warp runs the loop (waits are voted warp-wide so every lane
    // takes the same branch); one elected lane issues each MMA and commit.
    {
      constexpr uint32_t idesc_qk = idesc_bf16_f32(128, 128, false);
      constexpr uint32_t idesc_pv = idesc_bf16_f32(128, D, true);
      // Base descriptors are built once; an MMA's operand descriptor is its
      // base plus a compile-time offset (the start-address field holds
      // address >> 4 and every operand lies below 256 KB, so the add never
      // carries out of the field).  Rebuilding descriptors per MMA costs the
      // issuing warp about as long as the MMA itself takes.
      const uint64_t dQ[2] = {sdesc_sw128(smem_u32(sQ0), 16, 1024),
                              sdesc_sw128(smem_u32(sQ1), 16, 1024)};
      const uint64_t dK = sdesc_sw128(smem_u32(sK), 16, 1024);
      const uint64_t dV = sdesc_sw128(smem_u32(sV), C::kBoxBytes, 1024);
      constexpr uint64_t kTileStep = (uint64_t)(C::kTileBytes >> 4);
      // Under a block-sparse mask a query tile may skip a key tile the other
      // query tile attends: its S and PV MMAs are then not issued (the S
      // barrier is still committed, so every barrier completes once per
      // tile), and its first issued PV starts the accumulator.
      auto vis = [&](int b, int kt) {
        return !sparse || ((tmask[b][kt >> 5] >> (kt & 31)) & 1u) != 0u;
      };
      bool pv_started = false;  // this issuer's query tile has a PV in O
      // S_b = Q_b K_i^T into TMEM buffer `buf`, then a commit to S barrier `bar`
      auto issue_s = [&](int b, int buf, int bar, int i, bool v) {
        if (v) {
          const uint64_t kb = dK + (uint64_t)(i % C::kKStages) * kTileStep;
          const uint64_t qb = b == 0 ? dQ[0] : dQ[1];
          const uint32_t dcol = tbase + col_s<D>(buf);
          if constexpr (C::kOwnTile) {
            mma_ss_warp_x4(dcol, qb, kb, 2, idesc_qk);
          } else {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint64_t off = (uint64_t)(((kk >> 2) * C::kBoxBytes + (kk & 3) * 32) >> 4);
              mma_ss_warp(dcol, qb + off, kb + off, idesc_qk, kk > 0 ? 1u : 0u);
            }
          }
        }
        mma_commit_warp(&bars.s_full[bar]);
      };
      // O_b += P_b V_i with P_b read from TMEM over S_b in buffer `buf`
      auto issue_pv = [&](int b, int buf, int i) {
        const uint64_t vb = dV + (uint64_t)(i % C::kVStages) * kTileStep;
        const uint32_t ocol = tbase + col_o<D>(b);
        const uint32_t pcol = tbase + col_s<D>(buf);
        const uint32_t acc0 = (sparse ? pv_started : i > 0) ? 1u : 0u;
        if constexpr (C::kOwnTile)
          mma_ts_warp_x8(ocol, pcol, vb, idesc_pv, acc0);
        else
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk)
          mma_ts_warp(ocol, pcol + kk * 8, vb + (uint64_t)((kk * 2048) >> 4), idesc_pv,
                 kk > 0 ? 1u : acc0);
        if (sparse) pv_started = true;
      };
      auto wait = [&](uint64_t* bar, uint32_t parity) {
        return __all_sync(0xffffffffu, mbar_wait(bar, parity, &abort_flag, tmo));
      };
      auto wait_k = [&](int i) {
        return wait(&bars.k_full[i % C::kKStages], (uint32_t)(i / C::kKStages) & 1u);
      };
      const int bq = warp == 1 ? 0 : 1;  // the query tile this warp issues for (D = 128)
      bool ok = wait(&bars.q_full, 0);
      if constexpr (C::kOwnTile) {
        // Steps n = (key tile i, query tile b), b fastest, in S buffer n % 3:
        // when P_n is there, PV_n is issued and right behind it S_{n+3}, which
        // overwrites the buffer that PV_n reads (the MMAs of one thread
        // execute in issue order).  Two issuers: warp 1 takes the even n (PV
        // of query tile 0, S of query tile 1), warp 3 the odd n (PV of query
        // tile 1, S of query tile 0).  With one query tile warp 1 takes all.
        const int nb = has_q1 ? 2 : 1;
        if (bq < nb) {
          const int qs = nb - 1 - bq;  // the query tile whose S this warp issues
          TileWalk<kSparse ? kMaskWords : 1> walk_s, walk_p;
          if constexpr (sparse) {
            walk_s.start(tmask, t_begin, n_all);
            walk_p.start(tmask, t_begin, n_all);
          }
          int si = 0, skt = 0;  // tile of the next S and its key tile of the node
          auto next_kt_s = [&]() {
            if constexpr (sparse) skt = walk_s.next();
          };
          // ahead: S steps issued before the first PV (of the first three steps)
          const int ahead = nb == 1 ? 3 : 1 + bq;
          for (int k = 0; ok && k < ahead && si < n_tiles; ++k, ++si) {
            next_kt_s();
            ok = wait_k(si);
            if (!ok) break;
            tc_fence_after();
            issue_s(qs, nb == 1 ? k : qs + 2 * k, qs * 3 + k, si, vis(qs, skt));
          }
          int buf = bq;             // S buffer of step n = nb * i + bq
          int bar = 0;              // i % 3 and the phase of that P barrier
          uint32_t par = 0;
          for (int i = 0; ok && i < n_tiles; ++i) {
            const bool more = si < n_tiles;
            int pkt = 0;
            if constexpr (sparse) pkt = walk_p.next();
            if (more) next_kt_s();
            // V_i and the next S's K normally landed long ago: one round trip
            // tests both
            uint64_t* vbar = &bars.v_full[i % C::kVStages];
            uint64_t* kbar = &bars.k_full[more ? si % C::kKStages : 0];
            const uint32_t vpar = (uint32_t)(i / C::kVStages) & 1u;
            const uint32_t kpar = (uint32_t)(si / C::kKStages) & 1u;
            const bool vok = mbar_try_wait(vbar, vpar);
            const bool kok = !more || mbar_try_wait(kbar, kpar);
            if (!__all_sync(0xffffffffu, vok && kok))
              ok = wait(vbar, vpar) && (!more || wait(kbar, kpar));
            if (!ok || !wait(&bars.p_full[bq * 3 + bar], par)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (vis(bq, pkt)) issue_pv(bq, buf, i);
            mma_commit_warp(&bars.v_empty[i % C::kVStages]);
            if (more) {
              issue_s(qs, buf, qs * 3 + si % 3, si, vis(qs, skt));
              ++si;
            }
            buf += nb;
            if (buf >= 3) buf -= 3;
            if (++bar == 3) {
              bar = 0;
              par ^= 1u;
            }
          }
        }
      } else if (bq == 0 || has_q1) {
        TileWalk<kSparse ? kMaskWords : 1> walk;
        if constexpr (sparse) walk.start(tmask, t_begin, n_all);
        int kt = sparse ? walk.next() : t_begin;  // key tile of the node at iteration i
        if (n_tiles > 0) {  // a block-sparse range may be empty: then only o_final is committed
          ok = ok && wait_k(0);
          if (ok) {
            tc_fence_after();
            issue_s(bq, bq, bq, 0, vis(bq, kt));
          }
        }
        for (int i = 0; ok && i < n_tiles; ++i) {
          const uint32_t par = (uint32_t)i & 1u;
          const bool more = i + 1 < n_tiles;
          const int kt_next = !more ? kt : (sparse ? walk.next() : next_kt(kt));
          const bool vis_cur = vis(bq, kt), vis_next = more && vis(bq, kt_next);
          // V_i and K_{i+1} normally land before the softmax hands over P_b,
          // so their waits go first, off the path from P_b to the next MMA.
          if (!wait(&bars.v_full[i % C::kVStages], (uint32_t)(i / C::kVStages) & 1u) ||
              (more && !wait_k(i + 1)) || !wait(&bars.p_full[bq], par)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (vis_cur) issue_pv(bq, bq, i);
          if (more) issue_s(bq, bq, bq, i + 1, vis_next);
          kt = kt_next;
        }
      }
      if (ok) {
        mma_commit_warp(&bars.o_final);
      } else if (lane == 0) {
        record_timeout(p, &abort_flag);
      }
    }
    }
    // ---------------------------------------------------------------- teardown (warpgroup 0)
    __syncwarp();
    if constexpr (kCluster) {  // the two barriers of the merge
      cluster_sync();
      cluster_sync();
    }
    tc_fence_before();
    __syncthreads();
    if (abort_flag) {
      // Some wait expired.  Before the CTA exits, wait (bounded, ignoring
      // the abort flag) for what this CTA still has in flight: the TMA
      // copies the producer started (a stage's barrier cannot run ahead of
      // the last copy started into it) and every MMA the issuers started.
      const int zero = 0;
      if (warp == 0 && lane == 0) {
        mbar_wait(&bars.q_full, 0, &zero, tmo);
        for (int i = (k_issued > C::kKStages ? k_issued - C::kKStages : 0); i < k_issued; ++i)
          mbar_wait(&bars.k_full[i % C::kKStages], (uint32_t)(i / C::kKStages) & 1u, &zero, tmo);
        for (int i = (v_issued > C::kVStages ? v_issued - C::kVStages : 0); i < v_issued; ++i) {
          if (p.fault_mode == 1 && i == 1) continue;  // the copy the test hook withheld
          mbar_wait(&bars.v_full[i % C::kVStages], (uint32_t)(i / C::kVStages) & 1u, &zero, tmo);
        }
      } else if (warp == 1 || warp == 3) {
        mma_commit_warp(&bars.drain);  // the same elected lane that issued the MMAs
        mbar_wait(&bars.drain, 0, &zero, tmo);
      }
    }
    __syncwarp();
    if (warp == 1) {
      tc_fence_after();
      tmem_dealloc(tbase, C::kTmemCols);
    }
  } else {
    regs_inc<AttnRegs<D>::kHigh>();
    // ------------------------------------------------------------ softmax + epilogue
    // D = 128: all eight softmax warps work on one query tile at a time (tile
    // 0, then tile 1, of every key tile).  A warp covers 16 rows, half of its
    // TMEM lane quarter, with two threads per row (16x32bx2 shape): thread t <
    // 16 holds keys 0..63 of its row, thread t + 16 keys 64..127 of the same
    // row.  Both threads of a row keep the same running max (the two halves'
    // maxima are exchanged with one shuffle) and each its part of the sum,
    // so each thread exponentiates 64 keys per tile instead of 128 and the
    // two warps sharing a sub-partition overlap their MUFU and FMA work.
    // D = 64: warps 4-7 take query tile 0, warps 8-11 tile 1, a thread per row
    // with all 128 keys; see the note above the kernel.
    constexpr int NT = C::kTilesPerWarp;           // query tiles this warp works on
    constexpr int NC = C::kChunks;                 // 32-key chunks per thread
    constexpr int DH = D / C::kRowThreads;         // output columns per thread
    const int q4 = warp & 3;                       // TMEM lane quarter this warp may access
    const int hi = warp >> 3;                      // D = 128: which 16 lanes of the quarter
    const int half = C::kOwnTile ? 0 : lane >> 4;  // which 64 keys, which D/2 columns
    // query row inside a tile, and the warp's first TMEM lane
    const int row = C::kOwnTile ? q4 * 32 + lane : q4 * 32 + hi * 16 + (lane & 15);
    const uint32_t lane_off = (uint32_t)(C::kOwnTile ? q4 * 32 : q4 * 32 + hi * 16) << 16;
    const int b_own = hi;                          // D = 64: this warpgroup's query tile
    const int nb = has_q1 ? 2 : 1;
    const float sl2 = p.scale_log2;
    const uint64_t sl2x2 = f2u(sl2, sl2);
    const int frame_causal = nd.frame_causal;
    // 32 output columns of this thread's row in O, from TMEM and back
    auto ld_o = [&](uint32_t col, uint32_t (&o)[32]) {
      if constexpr (C::kOwnTile)
        tmem_ld32(tbase + lane_off + col, o);
      else
        tmem_ld16x2_32<DH>(tbase + lane_off + col, o);
      tmem_wait_ld(o);
    };
    auto st_o = [&](uint32_t col, const uint32_t (&o)[32]) {
      if constexpr (C::kOwnTile)
        tmem_st32(tbase + lane_off + col, o);
      else
        tmem_st16x2_32<DH>(tbase + lane_off + col, o);
    };
    bool o_has[NT];       // O_b holds a PV (some key tile was attended)
    float m[NT];          // running max of scale*log2(e)*logit per query tile
    float l[NT];          // this thread's part of the running sum of 2^(x - m)
    int frame_end[NT];    // first token of the latent frame after this row's (frame-causal mask)
#pragma unroll
    for (int x = 0; x < NT; ++x) {
      const int b = C::kOwnTile ? b_own : x;
      o_has[x] = false;
      m[x] = -INFINITY;
      l[x] = 0.0f;
      frame_end[x] = ((qt0 + b) * kTile + row) / p.frame_tokens * p.frame_tokens + p.frame_tokens;
    }
    // D = 128: the softmax sees S_0 and then S_1 of key tile i complete.
    // S_b,i follows PV_b,i-1 in its issuer's order, so once both are seen every
    // MMA that reads K stage i or V stage i-1 has completed, and one softmax
    // thread hands both stages back to the producer when it sees the last S
    // of the tile (S_1, or S_0 without a second query tile).  The MMA warps
    // then commit only to their S barriers (a commit costs an issuer about
    // as long as an MMA).  D = 64: one thread per query tile hands back K
    // stage i when it sees S_b,i; the issuers' commits hand back the V stages.
    const bool releaser = (C::kOwnTile ? q4 == 0 : warp == 4) && lane == 0;
    bool ok = true;
    TileWalk<kSparse ? kMaskWords : 1> walk;
    if constexpr (sparse) walk.start(tmask, t_begin, n_all);
    int kt = sparse ? walk.next() : t_begin;  // key tile of the node
    // Key state (0 own, then the visible contexts) of a key tile: a division
    // by a reciprocal, exact for the tiles of the masked instances (kt < 2^12,
    // nt_slot <= 2^9).
    const uint32_t inv_nt = p.nt_slot > 1 ? 0xFFFFFFFFu / (uint32_t)p.nt_slot + 1u : 0u;
    auto state_of = [&](int tile) { return inv_nt ? (int)__umulhi((uint32_t)tile, inv_nt) : tile; };
    // Token-mask instance: this thread's bits of its row for a key tile, from
    // the own-chunk mask or from the history mask of the tile's key state (the
    // caller's context index); all ones without such a mask and for rows past
    // T, which are never stored.  Each is fetched a key tile ahead of its use:
    // its L2 latency, on the path from S to P, cost about 0.1 us a tile.  The
    // rows' addresses are worked out once.
    const uint32_t* own_row[NT];
    const uint32_t* hist_row[NT];
#pragma unroll
    for (int x = 0; x < NT; ++x) {
      const int u = (qt0 + (C::kOwnTile ? b_own : x)) * kTile + row;
      const size_t qrow = (size_t)nd.q_index * p.T + u;
      own_row[x] =
          kToken && p.own_mask && u < p.T ? p.own_mask + qrow * p.own_words + half * 2 : nullptr;
      hist_row[x] = kToken && p.hist_mask && u < p.T
                        ? p.hist_mask + qrow * p.hist_states * p.hist_words + half * 2
                        : nullptr;
    }
    auto token_bits = [&](int x, int tile, uint32_t (&ow)[NC]) {
      const int st = state_of(tile);
      const int tt = tile - st * p.nt_slot;
      const uint32_t* r = own_row[x];
      int words = p.own_words;
      if (st != 0) {
        r = hist_row[x] ? hist_row[x] + (nd.src[st] - 1) * p.hist_words : nullptr;
        words = p.hist_words;
      }
      words -= tt * 4 + half * 2;  // of this row from this thread's first on; < NC in the last tile only
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        ow[c] = ~0u;
        if (r) ow[c] = ld_global_u32_if(r + tt * 4 + c, c < words, 0u);
      }
    };
    if constexpr (C::kOwnTile) {
      const int b = b_own;
      int kst = kt / p.nt_slot;                 // its key state: 0 own, then the visible contexts
      int t = kt - kst * p.nt_slot;             // and its place in the state's slot
      // Steps to the next key tile of the walk.  A dense walk visits the tiles
      // of a slot in order (with the frame-causal gap at the end of the own
      // slot), so no division is needed.
      auto advance = [&](int next) {
        if constexpr (sparse) {
          kst = state_of(next);
          t = next - kst * p.nt_slot;
        } else {
          t += next - kt;
          if (t >= p.nt_slot) {  // also from a tile before the gap to the next slot's first
            t = 0;
            ++kst;
          }
        }
        kt = next;
      };
      auto attends = [&](int tile) {
        return !sparse || ((tmask[b][tile >> 5] >> (tile & 31)) & 1u) != 0u;
      };
      auto wait_s = [&](int bar, uint32_t par) {
        return __all_sync(0xffffffffu, mbar_wait(&bars.s_full[b * 3 + bar], par, &abort_flag, tmo)) != 0;
      };
      // One step from its scores s (with the maximum cmax of each 32-key chunk)
      // up to the row's running max: masks, then moves m and rescales O and l
      // where a row needs it.  False: a wait expired.
      // Token masks: w receives the visible keys, for expo.
      auto row_max = [&](int i, uint32_t (&s)[NC][32], const float (&cmax)[NC],
                         const uint32_t (&ow)[NC], uint32_t (&w)[NC]) {
        float m_part = cmax[0];
#pragma unroll
        for (int c = 1; c < NC; ++c) m_part = fmaxf(m_part, cmax[c]);
        const int valid_tile = (t == p.nt_slot - 1) ? p.valid_last : kTile;
        const bool own_fc = frame_causal && kst == 0;
        // The loads also reduce each 32-column chunk to its maximum, so a full
        // tile needs no max tree.  Tiles that can hold masked keys (a slot's
        // ragged last tile, the own chunk under frame causality, token masks)
        // take mask_tile; the test is the same for every thread.
        if (kToken || valid_tile < kTile || own_fc) {
          // own-chunk tile under frame causality: keys up to the end of this
          // row's latent frame are visible (tile 0, frame 0, always is)
          const int valid = own_fc ? min(valid_tile, frame_end[0] - t * kTile) : valid_tile;
#pragma unroll
          for (int c = 0; c < NC; ++c) w[c] = ow[c];
          if (valid_tile < kTile || own_fc)
#pragma unroll
            for (int c = 0; c < NC; ++c) w[c] &= first_bits(valid - c * 32);
          if constexpr (!kToken) mask_tile(s, w, m_part, m[0], sl2);
        }
        float m_new = fmaxf(m[0], m_part * sl2);
        bool move = __any_sync(0xffffffffu, m_new > m[0] + kRescaleThreshold) != 0;
        if constexpr (kToken) {
          if (move) {  // m_part was an upper bound: hidden keys counted
            m_new = fmaxf(m[0], max_visible(s, w) * sl2);
            move = __any_sync(0xffffffffu, m_new > m[0] + kRescaleThreshold) != 0;
          }
        }
        if (move) {
          // 0 when the row's first visible keys arrive (m = -inf); 1 for a row
          // of the warp whose max did not move (also when it is still -inf:
          // -inf - -inf would be NaN)
          const float alpha = m_new > m[0] ? ex2(m[0] - m_new) : 1.0f;
          if (sparse ? o_has[0] : i > 0) {
            // O_b holds the sum over earlier tiles.  S runs ahead of the PVs, so
            // the commit that follows PV of the previous tile and frees its V
            // stage is waited for (that stage's next phase cannot end before
            // this step's PV).
            const bool pv = mbar_wait(&bars.v_empty[(i - 1) % C::kVStages],
                                      (uint32_t)((i - 1) / C::kVStages) & 1u, &abort_flag, tmo);
            if (!__all_sync(0xffffffffu, pv)) return false;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < DH / 32; ++c) {
              uint32_t o[32];
              ld_o(col_o<D>(b) + c * 32, o);
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
              st_o(col_o<D>(b) + c * 32, o);
            }
            tmem_wait_st();
          }
          l[0] *= alpha;
          m[0] = m_new;
        }
        return true;
      };
      // P of a chunk of 32 keys, packed into the first 16 registers of its
      // scores (word e/2 is written after elements e, e+1 are read), and its
      // part of the row sum.  m stays -inf while a row has seen no visible key
      // (possible in a key range that starts past a row's frame under frame
      // causality); its scores are then all -inf and must give P = 0, not NaN.
      auto expo = [&](uint32_t (&sc)[32], uint32_t wc, uint64_t negm, uint64_t (&acc)[4]) {
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          float x0, x1;
          ffma2(x0, x1, __uint_as_float(sc[e]), __uint_as_float(sc[e + 1]), sl2x2, negm);
          if constexpr (kToken) {
            if (!((wc >> e) & 1u)) x0 = -INFINITY;
            if (!((wc >> (e + 1)) & 1u)) x1 = -INFINITY;
          }
          const float p0 = ex2(x0);
          const float p1 = ex2(x1);
          acc[(e >> 1) & 3] = fadd2(acc[(e >> 1) & 3], p0, p1);
          sc[e >> 1] = pack_bf16(p0, p1);
        }
      };
      auto neg_max = [&]() {
        const float m_sub = (m[0] == -INFINITY) ? 0.0f : m[0];
        return f2u(-m_sub, -m_sub);
      };
      auto add_sum = [&](const uint64_t (&acc)[4]) {
        float a0, a1, a2, a3, a4, a5, a6, a7;
        u2f(acc[0], a0, a1);
        u2f(acc[1], a2, a3);
        u2f(acc[2], a4, a5);
        u2f(acc[3], a6, a7);
        l[0] += ((a0 + a1) + (a2 + a3)) + ((a4 + a5) + (a6 + a7));
      };
      const int my_tiles = b < nb ? n_tiles : 0;
      int buf = b, bar = 0;  // S buffer of step n = nb * i + b; i % 3 and that barrier's phase
      uint32_t par = 0;
      uint32_t ow[NC];  // token masks: the bits of key tile kt
#pragma unroll
      for (int c = 0; c < NC; ++c) ow[c] = ~0u;
      if constexpr (kToken)
        if (my_tiles > 0) token_bits(0, kt, ow);
      for (int i = 0; ok && i < my_tiles; ++i) {
        const int kt_next = sparse ? walk.next() : next_kt(kt);
        uint64_t* p_bar = &bars.p_full[b * 3 + bar];
        ok = wait_s(bar, par);
        if (!ok) break;
        if (releaser) mbar_arrive(&bars.k_empty[i % C::kKStages]);
        if (attends(kt)) {  // else no S was computed and no P is due
          tc_fence_after();
          const uint32_t scol = tbase + lane_off + col_s<D>(buf);
          uint32_t s[NC][32];
          float cmax[NC];
#pragma unroll
          for (int c = 0; c < NC; ++c) tmem_ld32_max(scol + c * 32, s[c], cmax[c]);
#pragma unroll
          for (int c = 0; c < NC; ++c) tmem_wait_ld(s[c]);
          tmem_wait_ld_max(cmax);
          uint32_t w[NC];  // token masks: the visible keys
          ok = row_max(i, s, cmax, ow, w);
          if (!ok) break;
          if constexpr (kToken)
            if (i + 1 < my_tiles) token_bits(0, kt_next, ow);
          const uint64_t negm = neg_max();
          uint64_t acc[4] = {0, 0, 0, 0};
          expo(s[0], w[0], negm, acc);
          expo(s[1], w[1], negm, acc);
          tmem_st32_halves(scol, s[0], s[1]);
          expo(s[2], w[2], negm, acc);
          expo(s[3], w[3], negm, acc);
          tmem_st32_halves(scol + 32, s[2], s[3]);
          tmem_wait_st();
          tc_fence_before();
          add_sum(acc);
          o_has[0] = true;
        } else if constexpr (kToken) {
          if (i + 1 < my_tiles) token_bits(0, kt_next, ow);
        }
        mbar_arrive(p_bar);
        advance(kt_next);
        buf += nb;
        if (buf >= 3) buf -= 3;
        if (++bar == 3) {
          bar = 0;
          par ^= 1u;
        }
      }
    } else {
      int kt_next = kt;
      uint32_t ow[2][NC];  // token masks: the bits of key tile kt per query tile
#pragma unroll
      for (int b = 0; b < 2; ++b) {
#pragma unroll
        for (int c = 0; c < NC; ++c) ow[b][c] = ~0u;
        if constexpr (kToken)
          if (n_tiles > 0) token_bits(b, kt, ow[b]);
      }
      for (int i = 0; ok && i < n_tiles; ++i, kt = kt_next) {
        // The next tile of the walk and, under a tile mask, which query tiles
        // attend this one: read from shared memory before the S wait, so their
        // latency is not added to the path from S to P.
        kt_next = sparse ? walk.next() : next_kt(kt);
        const uint32_t attends = sparse ? ((tmask[0][kt >> 5] >> (kt & 31)) & 1u) |
                                              (((tmask[1][kt >> 5] >> (kt & 31)) & 1u) << 1)
                                        : 3u;
        const int t = sparse ? kt - state_of(kt) * p.nt_slot : kt % p.nt_slot;  // key tile inside its slot
        const int valid_tile = (t == p.nt_slot - 1) ? p.valid_last : kTile;
        const bool own_fc = frame_causal && kt < p.nt_slot;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          if (b == 1 && !has_q1) break;
          ok = mbar_wait(&bars.s_full[b], (uint32_t)i & 1u, &abort_flag, tmo);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (releaser && b == nb - 1) {
            mbar_arrive(&bars.k_empty[i % C::kKStages]);
            if (i > 0) mbar_arrive(&bars.v_empty[(i - 1) % C::kVStages]);
          }
          if (sparse && !((attends >> b) & 1u)) {
            // query tile b skips this key tile: no S was computed, no P is due
            mbar_arrive(&bars.p_full[b]);
            if constexpr (kToken)
              if (i + 1 < n_tiles) token_bits(b, kt_next, ow[b]);
            continue;
          }
          tc_fence_after();
          const uint32_t scol = tbase + lane_off + col_s<D>(b);
          const uint32_t ocol = tbase + lane_off + col_o<D>(b);
          // The loads also reduce each 32-column chunk to its maximum, so a
          // full tile needs no max tree.
          uint32_t s[2][32];
          float cmax[2];
          tmem_ld16x2_32_max<64>(scol, s[0], cmax[0]);
          tmem_ld16x2_32_max<64>(scol + 32, s[1], cmax[1]);
          tmem_wait_ld(s[0]);
          tmem_wait_ld(s[1]);
          tmem_wait_ld_max2(cmax);
          float m_part = fmaxf(cmax[0], cmax[1]);
          // Tiles that can hold masked keys (a slot's ragged last tile, the own
          // chunk under frame causality) take mask_tile; the test is the same
          // for every thread.  Under token masks every tile's exponents are
          // masked below instead, with the scores left as they are: a path
          // that changes them and one that does not had their registers copied
          // where the two meet (451 us against 400 with random masks).
          uint32_t wm[2] = {~0u, ~0u};
          if (kToken || valid_tile < kTile || own_fc) {
            // own-chunk tile under frame causality: keys up to the end of this
            // row's latent frame are visible (tile 0, frame 0, always is)
            const int valid = own_fc ? min(valid_tile, frame_end[b] - t * kTile) : valid_tile;
            const int vrel = valid - half * 64;  // visible keys among this thread's 64
            uint32_t w[2] = {ow[b][0], ow[b][1]};
            if (valid_tile < kTile || own_fc) {
              w[0] &= first_bits(vrel);
              w[1] &= first_bits(vrel - 32);
            }
            if constexpr (kToken) {
              wm[0] = w[0];
              wm[1] = w[1];
              if (i + 1 < n_tiles) token_bits(b, kt_next, ow[b]);
            } else {
              mask_tile(s, w, m_part, m[b], sl2);
            }
          }
          float m_tile = fmaxf(m_part, __shfl_xor_sync(0xffffffffu, m_part, 16)) * sl2;
          float m_new = fmaxf(m[b], m_tile);
          bool move = __any_sync(0xffffffffu, m_new > m[b] + kRescaleThreshold) != 0;
          if constexpr (kToken) {
            // m_part is the maximum with the hidden keys, an upper bound: only
            // where that could move m is the one over the visible keys taken
            if (move) {
              m_part = max_visible(s, wm);
              m_tile = fmaxf(m_part, __shfl_xor_sync(0xffffffffu, m_part, 16)) * sl2;
              m_new = fmaxf(m[b], m_tile);
              move = __any_sync(0xffffffffu, m_new > m[b] + kRescaleThreshold) != 0;
            }
          }
          if (move) {
            // 0 when the row's first visible keys arrive (m = -inf); 1 for a row
            // of the warp whose max did not move (also when it is still -inf:
            // -inf - -inf would be NaN)
            const float alpha = m_new > m[b] ? ex2(m[b] - m_new) : 1.0f;
            if (sparse ? o_has[b] : i > 0) {
              // O_b holds the sum over earlier tiles: the commit that completed
              // S_b of this tile came after PV_b of the previous one.
#pragma unroll
              for (int c = 0; c < DH / 32; ++c) {
                uint32_t o[32];
                tmem_ld16x2_32<DH>(ocol + c * 32, o);
                tmem_wait_ld(o);
#pragma unroll
                for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                tmem_st16x2_32<DH>(ocol + c * 32, o);
              }
              tmem_wait_st();
            }
            l[b] *= alpha;
            m[b] = m_new;
          }
          // m stays -inf while a row has seen no visible key (possible in a key
          // range that starts past a row's frame under frame causality); its
          // scores are then all -inf and must give P = 0, not NaN.
          const float m_sub = (m[b] == -INFINITY) ? 0.0f : m[b];
          const uint64_t negm = f2u(-m_sub, -m_sub);
          uint64_t acc[4] = {0, 0, 0, 0};
          // P of 32 keys packs into 16 words, written over the first half of
          // the same registers (word e/2 is written after elements e, e+1 are
          // read); the two halves make one 32-column store over S (keys
          // 0..63 of the row at columns 0..31, keys 64..127 at 32..63).
#pragma unroll
          for (int c = 0; c < 2; ++c) {
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              float x0, x1;
              ffma2(x0, x1, __uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1]), sl2x2, negm);
              if constexpr (kToken) {
                if (!((wm[c] >> e) & 1u)) x0 = -INFINITY;
                if (!((wm[c] >> (e + 1)) & 1u)) x1 = -INFINITY;
              }
              const float p0 = ex2(x0);
              const float p1 = ex2(x1);
              acc[(e >> 1) & 3] = fadd2(acc[(e >> 1) & 3], p0, p1);
              s[c][e >> 1] = pack_bf16(p0, p1);
            }
          }
          tmem_st16x2_32_halves<32>(scol, s[0], s[1]);
          float a0, a1, a2, a3, a4, a5, a6, a7;
          u2f(acc[0], a0, a1);
          u2f(acc[1], a2, a3);
          u2f(acc[2], a4, a5);
          u2f(acc[3], a6, a7);
          l[b] += ((a0 + a1) + (a2 + a3)) + ((a4 + a5) + (a6 + a7));
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(&bars.p_full[b]);
          if (sparse) o_has[b] = true;
        }
      }
    }
    if (ok) {
      ok = mbar_wait(&bars.o_final, 0, &abort_flag, tmo);
      ok = __all_sync(0xffffffffu, ok);
    }
    if (!ok) record_timeout(p, &abort_flag);
    float l_row[NT];  // the row's whole sum: both halves, under the same max
#pragma unroll
    for (int x = 0; x < NT; ++x)
      l_row[x] = C::kOwnTile ? l[x] : l[x] + __shfl_xor_sync(0xffffffffu, l[x], 16);
    if constexpr (kCluster) {
      // Merge over distributed shared memory.  Every CTA owns 1/ns of the
      // output columns (whole groups of 8) for all 256 rows; each pushes its
      // normalised fp32 partial, and every row's m and l, to the owners, into
      // the shared memory that Q, K and V no longer need, and each owner adds
      // up its columns in order of the key ranges.  So the merge is spread
      // over the unit's CTAs (131 KB out and in per CTA at D = 128, whatever
      // ns), needs no workspace, and costs two cluster barriers instead of
      // stores to L2, a fence, an atomic and the last CTA's reads.  A range
      // that timed out sets every CTA's range_lost in place of its rows, and
      // no owner stores the unit: what the range's partial would have been is
      // not in shared memory.
      constexpr int kGroups8 = D / 8;
      const int per = (kGroups8 + ns - 1) / ns;  // column groups per owner
      const uint32_t data = smem_u32(smem);
      const uint32_t ml = data + (uint32_t)(ns * per) * 8192u;  // [ns][m, l][256] fp32
      __syncwarp();
      cluster_sync();  // every CTA's MMAs are complete: its tiles may be overwritten
      if (ok) {
        tc_fence_after();
#pragma unroll
        for (int x = 0; x < NT; ++x) {
          const int b = C::kOwnTile ? b_own : x;
          if (b >= nb) break;
          const int r = b * 128 + row;
          const float inv_l = l_row[x] > 0.0f ? 1.0f / l_row[x] : 0.0f;  // no visible key here
#pragma unroll
          for (int c = 0; c < DH / 32; ++c) {
            uint32_t o[32];
            if (sparse ? o_has[x] : n_tiles > 0) {  // some key tile was attended
              ld_o(col_o<D>(b) + c * 32, o);
            } else {
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = 0u;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const int g8 = (DH * half + c * 32) / 8 + v;
              const int owner = g8 / per;
              const uint32_t dst = mapa_shared(
                  data + (uint32_t)((split * per + g8 - owner * per) * 8192 + r * 16), (uint32_t)owner);
#pragma unroll
              for (int q = 0; q < 2; ++q)
                st_cluster_v4(dst + q * 4096, __uint_as_float(o[v * 8 + q * 4]) * inv_l,
                              __uint_as_float(o[v * 8 + q * 4 + 1]) * inv_l,
                              __uint_as_float(o[v * 8 + q * 4 + 2]) * inv_l,
                              __uint_as_float(o[v * 8 + q * 4 + 3]) * inv_l);
            }
          }
          if (half == 0)
            for (int k = 0; k < ns; ++k) {
              const uint32_t dst = mapa_shared(ml + (uint32_t)(split * 2048 + r * 4), (uint32_t)k);
              st_cluster_f32(dst, m[x]);
              st_cluster_f32(dst + 1024, l_row[x]);
            }
        }
      } else if (lane < ns) {
        st_cluster_f32(mapa_shared(smem_u32(&range_lost), (uint32_t)lane), 1.0f);
      }
      __syncwarp();
      cluster_sync();  // every partial has arrived; nothing is read from another CTA after this
      const int r = threadIdx.x - 128;  // this thread's row of the pair
      const int token = qt0 * kTile + r;
      if (ok && ld_shared_f32(smem_u32(&range_lost)) == 0.0f && token < p.T && r < nb * kTile) {
        float M = -INFINITY;
        for (int k = 0; k < ns; ++k) M = fmaxf(M, ld_shared_f32(ml + (uint32_t)(k * 2048 + r * 4)));
        const float M_sub = (M == -INFINITY) ? 0.0f : M;  // every range empty: O = 0
        float w[kMaxClusterSplit];
        float L = 0.0f;
#pragma unroll
        for (int k = 0; k < kMaxClusterSplit; ++k) {
          w[k] = 0.0f;
          if (k < ns) {
            const uint32_t at = ml + (uint32_t)(k * 2048 + r * 4);
            w[k] = ld_shared_f32(at + 1024) * ex2(ld_shared_f32(at) - M_sub);
            L += w[k];
          }
        }
        const float inv_L = L > 0.0f ? 1.0f / L : 0.0f;
        uint4* orow4 = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.out) +
                                                (((size_t)nd.q_index * p.T + token) * p.H + h) * D);
        for (int g = 0; g < per && split * per + g < kGroups8; ++g) {
          float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int k = 0; k < kMaxClusterSplit; ++k) {
            if (k < ns) {
              const uint32_t at = data + (uint32_t)((k * per + g) * 8192 + r * 16);
              const uint4 y0 = ld_shared_v4(at), y1 = ld_shared_v4(at + 4096);
              const float wk = w[k] * inv_L;
              a[0] += wk * __uint_as_float(y0.x); a[1] += wk * __uint_as_float(y0.y);
              a[2] += wk * __uint_as_float(y0.z); a[3] += wk * __uint_as_float(y0.w);
              a[4] += wk * __uint_as_float(y1.x); a[5] += wk * __uint_as_float(y1.y);
              a[6] += wk * __uint_as_float(y1.z); a[7] += wk * __uint_as_float(y1.w);
            }
          }
          orow4[split * per + g] = make_uint4(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]),
                                              pack_bf16(a[4], a[5]), pack_bf16(a[6], a[7]));
        }
        if (p.lse != nullptr && split == 0)
          p.lse[((size_t)nd.q_index * p.H + h) * p.T + token] = (M + __log2f(L)) * 0.69314718055994531f;
      }
    } else if (ns == 1) {
      // Each thread's row of O goes to the shared memory of its Q tile (no
      // longer needed; the 128-byte swizzle keeps the writes free of bank
      // conflicts), and the warp stores its rows whole: 256 or 128 contiguous
      // bytes a row, 512 a warp instruction.  Stores straight from the threads
      // touched 32 lines an instruction and took 6700 cycles a CTA; TMA tile
      // stores 3700, 2100 of them waiting for the copy to read 64 KB of shared
      // memory before the CTA may leave; these 3250.
      if (ok) {
        tc_fence_after();
#pragma unroll
        for (int x = 0; x < NT; ++x) {
          const int b = C::kOwnTile ? b_own : x;
          if (b >= nb) break;
          const int token = (qt0 + b) * kTile + row;
          const uint32_t srow = smem_u32(b ? sQ1 : sQ0) + (uint32_t)(half * C::kBoxBytes + row * 128);
          const float inv_l = l_row[x] > 0.0f ? 1.0f / l_row[x] : 0.0f;  // no visible key: O = 0
#pragma unroll
          for (int c = 0; c < DH / 32; ++c) {
            uint32_t o[32];
            if (sparse ? o_has[x] : n_tiles > 0) {  // some key tile was attended
              ld_o(col_o<D>(b) + c * 32, o);
            } else {  // no key tile attended in this range (block-sparse): no MMA wrote O
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = 0u;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              uint32_t w[4];
#pragma unroll
              for (int e = 0; e < 4; ++e)
                w[e] = pack_bf16(__uint_as_float(o[v * 8 + 2 * e]) * inv_l,
                                 __uint_as_float(o[v * 8 + 2 * e + 1]) * inv_l);
              st_shared_v4(srow + (uint32_t)(((c * 4 + v) ^ (row & 7)) << 4), w[0], w[1], w[2], w[3]);
            }
          }
          if (p.lse != nullptr && token < p.T && half == 0)
            p.lse[((size_t)nd.q_index * p.H + h) * p.T + token] =
                (m[x] + __log2f(l_row[x])) * 0.69314718055994531f;
        }
        __syncwarp();
        constexpr int kPieces = D / 8;                     // 16-byte pieces of a row
        constexpr int kRows = 32 / C::kRowThreads;         // rows of this warp per query tile
        const int r0 = row - (C::kOwnTile ? lane : lane & 15);
        const int piece = lane % kPieces;
#pragma unroll
        for (int x = 0; x < NT; ++x) {
          const int b = C::kOwnTile ? b_own : x;
          if (b >= nb) break;
          const uint32_t box = smem_u32(b ? sQ1 : sQ0) + (uint32_t)((piece >> 3) * C::kBoxBytes);
          __nv_bfloat16* o0 = static_cast<__nv_bfloat16*>(p.out) +
                              (((size_t)nd.q_index * p.T + (qt0 + b) * kTile) * p.H + h) * D + piece * 8;
#pragma unroll
          for (int k = 0; k < kRows * kPieces / 32; ++k) {
            const int r = r0 + k * (32 / kPieces) + lane / kPieces;
            const uint4 v = ld_shared_v4(box + (uint32_t)(r * 128 + (((piece & 7) ^ (r & 7)) << 4)));
            if ((qt0 + b) * kTile + r < p.T)
              *reinterpret_cast<uint4*>(o0 + (size_t)r * p.H * D) = v;
          }
        }
      }
    } else {
      // Split unit.  Partial layout per (unit, split): O as [D/4][256]
      // float4 (rows of both query tiles), then m[256], then l[256].
      constexpr size_t kItem = (size_t)256 * (D + 2);
      float* part = p.ws + ((size_t)sunit * ns + split) * kItem;
      if (ok) {
        tc_fence_after();
        float4* part4 = reinterpret_cast<float4*>(part);
#pragma unroll
        for (int x = 0; x < NT; ++x) {
          const int b = C::kOwnTile ? b_own : x;
          if (b >= nb) break;
          const int r = b * 128 + row;
          const float inv_l = l_row[x] > 0.0f ? 1.0f / l_row[x] : 0.0f;  // no visible key here
#pragma unroll
          for (int c = 0; c < DH / 32; ++c) {
            uint32_t o[32];
            if (sparse ? o_has[x] : n_tiles > 0) {  // some key tile was attended
              ld_o(col_o<D>(b) + c * 32, o);
            } else {  // no key tile attended in this range (block-sparse): no MMA wrote O
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = 0u;
            }
#pragma unroll
            for (int v = 0; v < 8; ++v)
              part4[(DH * half / 4 + c * 8 + v) * 256 + r] =
                  make_float4(__uint_as_float(o[v * 4 + 0]) * inv_l, __uint_as_float(o[v * 4 + 1]) * inv_l,
                              __uint_as_float(o[v * 4 + 2]) * inv_l, __uint_as_float(o[v * 4 + 3]) * inv_l);
          }
          if (half == 0) {
            part[D * 256 + r] = m[x];
            part[D * 256 + 256 + r] = l_row[x];
          }
        }
      }
      __threadfence();
      // Every softmax thread of the CTA passes both barriers, whatever its
      // wait results were, so none can be left waiting here.
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (threadIdx.x == 128) {
        int last = 0;
        if (!abort_flag) last = atomicAdd(&p.ws_count[sunit], 1) == ns - 1;
        last_split = last;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (last_split) {
        __threadfence();
        const float* base = p.ws + (size_t)sunit * ns * kItem;
#pragma unroll
        for (int x = 0; x < NT; ++x) {
          const int b = C::kOwnTile ? b_own : x;
          if (b >= nb) break;
          const int r = b * 128 + row;
          const int token = (qt0 + b) * kTile + row;
          if (token >= p.T) continue;
          float mk[kMaxSplit], wk[kMaxSplit];
          float M = -INFINITY;
#pragma unroll
          for (int k = 0; k < kMaxSplit; ++k) {
            mk[k] = k < ns ? __ldcg(base + k * kItem + D * 256 + r) : -INFINITY;
            M = fmaxf(M, mk[k]);
          }
          const float M_sub = (M == -INFINITY) ? 0.0f : M;  // every range empty: O = 0
          float L = 0.0f;
#pragma unroll
          for (int k = 0; k < kMaxSplit; ++k) {
            wk[k] = k < ns
                        ? __ldcg(base + k * kItem + D * 256 + 256 + r) * ex2(mk[k] - M_sub)
                        : 0.0f;
            L += wk[k];
          }
          const float inv_L = L > 0.0f ? 1.0f / L : 0.0f;
#pragma unroll
          for (int k = 0; k < kMaxSplit; ++k) wk[k] *= inv_L;
          uint4* orow4 = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.out) +
                                                  (((size_t)nd.q_index * p.T + token) * p.H + h) * D);
          // Loads of absent splits are predicated off rather than broken out
          // of, so every load of an iteration is in flight at once (a loop
          // that waited for each L2 round trip in turn took ~9 us per CTA).
#pragma unroll 2
          for (int c8 = half * (DH / 8); c8 < (half + 1) * (DH / 8); ++c8) {
            float4 x[kMaxSplit], y[kMaxSplit];
#pragma unroll
            for (int k = 0; k < kMaxSplit; ++k) {
              const float4* b4 = reinterpret_cast<const float4*>(base + k * kItem);
              x[k] = k < ns ? __ldcg(b4 + (c8 * 2 + 0) * 256 + r) : make_float4(0.f, 0.f, 0.f, 0.f);
              y[k] = k < ns ? __ldcg(b4 + (c8 * 2 + 1) * 256 + r) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < kMaxSplit; ++k) {
              a[0] += wk[k] * x[k].x; a[1] += wk[k] * x[k].y; a[2] += wk[k] * x[k].z; a[3] += wk[k] * x[k].w;
              a[4] += wk[k] * y[k].x; a[5] += wk[k] * y[k].y; a[6] += wk[k] * y[k].z; a[7] += wk[k] * y[k].w;
            }
            uint4 w;
            w.x = pack_bf16(a[0], a[1]);
            w.y = pack_bf16(a[2], a[3]);
            w.z = pack_bf16(a[4], a[5]);
            w.w = pack_bf16(a[6], a[7]);
            orow4[c8] = w;
          }
          if (p.lse != nullptr && half == 0)
            p.lse[((size_t)nd.q_index * p.H + h) * p.T + token] = (M + __log2f(L)) * 0.69314718055994531f;
        }
        if (threadIdx.x == 128) p.ws_count[sunit] = 0;  // ready for the next launch
      }
    }
    // ---------------------------------------------------------------- teardown (softmax)
    __syncwarp();
    tc_fence_before();
    __syncthreads();
  }
}

}  // namespace

// The kernel's instances are compiled in three units (attend_dense.cu,
// attend_cluster.cu, attend_masked.cu), because in one the speed of the dense
// instance was seen to change with the code of the others (a 4680-token layer
// between 367 and 381 us for the same source of its own).  Why is not known:
// after a change to this file, time the dense launches too, whichever instance
// it was for.
using AttendKernel = void (*)(const AttnParams);

// Without splits inside clusters: dense; block-sparse, and with token masks.
AttendKernel attend_dense_kernel(int head_dim);
AttendKernel attend_masked_kernel(int head_dim, bool token);
// Each unit split over a cluster.
AttendKernel attend_cluster_kernel(int head_dim, bool masked, bool token);

}  // namespace sva
