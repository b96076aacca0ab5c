// Fused 3D-RoPE + KV-cache scatter.
//
// Writing a node's keys and values into the (chunk, level)-indexed cache is
// what makes its features available to later nodes and, under progressive
// history, to the other nodes of the same pipeline round (Section 3.3).  The
// rotary embedding is this library's reading of the positional encoding (the
// paper names none): 3D RoPE over (t, h, w) at absolute positions, pairs of
// adjacent head-dimension elements, rotated in fp32 with cos/sin tables that
// the host computed in fp64 and rounded once to fp32.
//
// Bandwidth-bound: each warp moves one token's K, V (and Q) rows for all heads
// as 16-byte vectors, so the position and table work is shared by the heads
// and the three tensors.  Reads are contiguous per token; every store covers
// whole 256-byte (or 128-byte) cache rows per half-warp.
//
// These kernels wait for the ones before them but do not let the next one in
// before their blocks leave: several blocks fit an SM, and the next launch's,
// taking each place as it came free, were spread so unevenly that writes back
// to back lost up to 25% (2340 tokens of 16 x 128 with Q, graph replays: 7.5 us
// without programmatic launches, 8.9 with an early trigger, 7.0 so).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace sva {
namespace {

__device__ __forceinline__ uint4 ld_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

__device__ __forceinline__ uint32_t rotate_pair_f(float x, float y, float c, float s) {
  const float rx = __fmaf_rn(x, c, -(y * s));
  const float ry = __fmaf_rn(x, s, y * c);
  __nv_bfloat162 r = __floats2bfloat162_rn(rx, ry);  // .x (rx) in the low half
  return *reinterpret_cast<uint32_t*>(&r);
}

// bf16 pair (element 2k in the low half) times g0, g1, then rotated
__device__ __forceinline__ uint32_t norm_rotate_pair(uint32_t xy, float g0, float g1, float c,
                                                     float s) {
  return rotate_pair_f(__uint_as_float(xy << 16) * g0, __uint_as_float(xy & 0xFFFF0000u) * g1, c,
                       s);
}

__device__ __forceinline__ float sumsq8(uint4 v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  float a = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float x = __uint_as_float(w[k] << 16), y = __uint_as_float(w[k] & 0xFFFF0000u);
    a = __fmaf_rn(x, x, a);
    a = __fmaf_rn(y, y, a);
  }
  return a;
}

__device__ __forceinline__ uint32_t rotate_pair(uint32_t xy, float c, float s) {
  const float x = __uint_as_float(xy << 16);
  const float y = __uint_as_float(xy & 0xFFFF0000u);
  const float rx = __fmaf_rn(x, c, -(y * s));
  const float ry = __fmaf_rn(x, s, y * c);
  __nv_bfloat162 r = __floats2bfloat162_rn(rx, ry);  // .x (rx) in the low half
  return *reinterpret_cast<uint32_t*>(&r);
}

// The gammas of a vector of eight.  They come by ordinary loads, which the
// compiler keeps behind the stores in front of them, so both kernels fetch a
// vector's gammas ahead of the stores of the vector before it.  (Fetched at
// their use the write with Q took 3 to 10% longer at every size; all fetched
// ahead of the first store they spill, up to 40% longer.)
struct Gamma8 {
  float4 lo, hi;
};
__device__ __forceinline__ Gamma8 gamma_at(const float* gamma, int v) {
  return {ptx::ld_global_f4(gamma + (size_t)v * 8), ptx::ld_global_f4(gamma + (size_t)v * 8 + 4)};
}

// x * gamma * r of one vector, rotated
__device__ __forceinline__ uint4 norm_rotate(uint4 x, const Gamma8& g, float r,
                                             const float2 (&cs)[4]) {
  return make_uint4(norm_rotate_pair(x.x, g.lo.x * r, g.lo.y * r, cs[0].x, cs[0].y),
                    norm_rotate_pair(x.y, g.lo.z * r, g.lo.w * r, cs[1].x, cs[1].y),
                    norm_rotate_pair(x.z, g.hi.x * r, g.hi.y * r, cs[2].x, cs[2].y),
                    norm_rotate_pair(x.w, g.hi.z * r, g.hi.w * r, cs[3].x, cs[3].y));
}

// One warp per (node, token).  A token's H*d values are contiguous in the
// token-major inputs, so the warp walks them as 16-byte vectors; lane l always
// holds vector l mod (d/8) of a head row, i.e. the same four pairs for every
// head, so its cos/sin come from the tables once per token.
// kWave holds the kernel to 64 registers (loads in batches of two), so four
// 256-thread blocks fit an SM and a launch of one 4680-token node (585
// blocks) runs in a single wave: such a launch is bound by memory latency,
// and occupancy is what hides it.  Larger launches loop over their tokens
// and do better with batches of four at two blocks per SM.
// kNorm: the RMSNorm of K (and Q) in front, for the launches that
// launch_rope_kv gives to this kernel rather than to rope_norm_kernel.
template <bool kNorm, bool kWave>
__global__ void __launch_bounds__(256, kWave ? 4 : 2) rope_kv_kernel(const __grid_constant__ RopeParams p) {
  const int lane = threadIdx.x & 31;
  const int vpr = p.d >> 3;                        // 16-byte vectors per (token, head) row
  const int vshift = (vpr == 16) ? 4 : 3;
  const int c8 = lane & (vpr - 1);
  const int per_tok = p.H * vpr;                   // vectors per token
  const int HpWp = p.Hp * p.Wp;
  const size_t kv_stride = (size_t)p.H * p.Tpad * p.d;  // elements between K and V of a slot
  const __nv_bfloat16* kin = static_cast<const __nv_bfloat16*>(p.k_new);
  const __nv_bfloat16* vin = static_cast<const __nv_bfloat16*>(p.v_new);
  __nv_bfloat16* qio = static_cast<__nv_bfloat16*>(p.q);
  __nv_bfloat16* cache = static_cast<__nv_bfloat16*>(p.cache);
  const int warps_per_block = blockDim.x >> 5;
  const int n_tok = p.n_nodes * p.T;
  ptx::pdl_wait();

  for (int tok = blockIdx.x * warps_per_block + (threadIdx.x >> 5); tok < n_tok;
       tok += gridDim.x * warps_per_block) {
    const int node = tok / p.T;
    const int u = tok - node * p.T;
    const int f = u / HpWp;
    const int hw = u - f * HpWp;
    const int hh = hw / p.Wp;
    const int ww = hw - hh * p.Wp;
    const RopeNode nd = p.nodes[node];
    const int tpos = nd.t_base + f;
    float2 cs[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int pi = c8 * 4 + k;  // pair index within the head dimension
      if (pi < p.P0)
        cs[k] = __ldg(p.tab_t + (size_t)tpos * p.P0 + pi);
      else if (pi < p.P0 + p.P1)
        cs[k] = __ldg(p.tab_h + (size_t)hh * p.P1 + (pi - p.P0));
      else
        cs[k] = __ldg(p.tab_w + (size_t)ww * p.P2 + (pi - p.P0 - p.P1));
    }
    const size_t in_tok = (size_t)tok * per_tok * 8;
    const size_t out_slot = ((size_t)nd.slot * 2 * p.H) * p.Tpad;  // row of (slot, K, head 0)
    // RMSNorm scale of the token's K and Q vectors: a pass over the rows and a
    // warp reduction; the pass below reads them again from L1 or L2.
    float rk = 1.0f, rq = 1.0f;
    if constexpr (kNorm) {
      float sk = 0.0f, sq = 0.0f;
      for (int v = lane; v < per_tok; v += 32) {
        const size_t off = in_tok + (size_t)v * 8;
        sk += sumsq8(*reinterpret_cast<const uint4*>(kin + off));
        if (qio) sq += sumsq8(*reinterpret_cast<const uint4*>(qio + off));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        sk += __shfl_xor_sync(0xffffffffu, sk, o);
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
      }
      const float inv_n = 1.0f / (float)(per_tok * 8);
      rk = __frsqrt_rn(__fmaf_rn(sk, inv_n, p.norm_eps));
      rq = __frsqrt_rn(__fmaf_rn(sq, inv_n, p.norm_eps));
    }
    // Batches of kBatch vectors per lane: every load of a batch is issued
    // before any of its stores (q is rotated in place, so without the split
    // the compiler keeps each iteration's loads behind the previous stores).
    // The single-wave instance runs four blocks per SM, so half the batch
    // keeps as many bytes in flight per SM as the others' two blocks.
    constexpr int kBatch = kWave ? 2 : 4;
    for (int v0 = lane; v0 < per_tok; v0 += 32 * kBatch) {
      uint4 kv[kBatch], vv[kBatch], qv[kBatch];
      Gamma8 next{};  // the gammas of the next vector to be stored
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int v = v0 + 32 * j;
        if (v < per_tok) {
          const size_t in_off = in_tok + (size_t)v * 8;
          kv[j] = ld_stream(kin + in_off);
          vv[j] = ld_stream(vin + in_off);
          qv[j] = qio ? *reinterpret_cast<const uint4*>(qio + in_off) : make_uint4(0, 0, 0, 0);
        }
      }
      if constexpr (kNorm) next = gamma_at(p.gamma_k, v0);
      auto turn = [&](uint4 x, const Gamma8& g, float r) {
        if constexpr (kNorm) return norm_rotate(x, g, r, cs);
        return make_uint4(rotate_pair(x.x, cs[0].x, cs[0].y), rotate_pair(x.y, cs[1].x, cs[1].y),
                          rotate_pair(x.z, cs[2].x, cs[2].y), rotate_pair(x.w, cs[3].x, cs[3].y));
      };
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int v = v0 + 32 * j;
        if (v >= per_tok) break;
        const int h = v >> vshift;
        const size_t in_off = in_tok + (size_t)v * 8;
        __nv_bfloat16* kdst = cache + ((out_slot + (size_t)h * p.Tpad + u) * p.d + c8 * 8);
        const bool more = j + 1 < kBatch && v + 32 < per_tok;
        Gamma8 g = next;  // of this vector's K, then of its Q
        if constexpr (kNorm) {
          if (qio)
            next = gamma_at(p.gamma_q, v);
          else if (more)
            next = gamma_at(p.gamma_k, v + 32);
        }
        *reinterpret_cast<uint4*>(kdst) = turn(kv[j], g, rk);
        *reinterpret_cast<uint4*>(kdst + kv_stride) = vv[j];
        if (qio) {
          g = next;
          if (kNorm && more) next = gamma_at(p.gamma_k, v + 32);
          *reinterpret_cast<uint4*>(qio + in_off) = turn(qv[j], g, rq);
        }
      }
    }
  }
}

// The same with an RMSNorm of the token's K (and Q) vector of H*d elements in
// front of the rotation.  kWarps warps share a token and keep its K and Q in
// registers (at most kVec 16-byte vectors a lane and tensor) from the sum of
// squares to the rotation, so every input is read once; V is stored once the
// sums are reduced (shuffles, then shared memory across the token's warps).
// One block of eight warps takes 8 / kWarps tokens, all their loads in flight
// at once; two or three blocks an SM (registers) is what its bandwidth needs:
// one block gave 4.6 TB/s where two give 6.3, and fewer registers spill.
// Against reading the rows twice with one warp a token (all with CUDA graphs,
// three sets of buffers): 4680 tokens x 40 x 128, K and V (192 MB) 37.9 -> 35.0
// us; 4 x 4680 tokens x 12 x 128 with Q (345 MB) 68.7 -> 58.7 us, x 40 x 128
// (1150 MB) 204 -> 183 us; one node of 12 x 128 with Q 19.5 -> 19.4 us (a
// device copy of its 43 MB takes 20.5 us in the same loop).
template <int kWarps, int kVec, bool kQ>
__global__ void __launch_bounds__(256, kVec <= 3 || (kVec <= 5 && !kQ) ? 3 : (kVec <= 5 || !kQ ? 2 : 1))
    rope_norm_kernel(const __grid_constant__ RopeParams p) {
  __shared__ float part[8][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int vpr = p.d >> 3;                        // 16-byte vectors per (token, head) row
  const int vshift = (vpr == 16) ? 4 : 3;
  const int c8 = lane & (vpr - 1);
  const int per_tok = p.H * vpr;                   // vectors per token
  const int tok = blockIdx.x * (8 / kWarps) + warp / kWarps;
  const bool live = tok < p.n_nodes * p.T;         // the last block may have tokens to spare
  const __nv_bfloat16* kin = static_cast<const __nv_bfloat16*>(p.k_new);
  const __nv_bfloat16* vin = static_cast<const __nv_bfloat16*>(p.v_new);
  __nv_bfloat16* qio = static_cast<__nv_bfloat16*>(p.q);
  __nv_bfloat16* cache = static_cast<__nv_bfloat16*>(p.cache);
  const size_t kv_stride = (size_t)p.H * p.Tpad * p.d;  // elements between K and V of a slot
  const int v0 = (warp % kWarps) * 32 + lane;
  const size_t in_tok = (size_t)tok * per_tok * 8;
  ptx::pdl_wait();
  uint4 kv[kVec], qv[kQ ? kVec : 1], vv[kVec];
#pragma unroll
  for (int j = 0; j < kVec; ++j) {
    const int v = v0 + j * 32 * kWarps;
    const bool in = live && v < per_tok;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    kv[j] = in ? ld_stream(kin + in_tok + (size_t)v * 8) : zero;
    if constexpr (kQ) qv[j] = in ? *reinterpret_cast<const uint4*>(qio + in_tok + (size_t)v * 8) : zero;
    vv[j] = in ? ld_stream(vin + in_tok + (size_t)v * 8) : zero;
  }
  const int HpWp = p.Hp * p.Wp;
  const int node = live ? tok / p.T : 0;
  const int u = live ? tok - node * p.T : 0;
  const int f = u / HpWp;
  const int hw = u - f * HpWp;
  const int hh = hw / p.Wp;
  const int ww = hw - hh * p.Wp;
  const RopeNode nd = p.nodes[node];
  const int tpos = nd.t_base + f;
  float2 cs[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int pi = c8 * 4 + k;  // pair index within the head dimension
    if (pi < p.P0)
      cs[k] = __ldg(p.tab_t + (size_t)tpos * p.P0 + pi);
    else if (pi < p.P0 + p.P1)
      cs[k] = __ldg(p.tab_h + (size_t)hh * p.P1 + (pi - p.P0));
    else
      cs[k] = __ldg(p.tab_w + (size_t)ww * p.P2 + (pi - p.P0 - p.P1));
  }
  const size_t out_slot = ((size_t)nd.slot * 2 * p.H) * p.Tpad;  // row of (slot, K, head 0)
  auto cache_at = [&](int v) {
    return cache + ((out_slot + (size_t)(v >> vshift) * p.Tpad + u) * p.d + c8 * 8);
  };
  float sk = 0.0f, sq = 0.0f;
#pragma unroll
  for (int j = 0; j < kVec; ++j) {
    sk += sumsq8(kv[j]);
    if constexpr (kQ) sq += sumsq8(qv[j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sk += __shfl_xor_sync(0xffffffffu, sk, o);
    sq += __shfl_xor_sync(0xffffffffu, sq, o);
  }
  if constexpr (kWarps > 1) {
    if (lane == 0) {
      part[warp][0] = sk;
      part[warp][1] = sq;
    }
    __syncthreads();
    sk = 0.0f;
    sq = 0.0f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      sk += part[warp / kWarps * kWarps + w][0];
      sq += part[warp / kWarps * kWarps + w][1];
    }
  }
  if (!live) return;
#pragma unroll
  for (int j = 0; j < kVec; ++j) {
    const int v = v0 + j * 32 * kWarps;
    if (v < per_tok) *reinterpret_cast<uint4*>(cache_at(v) + kv_stride) = vv[j];
  }
  Gamma8 next{};  // the gammas of the next vector to be stored
  if (v0 < per_tok) next = gamma_at(p.gamma_k, v0);
  const float inv_n = 1.0f / (float)(per_tok * 8);
  const float rk = __frsqrt_rn(__fmaf_rn(sk, inv_n, p.norm_eps));
  const float rq = __frsqrt_rn(__fmaf_rn(sq, inv_n, p.norm_eps));
#pragma unroll
  for (int j = 0; j < kVec; ++j) {
    const int v = v0 + j * 32 * kWarps;
    if (v < per_tok) {
      const bool more = j + 1 < kVec && v + 32 * kWarps < per_tok;
      Gamma8 g = next;  // of this vector's K, then of its Q
      if constexpr (kQ) next = gamma_at(p.gamma_q, v);
      const uint4 k = norm_rotate(kv[j], g, rk, cs);
      if (!kQ && more) next = gamma_at(p.gamma_k, v + 32 * kWarps);
      *reinterpret_cast<uint4*>(cache_at(v)) = k;
      if constexpr (kQ) {
        g = next;
        if (more) next = gamma_at(p.gamma_k, v + 32 * kWarps);
        *reinterpret_cast<uint4*>(qio + in_tok + (size_t)v * 8) = norm_rotate(qv[j], g, rq, cs);
      }
    }
  }
}

template <int kWarps, int kVec>
cudaError_t launch_norm(const RopeParams& p, cudaStream_t s) {
  const long long tokens = (long long)p.n_nodes * p.T;
  constexpr int per_block = 8 / kWarps;
  LaunchConfig l(dim3((unsigned)((tokens + per_block - 1) / per_block)), 256, 0, s);
  return p.q != nullptr ? cudaLaunchKernelEx(&l.cfg, rope_norm_kernel<kWarps, kVec, true>, p)
                        : cudaLaunchKernelEx(&l.cfg, rope_norm_kernel<kWarps, kVec, false>, p);
}

}  // namespace

cudaError_t launch_rope_kv(const RopeParams& p, int num_sms, cudaStream_t s) {
  const long long tokens = (long long)p.n_nodes * p.T;
  const long long sms = num_sms;
  const int per_tok = p.H * (p.d >> 3);  // 16-byte vectors, at most 2048
  LaunchConfig l(dim3((unsigned)p.grid_blocks), 256, 0, s);
  const bool wave = tokens <= 32 * sms;  // one warp a token, four blocks of eight warps per SM
  if (p.gamma_k == nullptr)
    return wave ? cudaLaunchKernelEx(&l.cfg, rope_kv_kernel<false, true>, p)
                : cudaLaunchKernelEx(&l.cfg, rope_kv_kernel<false, false>, p);
  const bool q = p.q != nullptr;
  // The kernel that reads its rows twice with one warp a token is the faster
  // one where the tokens fill most of a wave of it and rope_norm_kernel, with
  // two to eight warps a token, needs the better part of two.
  // At two blocks per SM (16 tokens): 2340 tokens of 16 x 128, K and V, 7.0 us
  // against 8.6, of 12 x 128 with Q 7.8 against 9.0.  Below 8 or 12 tokens per
  // SM the instances of two warps a token need one wave; past 448 vectors with
  // Q, 768 without, the second read no longer finds the rows in L1.
  // At four (32 tokens): 4680 tokens of 18 x 128, K and V, 13.7 us against 16.6,
  // with Q 20.8 against 24.6.  At 24 tokens per SM the others fill their last
  // wave (3120 tokens of 24 x 128, 14.4 against 12.9); narrower rows are no
  // slower there on two warps a token, and with Q the rows that fill all lanes
  // of <4, 3> are not either (24 x 128, three sets of buffers, 35.9 against
  // 34.2).
  if (tokens > (q && per_tok > 192 && per_tok <= 256 ? 8 : 12) * sms && tokens <= 16 * sms &&
      per_tok > 128 && per_tok <= (q ? 448 : 768))
    return cudaLaunchKernelEx(&l.cfg, rope_kv_kernel<true, false>, p);
  if (tokens > 24 * sms && wave && per_tok > (q ? 192 : 256) && per_tok <= 448 &&
      !(q && per_tok > 320 && per_tok <= 384))
    return cudaLaunchKernelEx(&l.cfg, rope_kv_kernel<true, true>, p);
  // Few vectors a lane where that costs no bandwidth (a small launch is as
  // long as one token takes: 320 tokens of 12 x 128, 5.4 us at six vectors,
  // 4.0 at three), more where three would leave warps short of loads (40 x
  // 128: 38 us at three, 35 at five; 16 x 64: 13.5 at three, 12.6 at four).
  // From 129 to 768 vectors each step keeps two thirds of its lanes busy or
  // more; in a wider one lanes idle through every load (18720 tokens of 13 x
  // 128 with Q: 80 us on <4, 3>, 69 on <2, 4>; of 41 x 128 251 on <8, 5>, 206
  // on <8, 3>).
  if (per_tok <= 64) return launch_norm<1, 2>(p, s);
  if (per_tok <= 128) return launch_norm<1, 4>(p, s);
  if (per_tok <= 192) return launch_norm<2, 3>(p, s);
  // within one wave of <4, 3>: 600 tokens of 16 x 128, 3.6 us, 4.0 on <2, 4>
  if (per_tok <= 256 && tokens > 6 * sms) return launch_norm<2, 4>(p, s);
  if (per_tok <= 384) return launch_norm<4, 3>(p, s);
  if (per_tok <= 512) return launch_norm<4, 4>(p, s);
  if (per_tok <= 640) return launch_norm<4, 5>(p, s);
  // within two waves of <8, 5>: 600 tokens of 48 x 128 with Q, 9.0 us, 11.1 on <8, 3>
  if (per_tok <= 768 && tokens > 4 * sms) return launch_norm<8, 3>(p, s);
  if (per_tok <= 1280) return launch_norm<8, 5>(p, s);
  return launch_norm<8, 8>(p, s);
}

}  // namespace sva
