// Which key tiles the token masks of a launch leave anything of.
//
// The attention kernel reads token masks a tile at a time, after S is already
// computed; without a block-sparse tile mask it therefore walks every key
// tile, also those whose bits are all clear.  Masks used in earnest (local
// windows, selected history tokens) clear most of a query tile's key tiles, so
// a launch with token masks first reduces them to one byte per (node, query
// tile, key tile): 1 if any of the tile's 128 x 128 bits is set.  The bytes
// then act as a tile mask (on top of the caller's, if any).
//
// Bound by the read of the masks: one block per (node, query tile, key state),
// two rows per warp at a time, 32 words (8 key tiles) a load, up to sixteen
// loads in flight.  A warp whose rows so far have set a bit in every tile
// stops reading, so dense random masks cost a few rows per block.  Times (one
// launch under ncu): one 4680-token node, 3 history states, bits within 6 patch
// rows and columns (11 MB of masks) 7 us, random bits of the same size 4 us;
// 8220 tokens, one history state, bits within 12 rows and columns (17 MB) 9 us.
// The first two are followed by an attention launch of 259 us over the 58% of
// key tiles that keep a bit for their query-tile pair, and of 388 us over all.
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace sva {
namespace {

constexpr int kWarps = 16;
constexpr int kGroup = 8;  // 32-word loads per row and pass: 64 key tiles

__global__ void __launch_bounds__(kWarps * 32) mask_scan_kernel(const __grid_constant__ ScanParams p) {
  __shared__ uint32_t seen[kWarps][kGroup * 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int state = blockIdx.x, qt = blockIdx.y, node = blockIdx.z;
  const int nt = (p.T + kTile - 1) / kTile;
  const uint32_t* mask = state == 0 ? p.own_mask : p.hist_mask;
  uint8_t* out = p.any + ((size_t)node * p.n_qt + qt) * p.row_bytes + (size_t)state * nt;
  ptx::pdl_launch_dependents();
  ptx::pdl_wait();
  if (state > p.n_ctx[node]) return;
  if (mask == nullptr) {
    for (int t = threadIdx.x; t < nt; t += kWarps * 32) out[t] = 1;
    return;
  }
  const int words = (p.T + 31) / 32;  // of a row: rows may be longer, the rest has no meaning
  const int u_end = min((qt + 1) * kTile, p.T);
  for (int base = 0; base < words; base += kGroup * 32) {
    uint32_t acc[kGroup];
#pragma unroll
    for (int j = 0; j < kGroup; ++j) acc[j] = 0;
    for (int u = qt * kTile + warp; u < u_end; u += 2 * kWarps) {
      const size_t q = (size_t)node * p.T + u;
      const size_t step = state == 0 ? (size_t)p.own_words : (size_t)p.hist_states * p.hist_words;
      const uint32_t* row = mask + q * step + (state == 0 ? 0 : (size_t)(state - 1) * p.hist_words);
      const uint32_t* row2 = u + kWarps < u_end ? row + kWarps * step : row;
      uint32_t v[kGroup], v2[kGroup];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const int w = base + j * 32 + lane;
        v[j] = ptx::ld_global_u32_if(row + w, w < words, 0u);
        v2[j] = ptx::ld_global_u32_if(row2 + w, w < words, 0u);
      }
      // every tile (four words, four neighbouring lanes) has a bit by now, or
      // lies past the row's end?  The words that the last tile lacks must not
      // stand in for the ones it has.
      bool all = true;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        acc[j] |= v[j] | v2[j];
        const bool past = base + j * 32 + (lane & ~3) >= words;
        const uint32_t has = __ballot_sync(0xffffffffu, past || acc[j] != 0u);
        const uint32_t pair = has | (has >> 1);
        all = all && ((pair | (pair >> 2)) & 0x11111111u) == 0x11111111u;
      }
      if (all) break;
    }
#pragma unroll
    for (int j = 0; j < kGroup; ++j) seen[warp][j * 32 + lane] = acc[j];
    __syncthreads();
    // one tile per thread: 4 words of every warp
    const int t = base / 4 + threadIdx.x;
    if (threadIdx.x < kGroup * 8 && t < nt) {
      uint32_t any = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w)
#pragma unroll
        for (int k = 0; k < 4; ++k) any |= seen[w][threadIdx.x * 4 + k];
      out[t] = any != 0u;
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_mask_scan(const ScanParams& p, int n_nodes, int max_states, cudaStream_t s) {
  LaunchConfig l(dim3(max_states, p.n_qt, n_nodes), kWarps * 32, 0, s);
  return cudaLaunchKernelEx(&l.cfg, mask_scan_kernel, p);
}

}  // namespace sva
