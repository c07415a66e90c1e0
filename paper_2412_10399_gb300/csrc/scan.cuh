// Tile sums of the block histogram, shared by the binning (a state that came
// from outside a step) and the float64 pass (every step, for the next one).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "launch.h"

namespace ck {

// Particles and non-empty keys of every tile of TILE keys; T threads per CTA, a
// loop over tiles.  cnt is 16-byte aligned.
template <int T, int TILE>
__device__ __forceinline__ void write_tile_sums(const uint32_t* cnt, uint32_t n_keys, uint32_t* tile_cnt,
                                                uint32_t* tile_ne) {
  static_assert(TILE % (4 * T) == 0, "a thread takes whole 16-byte groups");
  __shared__ uint32_t sc[T / 32], sn[T / 32];
  const uint32_t ntiles = scan_tiles(n_keys);
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    uint32_t c = 0, ne = 0;
#pragma unroll
    for (int q = 0; q < TILE / (4 * T); ++q) {
      const uint64_t k = (uint64_t)tile * TILE + 4u * (q * T + threadIdx.x);
      if (k + 4 <= n_keys) {
        const uint4 x = *reinterpret_cast<const uint4*>(cnt + k);
        c += x.x + x.y + x.z + x.w;
        ne += (x.x != 0u) + (x.y != 0u) + (x.z != 0u) + (x.w != 0u);
      } else {
        for (uint64_t j = k; j < n_keys; ++j) {
          const uint32_t x = cnt[j];
          c += x;
          ne += x != 0u;
        }
      }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    ne = __reduce_add_sync(0xffffffffu, ne);
    __syncthreads();  // the previous tile's sums have been read
    if ((threadIdx.x & 31) == 0) {
      sc[threadIdx.x >> 5] = c;
      sn[threadIdx.x >> 5] = ne;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t tc = 0, tn = 0;
#pragma unroll
      for (int w = 0; w < T / 32; ++w) {
        tc += sc[w];
        tn += sn[w];
      }
      tile_cnt[tile] = tc;
      tile_ne[tile] = tn;
    }
  }
}

}  // namespace ck
