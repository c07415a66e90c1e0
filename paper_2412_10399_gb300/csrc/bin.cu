// Per-step particle binning by particle block (counting sort on block keys).
//
// The histogram of the keys is produced by the previous G2P (or by admission
// / re-keying), and its sums per tile of kScanTile keys by the float64 pass
// that follows it.  One step then runs two kernels:
//   scan_final    per non-empty key: first slot and scatter cursor; non-empty
//                 keys become the particle-block list (in key order, so the
//                 list is deterministic) and flag the 2x2x2 grid blocks they
//                 touch.  Each CTA takes one tile and sums the tiles before it
//                 (a few tiles: their keys, without tile sums).
//   scatter_glist perm[cursor[key]++] = particle (warp-aggregated atomics) in
//                 one part of its CTAs; in the other the flagged grid blocks
//                 become the active grid-block list, flags cleared
// (A state that changed outside a step first takes its tile sums with
// scan_tiles; a key space of more than kScanFusedTiles tiles runs scan_tiles
// and scan_top, one CTA's exclusive scan over the sums of tiles of
// kScanTileWide keys, every step.)
// (The float64 pass clears the histogram entries of the step's blocks, so the
// buffer that G2P fills next step starts at zero without a pass over the whole
// key space.)
// Against a scan of three kernels over 4096-key tiles and two further ones
// (five launches), with the float64 pass that takes the tile sums: 14.2 -> 8.2
// us a step on the elastic cube (32,768 particles, 64^3), 17.2 -> 9.7 on the
// granular column (346,112, 128^3), 60 -> 50 on 16.27 M particles (512^3).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "launch.h"
#include "scan.cuh"

namespace ck {

constexpr int kScanThreads = 256;

template <int TILE>
__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(StepView v, BinScratch bs) {
  write_tile_sums<kScanThreads, TILE>(v.cnt_cur, v.n_keys, bs.tile_cnt, bs.tile_ne);
}

// Exclusive scan of (tile_cnt, tile_ne) in place by one CTA of 1024 threads.
__global__ void __launch_bounds__(1024) k_scan_top(BinScratch bs, uint32_t ntiles) {
  __shared__ uint32_t wc[32], wn[32];
  __shared__ uint32_t carry_c, carry_n;
  if (threadIdx.x == 0) {
    carry_c = 0;
    carry_n = 0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t b0 = 0; b0 < ntiles; b0 += 1024) {
    uint32_t i = b0 + threadIdx.x;
    uint32_t c = i < ntiles ? bs.tile_cnt[i] : 0u;
    uint32_t n = i < ntiles ? bs.tile_ne[i] : 0u;
    uint32_t ic = c, in = n;  // inclusive within warp
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t yc = __shfl_up_sync(0xffffffffu, ic, o);
      uint32_t yn = __shfl_up_sync(0xffffffffu, in, o);
      if (lane >= o) {
        ic += yc;
        in += yn;
      }
    }
    if (lane == 31) {
      wc[warp] = ic;
      wn[warp] = in;
    }
    __syncthreads();
    if (warp == 0) {
      uint32_t xc = wc[lane], xn = wn[lane];
      for (int o = 1; o < 32; o <<= 1) {
        uint32_t yc = __shfl_up_sync(0xffffffffu, xc, o);
        uint32_t yn = __shfl_up_sync(0xffffffffu, xn, o);
        if (lane >= o) {
          xc += yc;
          xn += yn;
        }
      }
      wc[lane] = xc;
      wn[lane] = xn;
    }
    __syncthreads();
    uint32_t pc = (warp ? wc[warp - 1] : 0u) + ic - c + carry_c;
    uint32_t pn = (warp ? wn[warp - 1] : 0u) + in - n + carry_n;
    if (i < ntiles) {
      bs.tile_cnt[i] = pc;
      bs.tile_ne[i] = pn;
    }
    __syncthreads();
    if (threadIdx.x == 1023) {
      carry_c = pc + c;
      carry_n = pn + n;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int scene_of_key(const BinScratch& bs, uint32_t key) {
  int lo = 0, hi = bs.n_scene_tab - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (bs.scene_tab[2 * mid] <= key)
      lo = mid;
    else
      hi = mid - 1;
  }
  return (int)bs.scene_tab[2 * lo + 1];
}

// MODE: what precedes the CTA's tile comes from the tile sums' exclusive scan
// (0: a wide tile, 16 keys a thread), from the tiles' own sums (1) or from the
// histogram itself (2) (4 keys a thread: they are a serial chain).
template <int MODE>
__global__ void __launch_bounds__(kScanThreads) k_scan_final(StepView v, BinScratch bs) {
  constexpr int TILE = MODE == 0 ? kScanTileWide : kScanTile, PER = TILE / kScanThreads;
  static_assert(PER % 4 == 0 && (MODE == 0 || PER == 4), "keys in 16-byte loads, one of them where MODE 2 counts tiles");
  const uint64_t base = (uint64_t)blockIdx.x * TILE + threadIdx.x * PER;
  uint32_t c[PER];
  if (base + PER <= v.n_keys) {
#pragma unroll
    for (int q = 0; q < PER; q += 4) {
      const uint4 x = *reinterpret_cast<const uint4*>(v.cnt_cur + base + q);
      c[q] = x.x;
      c[q + 1] = x.y;
      c[q + 2] = x.z;
      c[q + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < PER; ++q) c[q] = base + q < v.n_keys ? v.cnt_cur[base + q] : 0u;
  }
  // particles and blocks of the tiles before this one
  uint32_t tpc = 0, tpn = 0;
  if (MODE != 0) {
    if (MODE == 1) {
      for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kScanThreads) {
        tpc += bs.tile_cnt[i];
        tpn += bs.tile_ne[i];
      }
    } else {
      const uint4* c4 = reinterpret_cast<const uint4*>(v.cnt_cur);
#pragma unroll 4
      for (uint32_t i = 0; i < blockIdx.x; ++i) {
        const uint4 y = c4[i * kScanThreads + threadIdx.x];
        tpc += y.x + y.y + y.z + y.w;
        tpn += (y.x != 0u) + (y.y != 0u) + (y.z != 0u) + (y.w != 0u);
      }
    }
    tpc = __reduce_add_sync(0xffffffffu, tpc);
    tpn = __reduce_add_sync(0xffffffffu, tpn);
  } else {
    tpc = bs.tile_cnt[blockIdx.x];
    tpn = bs.tile_ne[blockIdx.x];
  }
  uint32_t tc = 0, tn = 0, most = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    tc += c[q];
    tn += c[q] != 0u;
    most = max(most, c[q]);
  }
  if (v.fullest) {  // at most one atomic a warp, and none but in dense blocks
    most = __reduce_max_sync(0xffffffffu, most);
    if (most > kDenseBlock && (threadIdx.x & 31u) == 0u) atomicMax(v.fullest, most);
  }
  // block-wide exclusive scan of (tc, tn)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t ic = tc, in = tn;
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t yc = __shfl_up_sync(0xffffffffu, ic, o);
    uint32_t yn = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) {
      ic += yc;
      in += yn;
    }
  }
  constexpr int NW = kScanThreads / 32;
  __shared__ uint32_t wc[NW], wn[NW], pcs[NW], pns[NW];
  if (lane == 31) {
    wc[warp] = ic;
    wn[warp] = in;
    pcs[warp] = tpc;
    pns[warp] = tpn;
  }
  __syncthreads();
  uint32_t pc = ic - tc, pn = in - tn;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    if (MODE != 0 || w == 0) {
      pc += pcs[w];
      pn += pns[w];
    }
    if (w < warp) {
      pc += wc[w];
      pn += wn[w];
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // the step's counters
    *v.n_g = 0u;
    *v.fp64_count = 0ull;
    v.work[0] = v.work0[0];
    v.work[1] = v.work0[1];
    if (v.lo_count) *v.lo_count = 0u;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) {
    *v.n_pb = pn + tn;
    v.pb[pn + tn] = make_uint2(0u, pc + tc);
  }
  // the owning scene of the thread's keys, looked up once and kept in
  // registers while the keys stay inside its key range (the stores below
  // could alias the scene table, so reading it per key reloads it each time)
  int sl = -1, npb = 1, nb = 1;
  uint32_t klo = 1u;
  uint64_t khi = 0u;
  long long tbase = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    if (c[q]) {
      const uint32_t k = (uint32_t)base + q;
      v.cursor[k] = pc;
      if (!(k >= klo && (uint64_t)k < khi)) {
        sl = scene_of_key(bs, k);
        const SceneDev& s = v.scenes[sl];
        klo = s.key_base;
        npb = s.npb;
        nb = s.nb;
        tbase = s.table_base;
        khi = (uint64_t)klo + (uint64_t)npb * (uint64_t)npb * (uint64_t)npb;
      }
      v.pb[pn] = make_uint2(k, pc);
      v.pb_scene[pn] = (uint32_t)sl;
      int lb = (int)(k - klo);
      int bx = lb % npb, by = (lb / npb) % npb, bz = lb / (npb * npb);
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
          for (int dx = 0; dx < 2; ++dx)
            v.gflag[tbase + ((long long)(bz + dz) * nb + (by + dy)) * nb + (bx + dx)] = (uint32_t)sl + 1u;
      pn += 1;
    }
    pc += c[q];
  }
}

// Each warp handles kScatterUnroll groups of 32 particles per pass and issues
// the cursor atomics of all of them before it waits for the first result: the
// pass is one atomic round trip instead of kScatterUnroll.
constexpr int kScatterUnroll = 8;

// (CTA `cta` of `ctas`, 256 threads each)
__device__ __forceinline__ void scatter_particles(const StepView& v, uint32_t cta, uint32_t ctas) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t stride = ctas * blockDim.x * kScatterUnroll;
  // the loop runs on the warp's first index, so every lane of a warp takes
  // the same iterations (the full-mask warp intrinsics below need that)
  for (uint32_t w0 = cta * blockDim.x * kScatterUnroll + (threadIdx.x - lane) * kScatterUnroll;
       w0 < v.n_cur; w0 += stride) {
    const uint32_t j0 = w0 + lane;
    uint32_t key[kScatterUnroll], peers[kScatterUnroll], base[kScatterUnroll];
#pragma unroll
    for (int u = 0; u < kScatterUnroll; ++u) {
      const uint32_t j = j0 + 32u * u;
      key[u] = j < v.n_cur ? v.key_cur[j] : CK_DEAD_KEY;
    }
#pragma unroll
    for (int u = 0; u < kScatterUnroll; ++u) {
      peers[u] = __match_any_sync(0xffffffffu, key[u]);
      base[u] = 0u;
      if (key[u] != CK_DEAD_KEY && (int)lane == __ffs(peers[u]) - 1)
        base[u] = atomicAdd(&v.cursor[key[u]], (uint32_t)__popc(peers[u]));
    }
#pragma unroll
    for (int u = 0; u < kScatterUnroll; ++u) {
      const uint32_t b = __shfl_sync(0xffffffffu, base[u], __ffs(peers[u]) - 1);
      if (key[u] != CK_DEAD_KEY) v.perm[b + __popc(peers[u] & ((1u << lane) - 1u))] = j0 + 32u * u;
    }
  }
}

// Flagged virtual blocks get pool slots in list order; the block table maps
// each of them to its slot.  Entries of untouched blocks are stale and never
// read (P2G/G2P only look up the blocks their own particle block flagged).
// A warp reads 32 x 4 flags with one 16-byte load per lane; a warp scan of
// the lanes' flag counts and one atomic per warp give every flagged block its
// slot.  The tail (fewer than four flags) and an unaligned array are read one
// flag at a time.
__device__ __forceinline__ void glist_assign(const StepView& v, uint32_t g, uint32_t f, uint32_t idx) {
  if (idx < v.pool_cap) {
    v.g_list[idx] = g;
    v.g_scene[idx] = f - 1u;
    v.table[g] = idx;
  } else {
    v.table[g] = CK_NO_SLOT;
    flag_error(v.err, CK_ERR_POOL);
  }
  v.gflag[g] = 0u;
}

__device__ __forceinline__ void list_grid_blocks(const StepView& v, uint32_t n_vblocks, uint32_t cta, uint32_t ctas) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t n4 = (reinterpret_cast<uintptr_t>(v.gflag) & 15u) ? 0u : n_vblocks / 4u;
  const uint4* f4 = reinterpret_cast<const uint4*>(v.gflag);
  const uint32_t wstride = ctas * blockDim.x;
  // every lane of a warp runs the same iterations (full-mask intrinsics)
  for (uint32_t q0 = cta * blockDim.x + (threadIdx.x - lane); q0 < n4; q0 += wstride) {
    const uint32_t q = q0 + lane;
    const uint4 f = q < n4 ? f4[q] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t nf = (f.x != 0u) + (f.y != 0u) + (f.z != 0u) + (f.w != 0u);
    if (__ballot_sync(0xffffffffu, nf != 0u) == 0u) continue;
    uint32_t inc = nf;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if ((int)lane >= o) inc += y;
    }
    uint32_t start = 0u;
    if (lane == 31u) start = atomicAdd(v.n_g, inc);
    start = __shfl_sync(0xffffffffu, start, 31);
    uint32_t idx = start + inc - nf;
    if (f.x) glist_assign(v, 4u * q, f.x, idx++);
    if (f.y) glist_assign(v, 4u * q + 1u, f.y, idx++);
    if (f.z) glist_assign(v, 4u * q + 2u, f.z, idx++);
    if (f.w) glist_assign(v, 4u * q + 3u, f.w, idx++);
  }
  for (uint32_t g = 4u * n4 + cta * blockDim.x + threadIdx.x; g < n_vblocks; g += wstride) {
    const uint32_t f = v.gflag[g];
    if (f) glist_assign(v, g, f, atomicAdd(v.n_g, 1u));
  }
}

// The two passes read the scan's results and do not depend on each other: the
// first `sctas` CTAs scatter, the next `gctas` list.  In a step of split blocks
// one more sets the parts of a block for the transfers (in a warp that also
// lists it set the kernel's length on the diffusion bar: 0.2% of its step).
__global__ void __launch_bounds__(256) k_scatter_glist(StepView v, uint32_t n_vblocks, uint32_t sctas, uint32_t gctas) {
  if (blockIdx.x < sctas) {
    scatter_particles(v, blockIdx.x, sctas);
  } else if (blockIdx.x < sctas + gctas) {
    list_grid_blocks(v, n_vblocks, blockIdx.x - sctas, gctas);
  } else if (threadIdx.x == 0) {
    const uint32_t npb = *v.n_pb, fullest = *v.fullest;
    *v.fullest = 0u;
#pragma unroll
    for (int k = 0; k < 2; ++k) v.parts[k] = limit_units(v.units[k], npb, v.unit_most, fullest).splits;
  }
}

// Fused step: before a block table is filled again, the entries its last
// use assigned (the first *n_g entries of its list, slots claimed by the
// leftover P2G included) go back to CK_NO_SLOT, so that every entry not
// assigned in this step reads as unassigned.
__global__ void k_table_reset(uint32_t* table, const uint32_t* g_list, const uint32_t* n_g, uint32_t pool_cap) {
  const uint32_t n = min(*n_g, pool_cap);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    table[g_list[i]] = CK_NO_SLOT;
}

void launch_table_reset(cudaStream_t st, uint32_t* table, const uint32_t* g_list, const uint32_t* n_g,
                        uint32_t pool_cap, int grid_ctas) {
  k_table_reset<<<grid_ctas, 256, 0, st>>>(table, g_list, n_g, pool_cap);
}

// Retire particles [start, start + n) of the current pool (a released scene):
// they get the dead key and leave the pool at the next step; the histogram and
// bounds of the scene's key range [k0, k0 + nk) go back to zero.
__global__ void k_retire(uint32_t* key, uint32_t start, uint32_t n, uint32_t* cnt, uint32_t* bnd, uint32_t k0,
                         uint32_t nk) {
  const uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint64_t i = t0; i < n; i += stride) key[start + i] = CK_DEAD_KEY;
  for (uint64_t i = t0; i < nk; i += stride) cnt[k0 + i] = 0u;
  for (uint64_t i = t0; i < 2ull * nk; i += stride) bnd[2ull * k0 + i] = 0u;
}

void launch_retire(cudaStream_t st, uint32_t* key, uint32_t start, uint32_t n, uint32_t* cnt, uint32_t* bnd,
                   uint32_t k0, uint32_t nk) {
  const uint64_t most = std::max<uint64_t>(n, 2ull * nk);
  const int blocks = (int)std::max<uint64_t>(1, std::min<uint64_t>(4096, (most + 255) / 256));
  k_retire<<<blocks, 256, 0, st>>>(key, start, n, cnt, bnd, k0, nk);
}

void launch_bin(cudaStream_t st, const StepView& v, const BinScratch& bs, int which, uint32_t n_gblocks,
                int grid_ctas) {
  const uint32_t ntiles = scan_tiles(v.n_keys);
  const bool fused = scan_fused(v.n_keys);
  // CTAs that have work, up to grid_ctas for each pass
  const uint32_t lim = (uint32_t)grid_ctas;
  const uint32_t sctas = std::max(1u, std::min(lim, (v.n_cur + 256u * kScatterUnroll - 1u) / (256u * kScatterUnroll)));
  const uint32_t gctas = std::max(1u, std::min(lim, (n_gblocks + 1023u) / 1024u));
  const uint32_t pctas = v.fullest ? 1u : 0u;
  switch (which) {
    case LB_SCAN_TILES:
      if (scan_direct(v.n_keys)) break;
      if (fused)
        k_scan_tiles<kScanTile><<<ntiles, kScanThreads, 0, st>>>(v, bs);
      else
        k_scan_tiles<kScanTileWide><<<ntiles, kScanThreads, 0, st>>>(v, bs);
      break;
    case LB_SCAN_TOP:
      if (!fused) k_scan_top<<<1, 1024, 0, st>>>(bs, ntiles);
      break;
    case LB_SCAN_FINAL:
      if (scan_direct(v.n_keys))
        k_scan_final<2><<<ntiles, kScanThreads, 0, st>>>(v, bs);
      else if (fused)
        k_scan_final<1><<<ntiles, kScanThreads, 0, st>>>(v, bs);
      else
        k_scan_final<0><<<ntiles, kScanThreads, 0, st>>>(v, bs);
      break;
    case LB_SCATTER_GLIST: k_scatter_glist<<<sctas + gctas + pctas, 256, 0, st>>>(v, n_gblocks, sctas, gctas); break;
    case LB_GLIST: k_scatter_glist<<<gctas + pctas, 256, 0, st>>>(v, n_gblocks, 0u, gctas); break;
  }
}

}  // namespace ck
