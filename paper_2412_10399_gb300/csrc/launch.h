// Host-side launchers of the CK-MPM kernels (internal to the library).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"

namespace ck {

struct LaunchCfg {
  cudaStream_t stream;
  int persistent_ctas;  // CTAs of the kernel that clears a probe's accumulators
  int sm_count = 1;     // SMs of the device (grid of the float64 pass)
  int g2p_minb = 4;     // resident G2P warps per SM / 4 the register budget targets
  int transfer = 0;     // 0 APIC + MLS, 1 PIC, 2 APIC with the kernel gradient
  int p2g_rep = 1;      // copies of the P2G shared accumulators (1 or 2)
  int p2g_rot = 0;      // one copy: components in the lane-rotated order (1) or in order (0)
  int p2g_fma = 0;      // APIC + MLS: fused-multiply-add rounding in blocks of >= 256 particles (1)
};

// One-warp CTAs per SM of the transfer kernels.  P2G of whole blocks launches
// more than fit (they take units until none is left); split blocks, where a
// CTA's first unit is its index, take one resident wave: what shared memory
// or registers leave room for (rep: copies of the APIC + MLS accumulators).
constexpr int p2g_warps(int kind, int transfer, int rep) {
  if (transfer == 2) return kind == 0 ? 14 : 12;
  if (transfer == 0 && rep == 2) return kind == 0 ? 12 : 16;
  return kind == 1 && transfer == 1 ? 16 : 18;
}
inline uint32_t p2g_ctas(int sm_count) { return (uint32_t)sm_count * 32u; }
// G2P and the fused kernel: one resident wave at their register budgets
constexpr int fused_warps(int kind) { return kind == 0 ? 20 : 16; }
inline int g2p_warps(int kind, int transfer, int minb) {
  if (transfer == 1) return kind == 0 ? 20 : 16;
  if (transfer == 2) return kind == 0 ? 16 : 12;
  return 4 * minb;
}

// Units of a step of n particles for a kernel of that many warps per SM.  A
// step with a full block of 512 for every G2P warp (20 per SM) keeps whole
// blocks, because a unit costs a warp several microseconds of its own (its
// chain of dependent loads, the staged nodes, a partly filled last chunk).  A
// smaller one is cut so that full blocks give about one unit per warp, in
// whole chunks; P2G, where a unit also clears and flushes its nodes, into no
// less than two chunks of 96 unless the step has not a G2P chunk per warp.
// Measured, P2G / G2P us on the granular column (346,112 particles, compact
// kernel): units of 96 24.9 / 29.4, 128 27.3 / 24.0, 192 20.6 / 26.9, 256
// 21.0 / 26.6; on the diffusion bar (224,000, PIC): 21.1 / 24.6, 20.6 / 29.2,
// 16.9 / 31.0, 21.1 / 39.7; on a sand box of 592,704 (with the events' 6 us),
// P2G in parts of 192 39.5, of 256 32.7.
// The count of parts is for blocks of 512; limit_units raises it on the device
// where blocks are fuller.  Step of 343,331 particles at 27 per cell / 346,111
// at 64, us, with the count for 512 and with limit_units': compact kernel 89 / 143
// and 69 / 67, quadratic 93 / 150 and 69 / 69; kernel-gradient APIC at 27: 114 and 76.
inline Units step_units(int which, int64_t n, int sm_count, int warps) {
  const int64_t sm = sm_count, block = 512;
  if (n >= sm * 20 * block) return Units{1u, (uint32_t)block};
  const int64_t want = std::max<int64_t>(2, std::min<int64_t>(16, sm * warps * block / std::max<int64_t>(n, 1)));
  const int64_t chunk = which == kUnitsP2G ? 96 : 32;
  int64_t unit = ((block + want - 1) / want + chunk - 1) / chunk * chunk;
  if (which == kUnitsP2G && n >= sm * 20 * 32) unit = std::max<int64_t>(192, unit);
  return Units{(uint32_t)((block + unit - 1) / unit), (uint32_t)unit};
}

// CTAs of the grid update, which loops over the listed blocks.  Many for a
// large step: each CTA's loop is short, so the dependent loads of one block
// (list entry, scene) overlap across CTAs.  A small step has few blocks (about
// n / 340 at 8 per cell; n / 64 leaves room), and launching 9728 empty CTAs took
// 2.5 us of it.  Whole waves of what an SM holds (registers: ten of the compact
// kernel's, eight of the quadratic's), up to 64 per SM, since a body spread over
// more blocks than the estimate keeps them all looping and a part of a wave
// takes as long as a whole one; rounded down, because empty CTAs cost a compact
// body 0.3 ns each (592,704 particles: 0.7% of a step in rounding up).
// Measured, us with 4, 8, 10, 12, 16 and 64 per SM: 30,000 particles in as many
// blocks (compact kernel) 233, 158, 148, 186, 159, 149; 150,000 in 111,000
// (quadratic, without 10) 344, 199, 248, 199, 162; the elastic cube and the
// granular column 7.9 and 8.1 (with the events' 6) up to 16, 10.4 with 64.
constexpr int update_wave(int kind) { return kind == 0 ? 10 : 8; }
inline int update_ctas(int kind, int sm_count, uint32_t pool_cap, uint32_t n_cur) {
  const uint32_t wave = (uint32_t)(sm_count * update_wave(kind)), most = 64u / (uint32_t)update_wave(kind);
  const uint32_t est = (std::min(pool_cap, n_cur / 64u + 256u) + 1u) / 2u;  // two blocks a CTA and turn
  return (int)(wave * std::max(1u, std::min(most, est / wave)));
}

enum { LK_P2G = 0, LK_UPDATE = 1, LK_G2P = 2, LK_CLEAR = 3, LK_G2P_FP64 = 4, LK_G2P2G = 5, LK_LEFTOVER = 6 };

// transfer.cu
void launch_transfer(int kind, const LaunchCfg& lc, const StepView& v, int which);
void launch_read_particles(int kind, bool pic, cudaStream_t st, Pool P, const SceneDev* scenes, const MatDev* mats,
                           int scene, uint32_t start, uint32_t n, int field, float* out);
void launch_write_particles(bool pic, cudaStream_t st, Pool P, const SceneDev* scenes, const MatDev* mats, int scene,
                            uint32_t start, uint32_t n, int field, const float* in);
void launch_read_grid(int kind, cudaStream_t st, const StepView& v, int scene, int which, float* out);
void launch_admit(int kind, cudaStream_t st, Pool P, uint32_t* key, uint32_t* cnt, uint32_t* bnd,
                  const SceneDev* scenes, const MatDev* mats, int scene, uint32_t mat_base, uint32_t nmat,
                  uint32_t start, uint32_t n, const float* x, const float* v, const uint8_t* mat, const float* E,
                  uint32_t* err);
void launch_rekey(int kind, cudaStream_t st, Pool P, uint32_t* key, uint32_t* cnt, uint32_t* bnd,
                  const SceneDev* scenes, const MatDev* mats, uint32_t n, uint32_t* err);

// The allocation-free entry point (noalloc.cu): scene parameters as a kernel
// argument, which the admission kernel leaves in device memory for the rest.
constexpr int kStaticMaxMats = 16;
struct StaticParams {
  SceneDev scene;
  MatDev mats[kStaticMaxMats];
  uint32_t tab[2];
};
void launch_static_admit(int kind, cudaStream_t st, const StepView& v, const StaticParams& prm, StaticParams* d_prm,
                         bool pic, uint32_t nmat, const float* x, const float* vel, const uint8_t* mat, const float* F,
                         const float* B);
void launch_static_grids(int kind, cudaStream_t st, const StepView& v, uint32_t n_vblocks, float* grid_m,
                         float* grid_p);

// bin.cu
constexpr int kScanTile = 1024;  // keys per scan tile
// Up to this many tiles every CTA of the scan sums the tiles before its own
// (two arrays: at most 32 loads a thread).  Beyond, one CTA scans the tile sums
// first, 1024 an iteration, and tiles are wide: with 1024 keys its chain was
// four times as long and the other kernels had four times the CTAs, us a step's
// binning for res 1024 / 2048 (16.8 M and 134 M keys, 32,767 particles): 67 / 470
// against 43 / 250.
constexpr uint32_t kScanFusedTiles = 4096;
constexpr int kScanTileWide = 4096;
__host__ __device__ inline bool scan_fused(uint32_t n_keys) { return n_keys <= kScanFusedTiles * kScanTile; }
__host__ __device__ inline uint32_t scan_tiles(uint32_t n_keys) {
  const uint32_t tile = scan_fused(n_keys) ? kScanTile : kScanTileWide;
  return n_keys ? (n_keys - 1u) / tile + 1u : 1u;
}
// Up to this many tiles the scan needs no tile sums: every CTA counts the keys
// before its own tile itself (at most 7 loads of 16 bytes a thread).
constexpr uint32_t kScanDirectTiles = 8;
inline bool scan_direct(uint32_t n_keys) { return scan_tiles(n_keys) <= kScanDirectTiles; }
struct BinScratch {
  uint32_t* tile_cnt;   // per tile: sum of counts
  uint32_t* tile_ne;    // per tile: non-empty keys
  const uint32_t* scene_tab;  // sorted (key_base, slot) pairs of the scenes at the last admission
  int n_scene_tab;
};
void launch_bin(cudaStream_t st, const StepView& v, const BinScratch& bs, int which, uint32_t n_gblocks,
                int grid_ctas);
// LB_SCAN_TOP launches nothing when the scan is fused (scan_fused)
enum { LB_SCAN_TILES = 0, LB_SCAN_TOP = 1, LB_SCAN_FINAL = 2, LB_SCATTER_GLIST = 3, LB_GLIST = 4 };
void launch_retire(cudaStream_t st, uint32_t* key, uint32_t start, uint32_t n, uint32_t* cnt, uint32_t* bnd,
                   uint32_t k0, uint32_t nk);
void launch_table_reset(cudaStream_t st, uint32_t* table, const uint32_t* g_list, const uint32_t* n_g,
                        uint32_t pool_cap, int grid_ctas);

}  // namespace ck
