// Device-side data layout and helpers shared by the CK-MPM kernels.
//
// Particle pool (structure of arrays, double-buffered, 16-byte vectors):
//   X   float4 (x, y, z, material index as bits)
//   VM0 float4 (vx, vy, vz, M22)   VM1 (M00, M10, M01, M11)   VM2 (M02, M12, M20, M21)
//   F0  float4 (F00, F10, F01, F11)  F1 (F02, F12, F20, F21)  F2 float F22
// (rows 0 and 1 of a matrix side by side: the pairs of the packed arithmetic)
//   ID  uint32 scene-local particle index
// M = m B - dt V0 tau(F) is the per-particle matrix that P2G multiplies by
// D(x)^-1: it carries both the APIC affine momentum (Sec. 4.4) and the MLS
// stress force (Sec. 4.3.2 with reading R4).  Storing M instead of B lets P2G
// run without an SVD; B is recovered exactly as (M + dt V0 tau(F)) / m.
//
// Sparse grid: each scene's domain is a virtual array of 4x4x4-node blocks;
// a block table maps the blocks touched this step to slots of a compact pool
// (slot = position in the active-block list, reassigned every step).  Per
// pool slot and grid 64 float4:
//   Gacc  (m, p_x, p_y, p_z) accumulated by P2G, zeroed by the grid update
//   Gvel  (v~_x, v~_y, v~_z, m) written by the grid update, gathered by G2P
// CK uses two grids per block (0: G-, 1: G+), quadratic one.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#define CK_ERR_DOMAIN 1u
#define CK_ERR_NONFINITE 2u
#define CK_ERR_INTERNAL 4u
#define CK_ERR_TIMEOUT 8u
#define CK_ERR_POOL 16u
#define CK_NO_SLOT 0xFFFFFFFFu

#define CK_DEAD_KEY 0xFFFFFFFFu

namespace ck {

constexpr int kBlock = 4;        // nodes / cells per block edge
constexpr int kBlockNodes = 64;  // nodes per block and grid

struct SceneDev {
  float dx, inv_dx, dt, V0;
  float gx, gy, gz;
  float bc;           // sticky wall thickness in cells
  int res;            // cells per axis
  int npb;            // particle blocks per axis = ceil(res/4)
  int nb;             // grid blocks per axis = npb + 1
  uint32_t key_base;  // first particle-block key of this scene
  long long table_base;  // first entry of this scene's block table
  float j_tol, cond_tol, gap_tol;  // float64 SVD criteria
};

// Two 16-byte groups of what the update reads together, then the indices.
struct alignas(16) MatDev {
  float mass;     // rho * V0
  float mu, lam;  // Lame parameters
  float dpc;      // Drucker-Prager: (3 lam + 2 mu) / (2 mu) alpha = alpha (1 + nu) / (1 - 2 nu), any E
  float alpha;    // Drucker-Prager cone coefficient
  float E, nu;    // for per-particle E; the fluid's equation-of-state constant B is E
  float gamma;    // fluid equation-of-state exponent
  int model;      // 0 fixed-corotated, 1 Drucker-Prager, 2 J-based fluid
  int scene;      // owning scene slot
  int pad_[2];
};

// Pointers to one buffer of the particle pool.
struct Pool {
  float4* X;
  float4* VM0;
  float4* VM1;
  float4* VM2;
  float4* F0;
  float4* F1;
  float* F2;
  uint32_t* ID;
  float* E;  // optional per-particle Young's modulus (may be null)
  // APIC with the kernel gradient only (else null): T = -dt V0 tau in the
  // order of F (T0, T1, T2); VM then holds m B without the stress
  float4* T0;
  float4* T1;
  float* T2;
};

// Work units of a transfer kernel: `splits` parts of every particle block, of
// `unit` particles each (a block that holds more than splits * unit is cut into
// equal parts; the last parts of a thin one are empty; unit 0: a fixed count of
// parts).
struct Units {
  uint32_t splits, unit;
};
enum { kUnitsP2G = 0, kUnitsG2P = 1 };
// The host's count of parts is made for blocks of 8 particles per cell, 512,
// and holds up to this many particles a block; the scan records the fullest
// block beyond it.
constexpr uint32_t kDenseBlock = 640;
// The parts a step of npb blocks uses (a CTA of the listing kernel's launch
// takes them for both transfers, which then read them beside npb: worked out by
// each CTA they cost the elastic cube's step of 41 us 0.2 us).  Where the fullest block holds more than
// kDenseBlock particles, as many as cut that block into units (a part of it is
// the longest chain of the kernel: at 27 particles per cell the kernel-gradient
// G2P of 343,331 particles took 66 us in three parts a block, 41 in
// nine).  No more than give `most` units, so that a body spread over many thin
// blocks does not pay for parts without particles (a part then takes more than
// `unit`).
__host__ __device__ inline Units limit_units(Units w, uint32_t npb, uint32_t most, uint32_t fullest) {
  if (fullest > kDenseBlock && w.unit != 0u) {
    const uint32_t cut = (fullest + w.unit - 1u) / w.unit;
    w.splits = w.splits > cut ? w.splits : cut;
  }
  const uint32_t lim = npb ? (most + npb - 1u) / npb : 1u;
  w.splits = w.splits < lim ? w.splits : lim;
  return w;
}
// Particles of each part of a block of cnt, in whole chunks of `align`.
__host__ __device__ inline uint32_t part_size(const Units& w, uint32_t cnt, uint32_t align) {
  const uint32_t per = ((cnt + w.splits - 1u) / w.splits + align - 1u) / align * align;
  return w.unit > per ? w.unit : per;
}

// Everything the per-step kernels read; passed by value.
struct StepView {
  Pool cur, nxt;
  uint32_t* key_cur;    // keys of cur (input of the sort)
  uint32_t* key_nxt;    // keys written by G2P for nxt
  uint32_t* cnt_cur;    // histogram of key_cur over the key space
  uint32_t* cnt_nxt;    // histogram written by G2P (all zero before it: the float64 pass, behind the step's
                        // transfers, clears cnt_cur's entries of the step's blocks)
  uint32_t* bnd_cur;    // per key: P2G contribution bounds (mass, momentum) of cur, float
                        // bits; cleared with cnt_cur
  uint32_t* bnd_nxt;    // the same for nxt, written by G2P (all zero before it)
  uint32_t* cursor;     // scatter cursors
  uint32_t* perm;       // sorted slot -> index into cur
  uint2* pb;            // non-empty particle blocks in key order: (key, first sorted slot), and one
                        // more entry whose slot ends the last block
  uint32_t* pb_scene;   // and owning scene
  uint32_t* tile_cnt;   // per tile of kScanTile keys: particles and non-empty keys (the input of the
  uint32_t* tile_ne;    // next scan); null: the float64 pass leaves them to a kernel of their own
  uint32_t* n_pb;       // number of non-empty particle blocks
  uint32_t* gflag;      // per virtual grid block: scene+1 if touched this step
  uint32_t* table;      // per virtual grid block: pool slot (valid if touched this step)
  uint32_t* g_list;     // pool slot -> virtual grid block
  uint32_t* g_scene;    // pool slot -> owning scene
  uint32_t* n_g;        // number of active grid blocks (may exceed pool_cap on overflow)
  uint32_t pool_cap;    // pool capacity in blocks
  float4* Gacc;
  float4* Gvel;
  const SceneDev* scenes;
  const MatDev* mats;
  uint32_t* err;
  unsigned long long* fp64_count;  // particles listed for the float64 pass this step
  uint32_t* fp64_list;  // their slots in nxt (capacity: the pool)
  uint32_t* work;       // [0] next P2G block, [1] next G2P block (dynamic scheduling)
  uint32_t n_keys;      // size of the key space
  uint32_t n_cur;       // particles in cur (including dead ones)
  uint32_t keep_gacc;   // probe: the grid update leaves Gacc
  Units units[2];       // work units of P2G and of G2P
  uint32_t work0[2];    // what the scan sets work[] to: the CTAs of a step of split blocks, else 0
  uint32_t unit_most;   // limit_units' bound (32 per SM)
  uint32_t* fullest;    // split blocks only (else null): particles of the step's fullest block if above
                        // kDenseBlock, else 0 (from the scan; the CTA that sets parts returns it to 0)
  uint32_t* parts;      // limit_units of the step: parts of a block for P2G and for G2P
  uint32_t n_mats;      // entries of the material table
  // fused G2P2G step only (else null): the block table of the next step's
  // grid (the gather reads Gvel through `table`, the scatter adds to Gacc
  // through these), and the list of particles the fused kernel leaves to the
  // leftover P2G (changed block, float64 pass, non-finite)
  uint32_t* table_nxt;
  uint32_t* g_list_nxt;
  uint32_t* g_scene_nxt;
  uint32_t* n_g_nxt;
  uint32_t* lo_list;
  uint32_t* lo_count;
};

__device__ __forceinline__ void flag_error(uint32_t* err, uint32_t bit) { atomicOr(err, bit); }

struct Unit {
  uint32_t key, scene, start, cnt;  // the block
  uint32_t lo, hi;                  // the unit's particles: [lo, hi) of [0, cnt)
};

// Unit u: block u / splits, part u % splits, in whole chunks of ALIGN
// particles; false when the part is empty.  A block's entries are three
// independent loads: its key and first slot, the next block's first slot, its
// scene.
template <uint32_t ALIGN, bool SPLIT = true>
__device__ __forceinline__ bool unit_of(const StepView& v, const Units& w, uint32_t u, Unit& q) {
  const uint32_t bi = SPLIT ? u / w.splits : u, part = SPLIT ? u - bi * w.splits : 0u;
  const uint2 b = v.pb[bi];
  const uint32_t end = v.pb[bi + 1].y;
  q.scene = v.pb_scene[bi];
  q.key = b.x;
  q.start = b.y;
  q.cnt = end - b.y;
  if (!SPLIT) {
    q.lo = 0u;
    q.hi = q.cnt;
    return true;  // listed blocks hold particles
  }
  const uint32_t per = part_size(w, q.cnt, ALIGN);
  q.lo = part * per;
  q.hi = min(q.cnt, q.lo + per);
  return q.lo < q.hi;
}

// Unit schedule of a persistent one-warp CTA.  Units come one at a time from
// the step's counter; a few thousand CTAs asking one address at once are
// served one after the other (about 3 ns each), so in a step of split blocks
// the first unit is the CTA's own index.  A step of whole blocks keeps that
// first queue: it staggers the CTAs, which otherwise gather and compute in
// step (G2P of 16.27 M particles 0.64 -> 0.67 ms).
// (The scan starts the counter at the number of CTAs then: work0.)
__device__ __forceinline__ uint32_t next_unit(uint32_t* work) {
  uint32_t u = 0;
  if (threadIdx.x == 0) u = atomicAdd(work, 1u);
  return __shfl_sync(0xffffffffu, u, 0);
}
// Cell decomposition shared by every kernel that maps a position to nodes.
// u0 = x/dx.  CK: t = u0 + 1/4, b+ = floor(t), f+ = t - b+ (exact when dx is a
// power of two), b- = b+ or b+ - 1 with f- = f+ -+ 1/2 (Sec. 4.2 offsets).
// The particle block is floor(b-/4) for CK (G- blocks are the reference
// blocks, Sec. 5.1) and floor(base/4) for the quadratic stencil.
template <int KIND>
struct Cell;

template <>
struct Cell<0> {
  int bp, bm;   // base node on G+ and G-
  float fp, fm; // fractions in [0,1)
  __device__ __forceinline__ void set(float u0) {
    float t = u0 + 0.25f;
    float fb = floorf(t);
    bp = (int)fb;
    fp = t - fb;
    if (fp >= 0.5f) {
      bm = bp;
      fm = fp - 0.5f;
    } else {
      bm = bp - 1;
      fm = fp + 0.5f;
    }
  }
  __device__ __forceinline__ int block() const { return bm >> 2; }
};

template <>
struct Cell<1> {
  int b;
  float f;  // in [0.5, 1.5)
  __device__ __forceinline__ void set(float u0) {
    float t = u0 - 0.5f;
    float fb = floorf(t);
    b = (int)fb;
    f = u0 - fb;
  }
  __device__ __forceinline__ int block() const { return b >> 2; }
};

// Valid interior for both stencils: 0.5 <= x/dx < res - 0.5.
__device__ __forceinline__ bool in_domain(float u, int res) {
  return u >= 0.5f && u < (float)res - 0.5f;
}

template <int KIND, typename SceneT>
__device__ __forceinline__ uint32_t particle_key(const SceneT& s, float ux, float uy, float uz) {
  Cell<KIND> cx, cy, cz;
  cx.set(ux);
  cy.set(uy);
  cz.set(uz);
  int bx = cx.block(), by = cy.block(), bz = cz.block();
  return s.key_base + (uint32_t)((bz * s.npb + by) * s.npb + bx);
}

// Histogram increment and P2G contribution bounds of particles binned under
// `key` (lanes with equal keys add once).  The bounds are non-negative floats
// kept as bit patterns (whose unsigned order is the float order); each warp
// contributes the largest bound over all its active lanes, which may only
// overestimate a block's bound.
__device__ __forceinline__ void warp_aggregated_bin(uint32_t* cnt, uint32_t* bnd, uint32_t key, float bmass,
                                                    float bmom) {
  const unsigned mask = __activemask();
  const uint32_t bm = __reduce_max_sync(mask, __float_as_uint(bmass));
  const uint32_t bp = __reduce_max_sync(mask, __float_as_uint(bmom));
  const unsigned peers = __match_any_sync(mask, key);
  if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) {
    atomicAdd(&cnt[key], (uint32_t)__popc(peers));
    atomicMax(&bnd[2 * key], bm);
    atomicMax(&bnd[2 * key + 1], bp);
  }
}

}  // namespace ck
