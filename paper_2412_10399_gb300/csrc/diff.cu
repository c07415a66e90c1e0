// Differentiable CK-MPM step: forward and hand-written adjoint kernels.
//
// One step of the compact-kernel MPM on the dual grid (Sec. 4.3-4.5) with the
// fixed-corotated model, written as a pure function of the particle state
// (x, v, B, F) and a per-particle Young's modulus E, with particles kept in
// the caller's order and every node of both grids resident:
//   P2G   m_i = sum w m,  P_i = sum w (m v + A d),  A = (m B - dt V0 tau(F)) D^-1
//   grid  v~_i = mask (P_i / m_i + dt g)   (m_i > 0; sticky walls)
//   G2P   v' = 1/2 sum w v~,  B' = 1/2 sum w v~ (x_i - x_p)^T,
//         F' = (I + dt B' D^-1) F,  x' = x + dt v'
// (readings R4-R8 of the forward engine).  The adjoint of a step runs the
// reverse of these three stages: G2P^T scatters the velocity adjoint to the
// grid, the grid stage maps it to momentum and mass adjoints, and P2G^T
// gathers them back to the particles; weights, offsets and D depend on x and
// are differentiated in closed form (K1 is C^2, so dK1 is continuous).  The
// stress adjoint goes through the polar decomposition F = R S with
// dR = R Omega, Omega S + S Omega = R^T dF - dF^T R: a 3x3 system in the axial
// vector of Omega whose determinant, the product of the sigma_i + sigma_j,
// stays well conditioned when singular values coincide.
//
// Grid layout and its upkeep.  A node holds one float4 (m, P), (v~, 0) or
// (p_bar, m_bar), so that a scatter is one 16-byte vector reduction per node
// and a gather one 16-byte load, and nodes lie in 4x4x4 blocks (1 KiB).  P2G
// lists the blocks its particles touch (a flag per block, taken once by an
// exchange); the grid kernels run over that list alone and leave behind what
// the next call expects: accumulators and flags at zero, and the last kernel
// of a call returns the list's count to zero.  No call clears or sweeps the
// whole domain (a body fills a few per cent of it), and the state lives in
// device memory only, so a captured sequence can be replayed.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>

#include "../../include/ckmpm.h"
#include "svd3.cuh"

namespace ckd {

using ck::svd3;

// Launches of a step's kernels, with programmatic stream serialisation: a
// kernel's CTAs may become resident while the kernel before it drains, and
// wait there (grid_begin, the first statement of each) until it has finished
// and its writes are visible; each lets the next do the same from its own
// start.  That hides the launch latency and the ramp of kernels of a few
// microseconds; a kernel behind anything else (a copy, an event, a kernel of
// the caller) starts as usual.  Measured (262,144 particles): a forward step
// 60.3 -> 54.5 us, its adjoint 128.4 -> 116.3.  (The forward engine's steps
// are replayed as graphs, where it gained 2% on the smallest and lost 5% on
// the diffusion bar, so they are launched plainly.)
template <typename... P, typename... A>
inline void launch_step(void (*kernel)(P...), uint32_t grid, uint32_t block, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
// Wait for the kernel before this one, and let the one after it take its place.
__device__ __forceinline__ void grid_begin() {
  asm volatile("griddepcontrol.launch_dependents;\ngriddepcontrol.wait;" ::: "memory");
}

struct DP {
  float dx, inv_dx, dt, V0, mass, nu, gx, gy, gz, bc;
  int res, nb, n;  // nb: 4x4x4-node blocks per axis, ceil((res + 1) / 4)
};

// The grids and their active blocks.
struct DGrid {
  float4* G;        // (m, P) per node: [grid][block][64]; zero between calls
  float4* V;        // (v~, unused), valid in listed blocks
  float4* A;        // adjoint: v~_bar, then (p_bar, m_bar), valid in listed blocks
  uint32_t* flag;   // per block: 1 while listed
  uint32_t* list;   // listed blocks
  uint32_t* count;  // their number; zero between calls
  uint32_t* err;
};

constexpr float kInv2Pi = 0.15915494309189535f;

// Per-particle stencil on both grids with derivatives with respect to x.
struct DS {
  int base[2][3];      // base node per grid (0: G-, 1: G+) and axis
  float W[2][3][2];    // 1-D weights
  float dW[2][3];      // d W / d x of node 1 (per unit length); node 0 has the negative
  float f[2][3];       // fraction: x_i - x_p = (node - f) cells
  float Di[9];         // D^-1 (cells^-2)
  float sg[3], dsg[3]; // sigma = sin(2 pi f+)/(2 pi) and d sigma / dx
  float dLam[3];       // d Lambda / dx
  __device__ __forceinline__ void set(const DP& p, float x0, float x1, float x2) {
    const float xs[3] = {x0, x1, x2};
    float lam[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float u = xs[a] * p.inv_dx;
      float t = u + 0.25f;
      float fb = floorf(t);
      int bp = (int)fb;
      float fp = t - fb, fm;
      int bm;
      if (fp >= 0.5f) {
        bm = bp;
        fm = fp - 0.5f;
      } else {
        bm = bp - 1;
        fm = fp + 0.5f;
      }
      float s2, c2;
      sincospif(2.0f * fp, &s2, &c2);
      float s = s2 * kInv2Pi;
      base[0][a] = bm;
      base[1][a] = bp;
      W[1][a][0] = 1.0f - fp + s;
      W[1][a][1] = fp - s;
      W[0][a][0] = 1.0f - fm - s;
      W[0][a][1] = fm + s;
      dW[1][a] = (1.0f - c2) * p.inv_dx;
      dW[0][a] = (1.0f + c2) * p.inv_dx;
      f[1][a] = fp;
      f[0][a] = fm;
      float m2p = fp * (1.0f - fp) - s * (1.0f - 2.0f * fp);
      float m2m = fm * (1.0f - fm) + s * (1.0f - 2.0f * fm);
      lam[a] = 0.5f * (m2p + m2m) - s * s;
      float dm2p = (1.0f - 2.0f * fp) * (1.0f - c2) + 2.0f * s;
      float dm2m = (1.0f - 2.0f * fm) * (1.0f + c2) - 2.0f * s;
      dLam[a] = (0.5f * (dm2p + dm2m) - 2.0f * s * c2) * p.inv_dx;
      sg[a] = s;
      dsg[a] = c2 * p.inv_dx;
    }
    float li[3] = {1.0f / lam[0], 1.0f / lam[1], 1.0f / lam[2]};
    float y[3] = {li[0] * sg[0], li[1] * sg[1], li[2] * sg[2]};
    float den = 1.0f / (1.0f + sg[0] * y[0] + sg[1] * y[1] + sg[2] * y[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) Di[i * 3 + j] = (i == j ? li[i] : 0.0f) - y[i] * y[j] * den;
  }
  // x_bar contribution of an adjoint Dib on D^-1 (cells^-2)
  __device__ __forceinline__ void dinv_to_x(const float* Dib, float* xb) const {
    // D_bar = -Di^T Dib Di^T  (Di symmetric)
    float T[9], Db[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) T[i * 3 + j] = Di[i * 3 + 0] * Dib[0 * 3 + j] + Di[i * 3 + 1] * Dib[1 * 3 + j] + Di[i * 3 + 2] * Dib[2 * 3 + j];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) Db[i * 3 + j] = -(T[i * 3 + 0] * Di[0 * 3 + j] + T[i * 3 + 1] * Di[1 * 3 + j] + T[i * 3 + 2] * Di[2 * 3 + j]);
    // D_ab = Lam_a delta_ab + sg_a sg_b
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float sym = 0.f;
#pragma unroll
      for (int b = 0; b < 3; ++b) sym += (Db[c * 3 + b] + Db[b * 3 + c]) * sg[b];
      xb[c] += Db[c * 4] * dLam[c] + dsg[c] * sym;
    }
  }
};

// Offset of node i along an axis whose blocks are `bs` blocks apart and whose
// local nodes `ls` nodes apart; a node's index is the sum over the axes.
__device__ __forceinline__ uint32_t axis_off(int i, uint32_t bs, uint32_t ls) {
  return (uint32_t)(i >> 2) * (bs * 64u) + (uint32_t)(i & 3) * ls;
}

// Node offsets of a particle's stencil on one grid, per axis and node.
struct DOff {
  uint32_t o[3][2];
  __device__ __forceinline__ DOff(const DP& p, const DS& s, int g) {
    const uint32_t nb = (uint32_t)p.nb;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      o[0][k] = axis_off(s.base[g][0] + k, 1u, 1u);
      o[1][k] = axis_off(s.base[g][1] + k, nb, 4u);
      o[2][k] = axis_off(s.base[g][2] + k, nb * nb, 16u);
    }
  }
};

__device__ __forceinline__ size_t grid_size(const DP& p) { return (size_t)p.nb * p.nb * p.nb * 64u; }

__device__ __forceinline__ bool nodes_in_range(const DP& p, const DS& s) {
  bool ok = true;
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int a = 0; a < 3; ++a) ok = ok && s.base[g][a] >= 0 && s.base[g][a] + 1 <= p.res;
  return ok;
}

// *a += v as one 16-byte reduction (a quarter of the L2 operations of four
// scalar atomics).
__device__ __forceinline__ void red_add4(float4* a, float x, float y, float z, float w) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

__device__ __forceinline__ void list_block(const DGrid& D, uint32_t b) {
  // the plain read skips the exchange once the flag is seen; a stale 0 only
  // costs an exchange
  if (D.flag[b] == 0u && atomicExch(&D.flag[b], 1u) == 0u) D.list[atomicAdd(D.count, 1u)] = b;
}

// List the blocks of the nodes a warp's particles touch on either grid (nodes
// base[0] .. base[1] + 1 per axis; all lanes call, `on` marks those with a
// particle).  Neighbours in the caller's order are mostly neighbours in
// space, so the warp takes the bounding box of its blocks, one lane a block,
// when that is at most 32 blocks (a listed block without mass only costs its
// visit); each lane lists its own otherwise.  One exchange per warp and block
// instead of one per particle: the flags of a small body are contended.
__device__ __forceinline__ void list_blocks(const DP& p, const DGrid& D, const DS& s, bool on) {
  int lo[3], hi[3], wl[3], wn[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = s.base[0][a] >> 2;
    hi[a] = (s.base[1][a] + 1) >> 2;
    wl[a] = __reduce_min_sync(0xffffffffu, on ? lo[a] : 0x7fffffff);
    wn[a] = __reduce_max_sync(0xffffffffu, on ? hi[a] : -1) - wl[a] + 1;  // <= 0 without a particle
  }
  if (wn[0] <= 0) return;
  if (wn[0] <= 32 && wn[1] <= 32 && wn[2] <= 32 && wn[0] * wn[1] * wn[2] <= 32) {
    const int l = threadIdx.x & 31;
    if (l < wn[0] * wn[1] * wn[2]) {
      const int x = wl[0] + l % wn[0], y = wl[1] + (l / wn[0]) % wn[1], z = wl[2] + l / (wn[0] * wn[1]);
      list_block(D, ((uint32_t)z * p.nb + (uint32_t)y) * p.nb + (uint32_t)x);
    }
  } else if (on) {
    for (int z = lo[2]; z <= hi[2]; ++z)
      for (int y = lo[1]; y <= hi[1]; ++y)
        for (int x = lo[0]; x <= hi[0]; ++x) list_block(D, ((uint32_t)z * p.nb + (uint32_t)y) * p.nb + (uint32_t)x);
  }
}

// Rows of W consecutive floats per particle (the caller's arrays) of the 32
// particles of a warp, through shared memory: consecutive lanes move
// consecutive floats, and a lane's own row is read back at the odd pitch W.
// A kernel fetches all its arrays (each into its own region) before the one
// __syncwarp, so their loads are in flight together.  Scalar accesses: the
// caller's arrays are only 4-byte aligned.
template <int W>
__device__ __forceinline__ void fetch_rows(const float* g, size_t p0, int cnt, float* sm) {
  const int lane = threadIdx.x & 31;
  const float* src = g + p0 * W;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const int e = k * 32 + lane;
    if (e < cnt * W) sm[e] = src[e];
  }
}
template <int W>
__device__ __forceinline__ void take_row(const float* sm, float* r) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < W; ++q) r[q] = sm[lane * W + q];
}
// (begins with a __syncwarp: earlier rows in sm have been read)
template <int W>
__device__ __forceinline__ void store_rows(float* g, size_t p0, int cnt, float* sm, const float* r) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < W; ++q) sm[lane * W + q] = r[q];
  __syncwarp();
  float* dst = g + p0 * W;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const int e = k * 32 + lane;
    if (e < cnt * W) dst[e] = sm[e];
  }
}

// S = sum w a and M = sum w a (x_i - x_p)^T (cells; row c, column b) of the
// 3-vectors a = (node.x, node.y, node.z) over one grid's stencil, added to S
// and M: the weights are products, so x, y and z are reduced in turn.
__device__ __forceinline__ void gather_moments(const float4* g, const DS& s, const DOff& o, int k, float h, float* S,
                                               float* M) {
  const float wx0 = s.W[k][0][0], wx1 = s.W[k][0][1], mx0 = -s.f[k][0] * wx0, mx1 = (1.0f - s.f[k][0]) * wx1;
  const float wy0 = s.W[k][1][0], wy1 = s.W[k][1][1], my0 = -s.f[k][1] * wy0, my1 = (1.0f - s.f[k][1]) * wy1;
  const float wz[2] = {h * s.W[k][2][0], h * s.W[k][2][1]};
  const float mz[2] = {-s.f[k][2] * wz[0], (1.0f - s.f[k][2]) * wz[1]};
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    float R[2][3], Rx[2][3];
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const uint32_t row = o.o[2][z] + o.o[1][y];
      const float4 a = g[row + o.o[0][0]], b = g[row + o.o[0][1]];
      R[y][0] = wx0 * a.x + wx1 * b.x;
      R[y][1] = wx0 * a.y + wx1 * b.y;
      R[y][2] = wx0 * a.z + wx1 * b.z;
      Rx[y][0] = mx0 * a.x + mx1 * b.x;
      Rx[y][1] = mx0 * a.y + mx1 * b.y;
      Rx[y][2] = mx0 * a.z + mx1 * b.z;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float P = wy0 * R[0][c] + wy1 * R[1][c];
      S[c] += wz[z] * P;
      M[c * 3 + 0] += wz[z] * (wy0 * Rx[0][c] + wy1 * Rx[1][c]);
      M[c * 3 + 1] += wz[z] * (my0 * R[0][c] + my1 * R[1][c]);
      M[c * 3 + 2] += mz[z] * P;
    }
  }
}

__device__ __forceinline__ void mat3(const float* A, const float* B, float* C) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i * 3 + j] = A[i * 3] * B[j] + A[i * 3 + 1] * B[3 + j] + A[i * 3 + 2] * B[6 + j];
}
__device__ __forceinline__ void mat3_bt(const float* A, const float* B, float* C) {  // A B^T
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i * 3 + j] = A[i * 3] * B[j * 3] + A[i * 3 + 1] * B[j * 3 + 1] + A[i * 3 + 2] * B[j * 3 + 2];
}
__device__ __forceinline__ void mat3_at(const float* A, const float* B, float* C) {  // A^T B
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i * 3 + j] = A[i] * B[j] + A[3 + i] * B[3 + j] + A[6 + i] * B[6 + j];
}

__device__ __forceinline__ void lame(const DP& p, float E, float& mu, float& lam) {
  mu = E / (2.0f * (1.0f + p.nu));
  lam = E * p.nu / ((1.0f + p.nu) * (1.0f - 2.0f * p.nu));
}

// Rotation of the polar decomposition F = R S.  For det F well above zero by
// Newton's iteration R <- (R + R^-T) / 2 (Higham, "Computing the polar
// decomposition -- with applications", 1986), R^-T = cof(R) / det R: it
// converges quadratically, an update of size d leaving an error of d^2 / 2, so
// it stops after an update below 2^-12.  Elastic strains of some per cent take
// three to four rounds of about 35 instructions, where the singular value
// decomposition takes some 600; P2G and P2G^T need nothing else of it.
// Degenerate or inverted F goes through the decomposition (det R = +1).
__device__ __noinline__ void rotation_by_svd(const float* F, float* R) {
  float U[9], V[9], sig[3];
  svd3<float>(F, U, sig, V);
  mat3_bt(U, V, R);
}

__device__ __forceinline__ void cofactor(const float* F, float* C) {
  C[0] = F[4] * F[8] - F[5] * F[7];
  C[1] = F[5] * F[6] - F[3] * F[8];
  C[2] = F[3] * F[7] - F[4] * F[6];
  C[3] = F[2] * F[7] - F[1] * F[8];
  C[4] = F[0] * F[8] - F[2] * F[6];
  C[5] = F[1] * F[6] - F[0] * F[7];
  C[6] = F[1] * F[5] - F[2] * F[4];
  C[7] = F[2] * F[3] - F[0] * F[5];
  C[8] = F[0] * F[4] - F[1] * F[3];
}

// R of F, and cof(F) and J = det F
__device__ __forceinline__ void rotation(const float* F, float* R, float* cof, float& J) {
  cofactor(F, cof);
  J = F[0] * cof[0] + F[1] * cof[1] + F[2] * cof[2];
  bool ok = false;
  if (J > 0.05f) {
    float C[9], det = J;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      R[q] = F[q];
      C[q] = cof[q];
    }
#pragma unroll 1
    for (int it = 0; it < 10; ++it) {
      const float h = 0.5f / det;
      float d2 = 0.f;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const float n = fmaf(h, C[q], 0.5f * R[q]), d = n - R[q];
        R[q] = n;
        d2 = fmaf(d, d, d2);
      }
      if (d2 < 5.9604645e-8f) {  // (2^-12)^2
        ok = true;
        break;
      }
      cofactor(R, C);
      det = R[0] * C[0] + R[1] * C[1] + R[2] * C[2];
    }
  }
  if (!ok) {
    float Ft[9], Rt[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) Ft[q] = F[q];
    rotation_by_svd(Ft, Rt);
#pragma unroll
    for (int q = 0; q < 9; ++q) R[q] = Rt[q];
  }
}

// tau = 2 mu (F - R) F^T + lam J (J - 1) I
__device__ __forceinline__ void fc_stress(const float* F, const float* R, float J, float mu, float lam, float* tau) {
  float D[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) D[q] = F[q] - R[q];
  mat3_bt(D, F, tau);
  const float vol = lam * J * (J - 1.0f);
#pragma unroll
  for (int q = 0; q < 9; ++q) tau[q] = 2.0f * mu * tau[q] + (q % 4 == 0 ? vol : 0.0f);
}

// m(M) with M - M^T = [m]x
__device__ __forceinline__ void axial(const float* M, float* m) {
  m[0] = M[7] - M[5];
  m[1] = M[2] - M[6];
  m[2] = M[3] - M[1];
}

// Adjoint of tau(F; E) for the fixed-corotated model: F_bar += d tau/dF ^T : tb,
// E_bar += <tb, tau> / E (tau is proportional to E at fixed F).  (tau, R,
// cof F and J come from fc_stress and rotation.)
__device__ __forceinline__ void fc_stress_vjp(const float* F, const float* R, const float* cof, float J, float E,
                                              float mu, float lam, const float* tau, const float* tb, float* Fb,
                                              float& Eb) {
  float G[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) G[q] = F[q] - R[q];
  // 2 mu (tb F + tb^T G)
  float t1[9], t2[9];
  mat3(tb, F, t1);
  mat3_at(tb, G, t2);
#pragma unroll
  for (int q = 0; q < 9; ++q) Fb[q] += 2.0f * mu * (t1[q] + t2[q]);
  // lam (2J - 1) tr(tb) cof(F)
  const float kv = lam * (2.0f * J - 1.0f) * (tb[0] + tb[4] + tb[8]);
#pragma unroll
  for (int q = 0; q < 9; ++q) Fb[q] += kv * cof[q];
  // R_bar = -2 mu tb F.  dR = R [w]x with Omega S + S Omega = R^T dF - dF^T R,
  // Omega = [w]x, i.e. K w = m(R^T dF), K = tr(S) I - S; so <R_bar, dR> =
  // m(R^T R_bar) . w = z . m(R^T dF) with K z = m(R^T R_bar), and F_bar += R [z]x.
  // det K = prod (sigma_i + sigma_j).
  float S[9], N[9], m[3];
  mat3_at(R, F, S);
  mat3_at(R, t1, N);
  axial(N, m);
  const float tr = S[0] + S[4] + S[8];
  const float s01 = 0.5f * (S[1] + S[3]), s02 = 0.5f * (S[2] + S[6]), s12 = 0.5f * (S[5] + S[7]);
  const float K[9] = {tr - S[0], -s01, -s02, -s01, tr - S[4], -s12, -s02, -s12, tr - S[8]};
  float C[9];
  cofactor(K, C);
  // (K's eigenvalues are the sigma_i + sigma_j >= 0: at least 1e-6 each, by
  // the sum of their products)
  const float det = fmaxf(K[0] * C[0] + K[1] * C[1] + K[2] * C[2], fmaf(1e-6f, C[0] + C[4] + C[8], 1e-18f));
  const float h = -2.0f * mu / det;
  float z[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) z[i] = h * (C[3 * i] * m[0] + C[3 * i + 1] * m[1] + C[3 * i + 2] * m[2]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Fb[3 * i] += R[3 * i + 1] * z[2] - R[3 * i + 2] * z[1];
    Fb[3 * i + 1] += R[3 * i + 2] * z[0] - R[3 * i] * z[2];
    Fb[3 * i + 2] += R[3 * i] * z[1] - R[3 * i + 1] * z[0];
  }
  float dot = 0.f;
#pragma unroll
  for (int q = 0; q < 9; ++q) dot += tb[q] * tau[q];
  Eb += E > 0.f ? dot / E : 0.0f;
}

// --------------------------------------------------------------- forward
//
// One particle per thread, 64 threads per CTA, as many CTAs as particles
// need: the kernels are bound by the latency of their loads and of the
// decomposition's serial chain, so a small body (32,768 particles) should
// still give every scheduler several CTAs.  Measured on the differentiable
// cube (262,144 particles on 128^3), against 128-thread CTAs in a fixed grid
// stride with scalar atomics on dense grids that were cleared and swept whole:
// P2G 75 -> 30 us, grid 28 (with its clears) -> 5, G2P 25 -> 12, G2P^T 78 ->
// 35, P2G^T 71 -> 34 (its decomposition taken once, no local memory); a
// forward step 140 -> 62 us, its adjoint 302 -> 129 us (45 and 103 with the
// overlapped launches, the polar iteration and the late zeroing of k_fwd_grid).

constexpr int kDT = 64;

// A = (m B - dt V0 tau) D^-1 / dx, so that the affine momentum at a node is
// A times its offset in cells.
__device__ __forceinline__ void affine(const DP& p, const DS& s, const float* B, const float* tau, float* M, float* A) {
#pragma unroll
  for (int q = 0; q < 9; ++q) M[q] = p.mass * B[q] - p.dt * p.V0 * tau[q];
  mat3(M, s.Di, A);
#pragma unroll
  for (int q = 0; q < 9; ++q) A[q] *= p.inv_dx;
}

__global__ void __launch_bounds__(kDT, 10) k_fwd_p2g(DP p, DGrid D, const float* x, const float* v, const float* B,
                                                 const float* F, const float* E) {
  grid_begin();
  __shared__ float rows[kDT / 32][32 * 24];
  float* const sm = rows[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const size_t p0 = (size_t)blockIdx.x * kDT + (threadIdx.x - lane);
  if (p0 >= (size_t)p.n) return;
  const int cnt = (int)min((size_t)32, (size_t)p.n - p0);
  float xi[3], vi[3], Fi[9], Bi[9];
  fetch_rows<3>(x, p0, cnt, sm);
  fetch_rows<3>(v, p0, cnt, sm + 3 * 32);
  fetch_rows<9>(F, p0, cnt, sm + 6 * 32);
  fetch_rows<9>(B, p0, cnt, sm + 15 * 32);
  __syncwarp();
  take_row<3>(sm, xi);
  take_row<3>(sm + 3 * 32, vi);
  take_row<9>(sm + 6 * 32, Fi);
  take_row<9>(sm + 15 * 32, Bi);
  DS s;
  s.set(p, xi[0], xi[1], xi[2]);
  const bool on = lane < cnt && nodes_in_range(p, s);
  list_blocks(p, D, s, on);
  if (!on) {
    if (lane < cnt) atomicOr(D.err, 1u);
    return;
  }
  float tau[9], R[9], cof[9], J, mu, lam, M[9], A[9];
  lame(p, E[p0 + lane], mu, lam);
  rotation(Fi, R, cof, J);
  fc_stress(Fi, R, J, mu, lam, tau);
  affine(p, s, Bi, tau, M, A);
  const float mv[3] = {p.mass * vi[0], p.mass * vi[1], p.mass * vi[2]};
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const DOff o(p, s, g);
    float4* const G = D.G + g * grid_size(p);
#pragma unroll
    for (int z = 0; z < 2; ++z)
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        const float wyz = s.W[g][1][y] * s.W[g][2][z];
        const float dy = (float)y - s.f[g][1], dz = (float)z - s.f[g][2];
        float e[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) e[c] = mv[c] + A[c * 3 + 1] * dy + A[c * 3 + 2] * dz;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float w = s.W[g][0][k] * wyz, d = (float)k - s.f[g][0];
          red_add4(&G[o.o[2][z] + o.o[1][y] + o.o[0][k]], w * p.mass, w * (e[0] + A[0] * d), w * (e[1] + A[3] * d),
                   w * (e[2] + A[6] * d));
        }
      }
  }
}

// Whether a node of block (bx, by, bz) of grid g lies in a sticky wall.
__device__ __forceinline__ bool wall(const DP& p, int g, int ix, int iy, int iz) {
  const float off = g == 0 ? 0.25f : -0.25f;
  const float hi = (float)p.res - p.bc;
  const float a = ix + off, b = iy + off, c = iz + off;
  return a < p.bc || b < p.bc || c < p.bc || a > hi || b > hi || c > hi;
}

// The nodes of one listed block, both grids: thread t has node t & 63 of grid
// t >> 6.  Calls fn(index, in a wall).
template <typename Fn>
__device__ __forceinline__ void for_block_nodes(const DP& p, const DGrid& D, Fn&& fn) {
  const uint32_t n = *D.count;
  const int g = threadIdx.x >> 6, l = threadIdx.x & 63;
  for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) {
    const uint32_t b = D.list[i];
    const int bx = (int)(b % (uint32_t)p.nb), by = (int)((b / (uint32_t)p.nb) % (uint32_t)p.nb),
              bz = (int)(b / ((uint32_t)p.nb * (uint32_t)p.nb));
    if (threadIdx.x == 0) D.flag[b] = 0u;
    fn(g * grid_size(p) + (size_t)b * 64u + l, wall(p, g, bx * 4 + (l & 3), by * 4 + ((l >> 2) & 3), bz * 4 + (l >> 4)));
  }
}

// v~ = P / m + dt g (m > 0, off the walls).  The forward step returns the
// accumulators to zero; the adjoint keeps them for its own grid kernel and
// zeroes the velocity adjoints that G2P^T adds into.
// Here and in k_bwd_grid a node is read past L1 (it was last touched by
// reductions in L2) and zeroed after the store that needs its value: a store
// behind a pending load of the same address holds up the load-store unit.
// 100,000 particles spread over 36,000 blocks (compulsory: 220 MB and 295 MB),
// zeroed before and after: forward grid 113 -> 23 us, adjoint grid 116 -> 31; the
// differentiable cube's 800 blocks 5.8 -> 3.6.
template <bool ADJ>
__global__ void __launch_bounds__(128) k_fwd_grid(DP p, DGrid D) {
  grid_begin();
  for_block_nodes(p, D, [&](size_t q, bool w) {
    const float4 a = __ldcg(&D.G[q]), zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 o = zero;
    if (a.x > 0.f && !w) {
      o.x = a.y / a.x + p.dt * p.gx;
      o.y = a.z / a.x + p.dt * p.gy;
      o.z = a.w / a.x + p.dt * p.gz;
    }
    D.V[q] = o;
    if (ADJ)
      D.A[q] = zero;
    else
      D.G[q] = zero;
  });
}

__global__ void __launch_bounds__(kDT) k_fwd_g2p(DP p, DGrid D, const float* x, const float* F, float* x1, float* v1,
                                                 float* B1, float* F1) {
  grid_begin();
  __shared__ float rows[kDT / 32][32 * 12];
  float* const sm = rows[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  if (blockIdx.x == 0 && threadIdx.x == 0) *D.count = 0u;  // the list's last reader is done
  const size_t p0 = (size_t)blockIdx.x * kDT + (threadIdx.x - lane);
  if (p0 >= (size_t)p.n) return;
  const int cnt = (int)min((size_t)32, (size_t)p.n - p0);
  float xi[3], Fi[9];
  fetch_rows<3>(x, p0, cnt, sm);
  fetch_rows<9>(F, p0, cnt, sm + 3 * 32);
  __syncwarp();
  take_row<3>(sm, xi);
  take_row<9>(sm + 3 * 32, Fi);
  DS s;
  s.set(p, xi[0], xi[1], xi[2]);
  float vv[3] = {0.f, 0.f, 0.f}, Bh[9] = {0.f}, Fn[9], C[9];
  if (lane < cnt && nodes_in_range(p, s)) {
#pragma unroll
    for (int g = 0; g < 2; ++g) gather_moments(D.V + g * grid_size(p), s, DOff(p, s, g), g, 0.5f, vv, Bh);
    mat3(Bh, s.Di, C);
#pragma unroll
    for (int q = 0; q < 9; ++q) C[q] = (q % 4 == 0 ? 1.0f : 0.0f) + p.dt * p.inv_dx * C[q];
    mat3(C, Fi, Fn);
#pragma unroll
    for (int a = 0; a < 3; ++a) xi[a] += p.dt * vv[a];
#pragma unroll
    for (int q = 0; q < 9; ++q) Bh[q] *= p.dx;
  } else {  // reported by ckmpm_diff_sync; the particle is left in place
    if (lane < cnt) atomicOr(D.err, 1u);
#pragma unroll
    for (int q = 0; q < 9; ++q) Fn[q] = Fi[q];
  }
  store_rows<3>(x1, p0, cnt, sm, xi);
  store_rows<3>(v1, p0, cnt, sm, vv);
  store_rows<9>(B1, p0, cnt, sm, Bh);
  store_rows<9>(F1, p0, cnt, sm, Fn);
}

// --------------------------------------------------------------- adjoint

// The weight-derivative part of x_bar: sum over a grid's nodes of q dw/dx with
// q a scalar per node, q(z, y, k): x, y and z reduced in turn (dW of node 0 is
// minus that of node 1).
struct WeightAdjoint {
  float Q[2], Qx[2], Qy[2];  // of the current z: rows y reduced over x
  __device__ __forceinline__ void row(const DS& s, int g, int y, float q0, float q1) {
    Q[y] = s.W[g][0][0] * q0 + s.W[g][0][1] * q1;
    Qx[y] = s.dW[g][0] * (q1 - q0);
  }
  float T[2];
  __device__ __forceinline__ void plane(const DS& s, int g, int z, float* xb) {
    const float wz = s.W[g][2][z];
    xb[0] += wz * (s.W[g][1][0] * Qx[0] + s.W[g][1][1] * Qx[1]);
    xb[1] += wz * (s.dW[g][1] * (Q[1] - Q[0]));
    T[z] = s.W[g][1][0] * Q[0] + s.W[g][1][1] * Q[1];
    if (z == 1) xb[2] += s.dW[g][2] * (T[1] - T[0]);
  }
};

// G2P^T: given the step's output adjoints, write x_bar and F_bar (partial) of
// the step inputs and scatter the grid-velocity adjoint.
__global__ void __launch_bounds__(kDT, 6) k_bwd_g2p(DP p, DGrid D, const float* x, const float* F, const float* gx1,
                                                 const float* gv1, const float* gB1, const float* gF1, float* gx,
                                                 float* gF) {
  grid_begin();
  __shared__ float rows[kDT / 32][32 * 36];
  float* const sm = rows[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const size_t p0 = (size_t)blockIdx.x * kDT + (threadIdx.x - lane);
  if (p0 >= (size_t)p.n) return;
  const int cnt = (int)min((size_t)32, (size_t)p.n - p0);
  float xi[3], Fi[9], xb[3], vb[3], Bhb[9], Fb1[9], Fbo[9];
  fetch_rows<3>(x, p0, cnt, sm);
  fetch_rows<3>(gx1, p0, cnt, sm + 3 * 32);
  fetch_rows<3>(gv1, p0, cnt, sm + 6 * 32);
  fetch_rows<9>(F, p0, cnt, sm + 9 * 32);
  fetch_rows<9>(gB1, p0, cnt, sm + 18 * 32);
  fetch_rows<9>(gF1, p0, cnt, sm + 27 * 32);
  __syncwarp();
  take_row<3>(sm, xi);
  take_row<3>(sm + 3 * 32, xb);
  take_row<3>(sm + 6 * 32, vb);
  take_row<9>(sm + 9 * 32, Fi);
  take_row<9>(sm + 18 * 32, Bhb);
  take_row<9>(sm + 27 * 32, Fb1);
  DS s;
  s.set(p, xi[0], xi[1], xi[2]);
  if (lane < cnt && nodes_in_range(p, s)) {
    // the forward gather again
    float vv[3] = {0.f, 0.f, 0.f}, Bh[9] = {0.f};
#pragma unroll
    for (int g = 0; g < 2; ++g) gather_moments(D.V + g * grid_size(p), s, DOff(p, s, g), g, 0.5f, vv, Bh);
#pragma unroll
    for (int a = 0; a < 3; ++a) vb[a] += p.dt * xb[a];
    // F' = G F, G = I + k Bh Di, k = dt/dx
    const float k = p.dt * p.inv_dx;
    float C[9], Gb[9], Dib[9];
    mat3(Bh, s.Di, C);
#pragma unroll
    for (int q = 0; q < 9; ++q) C[q] = (q % 4 == 0 ? 1.0f : 0.0f) + k * C[q];
    mat3_at(C, Fb1, Fbo);   // G^T F'_bar
    mat3_bt(Fb1, Fi, Gb);   // F'_bar F^T
    // C = Bh Di: Bh_bar = k Gb Di^T, Di_bar = k Bh^T Gb ; plus B' = dx Bh
    float t[9];
    mat3_bt(Gb, s.Di, t);
#pragma unroll
    for (int q = 0; q < 9; ++q) Bhb[q] = k * t[q] + p.dx * Bhb[q];
    mat3_at(Bh, Gb, Dib);
#pragma unroll
    for (int q = 0; q < 9; ++q) Dib[q] *= k;
    // gather adjoints: v = 1/2 sum w v~, Bh = 1/2 sum w v~ d^T.  A node's
    // offset adjoint is w Bh_bar^T v~, which sums to Bh_bar^T v over the nodes.
#pragma unroll
    for (int b = 0; b < 3; ++b) xb[b] -= p.inv_dx * (Bhb[b] * vv[0] + Bhb[3 + b] * vv[1] + Bhb[6 + b] * vv[2]);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const DOff o(p, s, g);
      const float4* const V = D.V + g * grid_size(p);
      float4* const A = D.A + g * grid_size(p);
      WeightAdjoint wa;
#pragma unroll
      for (int z = 0; z < 2; ++z) {
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const float wyz = 0.5f * s.W[g][1][y] * s.W[g][2][z];
          const float dy = (float)y - s.f[g][1], dz = (float)z - s.f[g][2];
          float e[3], q[2];
#pragma unroll
          for (int a = 0; a < 3; ++a) e[a] = vb[a] + Bhb[a * 3 + 1] * dy + Bhb[a * 3 + 2] * dz;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float w = s.W[g][0][j] * wyz, d = (float)j - s.f[g][0];
            const float q0 = e[0] + Bhb[0] * d, q1 = e[1] + Bhb[3] * d, q2 = e[2] + Bhb[6] * d;
            const uint32_t ni = o.o[2][z] + o.o[1][y] + o.o[0][j];
            red_add4(&A[ni], w * q0, w * q1, w * q2, 0.f);
            const float4 c = V[ni];
            q[j] = 0.5f * (c.x * q0 + c.y * q1 + c.z * q2);
          }
          wa.row(s, g, y, q[0], q[1]);
        }
        wa.plane(s, g, z, xb);
      }
    }
    s.dinv_to_x(Dib, xb);
  } else {
#pragma unroll
    for (int q = 0; q < 9; ++q) Fbo[q] = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) xb[a] = 0.f;
  }
  store_rows<3>(gx, p0, cnt, sm, xb);
  store_rows<9>(gF, p0, cnt, sm, Fbo);
}

// grid^T: v~ = (P/m + dt g) on nodes with mass off the walls; A becomes
// (p_bar, m_bar) and the accumulators return to zero.
__global__ void __launch_bounds__(128) k_bwd_grid(DP p, DGrid D) {
  grid_begin();
  for_block_nodes(p, D, [&](size_t q, bool w) {
    const float4 a = __ldcg(&D.G[q]);
    const float4 b = __ldcg(&D.A[q]);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.x > 0.f && !w) {
      const float im = 1.0f / a.x;
      o.x = b.x * im;
      o.y = b.y * im;
      o.z = b.z * im;
      o.w = -(o.x * a.y + o.y * a.z + o.z * a.w) * im;
    }
    D.A[q] = o;
    D.G[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  });
}

// P2G^T: gather the grid adjoints back to the particles.
__global__ void __launch_bounds__(kDT, 6) k_bwd_p2g(DP p, DGrid D, const float* x, const float* v, const float* B,
                                                 const float* F, const float* E, float* gx, float* gv, float* gB,
                                                 float* gF, float* gE) {
  grid_begin();
  __shared__ float rows[kDT / 32][32 * 36];
  float* const sm = rows[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  if (blockIdx.x == 0 && threadIdx.x == 0) *D.count = 0u;  // the list's last reader is done
  const size_t p0 = (size_t)blockIdx.x * kDT + (threadIdx.x - lane);
  if (p0 >= (size_t)p.n) return;
  const int cnt = (int)min((size_t)32, (size_t)p.n - p0);
  float xi[3], vi[3], Fi[9], Bi[9], xb[3], Fb[9], Mb[9], vb[3] = {0.f, 0.f, 0.f};
  fetch_rows<3>(x, p0, cnt, sm);
  fetch_rows<3>(v, p0, cnt, sm + 3 * 32);
  fetch_rows<9>(F, p0, cnt, sm + 6 * 32);
  fetch_rows<9>(B, p0, cnt, sm + 15 * 32);
  fetch_rows<3>(gx, p0, cnt, sm + 24 * 32);
  fetch_rows<9>(gF, p0, cnt, sm + 27 * 32);
  __syncwarp();
  take_row<3>(sm, xi);
  take_row<3>(sm + 3 * 32, vi);
  take_row<9>(sm + 6 * 32, Fi);
  take_row<9>(sm + 15 * 32, Bi);
  take_row<3>(sm + 24 * 32, xb);
  take_row<9>(sm + 27 * 32, Fb);
  DS s;
  s.set(p, xi[0], xi[1], xi[2]);
  if (lane < cnt && nodes_in_range(p, s)) {
    float tau[9], R[9], cof[9], J, mu, lam, M[9], A[9];
    const float Ei = E[p0 + lane];
    lame(p, Ei, mu, lam);
    rotation(Fi, R, cof, J);
    fc_stress(Fi, R, J, mu, lam, tau);
    affine(p, s, Bi, tau, M, A);
    const float mv[3] = {p.mass * vi[0], p.mass * vi[1], p.mass * vi[2]};
    // S = sum w p_bar, Ab = sum w p_bar d^T; a node's contribution
    // c = m v + A d has x_bar through its weight (p_bar . c + m m_bar) and
    // through d, whose adjoint w A^T p_bar sums to A^T S
    float S[3] = {0.f, 0.f, 0.f}, Ab[9] = {0.f};
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const DOff o(p, s, g);
      const float4* const Pb = D.A + g * grid_size(p);
      gather_moments(Pb, s, o, g, 1.0f, S, Ab);
      WeightAdjoint wa;
#pragma unroll
      for (int z = 0; z < 2; ++z) {
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const float dy = (float)y - s.f[g][1], dz = (float)z - s.f[g][2];
          float e[3], q[2];
#pragma unroll
          for (int a = 0; a < 3; ++a) e[a] = mv[a] + A[a * 3 + 1] * dy + A[a * 3 + 2] * dz;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float d = (float)j - s.f[g][0];
            const float4 b = Pb[o.o[2][z] + o.o[1][y] + o.o[0][j]];
            q[j] = p.mass * b.w + b.x * (e[0] + A[0] * d) + b.y * (e[1] + A[3] * d) + b.z * (e[2] + A[6] * d);
          }
          wa.row(s, g, y, q[0], q[1]);
        }
        wa.plane(s, g, z, xb);
      }
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) xb[b] -= p.inv_dx * (A[b] * S[0] + A[3 + b] * S[1] + A[6 + b] * S[2]);
    // A = M Di / dx: M_bar = Ab Di^T / dx ; Di_bar = M^T Ab / dx
    float Dib[9];
    mat3_bt(Ab, s.Di, Mb);
    mat3_at(M, Ab, Dib);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      Mb[q] *= p.inv_dx;
      Dib[q] *= p.inv_dx;
    }
    s.dinv_to_x(Dib, xb);
    // M = m B - dt V0 tau
    float tb[9], Eb = 0.f;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      tb[q] = -p.dt * p.V0 * Mb[q];
      Mb[q] *= p.mass;
    }
    fc_stress_vjp(Fi, R, cof, J, Ei, mu, lam, tau, tb, Fb, Eb);
#pragma unroll
    for (int a = 0; a < 3; ++a) vb[a] = p.mass * S[a];
    gE[p0 + lane] += Eb;
  } else {
#pragma unroll
    for (int q = 0; q < 9; ++q) Mb[q] = 0.f;
  }
  store_rows<3>(gx, p0, cnt, sm, xb);
  store_rows<3>(gv, p0, cnt, sm, vb);
  store_rows<9>(gB, p0, cnt, sm, Mb);
  store_rows<9>(gF, p0, cnt, sm, Fb);
}

}  // namespace ckd

struct ckmpm_diff {
  ckd::DP p{};
  ckd::DGrid g{};
  cudaStream_t stream = nullptr;
  int grid_ctas = 1024;  // grid kernels (a loop over the listed blocks)
  int blocks = 1;        // particle kernels
};

extern "C" {

ckmpm_status ckmpm_diff_create(const ckmpm_scene* sc, void* stream, ckmpm_diff** out) {
  if (!out) return CKMPM_EINVAL;
  *out = nullptr;
  if (!sc || sc->n < 1 || sc->res < 4 || sc->res > 1024 || !(sc->dx > 0) || !(sc->dt > 0) || sc->ppc < 1 ||
      !sc->materials || sc->n_materials < 1 || sc->materials[0].model != CKMPM_FIXED_COROTATED ||
      !(sc->materials[0].rho > 0) || !(sc->materials[0].nu > -1.0 && sc->materials[0].nu < 0.5))
    return CKMPM_EINVAL;
  ckmpm_diff* d = new (std::nothrow) ckmpm_diff();
  if (!d) return CKMPM_ENOMEM;
  ckd::DP& p = d->p;
  p.dx = (float)sc->dx;
  p.inv_dx = (float)(1.0 / sc->dx);
  p.dt = (float)sc->dt;
  p.V0 = (float)(sc->dx * sc->dx * sc->dx / sc->ppc);
  p.mass = (float)(sc->materials[0].rho * sc->dx * sc->dx * sc->dx / sc->ppc);
  p.nu = (float)sc->materials[0].nu;
  p.gx = (float)sc->gravity[0];
  p.gy = (float)sc->gravity[1];
  p.gz = (float)sc->gravity[2];
  p.bc = (float)sc->bc_cells;
  p.res = sc->res;
  p.nb = (sc->res + 1 + 3) / 4;
  p.n = (int)sc->n;
  d->stream = (cudaStream_t)stream;
  const size_t nblk = (size_t)p.nb * p.nb * p.nb, bytes = 2 * nblk * 64 * sizeof(float4);
  ckd::DGrid& g = d->g;
  bool ok = cudaMalloc(&g.G, bytes) == cudaSuccess && cudaMalloc(&g.V, bytes) == cudaSuccess &&
            cudaMalloc(&g.A, bytes) == cudaSuccess && cudaMalloc(&g.flag, nblk * 4) == cudaSuccess &&
            cudaMalloc(&g.list, nblk * 4) == cudaSuccess && cudaMalloc(&g.count, 4) == cudaSuccess &&
            cudaMalloc(&g.err, 4) == cudaSuccess;
  // on the object's stream: the first call is ordered behind them
  if (!ok || cudaMemsetAsync(g.G, 0, bytes, d->stream) != cudaSuccess ||
      cudaMemsetAsync(g.flag, 0, nblk * 4, d->stream) != cudaSuccess ||
      cudaMemsetAsync(g.count, 0, 4, d->stream) != cudaSuccess ||
      cudaMemsetAsync(g.err, 0, 4, d->stream) != cudaSuccess) {
    cudaGetLastError();
    ckmpm_diff_destroy(d);
    return CKMPM_ENOMEM;
  }
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  d->grid_ctas = sms * 16;
  d->blocks = (int)(((int64_t)p.n + ckd::kDT - 1) / ckd::kDT);
  *out = d;
  return CKMPM_OK;
}

ckmpm_status ckmpm_diff_step(ckmpm_diff* d, const float* x, const float* v, const float* B, const float* F,
                             const float* E, float* x1, float* v1, float* B1, float* F1) {
  if (!d || !x || !v || !B || !F || !E || !x1 || !v1 || !B1 || !F1) return CKMPM_EINVAL;
  ckd::launch_step(ckd::k_fwd_p2g, d->blocks, ckd::kDT, d->stream, d->p, d->g, x, v, B, F, E);
  ckd::launch_step(ckd::k_fwd_grid<false>, d->grid_ctas, 128, d->stream, d->p, d->g);
  ckd::launch_step(ckd::k_fwd_g2p, d->blocks, ckd::kDT, d->stream, d->p, d->g, x, F, x1, v1, B1, F1);
  return cudaGetLastError() == cudaSuccess ? CKMPM_OK : CKMPM_ECUDA;
}

ckmpm_status ckmpm_diff_step_backward(ckmpm_diff* d, const float* x, const float* v, const float* B, const float* F,
                                      const float* E, const float* gx1, const float* gv1, const float* gB1,
                                      const float* gF1, float* gx, float* gv, float* gB, float* gF, float* gE) {
  if (!d || !x || !v || !B || !F || !E || !gx1 || !gv1 || !gB1 || !gF1 || !gx || !gv || !gB || !gF || !gE)
    return CKMPM_EINVAL;
  ckd::launch_step(ckd::k_fwd_p2g, d->blocks, ckd::kDT, d->stream, d->p, d->g, x, v, B, F, E);
  ckd::launch_step(ckd::k_fwd_grid<true>, d->grid_ctas, 128, d->stream, d->p, d->g);
  ckd::launch_step(ckd::k_bwd_g2p, d->blocks, ckd::kDT, d->stream, d->p, d->g, x, F, gx1, gv1, gB1, gF1, gx, gF);
  ckd::launch_step(ckd::k_bwd_grid, d->grid_ctas, 128, d->stream, d->p, d->g);
  ckd::launch_step(ckd::k_bwd_p2g, d->blocks, ckd::kDT, d->stream, d->p, d->g, x, v, B, F, E, gx, gv, gB, gF, gE);
  return cudaGetLastError() == cudaSuccess ? CKMPM_OK : CKMPM_ECUDA;
}

ckmpm_status ckmpm_diff_sync(ckmpm_diff* d) {
  if (!d) return CKMPM_EINVAL;
  if (cudaStreamSynchronize(d->stream) != cudaSuccess) return CKMPM_ECUDA;
  uint32_t e = 0;
  if (cudaMemcpy(&e, d->g.err, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return CKMPM_ECUDA;
  return e ? CKMPM_EDOMAIN : CKMPM_OK;
}

ckmpm_status ckmpm_diff_destroy(ckmpm_diff* d) {
  if (!d) return CKMPM_OK;
  if (d->stream) cudaStreamSynchronize(d->stream);
  cudaFree(d->g.G);
  cudaFree(d->g.V);
  cudaFree(d->g.A);
  cudaFree(d->g.flag);
  cudaFree(d->g.list);
  cudaFree(d->g.count);
  cudaFree(d->g.err);
  cudaGetLastError();
  delete d;
  return CKMPM_OK;
}

}  // extern "C"
