// P2G, grid update and fused G2P + constitutive kernels of the CK-MPM step,
// for the compact kernel on the dual grid (KIND 0) and the quadratic
// B-spline comparison path (KIND 1).
//
// One CTA works on one particle block (4x4x4 cells of the reference grid G-,
// Sec. 5.1) at a time and loops over the block list (persistent grid-stride
// launch over all resident scenes).  The nodes that the block's particles can
// touch are staged in shared memory:
//   CK:  G- nodes [4P, 4P+4]^3 (125) and G+ nodes [4P, 4P+5]^3 (216) = 341
//   quadratic: nodes [4P, 4P+5]^3 = 216
// P2G accumulates there with shared-memory atomics and flushes each touched
// node once with a 16-byte global atomic; G2P gathers from the staged copy.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "launch.h"
#include "pack.cuh"
#include "scan.cuh"
#include "svd3.cuh"

namespace ck {

constexpr float kInv2Pi = 0.15915494309189535f;

// Asynchronous global -> shared copies: a CTA issues the gathers of a whole
// chunk of particles before it waits for any.  The 16-byte copies stream
// through L2 only (.cg), so that the particle stream does not evict the small
// tables every particle reads through L1 (materials, scenes, block lists).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N of this thread's committed groups are still in flight
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Material tables of up to this many entries are staged in shared memory by
// the transfer kernels (one copy per CTA).
constexpr int kSmemMats = 8;

// The reduction of sin(2 pi f) and cos(2 pi f), f in [0, 1): t = f - rint(f) in
// [-1/2, 1/2], then |t| > 1/4 folds by t -> sign(t)/2 - t (both steps exact in
// float), which keeps the sine and flips the cosine's sign.
__device__ __forceinline__ float fold_2pi(float t) {
  const float h = copysignf(0.5f, t) - t;
  return fabsf(t) > 0.25f ? h : t;
}

// sin(2 pi f) per axis, f in [0, 1): the Taylor series of sin x at x = 2 pi t,
// |x| <= pi/2, through x^11: coefficients (-1)^k (2 pi)^(2k+1) / (2k+1)!,
// truncation error below (pi/2)^13 / 13! = 5.7e-8, about 1.6e-7 after float
// rounding.
__device__ __forceinline__ V3 sin_2pi(const V3& f) {
  V3 t = f - V3{pk(rintf(f.p.x), rintf(f.p.y)), rintf(f.z)};
  t = {pk(fold_2pi(t.p.x), fold_2pi(t.p.y)), fold_2pi(t.z)};
  const V3 t2 = t * t;
  V3 p = v3(-15.094642576822984f);
  p = fma3(p, t2, v3(42.058693944897634f));
  p = fma3(p, t2, v3(-76.70585975306136f));
  p = fma3(p, t2, v3(81.60524927607504f));
  p = fma3(p, t2, v3(-41.341702240399755f));
  p = fma3(p, t2, v3(6.283185307179586f));
  return t * p;
}

// cos(2 pi f) for f in [0, 1): the Taylor series of cos x at x = 2 pi t,
// |x| <= pi/2, through x^12: coefficients (-1)^k (2 pi)^(2k) / (2k)!,
// truncation error below (pi/2)^14 / 14! = 6.4e-9.
__device__ __forceinline__ float cos_2pi(float f) {
  float t = f - rintf(f);
  const bool fold = fabsf(t) > 0.25f;
  t = fold_2pi(t);
  const float t2 = t * t;
  float p = 7.903536371318465f;
  p = fmaf(p, t2, -26.426256783374388f);
  p = fmaf(p, t2, 60.24464137187664f);
  p = fmaf(p, t2, -85.45681720669371f);
  p = fmaf(p, t2, 64.93939402266828f);
  p = fmaf(p, t2, -19.739208802178716f);
  p = fmaf(p, t2, 1.0f);
  return fold ? -p : p;
}
// per axis: x and y packed, by the same steps
__device__ __forceinline__ V3 cos_2pi(const V3& f) {
  const f2 t = add2(f.p, pk(-rintf(f.p.x), -rintf(f.p.y)));
  const bool fx = fabsf(t.x) > 0.25f, fy = fabsf(t.y) > 0.25f;
  const f2 u = pk(fold_2pi(t.x), fold_2pi(t.y)), t2 = mul2(u, u);
  f2 p = dup(7.903536371318465f);
  p = fma2(p, t2, dup(-26.426256783374388f));
  p = fma2(p, t2, dup(60.24464137187664f));
  p = fma2(p, t2, dup(-85.45681720669371f));
  p = fma2(p, t2, dup(64.93939402266828f));
  p = fma2(p, t2, dup(-19.739208802178716f));
  p = fma2(p, t2, dup(1.0f));
  return {pk(fx ? -p.x : p.x, fy ? -p.y : p.y), cos_2pi(f.z)};
}

// 1/x for a normal float x: the hardware approximation refined by one
// Newton-Raphson step e = 1 - x y, y <- y + y e (the classical iteration for
// the reciprocal; the error after one step is about the square of the
// approximation's, below one ulp).  No special-case branches: callers pass
// values bounded away from 0 and infinity.
__device__ __forceinline__ float rcp_nr(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  const float e = fmaf(-x, y, 1.0f);
  return fmaf(y, e, y);
}
__device__ __forceinline__ V3 rcp_nr(const V3& x) {
  V3 y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.p.x) : "f"(x.p.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.p.y) : "f"(x.p.y));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.z) : "f"(x.z));
  return fma3(y, fma3(neg3(x), y, v3(1.0f)), y);
}

template <int KIND>
struct Geo;
template <>
struct Geo<0> {
  static constexpr int NG = 2;
  static constexpr int N = 2;  // nodes per axis of a stencil
  static constexpr int E0 = 5;
  static constexpr int N0 = 125;
  static constexpr int NS = 341;
};
template <>
struct Geo<1> {
  static constexpr int NG = 1;
  static constexpr int N = 3;
  static constexpr int E0 = 6;
  static constexpr int N0 = 216;
  static constexpr int NS = 216;
};

// staged index -> (slot, local node coordinates)
template <int KIND>
__device__ __forceinline__ void staged_coords(int j, int& slot, int& lx, int& ly, int& lz) {
  constexpr int E0 = Geo<KIND>::E0;
  if (j < Geo<KIND>::N0) {
    slot = 0;
    lx = j % E0;
    ly = (j / E0) % E0;
    lz = j / (E0 * E0);
  } else {
    j -= Geo<KIND>::N0;
    slot = 1;
    lx = j % 6;
    ly = (j / 6) % 6;
    lz = j / 36;
  }
}

// Pool index of a staged node (grid g, local coordinates relative to the
// particle block's origin 4P) from the pool slots of the 2x2x2 grid blocks
// the particle block touches; -1 if that block has no slot (pool overflow).
template <int KIND>
__device__ __forceinline__ long long pool_index(const uint32_t* bslot, int g, int lx, int ly, int lz) {
  uint32_t sl = bslot[((lz >> 2) * 2 + (ly >> 2)) * 2 + (lx >> 2)];
  if (sl == CK_NO_SLOT) return -1;
  int l = ((lz & 3) * 4 + (ly & 3)) * 4 + (lx & 3);
  return ((long long)sl * Geo<KIND>::NG + g) * kBlockNodes + l;
}

// Slots of the 2x2x2 grid blocks touched by particle block (bx, by, bz).
__device__ __forceinline__ void load_block_slots(const StepView& v, const SceneDev& s, int ox, int oy, int oz,
                                                 uint32_t* bslot) {
  if (threadIdx.x < 8) {
    int t = threadIdx.x;
    int bx = (ox >> 2) + (t & 1), by = (oy >> 2) + ((t >> 1) & 1), bz = (oz >> 2) + (t >> 2);
    bslot[t] = v.table[s.table_base + ((long long)bz * s.nb + by) * s.nb + bx];
  }
}

// ------------------------------------------------------------------ stencils

// Weights, node offsets (x_i - x_p in cells) and D^-1 (cells^-2) of one
// particle, per axis in a V3, computed from the fractions where they are used
// (a kernel holds one grid's weights at a time).  CK: K1 weights on both grids from one sine per
// axis (sin 2 pi f- = -sin 2 pi f+), D = Lambda + s s^T with the closed form
// Lambda_a = (m2(f+) + m2(f-))/2 - s_a^2, s_a = sin(2 pi f+_a)/(2 pi),
// inverted by Sherman-Morrison.  Quadratic: B-spline weights, D^-1 = 4 I.
template <int KIND>
struct Sten;

template <>
struct Sten<0> {
  int r[2][3];     // base node of each grid relative to the block origin
  V3 f[2];         // fractions on G- and G+
  V3 sg;           // sin(2 pi f+) / (2 pi)
  V3 c;            // kernel-gradient transfers: cos(2 pi f+) (set_grad)
  __device__ __forceinline__ bool set(float ux, float uy, float uz, int ox, int oy, int oz) {
    const int o[3] = {ox, oy, oz};
    bool ok = true;
    const V3 t = V3{pk(ux, uy), uz} + v3(0.25f);
    const float fb[3] = {floorf(t.p.x), floorf(t.p.y), floorf(t.z)};
    f[1] = t - V3{pk(fb[0], fb[1]), fb[2]};
    const float fp[3] = {f[1].p.x, f[1].p.y, f[1].z};
    float sh[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // Cell<0>: b- = b+ or b+ - 1, f- = f+ -+ 1/2
      const int bp = (int)fb[a];
      const bool up = fp[a] >= 0.5f;
      const int bm = up ? bp : bp - 1;
      sh[a] = up ? -0.5f : 0.5f;
      r[0][a] = bm - o[a];
      r[1][a] = bp - o[a];
      ok = ok && (unsigned)r[0][a] <= 3u;  // then the G+ base, r[0][a] or r[0][a] + 1, is in [0, 4]
    }
    f[0] = f[1] + V3{pk(sh[0], sh[1]), sh[2]};
    sg = kInv2Pi * sin_2pi(f[1]);
    return ok;
  }
  // K1 weights: 1 - f+ + s and f+ - s on G+, with -s on G-
  __device__ __forceinline__ V3 w(int g, int n) const {
    const V3 h = n == 0 ? v3(1.0f) - f[g] : f[g];
    return (g == 1) == (n == 0) ? h + sg : h - sg;
  }
  __device__ __forceinline__ V3 d(int g, int n) const { return n == 0 ? neg3(f[g]) : v3(1.0f) - f[g]; }
  // K1'(x) = sgn(x) (cos(2 pi |x|) - 1) at the node offsets d = -f, 1 - f:
  // with c = cos(2 pi f+), 1 - c and c - 1 on G+; cos(2 pi f-) = -c, so
  // 1 + c and -1 - c on G-.  Each pair sums to 0 (the weights sum to 1).
  __device__ __forceinline__ void set_grad() { c = cos_2pi(f[1]); }
  __device__ __forceinline__ V3 k(int g, int n) const {
    const V3 h = g == 1 ? v3(1.0f) - c : v3(1.0f) + c;
    return n == 0 ? h : neg3(h);
  }
  // D^-1 = diag(li) - den y y^T (cells^-2)
  __device__ __forceinline__ void dinv(V3& li, V3& y, float& den) const {
    const V3 one = v3(1.0f);
    const V3 m2p = fma3(f[1], one - f[1], neg3(sg * fma3(-2.0f, f[1], one)));
    const V3 m2m = fma3(f[0], one - f[0], sg * fma3(-2.0f, f[0], one));
    const V3 lam = fma3(0.5f, m2p + m2m, neg3(sg * sg));
    // Lambda_a in [0.0826, 0.1586] and 1 + s^T Lambda^-1 s in [1, 1.3]
    li = rcp_nr(lam);
    y = li * sg;
    den = rcp_nr(1.0f + sg.p.x * y.p.x + sg.p.y * y.p.y + sg.z * y.z);
  }
};

template <>
struct Sten<1> {
  int r[1][3];
  V3 f[1];  // in [0.5, 1.5)
  __device__ __forceinline__ bool set(float ux, float uy, float uz, int ox, int oy, int oz) {
    const float u[3] = {ux, uy, uz};
    const int o[3] = {ox, oy, oz};
    float fa[3];
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Cell<1> c;
      c.set(u[a]);
      r[0][a] = c.b - o[a];
      ok = ok && (unsigned)r[0][a] <= 3u;
      fa[a] = c.f;
    }
    f[0] = {pk(fa[0], fa[1]), fa[2]};
    return ok;
  }
  __device__ __forceinline__ V3 w(int, int n) const {
    const V3 p = n == 0 ? v3(1.5f) - f[0] : n == 1 ? v3(1.0f) - f[0] : f[0] - v3(0.5f);
    return n == 1 ? v3(0.75f) - p * p : 0.5f * (p * p);
  }
  __device__ __forceinline__ V3 d(int, int n) const { return n == 0 ? neg3(f[0]) : v3((float)n) - f[0]; }
  __device__ __forceinline__ void set_grad() {}
  // N'(x) of the quadratic B-spline at d = -f, 1 - f, 2 - f: 3/2 - f, 2 (f - 1), 1/2 - f
  __device__ __forceinline__ V3 k(int, int n) const {
    return n == 0 ? v3(1.5f) - f[0] : n == 1 ? 2.0f * (f[0] - v3(1.0f)) : v3(0.5f) - f[0];
  }
};

// Staged nodes of grid g: row pitch, first index, and a stencil's first node.
template <int KIND>
__device__ __forceinline__ constexpr int pitch(int g) {
  return KIND == 0 && g == 0 ? 5 : 6;
}
template <int KIND>
__device__ __forceinline__ int first_node(const Sten<KIND>& st, int g) {
  const int E = pitch<KIND>(g);
  return (g == 0 ? 0 : 125) + (st.r[g][2] * E + st.r[g][1]) * E + st.r[g][0];
}

// Visit every (node, weight, offset) of a stencil: fn(staged_index, w, dx, dy, dz).
template <int KIND, typename Fn>
__device__ __forceinline__ void for_nodes(const Sten<KIND>& st, Fn&& fn) {
  constexpr int N = Geo<KIND>::N;
#pragma unroll
  for (int g = 0; g < Geo<KIND>::NG; ++g) {
    const int E = pitch<KIND>(g), base = first_node<KIND>(st, g);
#pragma unroll
    for (int sz = 0; sz < N; ++sz)
#pragma unroll
      for (int sy = 0; sy < N; ++sy) {
        const float wyz = st.w(g, sy).p.y * st.w(g, sz).z;
#pragma unroll
        for (int sx = 0; sx < N; ++sx)
          fn(base + (sz * E + sy) * E + sx, st.w(g, sx).p.x * wyz, st.d(g, sx).p.x, st.d(g, sy).p.y, st.d(g, sz).z);
      }
  }
}

// Staged grid velocities: (x, y) and z apart, so that a node is an 8- and a
// 4-byte shared load (three wavefronts) instead of a 16-byte one (four).
template <int NS>
struct NodeVel {
  float2 xy[NS];
  float z[NS];
};
template <int NS>
__device__ __forceinline__ void stage_node(NodeVel<NS>& s, int j, const float4* g) {
  cp_async8(&s.xy[j], g);
  cp_async4(&s.z[j], reinterpret_cast<const float*>(g) + 2);
}
struct Nodes {
  const float2* xy;
  const float* z;
  __device__ __forceinline__ V3 operator[](int i) const { return {xy[i], z[i]}; }
  __device__ __forceinline__ Nodes operator+(int i) const { return {xy + i, z + i}; }
};

// G2P gather as a tensor-product contraction (a node's weight is the product
// of per-axis weights): over one grid's N^3 stencil, S = sum w v~ and the
// first moments M_a = sum w v~ s_a (s_a in 0..N-1: the node's offset in the
// stencil along axis a), reducing x, then y, then z.  With x_i - x_p =
// (s - f) dx per axis, sum w v~ (x_i - x_p)_a / dx = M_a - f_a S.  FIRST: M
// starts here (else it adds to the grid before).  wz carries the factor 1/2
// that averages the two CK grids: every sum is linear in the z weights, and
// scaling by a power of two is exact.
template <int KIND, bool FIRST>
__device__ __forceinline__ void gather_moments(const Nodes& sv, const Sten<KIND>& st, int g, V3& S, V3* M) {
  constexpr int N = Geo<KIND>::N;
  const int E = pitch<KIND>(g), base = first_node<KIND>(st, g);
#pragma unroll
  for (int sz = 0; sz < N; ++sz) {
    V3 Ps, Px, Py;
#pragma unroll
    for (int sy = 0; sy < N; ++sy) {
      const Nodes row = sv + base + (sz * E + sy) * E;
      V3 Rs, Rx;
      Rx = st.w(g, 1).p.x * row[1];
      Rs = fma3(st.w(g, 0).p.x, row[0], Rx);
      if constexpr (N == 3) {
        const V3 t = st.w(g, 2).p.x * row[2];
        Rs = Rs + t;
        Rx = fma3(2.0f, t, Rx);
      }
      const float wy = st.w(g, sy).p.y;
      if (sy == 0) {
        Ps = wy * Rs;
        Px = wy * Rx;
      } else {
        const V3 u = wy * Rs;
        Ps = Ps + u;
        Px = fma3(wy, Rx, Px);
        Py = sy == 1 ? u : fma3(2.0f, u, Py);
      }
    }
    const float wz = st.w(g, sz).z * (KIND == 0 ? 0.5f : 1.0f);
    if (sz == 0) {
      S = wz * Ps;
      M[0] = FIRST ? wz * Px : fma3(wz, Px, M[0]);
      M[1] = FIRST ? wz * Py : fma3(wz, Py, M[1]);
    } else {
      S = fma3(wz, Ps, S);
      M[0] = fma3(wz, Px, M[0]);
      M[1] = fma3(wz, Py, M[1]);
      M[2] = FIRST && sz == 1 ? wz * Ps : fma3((float)sz * wz, Ps, M[2]);
    }
  }
}

// v = h sum w v~ and Bh = h sum w v~ (x_i - x_p)^T / dx (column a: axis a) over
// the particle's stencil; h = 1/2 averages the two CK grids.
template <int KIND>
__device__ __forceinline__ void g2p_gather(const Sten<KIND>& st, const Nodes& sv, V3& vel, M3& Bh) {
  V3 S[Geo<KIND>::NG];
  gather_moments<KIND, true>(sv, st, 0, S[0], Bh.c);
  if constexpr (KIND == 0) gather_moments<KIND, false>(sv, st, 1, S[1], Bh.c);
#pragma unroll
  for (int a = 0; a < 3; ++a) {  // f_a = -d[g][0]
    if constexpr (KIND == 0) Bh.c[a] = fma3(at3(st.d(1, 0), a), S[1], Bh.c[a]);
    Bh.c[a] = fma3(at3(st.d(0, 0), a), S[0], Bh.c[a]);
  }
  vel = S[0];
  if constexpr (KIND == 0) vel = vel + S[1];
}

// Kernel-gradient transfers: S = sum w v~ and the derivative sums G_a = sum
// g_a v~ over one grid's N^3 stencil, g = (K'x Ky Kz, Kx K'y Kz, Kx Ky K'z)
// (so that grad w = -g / dx with respect to the particle position), by the
// same x, y, z reduction with the kernel derivative in place of the offset.
template <int KIND, bool FIRST>
__device__ __forceinline__ void gather_grad(const Nodes& sv, const Sten<KIND>& st, int g, V3& S, V3* G) {
  constexpr int N = Geo<KIND>::N;
  const int E = pitch<KIND>(g), base = first_node<KIND>(st, g);
  constexpr float h = KIND == 0 ? 0.5f : 1.0f;
#pragma unroll
  for (int sz = 0; sz < N; ++sz) {
    V3 Ps, Px, Py;
#pragma unroll
    for (int sy = 0; sy < N; ++sy) {
      const Nodes row = sv + base + (sz * E + sy) * E;
      V3 Rs, Rx;
#pragma unroll
      for (int sx = 0; sx < N; ++sx) {
        const V3 a = row[sx];
        Rs = sx == 0 ? st.w(g, sx).p.x * a : fma3(st.w(g, sx).p.x, a, Rs);
        Rx = sx == 0 ? st.k(g, sx).p.x * a : fma3(st.k(g, sx).p.x, a, Rx);
      }
      const float wy = st.w(g, sy).p.y, ky = st.k(g, sy).p.y;
      Ps = sy == 0 ? wy * Rs : fma3(wy, Rs, Ps);
      Px = sy == 0 ? wy * Rx : fma3(wy, Rx, Px);
      Py = sy == 0 ? ky * Rs : fma3(ky, Rs, Py);
    }
    const float wz = h * st.w(g, sz).z, kz = h * st.k(g, sz).z;
    const bool first = FIRST && sz == 0;
    S = first ? wz * Ps : fma3(wz, Ps, S);
    G[0] = first ? wz * Px : fma3(wz, Px, G[0]);
    G[1] = first ? wz * Py : fma3(wz, Py, G[1]);
    G[2] = first ? kz * Ps : fma3(kz, Ps, G[2]);
  }
}

// v = h sum w v~ and Gr = h sum v~ g^T (column a: axis a), so that grad v =
// -Gr / dx; h = 1/2 averages the two CK grids.  Needs set_grad().
template <int KIND>
__device__ __forceinline__ void g2p_gather_grad(const Sten<KIND>& st, const Nodes& sv, V3& vel, M3& Gr) {
  gather_grad<KIND, true>(sv, st, 0, vel, Gr.c);
  if constexpr (KIND == 0) gather_grad<KIND, false>(sv, st, 1, vel, Gr.c);
}

// R = scale Q D^-1.  CK: D^-1 = diag(li) - den y y^T, so with t = Q y a column
// costs one product and one fused update; quadratic: D^-1 = 4 I.
__device__ __forceinline__ M3 mul_dinv(const Sten<0>& st, const M3& Q, float scale) {
  V3 li, y;
  float den;
  st.dinv(li, y, den);
  const V3 t = fma3(y.z, Q.c[2], fma3(y.p.y, Q.c[1], y.p.x * Q.c[0]));
  const V3 ls = scale * li, ys = neg3((scale * den) * y);
  M3 R;
#pragma unroll
  for (int q = 0; q < 3; ++q) R.c[q] = fma3(at3(ys, q), t, at3(ls, q) * Q.c[q]);
  return R;
}
__device__ __forceinline__ M3 mul_dinv(const Sten<1>&, const M3& Q, float scale) {
  return {{(4.0f * scale) * Q.c[0], (4.0f * scale) * Q.c[1], (4.0f * scale) * Q.c[2]}};
}

__device__ __forceinline__ void decode_block(const SceneDev& s, uint32_t key, int& ox, int& oy, int& oz) {
  int lb = (int)(key - s.key_base);
  int bx = lb % s.npb;
  int by = (lb / s.npb) % s.npb;
  int bz = lb / (s.npb * s.npb);
  ox = bx * 4;
  oy = by * 4;
  oz = bz * 4;
}

// ------------------------------------------------------------------------ P2G

// Shared-memory accumulation is in 32-bit fixed point: integer shared
// atomics run about 4x faster than float ones on this part (measured), and
// integer sums do not depend on the order of the atomics.  Every contribution
// that a block's particles can make is bounded when they are binned
// (p2g_bounds, from the largest weight, weight times offset and row sum of
// D^-1 of the stencil), so with cnt particles no node sum can exceed cnt times
// the block's largest bound, and the scale maps that to 2^30 (no overflow).
// Rounding costs at most half a unit per contribution, cnt * bound * 2^-31.

// P2G runs one warp per CTA and streams a block's particles through shared
// memory in chunks of kP2GStage (cp.async gathers through the binned order,
// all in flight together); lanes take a chunk's particles C = kP2GStage / 32
// apart (C odd), so each quarter-warp's 16-byte reads fall on distinct bank
// groups and neighbouring lanes come from different cells.
constexpr int kP2GWarp = 32;
constexpr int kP2GStage = 96;  // 3 * 32

struct P2GPart {
  float4 X, a, b, c;
};

// Per-stencil bounds of one P2G contribution w (m v + A^ d) (d: node offset
// in cells); wmax and the product wd * dinv keep a margin of at least 0.3%
// over the exact maxima for float rounding:
//   wmax  largest node weight: CK 1 (K1(0)); quadratic 0.75^3;
//   wd    largest |w d_a|: max over one axis of |d| K(|d|) times the largest
//         weight of the other two: CK 0.27751 (at |d| = 0.394) x 1;
//         quadratic 0.25 (at |d| = 1/2) x 0.75^2 = 0.140625;
//   dinv  largest row abs-sum of D^-1 in cells^-2: CK 14.04 (over a 121^3
//         grid of fractions), quadratic 4 (D^-1 = 4 I).
template <int KIND>
struct P2GBound;
template <>
struct P2GBound<0> {
  static constexpr float wmax = 1.003f;
  static constexpr float wd = 0.2785f;
  static constexpr float dinv = 14.5f;
};
template <>
struct P2GBound<1> {
  static constexpr float wmax = 0.4232f;
  static constexpr float wd = 0.1411f;
  static constexpr float dinv = 4.0f;
};

// Bound of |w (m v + A^ d)|_inf over every node a particle touches:
// wmax m |v|_inf + wd * dinv * max_row sum_k |M_rk| / dx, since
// |w (A^ d)_r| <= sum_k |A^_rk| |w d_k| and the rows of A^ = M D^-1 / dx sum
// to at most sum_j |M_rj| * dinv / dx.
// The PIC transfer's contribution w m v + M grad w (M = -dt V0 tau) has the
// same bound with wd * dinv replaced by the largest |g_a| of a stencil:
// CK 2 (|K1'| <= 2, at |x| = 1/2, times weights <= 1), quadratic 0.5625
// (|N'| <= 1 times 0.75^2); both are below wd * dinv (4.04 and 0.5644), so
// one bound serves every transfer.  APIC with the kernel gradient keeps m B
// and T = -dt V0 tau apart and passes |m B| + |T| (elementwise) as M.
// The particle's two bounds (mass, momentum) go into its block's entry of
// the per-key bound table when it is binned (G2P for the next step, admission
// and re-keying otherwise), so P2G reads a block's bounds without a pass over
// its particles.
template <int KIND>
__device__ __forceinline__ void p2g_bounds(float inv_dx, float mass, const V3& v, const M3& M, float& bmass,
                                           float& bmom) {
  const float r0 = fabsf(M.c[0].p.x) + fabsf(M.c[1].p.x) + fabsf(M.c[2].p.x);
  const float r1 = fabsf(M.c[0].p.y) + fabsf(M.c[1].p.y) + fabsf(M.c[2].p.y);
  const float r2 = fabsf(M.c[0].z) + fabsf(M.c[1].z) + fabsf(M.c[2].z);
  const float rm = fmaxf(r0, fmaxf(r1, r2));
  bmass = P2GBound<KIND>::wmax * mass;
  bmom = bmass * fmaxf(fabsf(v.p.x), fmaxf(fabsf(v.p.y), fabsf(v.z))) +
         P2GBound<KIND>::wd * P2GBound<KIND>::dinv * rm * inv_dx;
}

// FMA: a block of at least kP2GFmaCount particles has every scaled
// contribution within 2^30 / count <= 2^22 in magnitude, where one fused
// multiply-add with 1.5 * 2^23 rounds w * (...) to the nearest integer in the
// low mantissa bits (the sum lies in [2^23, 2^24), whose spacing is 1): the
// integer is the float's bits minus those of 1.5 * 2^23.  That takes the
// conversion off the XU pipe; smaller blocks convert with __float2int_rn.
constexpr uint32_t kP2GFmaCount = 256;

// Two rounded contributions w * val into their planes.  FMA: one packed
// multiply-add with 1.5 * 2^23 rounds both halves; each is, in scalars,
//   __float_as_int(fmaf(w, val, 12582912.0f)) - 0x4B400000;
template <bool FMA>
__device__ __forceinline__ void p2g_add2(int* a, int* b, f2 w, f2 val) {
  if constexpr (FMA) {
    const f2 f = fma2(w, val, dup(12582912.0f));
    atomicAdd(a, __float_as_int(f.x) - 0x4B400000);
    atomicAdd(b, __float_as_int(f.y) - 0x4B400000);
  } else {
    const f2 f = mul2(w, val);
    atomicAdd(a, __float2int_rn(f.x));
    atomicAdd(b, __float2int_rn(f.y));
  }
}

// Scatter of one particle.  The four sums of a node lie in four planes (the
// three momenta, then the mass); plane c is a linear function of the node's
// offset, w (R0 + R1 dx + R2 dy + R3 dz), with the rows R = (p_c, row c of A^)
// of the momenta and (m, 0, 0, 0) of the mass, all pre-scaled.  Instruction
// slots 0, 1 and 2, 3 are computed packed.
// ROT: a shared atomic instruction costs about the largest number of its
// lanes that fall in one bank, and lanes on one address count like lanes on
// distinct addresses of that bank: about three lanes of an instruction share
// a cell and so every node of the stencil.  Slot c then adds plane
// (c + rot) & 3, rot = (3 lane) & 3, so neighbouring lanes of one cell write
// different planes (plane stride kP2GRotPlane, 24 banks apart); the lane's
// rows are permuted once per particle by two selects each, so no register
// array is indexed at run time.  pl[c] is the plane that slot c writes.
// TR: 0 APIC + MLS: A^ = M D^-1 / dx, so that A (x_i - x_p) = A^ (offset in
// cells).  1 PIC with the kernel gradient (Sec. 4.3): the state holds
// M = -dt V0 tau (B = 0) and a node receives w m v + M grad w with
// grad w = -g / dx: the rows multiply g in place of w d.  2 APIC with the
// kernel gradient: M = m B, T = -dt V0 tau apart, both terms.
template <int KIND>
struct P2GRotPlane {
  static constexpr int value = ((Geo<KIND>::NS + 7) / 32) * 32 + 24;  // >= NS, = 24 mod 32
};

// Rows of the four slots, packed by slots (0, 1) and (2, 3): e = 0 the
// constant, 1..3 the columns of an M3 (the mass row has none).
struct P2GRows {
  f2 a, b;
};
template <bool ROT>
__device__ __forceinline__ P2GRows p2g_rows(const V3& mom, float mass, bool r1, bool r2) {
  if constexpr (!ROT) {
    return {mom.p, pk(mom.z, mass)};
  } else {
    const float t0 = r1 ? mom.p.y : mom.p.x, t1 = r1 ? mom.z : mom.p.y, t2 = r1 ? mass : mom.z, t3 = r1 ? mom.p.x : mass;
    return {pk(r2 ? t2 : t0, r2 ? t3 : t1), pk(r2 ? t0 : t2, r2 ? t1 : t3)};
  }
}

template <int KIND, int TR, bool ROT, bool FMA>
__device__ __forceinline__ void p2g_scatter(const SceneDev& s, const MatDev* mats, uint32_t* err, const P2GPart& q,
                                            const M3& T, int ox, int oy, int oz, float Sm, float Sp, int* const* pl,
                                            uint32_t rot) {
  Sten<KIND> st;
  if (!st.set(q.X.x * s.inv_dx, q.X.y * s.inv_dx, q.X.z * s.inv_dx, ox, oy, oz)) {
    flag_error(err, CK_ERR_INTERNAL);
    return;
  }
  const M3 M = unpack_m3(q.b, q.c, q.a.w);
  const float mass = mats[__float_as_uint(q.X.w)].mass;
  const V3 p = (mass * Sp) * V3{pk(q.a.x, q.a.y), q.a.z};
  const bool r1 = (rot & 1u) != 0u, r2 = (rot & 2u) != 0u;
  // Q: constant and APIC columns; H: kernel-gradient columns
  P2GRows Q[4], H[4];
  Q[0] = p2g_rows<ROT>(p, mass * Sm, r1, r2);
  if constexpr (TR != 1) {
    const M3 A = mul_dinv(st, M, s.inv_dx * Sp);
#pragma unroll
    for (int e = 0; e < 3; ++e) Q[e + 1] = p2g_rows<ROT>(A.c[e], 0.f, r1, r2);
  }
  if constexpr (TR != 0) {
    st.set_grad();
    const float sc = -s.inv_dx * Sp;
#pragma unroll
    for (int e = 0; e < 3; ++e) H[e + 1] = p2g_rows<ROT>(sc * (TR == 1 ? M.c[e] : T.c[e]), 0.f, r1, r2);
  }
  constexpr int N = Geo<KIND>::N;
#pragma unroll
  for (int g = 0; g < Geo<KIND>::NG; ++g) {
    const int E = pitch<KIND>(g), jb = first_node<KIND>(st, g);
    int* const b0 = pl[0] + jb;
    int* const b1 = pl[1] + jb;
    int* const b2 = pl[2] + jb;
    int* const b3 = pl[3] + jb;
#pragma unroll
    for (int sz = 0; sz < N; ++sz)
#pragma unroll
      for (int sy = 0; sy < N; ++sy) {
        const float wy = st.w(g, sy).p.y, wz = st.w(g, sz).z, wyz = wy * wz;
        const float dy = st.d(g, sy).p.y, dz = st.d(g, sz).z;
        f2 ea = Q[0].a, eb = Q[0].b, ha, hb;
        if constexpr (TR != 1) {
          ea = fma2(Q[3].a, dup(dz), fma2(Q[2].a, dup(dy), ea));
          eb = fma2(Q[3].b, dup(dz), fma2(Q[2].b, dup(dy), eb));
        }
        if constexpr (TR != 0) {
          // w e + g H = wx (wyz e + K'y wz H2 + wy K'z H3) + K'x (wyz H1)
          const float kyz = st.k(g, sy).p.y * wz, ykz = wy * st.k(g, sz).z;
          ea = fma2(H[3].a, dup(ykz), fma2(H[2].a, dup(kyz), mul2(dup(wyz), ea)));
          eb = fma2(H[3].b, dup(ykz), fma2(H[2].b, dup(kyz), mul2(dup(wyz), eb)));
          ha = mul2(dup(wyz), H[1].a);
          hb = mul2(dup(wyz), H[1].b);
        }
#pragma unroll
        for (int sx = 0; sx < N; ++sx) {
          const int o = (sz * E + sy) * E + sx;
          const float wx = st.w(g, sx).p.x, dx = st.d(g, sx).p.x;
          if constexpr (TR == 0) {
            const f2 w = dup(wx * wyz);
            p2g_add2<FMA>(b0 + o, b1 + o, w, fma2(Q[1].a, dup(dx), ea));
            p2g_add2<FMA>(b2 + o, b3 + o, w, fma2(Q[1].b, dup(dx), eb));
          } else {
            f2 va = ea, vb = eb;
            if constexpr (TR == 2) {
              const float wdx = wyz * dx;
              va = fma2(Q[1].a, dup(wdx), va);
              vb = fma2(Q[1].b, dup(wdx), vb);
            }
            const float kx = st.k(g, sx).p.x;
            va = fma2(dup(kx), ha, mul2(dup(wx), va));
            vb = fma2(dup(kx), hb, mul2(dup(wx), vb));
            p2g_add2<FMA>(b0 + o, b1 + o, dup(1.0f), va);
            p2g_add2<FMA>(b2 + o, b3 + o, dup(1.0f), vb);
          }
        }
      }
  }
}

// Replicated accumulators: with REP = 2 the staged sums exist twice and a
// lane adds into copy (lane & 1).  Lanes of one cell are neighbours (they
// take particles C apart in binned order), and k lanes on one shared address
// cost about k cycles, so splitting neighbours over two copies halves those
// collisions; the copies start 16 banks apart, so the same node in both
// copies is on different banks.  The copies are summed at the flush.
template <int KIND, int REP>
struct P2GRep {
  static constexpr int NS = Geo<KIND>::NS;
  static constexpr int stride = REP == 1 ? 4 * NS : ((4 * NS + 15) / 32) * 32 + 16;  // ints per copy
};

// CTAs per SM that P2G's registers leave room for: what its shared memory
// allows, or fewer where that would spill (left to itself the compiler took up
// to 186 registers for the twin's 27 unrolled nodes: 32.8 us instead of 26.9
// on the granular column).
constexpr int p2g_min_ctas(int kind, int tr, int rep) {
  return tr == 2 ? (kind == 0 ? 16 : 12) : rep == 2 || (kind == 1 && tr == 1) ? 16 : 20;
}

// TR: transfer, 0 APIC + MLS, 1 PIC, 2 APIC with the kernel gradient.
// ROT (one copy): components issued in the lane-rotated order of p2g_scatter,
// planes kP2GRotPlane apart.  FMA: blocks of at least kP2GFmaCount particles
// round their contributions by p2g_add2's multiply-add instead of a
// conversion.
// SPLIT: blocks in parts; the form for whole blocks (a large step) is kept
// apart, because the units' arithmetic showed in it (16.27 M particles: 0.497
// against 0.491 ms here, 0.585 against 0.576 in G2P).
template <int KIND, int TR, int REP, int ROT, int FMA, bool SPLIT>
__global__ void __launch_bounds__(kP2GWarp, p2g_min_ctas(KIND, TR, REP)) k_p2g(StepView v) {
  constexpr int NS = Geo<KIND>::NS;
  static_assert(ROT == 0 || REP == 1, "the rotated order takes one copy");
  constexpr int PL = ROT ? P2GRotPlane<KIND>::value : NS;  // plane stride of the components
  constexpr int RS = ROT ? 4 * PL : P2GRep<KIND, REP>::stride;
  constexpr uint32_t CAP = kP2GStage, C = kP2GStage / 32;
  static_assert(C % 2 == 1, "lane stride must be odd");
  static_assert(RS % 4 == 0, "copies must keep 16-byte alignment");
  __shared__ __align__(16) int small[REP * RS];
  const uint32_t rot = ROT ? (threadIdx.x * 3u) & 3u : 0u;
  int* const copy = small + (REP == 1 ? 0 : (int)(threadIdx.x & 1u) * RS);
  int* const pl[4] = {copy + ((0u + rot) & 3u) * PL, copy + ((1u + rot) & 3u) * PL, copy + ((2u + rot) & 3u) * PL,
                      copy + ((3u + rot) & 3u) * PL};
  __shared__ float4 sX[CAP], sA[CAP], sB[CAP], sC[CAP];
  constexpr uint32_t TCAP = TR == 2 ? CAP : 1;  // the stress term T (kernel-gradient APIC only)
  __shared__ float4 sT0[TCAP], sT1[TCAP];
  __shared__ float sT2[TCAP];
  __shared__ uint32_t bslot[8];
  const uint32_t lane = threadIdx.x;
  // dynamic scheduling: one work unit (a block or a part of one) at a time
  const uint32_t npb = *v.n_pb;
  const Units units = SPLIT ? Units{v.parts[kUnitsP2G], v.units[kUnitsP2G].unit} : Units{1u, 0u};
  const uint32_t nunits = npb * units.splits;
  for (uint32_t u = SPLIT ? blockIdx.x : next_unit(&v.work[0]); u < nunits; u = next_unit(&v.work[0])) {
    Unit q;
    if (!unit_of<CAP, SPLIT>(v, units, u, q)) continue;
    const uint32_t key = q.key, start = q.start, cnt = q.cnt, lo = q.lo, hi = q.hi;
    const SceneDev s = v.scenes[q.scene];
    // the block's largest contribution bounds, recorded when its particles
    // were binned
    const float bmass = __uint_as_float(v.bnd_cur[2 * key]);
    const float bmom = __uint_as_float(v.bnd_cur[2 * key + 1]);
    int ox, oy, oz;
    decode_block(s, key, ox, oy, oz);
    load_block_slots(v, s, ox, oy, oz, bslot);
    for (int j = lane; j < REP * RS / 4; j += kP2GWarp) reinterpret_cast<int4*>(small)[j] = make_int4(0, 0, 0, 0);
    // the scale covers the block's whole count, so any part of it is bounded
    const float fcnt = (float)cnt;
    const float Sm = bmass > 0.f ? 1073741824.0f / (fcnt * bmass) : 1.0f;
    const float Sp = bmom > 0.f ? 1073741824.0f / (fcnt * bmom) : 1.0f;
    for (uint32_t c0 = lo; c0 < hi; c0 += CAP) {
      const uint32_t m = min(hi - c0, CAP);
#pragma unroll
      for (uint32_t r = 0; r < C; ++r) {
        const uint32_t i = lane + r * kP2GWarp;
        if (i < m) {
          const uint32_t p = v.perm[start + c0 + i];
          cp_async16(&sX[i], &v.cur.X[p]);
          cp_async16(&sA[i], &v.cur.VM0[p]);
          cp_async16(&sB[i], &v.cur.VM1[p]);
          cp_async16(&sC[i], &v.cur.VM2[p]);
          if constexpr (TR == 2) {
            cp_async16(&sT0[i], &v.cur.T0[p]);
            cp_async16(&sT1[i], &v.cur.T1[p]);
            cp_async4(&sT2[i], &v.cur.T2[p]);
          }
        }
      }
      cp_async_wait_all();
      __syncwarp();
#pragma unroll 1
      for (uint32_t r = 0; r < C; ++r) {
        const uint32_t i = lane * C + r;
        if (i < m) {
          const P2GPart part{sX[i], sA[i], sB[i], sC[i]};
          M3 T{};
          if constexpr (TR == 2) T = unpack_m3(sT0[i], sT1[i], sT2[i]);
          if (FMA && cnt >= kP2GFmaCount)
            p2g_scatter<KIND, TR, ROT != 0, true>(s, v.mats, v.err, part, T, ox, oy, oz, Sm, Sp, pl, rot);
          else
            p2g_scatter<KIND, TR, ROT != 0, false>(s, v.mats, v.err, part, T, ox, oy, oz, Sm, Sp, pl, rot);
        }
      }
      __syncwarp();  // the next chunk overwrites the staged copies
    }
    const float iSm = 1.0f / Sm, iSp = 1.0f / Sp;
    for (int j = lane; j < NS; j += kP2GWarp) {
      // the copies' sums: each copy's sum is bounded like the whole, and
      // their total too, so adding them as integers cannot overflow
      int q[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        q[c] = small[c * PL + j];
        if (REP == 2) q[c] += small[RS + c * NS + j];
      }
      if (q[3] != 0) {
        int g, lx, ly, lz;
        staged_coords<KIND>(j, g, lx, ly, lz);
        long long gi = pool_index<KIND>(bslot, g, lx, ly, lz);
        if (gi >= 0)
          atomicAdd(&v.Gacc[gi], make_float4((float)q[3] * iSm, (float)q[0] * iSp, (float)q[1] * iSp,
                                             (float)q[2] * iSp));
      }
    }
    // (the block's bounds are cleared after G2P, by the float64 pass: other
    // units of this block may still be reading them)
    __syncwarp();  // the next unit clears the accumulators
  }
}

// ---------------------------------------------------------------- grid update

// Sec. 4.3.3 per grid: v~ = (m v + dt f)/m + dt g on nodes with m > 0, zero
// elsewhere; sticky walls zero v~ where a node coordinate (in cells, node i of
// G- at i + 1/4, of G+ at i - 1/4, quadratic at i) is < bc or > res - bc.
template <int KIND>
__global__ void __launch_bounds__(128) k_grid_update(StepView v) {
  constexpr int NG = Geo<KIND>::NG;
  // blocks per iteration: their dependent loads (list entry, scene, sums)
  // overlap (four measured slower: registers)
  constexpr int PB = 2;
  const uint32_t ng = min(*v.n_g, v.pool_cap);
  for (uint32_t g0 = blockIdx.x * PB; g0 < ng; g0 += gridDim.x * PB) {
    uint32_t gb[PB];
    SceneDev sd[PB];
#pragma unroll
    for (int k = 0; k < PB; ++k) {
      const uint32_t gi = min(g0 + k, ng - 1);  // a missing second block repeats the first's reads
      gb[k] = v.g_list[gi];
      sd[k] = v.scenes[v.g_scene[gi]];
    }
    for (int t = threadIdx.x; t < NG * kBlockNodes; t += blockDim.x) {
      const int grid = t / kBlockNodes, l = t % kBlockNodes;
      float4 acc[PB];
#pragma unroll
      for (int k = 0; k < PB; ++k)
        acc[k] = g0 + k < ng ? v.Gacc[((long long)(g0 + k) * NG + grid) * kBlockNodes + l] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < PB; ++k) {
        if (g0 + k >= ng) break;
        const SceneDev& s = sd[k];
        const long long lb = (long long)gb[k] - s.table_base;
        const int gx = (int)(lb % s.nb), gy = (int)((lb / s.nb) % s.nb), gz = (int)(lb / ((long long)s.nb * s.nb));
        const int ix = gx * 4 + (l & 3), iy = gy * 4 + ((l >> 2) & 3), iz = gz * 4 + (l >> 4);
        const float off = KIND == 0 ? (grid == 0 ? 0.25f : -0.25f) : 0.0f;
        const long long idx = ((long long)(g0 + k) * NG + grid) * kBlockNodes + l;
        float4 o = make_float4(0.f, 0.f, 0.f, acc[k].x);
        if (acc[k].x > 0.f) {
          o.x = acc[k].y / acc[k].x + s.dt * s.gx;
          o.y = acc[k].z / acc[k].x + s.dt * s.gy;
          o.z = acc[k].w / acc[k].x + s.dt * s.gz;
        }
        const float px = ix + off, py = iy + off, pz = iz + off;
        const float hi = (float)s.res - s.bc;
        const bool wall = px < s.bc || py < s.bc || pz < s.bc || px > hi || py > hi || pz > hi;
        if (wall) o.x = o.y = o.z = 0.f;
        v.Gvel[idx] = o;
        if (!v.keep_gacc) v.Gacc[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
}

// ------------------------------------------------------ G2P + constitutive

__device__ __forceinline__ float min3(float a, float b, float c) { return fminf(a, fminf(b, c)); }

// G2P runs one warp per CTA: a particle block's ~400-500 particles leave a
// partly idle last round on 32 lanes instead of on 128, and the staging
// waits are warp-level, so a lane that finishes early never holds up three
// other warps at a block barrier.  MINB counts 4-warp equivalents per SM.
// The fused G2P2G kernel stages g2p_stage(MINB) particles per chunk (64 at
// 5 or more, so that shared memory admits the extra warps).
constexpr int kG2PWarp = 32;
__host__ __device__ constexpr int g2p_stage(int minb) { return minb >= 5 ? 64 : 128; }  // particles per chunk

// |A| + |B| elementwise (the bound of the kernel-gradient APIC's two terms)
__device__ __forceinline__ M3 abs_sum(const M3& A, const M3& B) {
  M3 r;
#pragma unroll
  for (int q = 0; q < 3; ++q)
    r.c[q] = {pk(fabsf(A.c[q].p.x) + fabsf(B.c[q].p.x), fabsf(A.c[q].p.y) + fabsf(B.c[q].p.y)),
              fabsf(A.c[q].z) + fabsf(B.c[q].z)};
  return r;
}

// Result of one particle's G2P: its next key and P2G contribution bounds,
// whether its constitutive update was deferred to the float64 pass, and
// whether its new state is finite.
struct G2POut {
  uint32_t nk;
  float bmass, bmom;
  bool use64, fin;
};

// What a particle's update reads of its scene, in 16-byte groups.
struct alignas(16) SceneStep {
  float inv_dx, dt, dx, mdtv;               // mdtv = -dt V0
  float gs, hi, j_tol, cond_tol;            // gs = dt / dx; hi = res - 1/2
  float gap_tol;
  int npb;
  uint32_t key_base;
  int res;
  __device__ __forceinline__ void set(const SceneDev& s) {
    inv_dx = s.inv_dx;
    dt = s.dt;
    dx = s.dx;
    mdtv = -s.dt * s.V0;
    gs = s.dt * s.inv_dx;
    hi = (float)s.res - 0.5f;
    j_tol = s.j_tol;
    cond_tol = s.cond_tol;
    gap_tol = s.gap_tol;
    npb = s.npb;
    key_base = s.key_base;
    res = s.res;
  }
};

// One particle's staged state (shared memory).  Read where it is used: the
// position and the material index a second time after the gather, instead of
// in registers across it.
struct G2PIn {
  const float4 *X, *F0, *F1;
  const float *F2, *E;
  const uint32_t* ID;
};

// A second read of a staged value that the compiler does not merge with the
// first (which would keep it in registers in between).
__device__ __forceinline__ float4 again(const float4* p) {
  float4 r;
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(a));
  return r;
}

// G2P of one particle (slot t of the current binned order): gather v and B
// (or the kernel-gradient sums) from the staged grid velocities sv, F update,
// constitutive update (or listing for the float64 pass), advection, next key
// and bounds; stores the new state at slot t of nxt.  Returns false (and
// flags CK_ERR_INTERNAL) for a particle outside its block.
template <int KIND, int TR>
__device__ __forceinline__ bool g2p_particle(const StepView& v, const SceneStep* sc, int ox, int oy, int oz,
                                             const Nodes& sv, uint32_t t, const G2PIn& in, G2POut& out,
                                             const MatDev* smat = nullptr) {
  out.use64 = false;
  Sten<KIND> st;
  {
    const float4 X = *in.X;
    const float inv_dx = sc->inv_dx;
    if (!st.set(X.x * inv_dx, X.y * inv_dx, X.z * inv_dx, ox, oy, oz)) {
      flag_error(v.err, CK_ERR_INTERNAL);
      return false;
    }
  }
  V3 vel;
  M3 Bh, C;  // C = dt grad v
  if constexpr (TR == 1) {
    // grad v = -Gr / dx (Gr in Bh)
    st.set_grad();
    g2p_gather_grad<KIND>(st, sv, vel, Bh);
    const float gs = -sc->gs;
#pragma unroll
    for (int q = 0; q < 3; ++q) C.c[q] = gs * Bh.c[q];
  } else if constexpr (TR == 2) {
    // B from the APIC moments, grad v = -Gr / dx from the derivative sums
    g2p_gather<KIND>(st, sv, vel, Bh);
    st.set_grad();
    V3 vg;
    g2p_gather_grad<KIND>(st, sv, vg, C);
    const float gs = -sc->gs;
#pragma unroll
    for (int q = 0; q < 3; ++q) C.c[q] = gs * C.c[q];
  } else {
    // grad v = B D^-1 = Bh D^-1 / dx
    g2p_gather<KIND>(st, sv, vel, Bh);
    C = mul_dinv(st, Bh, sc->gs);
  }
  const float vx = vel.p.x, vy = vel.p.y, vz = vel.z;
  const float4 X = again(in.X);
  const uint32_t mi = __float_as_uint(X.w);
  // the material table from shared memory when the kernel staged it there
  const MatDev* mt = (smat ? smat : v.mats) + mi;
  const float4 m4 = *reinterpret_cast<const float4*>(mt);  // mass, mu, lam, dpc
  const int model = mt->model;
  float mu = m4.y, lam = m4.z;
  float Ep = 0.f;
  if (v.cur.E) {
    Ep = *in.E;
    const float nu = mt->nu;
    mu = Ep / (2.0f * (1.0f + nu));
    lam = Ep * nu / ((1.0f + nu) * (1.0f - 2.0f * nu));
  }
  // F' = (I + dt grad v) F
  const M3 Fo = unpack_m3(*in.F0, *in.F1, *in.F2);
  M3 F = mul_add(C, Fo, Fo);
  // constitutive update in float32 from the left stretch; degenerate or
  // inverted F is deferred to the float64 pass (precision extension):
  // this kernel stores F' and M = m B' (no stress) and lists the particle.
  // ft: -dt V0 tau
  M3 ft;
  const float4 s4 = *reinterpret_cast<const float4*>(sc);  // inv_dx, dt, dx, mdtv
  const float inv_dx = s4.x, dt = s4.y, dx = s4.z, mdtv = s4.w;
  // Drucker-Prager at small stretch: matrix log/exp series, no eigen-
  // decomposition (such F is far from every float64 criterion)
  Sym Xs;
  const float xr = model == 1 ? left_strain(F, Xs) : 1.f;
  const bool small_dp = model == 1 && sc->gap_tol <= 0.f && sc->j_tol < 0.9f && sc->cond_tol < 0.9f &&
                        xr <= (1.f / 48.f);
  const int sdeg = dp_lane_degree(xr);
  if (small_dp) {
    Sym tau;
    dp_small_strain(F, Xs, sdeg, mu, lam, m4.w, mdtv, tau);
    ft = sym_m3(tau);
  } else {
    float Fr[9], tau[9];
    to_rows(F, Fr);
    if (model == 2) {
      // J-based fluid: volume ratio only, stress from J (no decomposition)
      fluid_update<float>(Fr, mt->E, mt->gamma, tau);
    } else {
      // b = F F^T = U diag(sigma^2) U^T
      float bq[9], U[9], e[3], sg[3];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int q = r; q < 3; ++q) {
          const float d = Fr[r * 3] * Fr[q * 3] + Fr[r * 3 + 1] * Fr[q * 3 + 1] + Fr[r * 3 + 2] * Fr[q * 3 + 2];
          bq[r * 3 + q] = d;
          bq[q * 3 + r] = d;
        }
      sym_eig3<float>(bq, U, e);
      sg[0] = sqrtf(fmaxf(e[0], 0.f));
      sg[1] = sqrtf(fmaxf(e[1], 0.f));
      sg[2] = sqrtf(fmaxf(e[2], 0.f));
      const float J = det3<float>(Fr);
      const float smax = fmaxf(sg[0], fmaxf(sg[1], sg[2]));
      const float smin = min3(sg[0], sg[1], sg[2]);
      const float gap = min3(fabsf(sg[0] - sg[1]), fabsf(sg[0] - sg[2]), fabsf(sg[1] - sg[2]));
      const bool use64 = !(J > 0.f) || (fabsf(J) < sc->j_tol) || (smin < sc->cond_tol * smax) ||
                         (gap < sc->gap_tol * smax);
      out.use64 = use64;
      if (use64) {
        const unsigned long long slot = atomicAdd(v.fp64_count, 1ull);
        v.fp64_list[slot] = t;
#pragma unroll
        for (int q = 0; q < 9; ++q) tau[q] = 0.f;
      } else {
        constitutive_left<float>(model, Fr, mu, lam, mt->alpha, tau, U, e, sg);
      }
    }
    F = from_rows(Fr);
    ft = from_rows(tau);
#pragma unroll
    for (int q = 0; q < 3; ++q) ft.c[q] = mdtv * ft.c[q];
  }
  // M' = m B' - dt V0 tau, B' = dx Bh (APIC) or 0 (PIC); the kernel-
  // gradient APIC keeps M' = m B' and T' = -dt V0 tau apart
  const float mdx = m4.x * dx;
  M3 Mn;
#pragma unroll
  for (int q = 0; q < 3; ++q) Mn.c[q] = TR == 1 ? ft.c[q] : TR == 2 ? mdx * Bh.c[q] : fma3(mdx, Bh.c[q], ft.c[q]);
  float4 Xn = make_float4(X.x + dt * vx, X.y + dt * vy, X.z + dt * vz, X.w);
  // next key; particles leaving the interior are clamped and flagged
  float ux = Xn.x * inv_dx, uy = Xn.y * inv_dx, uz = Xn.z * inv_dx;
  // x was finite, so x + dt v is finite when v is.  x * 0 is 0 for a finite
  // x and NaN for an infinite or NaN one, so one sum of such products tests
  // every value at one fused multiply-add each
  V3 z = 0.f * vel;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    z = fma3(0.f, F.c[q], fma3(0.f, Mn.c[q], z));
    if constexpr (TR == 2) z = fma3(0.f, ft.c[q], z);
  }
  const bool fin = z.p.x + z.p.y + z.z == 0.f;
  if (!fin) flag_error(v.err, CK_ERR_NONFINITE);
  out.fin = fin;
  const float uhi = sc->hi;
  if (!(ux >= 0.5f && ux < uhi && uy >= 0.5f && uy < uhi && uz >= 0.5f && uz < uhi)) {  // in_domain
    flag_error(v.err, CK_ERR_DOMAIN);
    const float lo = 0.5f, hi = (float)sc->res - 0.5f - 1e-3f;
    ux = fminf(fmaxf(isfinite(ux) ? ux : lo, lo), hi);
    uy = fminf(fmaxf(isfinite(uy) ? uy : lo, lo), hi);
    uz = fminf(fmaxf(isfinite(uz) ? uz : lo, lo), hi);
    Xn.x = ux * dx;
    Xn.y = uy * dx;
    Xn.z = uz * dx;
    ux = Xn.x * inv_dx;
    uy = Xn.y * inv_dx;
    uz = Xn.z * inv_dx;
  }
  const uint32_t nk = particle_key<KIND>(*sc, ux, uy, uz);
  v.nxt.X[t] = Xn;
  float4 a, b;
  float c;
  pack_m3(Mn, a, b, c);
  v.nxt.VM0[t] = make_float4(vx, vy, vz, c);
  v.nxt.VM1[t] = a;
  v.nxt.VM2[t] = b;
  pack_m3(F, a, b, c);
  v.nxt.F0[t] = a;
  v.nxt.F1[t] = b;
  v.nxt.F2[t] = c;
  v.nxt.ID[t] = *in.ID;
  if (v.nxt.E) v.nxt.E[t] = Ep;
  v.key_nxt[t] = nk;
  out.nk = nk;
  if constexpr (TR == 2) {
    pack_m3(ft, a, b, c);
    v.nxt.T0[t] = a;
    v.nxt.T1[t] = b;
    v.nxt.T2[t] = c;
    p2g_bounds<KIND>(inv_dx, m4.x, vel, abs_sum(Mn, ft), out.bmass, out.bmom);
  } else {
    p2g_bounds<KIND>(inv_dx, m4.x, vel, Mn, out.bmass, out.bmom);
  }
  return true;
}

// Bound by its issue slots and the packed multiply-adds (68% of the slots
// issue; DRAM 0.6 of the copy rate).  Measured against the scalar form (16.27 M
// particles / dam break, 4.18 M): 0.637 -> 0.590 ms / 0.165 -> 0.152, with the
// warp instructions per particle of the dam break down from 35 to 27; without
// the staged scene and the second read of the position 16-byte spills put it
// at 0.61 / 0.163, and a 16-byte node in place of NodeVel's 8 + 4 at 0.596 /
// 0.158.  (P2G, bound by its shared atomics: 0.507 -> 0.491 / 0.148 -> 0.145.)
//
// G2P with the next chunk's particle state in flight.  Chunks of 32
// particles (one per lane; each lane stages and reads only its own
// particle's slot) alternate between two staging buffers: while chunk k is
// computed, chunk k+1 is being gathered with cp.async.  The binned-order
// indices (perm) that address those gathers travel by cp.async into shared
// memory too, three chunks ahead, so inside a block no load result is waited
// on and no index is held in a register across a chunk's computation (held
// there, one was spilled to local memory at this register budget, and its
// spill store waited for the load).

// TR: transfer, 0 APIC + MLS, 1 PIC, 2 APIC with the kernel gradient.
// SPLIT as in k_p2g.
template <int KIND, int MINB, int TR, bool SPLIT>
__global__ void __launch_bounds__(kG2PWarp, 4 * MINB) k_g2p(StepView v) {
  constexpr int NS = Geo<KIND>::NS;
  constexpr int CH = 32;
  constexpr int NB = 2;       // staging buffers (four measured slower: registers)
  constexpr int D = NB - 1;   // chunks in flight ahead of the computed one
  constexpr int PS = 2 * NB;  // slots of binned-order indices (D + 2 live at a time)
  static_assert((NB & (NB - 1)) == 0, "NB must be a power of two");
  __shared__ NodeVel<NS> svel;
  __shared__ float4 sX[NB][CH], sF0[NB][CH], sF1[NB][CH];
  __shared__ float sF2[NB][CH], sE[NB][CH];
  __shared__ uint32_t sID[NB][CH];
  __shared__ uint32_t sP[PS][CH];
  __shared__ uint32_t bslot[8];
  __shared__ MatDev smat[kSmemMats];
  __shared__ SceneStep sstep;  // the unit's scene, read where it is used (registers)
  const uint32_t lane = threadIdx.x;
  const bool mat_smem = v.n_mats <= (uint32_t)kSmemMats;
  if (mat_smem) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(v.mats);
    uint32_t* dst = reinterpret_cast<uint32_t*>(smat);
    const uint32_t words = v.n_mats * (uint32_t)(sizeof(MatDev) / 4);
    for (uint32_t w = lane; w < words; w += CH) dst[w] = src[w];
  }
  __syncwarp();
  const uint32_t npb = *v.n_pb;
  const Units units = SPLIT ? Units{v.parts[kUnitsG2P], v.units[kUnitsG2P].unit} : Units{1u, 0u};
  const uint32_t nunits = npb * units.splits;
  for (uint32_t u = SPLIT ? blockIdx.x : next_unit(&v.work[1]); u < nunits; u = next_unit(&v.work[1])) {
    Unit q;
    if (!unit_of<32, SPLIT>(v, units, u, q)) continue;
    const uint32_t key = q.key, start = q.start, lo = q.lo, hi = q.hi;
    const SceneDev& s = v.scenes[q.scene];
    if (lane == 0) sstep.set(s);
    int ox, oy, oz;
    decode_block(s, key, ox, oy, oz);
    load_block_slots(v, s, ox, oy, oz, bslot);
    const uint32_t nch = (hi - lo + CH - 1) / CH;
    // Each lane stages and reads only its own slot of every buffer, so the
    // index and particle buffers need no cross-lane ordering; sv does.
    // Binned-order indices of chunks 0 .. 2D: loaded together; chunks
    // 0 .. D-1 are staged at once, D .. 2D parked in sP.  The index of chunk
    // c >= 2D + 1 is fetched by cp.async in the group of chunk c - D - 1,
    // which has landed before chunk c is staged.
    uint32_t pp[2 * D + 1];
#pragma unroll
    for (int j = 0; j <= 2 * D; ++j) {
      const uint32_t i = lo + (uint32_t)j * CH + lane;
      pp[j] = i < hi ? v.perm[start + i] : 0u;
    }
#pragma unroll
    for (int j = D; j <= 2 * D; ++j) sP[j % PS][lane] = pp[j];
    __syncwarp();  // bslot
    for (int j = lane; j < NS; j += CH) {
      int g, lx, ly, lz;
      staged_coords<KIND>(j, g, lx, ly, lz);
      const long long gi = pool_index<KIND>(bslot, g, lx, ly, lz);
      if (gi >= 0)
        stage_node(svel, j, &v.Gvel[gi]);
      else
        svel.xy[j] = make_float2(0.f, 0.f), svel.z[j] = 0.f;
    }
    auto stage = [&](uint32_t c, uint32_t p) {
      const uint32_t b = c & (NB - 1);
      if (lo + c * CH + lane < hi) {
        cp_async16(&sX[b][lane], &v.cur.X[p]);
        cp_async16(&sF0[b][lane], &v.cur.F0[p]);
        cp_async16(&sF1[b][lane], &v.cur.F1[p]);
        cp_async4(&sF2[b][lane], &v.cur.F2[p]);
        cp_async4(&sID[b][lane], &v.cur.ID[p]);
        if (v.cur.E) cp_async4(&sE[b][lane], &v.cur.E[p]);
      }
    };
    // chunks 0 .. D-1 (the grid velocities go with chunk 0's group)
#pragma unroll
    for (int j = 0; j < D; ++j) {
      if ((uint32_t)j < nch) stage((uint32_t)j, pp[j]);
      cp_async_commit();
    }
    for (uint32_t k = 0; k < nch; ++k) {
      const uint32_t kn = k + D;
      if (kn < nch) stage(kn, sP[kn % PS][lane]);
      const uint32_t kp = k + 2 * D + 1;
      if (kp < nch) {
        const uint32_t i = lo + kp * CH + lane;
        if (i < hi) cp_async4(&sP[kp % PS][lane], &v.perm[start + i]);
      }
      cp_async_commit();
      cp_async_wait<D>();  // the D newest groups may still be in flight: chunk k has landed
      __syncwarp();
      const uint32_t b = k & (NB - 1);
      const uint32_t i = lo + k * CH + lane;
      if (i < hi) {
        G2POut o;
        const G2PIn in{&sX[b][lane], &sF0[b][lane], &sF1[b][lane], &sF2[b][lane], &sE[b][lane], &sID[b][lane]};
        if (g2p_particle<KIND, TR>(v, &sstep, ox, oy, oz, Nodes{svel.xy, svel.z}, start + i, in, o, mat_smem ? smat : nullptr))
          warp_aggregated_bin(v.cnt_nxt, v.bnd_nxt, o.nk, o.bmass, o.bmom);
      }
      __syncwarp();  // chunk k + NB is staged into this buffer next
    }
  }
}

// ------------------------------------------------------------ fused G2P2G
//
// The paper's G2P2G (Sec. 5.1, after Wang 2020) gathers step n and scatters
// step n + 1 in one kernel.  Here one CTA (one warp) takes a particle block
// of step n and
//   1. runs G2P on every particle of the block exactly as k_g2p does
//      (new state, next key, histogram and bounds for the next binning);
//   2. scatters the particles that stay in the block (same key, float32
//      constitutive update, finite) into the block's staged nodes with the
//      fixed-point shared atomics of k_p2g, and flushes them into the next
//      step's grid through its block table.
// The fixed-point scale needs the bound of the block's new contributions
// before the first atomic, so the scatter is a second pass that reads the
// new state the first pass just wrote (contiguous, from L2), instead of a
// stash in shared memory that would cost occupancy.  Particles that moved to
// another block, took the float64 pass or became non-finite go to a list
// that k_p2g_leftover scatters after the float64 pass.
// The staged grid velocities of pass 1 and the accumulators of pass 2 share
// one shared-memory arena.
constexpr int kFuseMaxCnt = 4096;  // block particle count up to which stays are tracked (larger: all leftover)

template <int KIND, int MINB>
struct FuseSmem {
  static constexpr int NS = Geo<KIND>::NS;
  static constexpr int CAP = g2p_stage(MINB);
  struct Ph1 {
    NodeVel<NS> svel;
    float4 sX[CAP], sF0[CAP], sF1[CAP];
    float sF2[CAP], sE[CAP];
    uint32_t sID[CAP];
  };
  struct Ph2 {
    int sm[4][NS];
    float4 sX[kP2GStage], sA[kP2GStage], sB[kP2GStage], sC[kP2GStage];
  };
  static constexpr size_t bytes = sizeof(Ph1) > sizeof(Ph2) ? sizeof(Ph1) : sizeof(Ph2);
};

// Append value to a global list when pred holds (one atomic per warp).
__device__ __forceinline__ void warp_append(uint32_t* count, uint32_t* list, uint32_t value, bool pred) {
  const unsigned am = __activemask();
  const unsigned m = __ballot_sync(am, pred);
  if (!m) return;
  const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(count, (uint32_t)__popc(m));
  base = __shfl_sync(am, base, leader);
  if (pred) list[base + __popc(m & ((1u << lane) - 1u))] = value;
}

template <int KIND, int MINB>
__global__ void __launch_bounds__(kG2PWarp, 4 * MINB) k_g2p2g(StepView v) {
  using SM = FuseSmem<KIND, MINB>;
  constexpr int NS = SM::NS;
  constexpr int CAP = SM::CAP;
  constexpr uint32_t PCAP = kP2GStage, PC = kP2GStage / 32;
  static_assert(CAP % 32 == 0, "the stay mask takes one ballot per 32 particles");
  __shared__ __align__(16) unsigned char arena[SM::bytes];
  __shared__ uint32_t stay[kFuseMaxCnt / 32];
  __shared__ uint32_t bslot[8];
  __shared__ SceneStep sstep;
  auto& p1 = *reinterpret_cast<typename SM::Ph1*>(arena);
  auto& p2 = *reinterpret_cast<typename SM::Ph2*>(arena);
  const uint32_t lane = threadIdx.x;
  const uint32_t npb = *v.n_pb;
  const bool split = v.units[kUnitsG2P].splits > 1u;
  const Units units = split ? Units{v.parts[kUnitsG2P], v.units[kUnitsG2P].unit} : Units{1u, 0u};
  const uint32_t nunits = npb * units.splits;
  for (uint32_t u = split ? blockIdx.x : next_unit(&v.work[1]); u < nunits; u = next_unit(&v.work[1])) {
    Unit q;
    if (!unit_of<32>(v, units, u, q)) continue;
    const uint32_t key = q.key, start = q.start, lo = q.lo, hi = q.hi;
    const SceneDev s = v.scenes[q.scene];
    const bool track = hi - lo <= (uint32_t)kFuseMaxCnt;
    int ox, oy, oz;
    decode_block(s, key, ox, oy, oz);
    load_block_slots(v, s, ox, oy, oz, bslot);  // this step's grid (gather)
    if (lane == 0) sstep.set(s);
    __syncwarp();
    // ---- pass 1: G2P of the block
    float bm_max = 0.f, bp_max = 0.f;
    uint32_t nstay = 0;
    for (uint32_t c0 = lo; c0 < hi; c0 += CAP) {
      const uint32_t m = min(hi - c0, (uint32_t)CAP);
#pragma unroll 4
      for (uint32_t i = lane; i < m; i += 32) {
        const uint32_t p = v.perm[start + c0 + i];
        cp_async16(&p1.sX[i], &v.cur.X[p]);
        cp_async16(&p1.sF0[i], &v.cur.F0[p]);
        cp_async16(&p1.sF1[i], &v.cur.F1[p]);
        cp_async4(&p1.sF2[i], &v.cur.F2[p]);
        cp_async4(&p1.sID[i], &v.cur.ID[p]);
        if (v.cur.E) cp_async4(&p1.sE[i], &v.cur.E[p]);
      }
      if (c0 == lo) {
        for (int j = lane; j < NS; j += 32) {
          int g, lx, ly, lz;
          staged_coords<KIND>(j, g, lx, ly, lz);
          long long gi = pool_index<KIND>(bslot, g, lx, ly, lz);
          if (gi >= 0)
            stage_node(p1.svel, j, &v.Gvel[gi]);
          else
            p1.svel.xy[j] = make_float2(0.f, 0.f), p1.svel.z[j] = 0.f;
        }
      }
      cp_async_wait_all();
      __syncwarp();
      for (uint32_t i = lane; i < m; i += 32) {
        const uint32_t t = start + c0 + i;
        G2POut o;
        const G2PIn in{&p1.sX[i], &p1.sF0[i], &p1.sF1[i], &p1.sF2[i], &p1.sE[i], &p1.sID[i]};
        const bool ok = g2p_particle<KIND, 0>(v, &sstep, ox, oy, oz, Nodes{p1.svel.xy, p1.svel.z}, t, in, o);
        if (ok) warp_aggregated_bin(v.cnt_nxt, v.bnd_nxt, o.nk, o.bmass, o.bmom);
        const bool st = ok && track && o.nk == key && !o.use64 && o.fin;
        if (st) {
          bm_max = fmaxf(bm_max, o.bmass);
          bp_max = fmaxf(bp_max, o.bmom);
          nstay += 1;
        }
        warp_append(v.lo_count, v.lo_list, t, ok && !st);
        const unsigned am = __activemask();
        const unsigned w = __ballot_sync(am, st);
        if (track && (int)lane == __ffs(am) - 1) stay[(c0 - lo + i - lane) >> 5] = w;
      }
      __syncwarp();  // the next chunk overwrites the staged copies
    }
    // ---- pass 2: P2G of the particles that stayed, into the next grid
    bm_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(bm_max)));
    bp_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(bp_max)));
    nstay = __reduce_add_sync(0xffffffffu, nstay);
    if (nstay > 0) {
      if (lane < 8) {  // the next step's grid blocks (scatter)
        const int bx = (ox >> 2) + (lane & 1), by = (oy >> 2) + ((lane >> 1) & 1), bz = (oz >> 2) + (lane >> 2);
        bslot[lane] = v.table_nxt[s.table_base + ((long long)bz * s.nb + by) * s.nb + bx];
      }
      for (int j = lane; j < NS; j += 32) reinterpret_cast<int4*>(&p2.sm[0][0])[j] = make_int4(0, 0, 0, 0);
      int* const pl[4] = {p2.sm[0], p2.sm[1], p2.sm[2], p2.sm[3]};
      const float fst = (float)nstay;
      const float Sm = bm_max > 0.f ? 1073741824.0f / (fst * bm_max) : 1.0f;
      const float Sp = bp_max > 0.f ? 1073741824.0f / (fst * bp_max) : 1.0f;
      for (uint32_t c0 = lo; c0 < hi; c0 += PCAP) {
        const uint32_t m = min(hi - c0, PCAP);
#pragma unroll
        for (uint32_t r = 0; r < PC; ++r) {
          const uint32_t i = lane + r * 32;
          if (i < m) {
            const uint32_t t = start + c0 + i;
            cp_async16(&p2.sX[i], &v.nxt.X[t]);
            cp_async16(&p2.sA[i], &v.nxt.VM0[t]);
            cp_async16(&p2.sB[i], &v.nxt.VM1[t]);
            cp_async16(&p2.sC[i], &v.nxt.VM2[t]);
          }
        }
        cp_async_wait_all();
        __syncwarp();
#pragma unroll 1
        for (uint32_t r = 0; r < PC; ++r) {
          const uint32_t i = lane * PC + r;
          const uint32_t q = c0 - lo + i;
          if (i < m && ((stay[q >> 5] >> (q & 31)) & 1u)) {
            const P2GPart part{p2.sX[i], p2.sA[i], p2.sB[i], p2.sC[i]};
            p2g_scatter<KIND, 0, false, false>(s, v.mats, v.err, part, M3{}, ox, oy, oz, Sm, Sp, pl, 0u);
          }
        }
        __syncwarp();
      }
      const float iSm = 1.0f / Sm, iSp = 1.0f / Sp;
      for (int j = lane; j < NS; j += 32) {
        const int mi = p2.sm[3][j];
        if (mi != 0) {
          int g, lx, ly, lz;
          staged_coords<KIND>(j, g, lx, ly, lz);
          const long long gi = pool_index<KIND>(bslot, g, lx, ly, lz);
          if (gi >= 0)
            atomicAdd(&v.Gacc[gi], make_float4((float)mi * iSm, (float)p2.sm[0][j] * iSp,
                                               (float)p2.sm[1][j] * iSp, (float)p2.sm[2][j] * iSp));
          else
            flag_error(v.err, CK_ERR_POOL);
        }
      }
    }
    __syncwarp();  // the next unit reuses the arena and the slots
  }
}

// Pool slot of virtual grid block g in the next step's table; a block no
// fused scatter touched is claimed here: a slot is taken from the counter
// and offered to the table with one compare-and-swap; when another thread
// got there first its slot is used and this one stays empty (its
// accumulators are zero, so the grid update leaves it at rest).  No thread
// waits on another.
__device__ __forceinline__ uint32_t claim_slot(const StepView& v, long long g, uint32_t scene) {
  const uint32_t cur = v.table_nxt[g];
  if (cur != CK_NO_SLOT) return cur;
  const uint32_t ns = atomicAdd(v.n_g_nxt, 1u);
  if (ns >= v.pool_cap) {
    flag_error(v.err, CK_ERR_POOL);
    return CK_NO_SLOT;
  }
  v.g_list_nxt[ns] = (uint32_t)g;
  v.g_scene_nxt[ns] = scene;
  const uint32_t old = atomicCAS(&v.table_nxt[g], CK_NO_SLOT, ns);
  return old == CK_NO_SLOT ? ns : old;
}

// P2G of the particles the fused kernel left over (new state in nxt, after
// the float64 pass): one particle per thread, contributions in float added
// with one 16-byte global atomic per node (APIC + MLS; quadratic or CK).
template <int KIND>
__global__ void __launch_bounds__(128) k_p2g_leftover(StepView v) {
  constexpr int NG = Geo<KIND>::NG;
  const uint32_t n = min(*v.lo_count, v.n_cur);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t t = v.lo_list[i];
    const float4 X = v.nxt.X[t];
    const MatDev mt = v.mats[__float_as_uint(X.w)];
    const SceneDev s = v.scenes[mt.scene];
    const float ux = X.x * s.inv_dx, uy = X.y * s.inv_dx, uz = X.z * s.inv_dx;
    Cell<KIND> cx, cy, cz;
    cx.set(ux);
    cy.set(uy);
    cz.set(uz);
    const int ox = cx.block() * 4, oy = cy.block() * 4, oz = cz.block() * 4;
    Sten<KIND> st;
    if (!st.set(ux, uy, uz, ox, oy, oz)) {
      flag_error(v.err, CK_ERR_INTERNAL);
      continue;
    }
    const float4 a = v.nxt.VM0[t], b = v.nxt.VM1[t], c = v.nxt.VM2[t];
    float A[9];
    to_rows(mul_dinv(st, unpack_m3(b, c, a.w), s.inv_dx), A);
    const float mass = mt.mass;
    const float px = mass * a.x, py = mass * a.y, pz = mass * a.z;
    for_nodes<KIND>(st, [&](int j, float w, float dx, float dy, float dz) {
      int g, lx, ly, lz;
      staged_coords<KIND>(j, g, lx, ly, lz);
      const int ix = ox + lx, iy = oy + ly, iz = oz + lz;
      const long long gb = s.table_base + ((long long)(iz >> 2) * s.nb + (iy >> 2)) * s.nb + (ix >> 2);
      const uint32_t sl = claim_slot(v, gb, mt.scene);
      if (sl == CK_NO_SLOT) return;
      const int l = ((iz & 3) * 4 + (iy & 3)) * 4 + (ix & 3);
      atomicAdd(&v.Gacc[((long long)sl * NG + g) * kBlockNodes + l],
                make_float4(w * mass, w * (px + A[0] * dx + A[1] * dy + A[2] * dz),
                            w * (py + A[3] * dx + A[4] * dy + A[5] * dz), w * (pz + A[6] * dx + A[7] * dy + A[8] * dz)));
    });
  }
}

// One particle's matrices by rows (stored by pack.cuh's order).
__device__ __forceinline__ void load_F(const Pool& P, uint32_t t, float* F) {
  to_rows(unpack_m3(P.F0[t], P.F1[t], P.F2[t]), F);
}
__device__ __forceinline__ void store_F(const Pool& P, uint32_t t, const float* F) {
  float4 a, b;
  float c;
  pack_m3(from_rows(F), a, b, c);
  P.F0[t] = a;
  P.F1[t] = b;
  P.F2[t] = c;
}
__device__ __forceinline__ void load_M(const Pool& P, uint32_t t, float* M) {
  to_rows(unpack_m3(P.VM1[t], P.VM2[t], P.VM0[t].w), M);
}
__device__ __forceinline__ void store_M(const Pool& P, uint32_t t, const float* M) {
  float4 a, b;
  float c;
  pack_m3(from_rows(M), a, b, c);
  P.VM0[t].w = c;
  P.VM1[t] = a;
  P.VM2[t] = b;
}
__device__ __forceinline__ void store_T(const Pool& P, uint32_t t, const float* T) {
  float4 a, b;
  float c;
  pack_m3(from_rows(T), a, b, c);
  P.T0[t] = a;
  P.T1[t] = b;
  P.T2[t] = c;
}

// Float64 pass of the precision extension: the particles G2P listed (F
// degenerate, inverted or flagged by the scene's criteria) get the full
// rotation-variant SVD and constitutive update in float64.  G2P stored the
// advanced F' and M = m B'; this pass stores the projected F, subtracts
// dt V0 tau from M (with the kernel-gradient APIC: stores T = -dt V0 tau) and
// raises the particle's block bounds to cover the new M.
// Grid-stride over the list; an empty list returns at once.
template <int KIND>
__global__ void __launch_bounds__(128) k_g2p_fp64(StepView v) {
  // every transfer kernel of the step is done with the histogram entries and
  // P2G bounds of this step's blocks: clear them, so that this buffer is all
  // zero when G2P fills it for the step after next
  const uint32_t npb = *v.n_pb;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < npb; i += gridDim.x * blockDim.x) {
    const uint32_t key = v.pb[i].x;
    v.cnt_cur[key] = 0u;
    v.bnd_cur[2 * key] = 0u;
    v.bnd_cur[2 * key + 1] = 0u;
  }
  // the histogram G2P filled is complete: its tile sums for the next scan
  if (v.tile_cnt) write_tile_sums<128, kScanTile>(v.cnt_nxt, v.n_keys, v.tile_cnt, v.tile_ne);
  const uint32_t n = (uint32_t)min(*v.fp64_count, (unsigned long long)v.n_cur);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t t = v.fp64_list[i];
    const float4 X = v.nxt.X[t];
    const MatDev mt = v.mats[__float_as_uint(X.w)];
    const SceneDev s = v.scenes[mt.scene];
    double mu = mt.mu, lam = mt.lam;
    if (v.nxt.E) {
      const double E = v.nxt.E[t], nu = mt.nu;
      mu = E / (2.0 * (1.0 + nu));
      lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu));
    }
    float Ff[9];
    load_F(v.nxt, t, Ff);
    double F[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) F[q] = Ff[q];
    double tau[9], sg[3];
    constitutive<double>(mt.model, F, mu, lam, (double)mt.alpha, tau, sg);
    const double dtv = (double)s.dt * (double)s.V0;
    const float4 a = v.nxt.VM0[t];
    float Mn[9], Tn[9];
    load_M(v.nxt, t, Mn);
    const bool sep = v.nxt.T0 != nullptr;  // stress term kept apart from m B
    bool fin = true;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      Tn[q] = (float)(-dtv * tau[q]);
      if (!sep) Mn[q] = (float)(Mn[q] - dtv * tau[q]);
      Ff[q] = (float)F[q];
      fin = fin && isfinite(Mn[q]) && isfinite(Tn[q]) && isfinite(Ff[q]);
    }
    if (!fin) flag_error(v.err, CK_ERR_NONFINITE);
    if (sep)
      store_T(v.nxt, t, Tn);
    else
      store_M(v.nxt, t, Mn);
    store_F(v.nxt, t, Ff);
    const M3 Mb = sep ? abs_sum(from_rows(Mn), from_rows(Tn)) : from_rows(Mn);
    float bmass, bmom;
    p2g_bounds<KIND>(s.inv_dx, mt.mass, V3{pk(a.x, a.y), a.z}, Mb, bmass, bmom);
    const uint32_t nk = v.key_nxt[t];
    atomicMax(&v.bnd_nxt[2 * nk], __float_as_uint(bmass));
    atomicMax(&v.bnd_nxt[2 * nk + 1], __float_as_uint(bmom));
  }
}

// Zero the accumulators of the blocks listed by the last probe.
template <int KIND>
__global__ void k_clear_gacc(StepView v) {
  constexpr int NG = Geo<KIND>::NG;
  const uint32_t ng = min(*v.n_g, v.pool_cap);
  for (uint32_t gi = blockIdx.x; gi < ng; gi += gridDim.x) {
    for (int t = threadIdx.x; t < NG * kBlockNodes; t += blockDim.x)
      v.Gacc[((long long)gi * NG + (t / kBlockNodes)) * kBlockNodes + (t % kBlockNodes)] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// ------------------------------------------------------- readback / upload

// Kirchhoff stress of a stored F (no plasticity), any material.
__device__ __forceinline__ void stress_of(const MatDev& mt, const float* F, float mu, float lam, float* tau) {
  if (mt.model == 2)
    fluid_tau_of_J<float>(det3(F), mt.E, mt.gamma, tau);
  else
    stress_only<float>(mt.model, F, mu, lam, tau);
}

__device__ __forceinline__ void lame_of(const MatDev& mt, const Pool& P, uint32_t t, float& mu, float& lam) {
  mu = mt.mu;
  lam = mt.lam;
  if (P.E) {
    float E = P.E[t];
    mu = E / (2.0f * (1.0f + mt.nu));
    lam = E * mt.nu / ((1.0f + mt.nu) * (1.0f - 2.0f * mt.nu));
  }
}

// B = (M + dt V0 tau(F)) / m; with the stress term kept apart, B = M / m
__device__ __forceinline__ void recover_B(const Pool& P, const SceneDev& s, const MatDev& mt, uint32_t t, float* B) {
  float F[9], M[9], tau[9];
  load_M(P, t, M);
  if (P.T0) {
    const float im = 1.0f / mt.mass;
#pragma unroll
    for (int q = 0; q < 9; ++q) B[q] = M[q] * im;
    return;
  }
  load_F(P, t, F);
  float mu, lam;
  lame_of(mt, P, t, mu, lam);
  stress_of(mt, F, mu, lam, tau);
  float dtv = s.dt * s.V0, im = 1.0f / mt.mass;
#pragma unroll
  for (int q = 0; q < 9; ++q) B[q] = (M[q] + dtv * tau[q]) * im;
}

// Floats of a particle field (x, v: 3; B, C, F: 9; E: 1).
__host__ __device__ constexpr int field_width(int field) { return field <= 1 ? 3 : field == 5 ? 1 : 9; }

// One particle field in the scene's original order.  Bound by HBM: it reads
// the field (and the ids) once and writes it once.  Particles lie in binned
// order, so the output rows are scattered by id, but neighbours in memory are
// mostly neighbours in the original order too: a warp takes 32 particles,
// turns their rows through shared memory (row pitch = width, odd: no bank
// conflicts) and lets consecutive lanes write consecutive floats, so a store
// instruction covers whole 32-byte sectors instead of 32 separate ones.
// Only what the field needs is loaded (x and the material for B and C only).
// Measured on 16.27 M particles (x, v, F): 127, 123 and 267 us (3.6, 3.7 and
// 4.6 TB/s) against 1261 us for the three with one 4-byte store per lane and
// float, rows apart, and every load made for every field.
// pic: the PIC transfer keeps B = 0, so B and C read as 0.
template <int KIND, int FIELD>
__global__ void __launch_bounds__(256) k_read_particles(Pool P, const SceneDev* scenes, const MatDev* mats, int scene,
                                                        uint32_t start, uint32_t n, int pic, float* out) {
  constexpr int W = field_width(FIELD);
  constexpr int U = FIELD == 2 || FIELD == 3 ? 1 : 2;  // groups of 32 particles whose loads are in flight together
  __shared__ float rows[8][32 * W];
  const uint32_t lane = threadIdx.x & 31u;
  float* const row = rows[threadIdx.x >> 5];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x * U;
  // the loop runs on the warp's first particle: every lane takes every round
  for (uint64_t i0 = ((uint64_t)blockIdx.x * blockDim.x + (threadIdx.x - lane)) * U; i0 < n; i0 += stride) {
    const uint32_t cnt = (uint32_t)min((uint64_t)(32u * U), n - i0);
    uint32_t id[U];
    float r[U][W];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      id[u] = 0u;
      if (u * 32u + lane >= cnt) continue;
      const uint32_t t = start + (uint32_t)i0 + u * 32u + lane;
      id[u] = P.ID[t];
      if constexpr (FIELD == 0) {
        const float4 X = P.X[t];
        r[u][0] = X.x; r[u][1] = X.y; r[u][2] = X.z;
      } else if constexpr (FIELD == 1) {
        const float4 a = P.VM0[t];
        r[u][0] = a.x; r[u][1] = a.y; r[u][2] = a.z;
      } else if constexpr (FIELD == 4) {
        load_F(P, t, r[u]);
      } else if constexpr (FIELD == 5) {
        r[u][0] = P.E ? P.E[t] : 0.f;
      } else {
        if (pic) {
#pragma unroll
          for (int q = 0; q < 9; ++q) r[u][q] = 0.f;
        } else {
          const SceneDev s = scenes[scene];
          const float4 X = P.X[t];
          const MatDev mt = mats[__float_as_uint(X.w)];
          recover_B(P, s, mt, t, r[u]);
          if constexpr (FIELD == 3) {  // C = B D^-1 = B Di / dx^2
            Sten<KIND> st;
            const float ux = X.x * s.inv_dx, uy = X.y * s.inv_dx, uz = X.z * s.inv_dx;
            Cell<KIND> cx, cy, cz;
            cx.set(ux); cy.set(uy); cz.set(uz);
            st.set(ux, uy, uz, cx.block() * 4, cy.block() * 4, cz.block() * 4);
            to_rows(mul_dinv(st, from_rows(r[u]), s.inv_dx * s.inv_dx), r[u]);
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u * 32u + lane < cnt) {
#pragma unroll
        for (int q = 0; q < W; ++q) row[lane * W + q] = r[u][q];
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const uint32_t e = (uint32_t)k * 32u + lane, p = e / W;
        const uint32_t idp = __shfl_sync(0xffffffffu, id[u], p);
        if (u * 32u + p < cnt) out[(size_t)idp * W + (e - p * W)] = row[e];
      }
      __syncwarp();  // the next group overwrites the rows
    }
  }
}

// Overwrite one field from original-order input; keeps M = m B - dt V0 tau(F)
// (pic: B = 0, the host refuses uploads of B).
__global__ void k_write_particles(Pool P, const SceneDev* scenes, const MatDev* mats, int scene, uint32_t start,
                                  uint32_t n, int field, int pic, const float* in) {
  const SceneDev s = scenes[scene];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint32_t t = start + i;
    uint32_t id = P.ID[t];
    float4 X = P.X[t];
    const MatDev mt = mats[__float_as_uint(X.w)];
    float dtv = s.dt * s.V0;
    if (field == 0) {
      P.X[t] = make_float4(in[3 * id], in[3 * id + 1], in[3 * id + 2], X.w);
    } else if (field == 1) {
      float4 a = P.VM0[t];
      P.VM0[t] = make_float4(in[3 * id], in[3 * id + 1], in[3 * id + 2], a.w);
    } else if (field == 2) {
      float F[9], tau[9], M[9], mu, lam;
      load_F(P, t, F);
      lame_of(mt, P, t, mu, lam);
      stress_of(mt, F, mu, lam, tau);
      for (int q = 0; q < 9; ++q) M[q] = mt.mass * in[9 * id + q] - (P.T0 ? 0.f : dtv * tau[q]);
      store_M(P, t, M);
    } else if (field == 4 || field == 5) {
      float B[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (!pic) recover_B(P, s, mt, t, B);
      if (field == 4) {
        store_F(P, t, in + 9 * (size_t)id);
      } else if (P.E) {
        P.E[t] = in[id];
      }
      float F[9], tau[9], M[9], mu, lam;
      load_F(P, t, F);
      lame_of(mt, P, t, mu, lam);
      stress_of(mt, F, mu, lam, tau);
      if (P.T0) {  // m B stays; the stress term follows the new F (or E)
        for (int q = 0; q < 9; ++q) tau[q] *= -dtv;
        store_T(P, t, tau);
      } else {
        for (int q = 0; q < 9; ++q) M[q] = mt.mass * B[q] - dtv * tau[q];
        store_M(P, t, M);
      }
    }
  }
}

// Dense grid fields of one scene: out[grid][iz][iy][ix] (x fastest) over
// 0..res per axis, written from the active blocks of the last step (the
// caller zeroes out first); which: 0 mass, 1 momentum (3), 2 velocity (3)
// from a probe's accumulators; 3 mass, 4 velocity (3) from the grid a fused
// step left (velocity and mass after its update), nodes with mass only, so
// that a slot the leftover P2G claimed in vain (empty) writes nothing.
template <int KIND>
__global__ void k_read_grid(const float4* Gacc, const float4* Gvel, const uint32_t* g_list, const uint32_t* g_scene,
                            const uint32_t* n_g, uint32_t pool_cap, const SceneDev* scenes, int scene, int which,
                            float* out) {
  constexpr int NG = Geo<KIND>::NG;
  const SceneDev s = scenes[scene];
  const int n = s.res + 1;
  const long long nnode = (long long)n * n * n;
  const uint32_t ng = min(*n_g, pool_cap);
  for (uint32_t gi = blockIdx.x; gi < ng; gi += gridDim.x) {
    if ((int)g_scene[gi] != scene) continue;
    long long lb = (long long)g_list[gi] - s.table_base;
    int gx = (int)(lb % s.nb), gy = (int)((lb / s.nb) % s.nb), gz = (int)(lb / ((long long)s.nb * s.nb));
    for (int t = threadIdx.x; t < NG * kBlockNodes; t += blockDim.x) {
      int grid = t / kBlockNodes, l = t % kBlockNodes;
      int ix = gx * 4 + (l & 3), iy = gy * 4 + ((l >> 2) & 3), iz = gz * 4 + (l >> 4);
      if (ix >= n || iy >= n || iz >= n) continue;
      long long q = grid * nnode + ((long long)iz * n + iy) * n + ix;
      long long idx = ((long long)gi * NG + grid) * kBlockNodes + l;
      if (which >= 3) {
        const float4 g = Gvel[idx];
        if (g.w > 0.f) {
          if (which == 3) {
            out[q] = g.w;
          } else {
            out[3 * q] = g.x; out[3 * q + 1] = g.y; out[3 * q + 2] = g.z;
          }
        }
        continue;
      }
      float4 a = Gacc[idx];
      if (which == 0) {
        out[q] = a.x;
      } else if (which == 1) {
        out[3 * q] = a.y; out[3 * q + 1] = a.z; out[3 * q + 2] = a.w;
      } else {
        float4 g = Gvel[idx];
        bool has = a.x > 0.f;
        out[3 * q] = has ? g.x : 0.f;
        out[3 * q + 1] = has ? g.y : 0.f;
        out[3 * q + 2] = has ? g.z : 0.f;
      }
    }
  }
}

// The allocation-free entry point's admission: the state that k_admit, an
// upload of F and one of B would leave (M = m B - dt V0 tau(F); pic: no B), its
// keys, histogram and bounds in one pass.
template <int KIND>
__global__ void __launch_bounds__(128) k_static_admit(StepView v, const __grid_constant__ StaticParams prm,
                                                      StaticParams* d_prm, int pic, uint32_t nmat, const float* x,
                                                      const float* vel, const uint8_t* mat, const float* Fin,
                                                      const float* Bin) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *d_prm = prm;
  const SceneDev& s = prm.scene;
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= v.n_cur) return;
  float px = x[3 * t], py = x[3 * t + 1], pz = x[3 * t + 2];
  float ux = px * s.inv_dx, uy = py * s.inv_dx, uz = pz * s.inv_dx;
  if (!(in_domain(ux, s.res) && in_domain(uy, s.res) && in_domain(uz, s.res))) {
    flag_error(v.err, CK_ERR_DOMAIN);
    const float lo = 0.5f, hi = (float)s.res - 0.5f - 1e-3f;
    ux = fminf(fmaxf(isfinite(ux) ? ux : lo, lo), hi);
    uy = fminf(fmaxf(isfinite(uy) ? uy : lo, lo), hi);
    uz = fminf(fmaxf(isfinite(uz) ? uz : lo, lo), hi);
    px = ux * s.dx; py = uy * s.dx; pz = uz * s.dx;
    ux = px * s.inv_dx; uy = py * s.inv_dx; uz = pz * s.inv_dx;
  }
  uint32_t m = mat ? (uint32_t)mat[t] : 0u;
  if (m >= nmat) {  // unknown material index: use material 0 and report
    flag_error(v.err, CK_ERR_INTERNAL);
    m = 0;
  }
  const MatDev& mt = prm.mats[m];
  const float vx = vel ? vel[3 * t] : 0.f, vy = vel ? vel[3 * t + 1] : 0.f, vz = vel ? vel[3 * t + 2] : 0.f;
  float M[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (Bin && !pic) {
#pragma unroll
    for (int q = 0; q < 9; ++q) M[q] = mt.mass * Bin[9 * t + q];
  }
  if (Fin) {  // tau(I) = 0 for every model
    float F[9], tau[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) F[q] = Fin[9 * t + q];
    stress_of(mt, F, mt.mu, mt.lam, tau);
    const float dtv = s.dt * s.V0;
#pragma unroll
    for (int q = 0; q < 9; ++q) M[q] -= dtv * tau[q];
  }
  v.cur.X[t] = make_float4(px, py, pz, __uint_as_float(m));
  v.cur.VM0[t] = make_float4(vx, vy, vz, 0.f);
  Pool P = v.cur;
  store_M(P, t, M);
  const uint32_t k = particle_key<KIND>(s, ux, uy, uz);
  v.key_cur[t] = k;
  float bmass, bmom;
  p2g_bounds<KIND>(s.inv_dx, mt.mass, V3{pk(vx, vy), vz}, from_rows(M), bmass, bmom);
  warp_aggregated_bin(v.cnt_cur, v.bnd_cur, k, bmass, bmom);
}

// Its results: mass and momentum of every node of the domain, read from the
// active blocks (a block is active when its table entry and the slot's list
// entry agree; entries of other blocks are stale) and zero elsewhere, in one
// pass that writes each output once.
template <int KIND>
__global__ void __launch_bounds__(128) k_static_grids(StepView v, uint32_t n_vblocks, float* gm, float* gp) {
  constexpr int NG = Geo<KIND>::NG;
  const int n = v.scenes[0].res + 1, nb = v.scenes[0].nb;
  const size_t nnode = (size_t)n * n * n;
  const uint32_t ng = min(*v.n_g, v.pool_cap);
  for (uint32_t b = blockIdx.x; b < n_vblocks; b += gridDim.x) {
    const uint32_t sl = v.table[b];
    const bool on = sl < ng && v.g_list[sl] == b;
    const int bx = (int)(b % (uint32_t)nb), by = (int)((b / (uint32_t)nb) % (uint32_t)nb), bz = (int)(b / ((uint32_t)nb * nb));
    for (int t = threadIdx.x; t < NG * kBlockNodes; t += 128) {
      const int g = t / kBlockNodes, l = t % kBlockNodes;
      const int ix = bx * 4 + (l & 3), iy = by * 4 + ((l >> 2) & 3), iz = bz * 4 + (l >> 4);
      if (ix >= n || iy >= n || iz >= n) continue;
      const float4 a = on ? v.Gacc[((size_t)sl * NG + g) * kBlockNodes + l] : make_float4(0.f, 0.f, 0.f, 0.f);
      const size_t q = g * nnode + ((size_t)iz * n + iy) * n + ix;
      gm[q] = a.x;
      gp[3 * q] = a.y;
      gp[3 * q + 1] = a.z;
      gp[3 * q + 2] = a.w;
    }
  }
}

// Append a new scene's particles: X (x, mat_base + mat), v, M = 0 (B = 0 and
// tau(I) = 0), F = I, ID = index; plus keys and the histogram.
template <int KIND>
__global__ void k_admit(Pool P, uint32_t* key, uint32_t* cnt, uint32_t* bnd, const SceneDev* scenes,
                        const MatDev* mats, int scene, uint32_t mat_base, uint32_t nmat, uint32_t start, uint32_t n,
                        const float* x, const float* vel, const uint8_t* mat, const float* E, uint32_t* err) {
  const SceneDev s = scenes[scene];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint32_t t = start + i;
    float px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2];
    float ux = px * s.inv_dx, uy = py * s.inv_dx, uz = pz * s.inv_dx;
    if (!(in_domain(ux, s.res) && in_domain(uy, s.res) && in_domain(uz, s.res))) {
      flag_error(err, CK_ERR_DOMAIN);
      const float lo = 0.5f, hi = (float)s.res - 0.5f - 1e-3f;
      ux = fminf(fmaxf(isfinite(ux) ? ux : lo, lo), hi);
      uy = fminf(fmaxf(isfinite(uy) ? uy : lo, lo), hi);
      uz = fminf(fmaxf(isfinite(uz) ? uz : lo, lo), hi);
      px = ux * s.dx; py = uy * s.dx; pz = uz * s.dx;
      ux = px * s.inv_dx; uy = py * s.inv_dx; uz = pz * s.inv_dx;
    }
    uint32_t mloc = mat ? (uint32_t)mat[i] : 0u;
    if (mloc >= nmat) {  // unknown material index: use material 0 and report
      flag_error(err, CK_ERR_INTERNAL);
      mloc = 0;
    }
    uint32_t m = mat_base + mloc;
    P.X[t] = make_float4(px, py, pz, __uint_as_float(m));
    float vx = vel ? vel[3 * i] : 0.f, vy = vel ? vel[3 * i + 1] : 0.f, vz = vel ? vel[3 * i + 2] : 0.f;
    P.VM0[t] = make_float4(vx, vy, vz, 0.f);
    P.VM1[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    P.VM2[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    P.F0[t] = make_float4(1.f, 0.f, 0.f, 1.f);
    P.F1[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    P.F2[t] = 1.f;
    P.ID[t] = i;
    if (P.E) P.E[t] = E ? E[i] : 0.f;
    if (P.T0) {  // tau(I) = 0 for every model
      P.T0[t] = make_float4(0.f, 0.f, 0.f, 0.f);
      P.T1[t] = make_float4(0.f, 0.f, 0.f, 0.f);
      P.T2[t] = 0.f;
    }
    uint32_t k = particle_key<KIND>(s, ux, uy, uz);
    key[t] = k;
    const M3 M0 = {{v3(0.f), v3(0.f), v3(0.f)}};
    float bmass, bmom;
    p2g_bounds<KIND>(s.inv_dx, mats[m].mass, V3{pk(vx, vy), vz}, M0, bmass, bmom);
    warp_aggregated_bin(cnt, bnd, k, bmass, bmom);
  }
}

// Recompute keys and the histogram of the whole current pool (after an
// upload of positions); particles already retired by a release keep the dead
// key and leave the pool at the next step.
template <int KIND>
__global__ void k_rekey(Pool P, uint32_t* key, uint32_t* cnt, uint32_t* bnd, const SceneDev* scenes,
                        const MatDev* mats, uint32_t n, uint32_t* err) {
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    if (key[t] == CK_DEAD_KEY) continue;  // retired by a release; its slot may already be reused
    float4 X = P.X[t];
    const MatDev mt = mats[__float_as_uint(X.w)];
    const SceneDev s = scenes[mt.scene];
    float ux = X.x * s.inv_dx, uy = X.y * s.inv_dx, uz = X.z * s.inv_dx;
    if (!(in_domain(ux, s.res) && in_domain(uy, s.res) && in_domain(uz, s.res))) {
      flag_error(err, CK_ERR_DOMAIN);
      const float lo = 0.5f, hi = (float)s.res - 0.5f - 1e-3f;
      ux = fminf(fmaxf(isfinite(ux) ? ux : lo, lo), hi);
      uy = fminf(fmaxf(isfinite(uy) ? uy : lo, lo), hi);
      uz = fminf(fmaxf(isfinite(uz) ? uz : lo, lo), hi);
      X.x = ux * s.dx; X.y = uy * s.dx; X.z = uz * s.dx;
      P.X[t] = X;
      ux = X.x * s.inv_dx; uy = X.y * s.inv_dx; uz = X.z * s.inv_dx;
    }
    uint32_t k = particle_key<KIND>(s, ux, uy, uz);
    key[t] = k;
    const float4 a = P.VM0[t];
    M3 M = unpack_m3(P.VM1[t], P.VM2[t], a.w);
    if (P.T0) M = abs_sum(M, unpack_m3(P.T0[t], P.T1[t], P.T2[t]));
    float bmass, bmom;
    p2g_bounds<KIND>(s.inv_dx, mt.mass, V3{pk(a.x, a.y), a.z}, M, bmass, bmom);
    warp_aggregated_bin(cnt, bnd, k, bmass, bmom);
  }
}

// ------------------------------------------------------------ host launchers

template <int KIND, int TR, int REP, int ROT, int FMA>
static void launch_p2g(const LaunchCfg& lc, const StepView& v) {
  if (v.units[kUnitsP2G].splits > 1u)
    k_p2g<KIND, TR, REP, ROT, FMA, true><<<v.work0[kUnitsP2G], kP2GWarp, 0, lc.stream>>>(v);
  else
    k_p2g<KIND, TR, REP, ROT, FMA, false><<<p2g_ctas(lc.sm_count), kP2GWarp, 0, lc.stream>>>(v);
}

// P2G of the APIC + MLS transfer: accumulator copies, component order and
// rounding as the launch configuration asks.
template <int KIND>
static void launch_p2g_apic(const LaunchCfg& lc, const StepView& v) {
  if (lc.p2g_rep == 2) {
    if (lc.p2g_fma)
      launch_p2g<KIND, 0, 2, 0, 1>(lc, v);
    else
      launch_p2g<KIND, 0, 2, 0, 0>(lc, v);
  } else if (lc.p2g_rot) {
    if (lc.p2g_fma)
      launch_p2g<KIND, 0, 1, 1, 1>(lc, v);
    else
      launch_p2g<KIND, 0, 1, 1, 0>(lc, v);
  } else {
    if (lc.p2g_fma)
      launch_p2g<KIND, 0, 1, 0, 1>(lc, v);
    else
      launch_p2g<KIND, 0, 1, 0, 0>(lc, v);
  }
}

template <int KIND, int MINB, int TR>
static void launch_g2p(const LaunchCfg& lc, const StepView& v, uint32_t g) {
  if (v.units[kUnitsG2P].splits > 1u)
    k_g2p<KIND, MINB, TR, true><<<g, kG2PWarp, 0, lc.stream>>>(v);
  else
    k_g2p<KIND, MINB, TR, false><<<g, kG2PWarp, 0, lc.stream>>>(v);
}

template <int KIND>
static void launch_all(const LaunchCfg& lc, StepView v, int which) {
  switch (which) {
    case LK_P2G:
      if (lc.transfer == 1)
        launch_p2g<KIND, 1, 1, KIND == 0, 1>(lc, v);
      else if (lc.transfer == 2)
        launch_p2g<KIND, 2, 1, KIND == 0, 1>(lc, v);
      else
        launch_p2g_apic<KIND>(lc, v);
      break;
    case LK_UPDATE:
      k_grid_update<KIND><<<update_ctas(KIND, lc.sm_count, v.pool_cap, v.n_cur), 128, 0, lc.stream>>>(v);
      break;
    case LK_G2P:
      // register budget of G2P: 20 warps/SM (96 registers) by default, the
      // faster for both kernels on the large-impact scene; 16 (119-124
      // registers) or 24 (80) on request.  One resident wave.  The kernel-
      // gradient transfers run one budget each: PIC the APIC default (16
      // warps/SM for the quadratic twin); the kernel-gradient APIC (two
      // gathers) 16 warps/SM for CK and 12 (168 registers, no spills) for
      // the quadratic twin.
      {
        const uint32_t g = (uint32_t)(lc.sm_count * g2p_warps(KIND, lc.transfer, lc.g2p_minb));
        if (lc.transfer == 1)
          launch_g2p<KIND, KIND == 0 ? 5 : 4, 1>(lc, v, g);
        else if (lc.transfer == 2)
          launch_g2p<KIND, KIND == 0 ? 4 : 3, 2>(lc, v, g);
        else if (lc.g2p_minb >= 6)
          launch_g2p<KIND, 6, 0>(lc, v, g);
        else if (lc.g2p_minb == 5)
          launch_g2p<KIND, 5, 0>(lc, v, g);
        else
          launch_g2p<KIND, 4, 0>(lc, v, g);
      }
      break;
    case LK_G2P_FP64: k_g2p_fp64<KIND><<<lc.sm_count * 4, 128, 0, lc.stream>>>(v); break;
    // fused step (APIC + MLS): one resident wave at the G2P register budget
    case LK_G2P2G:
      k_g2p2g<KIND, fused_warps(KIND) / 4><<<lc.sm_count * fused_warps(KIND), kG2PWarp, 0, lc.stream>>>(v);
      break;
    case LK_LEFTOVER: k_p2g_leftover<KIND><<<lc.sm_count * 4, 128, 0, lc.stream>>>(v); break;
    case LK_CLEAR: k_clear_gacc<KIND><<<lc.persistent_ctas, 128, 0, lc.stream>>>(v); break;
  }
}

void launch_transfer(int kind, const LaunchCfg& lc, const StepView& v, int which) {
  if (kind == 0)
    launch_all<0>(lc, v, which);
  else
    launch_all<1>(lc, v, which);
}

template <int KIND>
static void launch_read_field(int blocks, bool pic, cudaStream_t st, Pool P, const SceneDev* scenes,
                              const MatDev* mats, int scene, uint32_t start, uint32_t n, int field, float* out) {
  const int pc = pic ? 1 : 0;
  switch (field) {
    case 0: k_read_particles<KIND, 0><<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, pc, out); break;
    case 1: k_read_particles<KIND, 1><<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, pc, out); break;
    case 2: k_read_particles<KIND, 2><<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, pc, out); break;
    case 3: k_read_particles<KIND, 3><<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, pc, out); break;
    case 4: k_read_particles<KIND, 4><<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, pc, out); break;
    case 5: k_read_particles<KIND, 5><<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, pc, out); break;
  }
}

void launch_read_particles(int kind, bool pic, cudaStream_t st, Pool P, const SceneDev* scenes, const MatDev* mats,
                           int scene, uint32_t start, uint32_t n, int field, float* out) {
  int blocks = (int)((n + 255) / 256);
  if (blocks < 1) blocks = 1;
  if (blocks > 16384) blocks = 16384;
  if (kind == 0)
    launch_read_field<0>(blocks, pic, st, P, scenes, mats, scene, start, n, field, out);
  else
    launch_read_field<1>(blocks, pic, st, P, scenes, mats, scene, start, n, field, out);
}

void launch_write_particles(bool pic, cudaStream_t st, Pool P, const SceneDev* scenes, const MatDev* mats, int scene,
                            uint32_t start, uint32_t n, int field, const float* in) {
  int blocks = (int)((n + 255) / 256);
  if (blocks < 1) blocks = 1;
  if (blocks > 4096) blocks = 4096;
  k_write_particles<<<blocks, 256, 0, st>>>(P, scenes, mats, scene, start, n, field, pic ? 1 : 0, in);
}

void launch_read_grid(int kind, cudaStream_t st, const StepView& v, int scene, int which, float* out) {
  if (kind == 0)
    k_read_grid<0><<<1024, 128, 0, st>>>(v.Gacc, v.Gvel, v.g_list, v.g_scene, v.n_g, v.pool_cap, v.scenes, scene,
                                          which, out);
  else
    k_read_grid<1><<<1024, 128, 0, st>>>(v.Gacc, v.Gvel, v.g_list, v.g_scene, v.n_g, v.pool_cap, v.scenes, scene,
                                          which, out);
}

void launch_static_admit(int kind, cudaStream_t st, const StepView& v, const StaticParams& prm, StaticParams* d_prm,
                         bool pic, uint32_t nmat, const float* x, const float* vel, const uint8_t* mat, const float* F,
                         const float* B) {
  const uint32_t blocks = (v.n_cur + 127u) / 128u;
  if (kind == 0)
    k_static_admit<0><<<blocks, 128, 0, st>>>(v, prm, d_prm, pic ? 1 : 0, nmat, x, vel, mat, F, B);
  else
    k_static_admit<1><<<blocks, 128, 0, st>>>(v, prm, d_prm, pic ? 1 : 0, nmat, x, vel, mat, F, B);
}

void launch_static_grids(int kind, cudaStream_t st, const StepView& v, uint32_t n_vblocks, float* grid_m,
                         float* grid_p) {
  if (kind == 0)
    k_static_grids<0><<<n_vblocks, 128, 0, st>>>(v, n_vblocks, grid_m, grid_p);
  else
    k_static_grids<1><<<n_vblocks, 128, 0, st>>>(v, n_vblocks, grid_m, grid_p);
}

void launch_admit(int kind, cudaStream_t st, Pool P, uint32_t* key, uint32_t* cnt, uint32_t* bnd,
                  const SceneDev* scenes, const MatDev* mats, int scene, uint32_t mat_base, uint32_t nmat,
                  uint32_t start, uint32_t n, const float* x, const float* v, const uint8_t* mat, const float* E,
                  uint32_t* err) {
  int blocks = (int)((n + 255) / 256);
  if (blocks < 1) blocks = 1;
  if (blocks > 8192) blocks = 8192;
  if (kind == 0)
    k_admit<0><<<blocks, 256, 0, st>>>(P, key, cnt, bnd, scenes, mats, scene, mat_base, nmat, start, n, x, v, mat, E,
                                        err);
  else
    k_admit<1><<<blocks, 256, 0, st>>>(P, key, cnt, bnd, scenes, mats, scene, mat_base, nmat, start, n, x, v, mat, E,
                                        err);
}

void launch_rekey(int kind, cudaStream_t st, Pool P, uint32_t* key, uint32_t* cnt, uint32_t* bnd,
                  const SceneDev* scenes, const MatDev* mats, uint32_t n, uint32_t* err) {
  int blocks = (int)((n + 255) / 256);
  if (blocks < 1) blocks = 1;
  if (blocks > 8192) blocks = 8192;
  if (kind == 0)
    k_rekey<0><<<blocks, 256, 0, st>>>(P, key, cnt, bnd, scenes, mats, n, err);
  else
    k_rekey<1><<<blocks, 256, 0, st>>>(P, key, cnt, bnd, scenes, mats, n, err);
}

}  // namespace ck
