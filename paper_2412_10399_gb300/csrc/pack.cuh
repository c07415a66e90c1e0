// Packed float32 arithmetic (two lanes per instruction, sm_100 and later) and
// the small matrix types the transfer kernels keep in it.
//
// Why: G2P and P2G are bound by their issue slots, not by the FMA pipe (72%
// of the slots issue while the pipe is 42% busy).  A packed multiply-add does
// the work of two in one slot; measured on GB300 it takes the pipe twice as
// long (1.94 against 3.50 warp instructions per clock and SM, 3.87 against
// 3.50 multiply-adds), leaves the other slot to the remaining instructions,
// and takes a scalar as both halves of an operand, or two separately computed
// scalars as its two halves, without a move.
// Rounding is that of the scalar operations.
//
// Which pairs: rows 0 and 1 of every 3x3 matrix (and the x and y components of
// every vector), with row 2 (z) in scalars.  The gather then works on the
// (x, y) half of a node's float4 as it was loaded, every product with the
// matrix from the right keeps the pairing, and the particle arrays store F
// and M in that order (common.cuh), so that no component is moved.
#pragma once
#include <cuda_runtime.h>

namespace ck {

using f2 = float2;

__device__ __forceinline__ f2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 neg2(f2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }

// A 3-vector (per axis or per component): x and y packed.
struct V3 {
  f2 p;
  float z;
};
__device__ __forceinline__ V3 v3(float a) { return {dup(a), a}; }
__device__ __forceinline__ V3 operator+(const V3& a, const V3& b) { return {add2(a.p, b.p), a.z + b.z}; }
__device__ __forceinline__ V3 operator-(const V3& a, const V3& b) { return {add2(a.p, neg2(b.p)), a.z - b.z}; }
__device__ __forceinline__ V3 operator*(const V3& a, const V3& b) { return {mul2(a.p, b.p), a.z * b.z}; }
__device__ __forceinline__ V3 operator*(float a, const V3& b) { return {mul2(dup(a), b.p), a * b.z}; }
__device__ __forceinline__ V3 fma3(const V3& a, const V3& b, const V3& c) {
  return {fma2(a.p, b.p, c.p), fmaf(a.z, b.z, c.z)};
}
__device__ __forceinline__ V3 fma3(float a, const V3& b, const V3& c) {
  return {fma2(dup(a), b.p, c.p), fmaf(a, b.z, c.z)};
}
__device__ __forceinline__ V3 neg3(const V3& a) { return {neg2(a.p), -a.z}; }
// component a (0..2) of a 3-vector, a known at compile time
__device__ __forceinline__ float at3(const V3& v, int a) { return a == 0 ? v.p.x : a == 1 ? v.p.y : v.z; }

// A 3x3 matrix as its columns: c[q] = (M0q, M1q, M2q).
struct M3 {
  V3 c[3];
};
__device__ __forceinline__ float at(const M3& m, int r, int q) { return at3(m.c[q], r); }
__device__ __forceinline__ void to_rows(const M3& m, float* r) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 3; ++q) r[i * 3 + q] = at(m, i, q);
}
__device__ __forceinline__ M3 from_rows(const float* r) {
  M3 m;
#pragma unroll
  for (int q = 0; q < 3; ++q) m.c[q] = {pk(r[q], r[3 + q]), r[6 + q]};
  return m;
}
// acc + A B
__device__ __forceinline__ M3 mul_add(const M3& A, const M3& B, const M3& acc) {
  M3 r;
#pragma unroll
  for (int q = 0; q < 3; ++q)
    r.c[q] = fma3(at(B, 0, q), A.c[0], fma3(at(B, 1, q), A.c[1], fma3(at(B, 2, q), A.c[2], acc.c[q])));
  return r;
}

// The stored order of a 3x3 matrix: (00, 10, 01, 11), (02, 12, 20, 21), 22.
__device__ __forceinline__ M3 unpack_m3(const float4& a, const float4& b, float c) {
  return {{{pk(a.x, a.y), b.z}, {pk(a.z, a.w), b.w}, {pk(b.x, b.y), c}}};
}
__device__ __forceinline__ void pack_m3(const M3& m, float4& a, float4& b, float& c) {
  a = make_float4(m.c[0].p.x, m.c[0].p.y, m.c[1].p.x, m.c[1].p.y);
  b = make_float4(m.c[2].p.x, m.c[2].p.y, m.c[0].z, m.c[1].z);
  c = m.c[2].z;
}

// A symmetric 3x3 matrix: d = (00, 11), o = (02, 12), c = 22, e = 01.
struct Sym {
  f2 d, o;
  float c, e;
};
__device__ __forceinline__ Sym scale(float s, const Sym& a) { return {mul2(dup(s), a.d), mul2(dup(s), a.o), s * a.c, s * a.e}; }
__device__ __forceinline__ Sym add_diag(float t, const Sym& a) { return {add2(dup(t), a.d), a.o, t + a.c, a.e}; }
// t I + A B for commuting A and B (polynomials in one matrix; the result is
// symmetric): 12 instructions.
__device__ __forceinline__ Sym sym_mul(const Sym& a, const Sym& b, float t) {
  Sym r;
  r.d = fma2(a.d, b.d, fma2(dup(a.e), dup(b.e), fma2(a.o, b.o, dup(t))));
  r.o = fma2(a.d, b.o, fma2(dup(a.e), pk(b.o.y, b.o.x), mul2(a.o, dup(b.c))));
  r.c = fmaf(a.o.x, b.o.x, fmaf(a.o.y, b.o.y, fmaf(a.c, b.c, t)));
  r.e = fmaf(a.d.x, b.e, fmaf(a.e, b.d.y, a.o.x * b.o.y));
  return r;
}
// the matrix by columns (as M3)
__device__ __forceinline__ M3 sym_m3(const Sym& a) {
  return {{{pk(a.d.x, a.e), a.o.x}, {pk(a.e, a.d.y), a.o.y}, {a.o, a.c}}};
}

}  // namespace ck
