// gd_boxes.cuh -- bounding boxes over Morton-ordered points, and exact pruning by
// them.  32 consecutive points form a chunk, 32 chunks a super-chunk; in octree
// order both are compact in space, so most of them lie farther from a query than
// the distance that still matters, and are skipped whole.
//
// The pruning is exact in the arithmetic of the method, not up to a rounding
// slack.  FP32 subtraction, multiplication and fused multiply-add round
// monotonically, so for a query q and any point x of a box [lo, hi], per axis,
// gap = max(0, fl(lo - q), fl(q - hi)) <= |fl(x - q)|, and the squared distance
// formed from the three gaps by the same operations (fma(dz, dz, fma(dy, dy,
// dx * dx))) never exceeds the computed d^2 of any point in the box.  The same
// holds for a box of queries, and, with the far corners, for the upper bound.
#pragma once

#include "gd_common.cuh"

namespace gd {

constexpr uint32_t kBoxChunk = 32;    // points per chunk: one per lane
constexpr uint32_t kBoxSuper = 1024;  // points per super-chunk: one chunk per lane

struct Box {
  float lo[3], hi[3];  // empty: lo > hi
};

// Chunk boxes and super-chunk boxes of an array of points: lo at [2 i], hi at [2 i + 1].
struct BoxIndex {
  float4 *chunk, *super;
};
__host__ __device__ __forceinline__ uint32_t box_chunks(uint32_t n) { return (n + kBoxChunk - 1) / kBoxChunk; }
__host__ __device__ __forceinline__ uint32_t box_supers(uint32_t n) { return (n + kBoxSuper - 1) / kBoxSuper; }
// bytes of the index of n points (a multiple of 32)
__host__ __device__ __forceinline__ size_t box_bytes(uint32_t n) {
  return 32ull * ((size_t)box_chunks(n) + box_supers(n));
}
__host__ __device__ __forceinline__ BoxIndex box_index(unsigned char *p, uint32_t n) {
  return BoxIndex{reinterpret_cast<float4 *>(p), reinterpret_cast<float4 *>(p + 32ull * box_chunks(n))};
}

__device__ __forceinline__ Box box_load(const float4 *__restrict__ b, uint32_t i) {
  const float4 l = b[2ull * i], h = b[2ull * i + 1];
  return Box{{l.x, l.y, l.z}, {h.x, h.y, h.z}};
}
__device__ __forceinline__ void box_store(float4 *b, uint32_t i, const Box &x) {
  b[2ull * i] = make_float4(x.lo[0], x.lo[1], x.lo[2], 0.0f);
  b[2ull * i + 1] = make_float4(x.hi[0], x.hi[1], x.hi[2], 0.0f);
}

// smallest / largest value over the warp (floats through their ordered integers; no NaN)
__device__ __forceinline__ float warp_fmin(float v) { return ord2f(__reduce_min_sync(0xFFFFFFFFu, f2ord(v))); }
__device__ __forceinline__ float warp_fmax(float v) { return ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(v))); }

// the warp's union of one box per lane
__device__ __forceinline__ Box box_warp_union(Box b) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    b.lo[a] = warp_fmin(b.lo[a]);
    b.hi[a] = warp_fmax(b.hi[a]);
  }
  return b;
}
__device__ __forceinline__ Box box_empty() {
  return Box{{INFINITY, INFINITY, INFINITY}, {-INFINITY, -INFINITY, -INFINITY}};
}
__device__ __forceinline__ Box box_point(float x, float y, float z) { return Box{{x, y, z}, {x, y, z}}; }

// Lower bound of the computed d^2 between any point of b and any point of q;
// +infinity for an empty box (the caller skips an empty box by its own test where
// an infinite bound is not above its limit).
__device__ __forceinline__ float box_lower(const Box &b, const Box &q) {
  float g[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    g[a] = fmaxf(0.0f, fmaxf(__fsub_rn(b.lo[a], q.hi[a]), __fsub_rn(q.lo[a], b.hi[a])));
  return __fmaf_rn(g[2], g[2], __fmaf_rn(g[1], g[1], __fmul_rn(g[0], g[0])));
}
// Upper bound of the same (the far corners).
__device__ __forceinline__ float box_upper(const Box &b, const Box &q) {
  float g[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    g[a] = fmaxf(__fsub_rn(b.hi[a], q.lo[a]), __fsub_rn(q.hi[a], b.lo[a]));
  return __fmaf_rn(g[2], g[2], __fmaf_rn(g[1], g[1], __fmul_rn(g[0], g[0])));
}
__device__ __forceinline__ bool box_is_empty(const Box &b) { return b.lo[0] > b.hi[0]; }

}  // namespace gd
