// gd_eval_box.cu -- the two cross-set passes of gd_eval.cu (nearest squared
// distance, count within a radius) for large clouds, without comparing every pair:
// both clouds are brought into octree order by the front end (as two frames of one
// batch), 32-point chunks and 1,024-point super-chunks get boxes (gd_boxes.cuh), and
// a query reads only the chunks that can change its result.  The pruning is exact in
// the method's FP32 arithmetic, so every distance and count equals the full pass's.
//
// One warp takes a chunk of 32 consecutive queries, one a lane, and reads the needed
// candidate chunks through shared memory.  Queries far apart (outliers share chunks
// with points of other regions) would make their warp read the union of many
// regions; they go on a list and get a warp of their own, with the candidates
// across the lanes.
//
// 500,000 against 510,000 points (two passes): 96.8 ms -> 0.95 ms, 0.77 ms of it the
// four search kernels; counts within 8 % of the extent among 560,000 points: 73.0 ms
// -> 2.27 ms.  The full pass is bound by the FP32 pipe; these by the box tests and the
// chunks that the spheres' borders cross: issue in 62 % (nearest) and 67 % (counts) of the
// cycles with 37 and 41 % of the warp slots occupied, no one stall on top.
#include "gd_boxes.cuh"
#include "gd_f32x2.cuh"

namespace gd {

namespace {
constexpr int kEbWarps = 4;
constexpr int kEbThreads = 32 * kEbWarps;
// A nearest-neighbour query is left to a warp of its own once its share of the chunks
// it wants (each split evenly over the queries that want it) is this many: a chunk
// costs the warp about 200 instructions, a query of its own about 700.  With fewer
// warps than fill the GPU the last warp's time counts, and queries leave earlier.
// Measured, us a call at shares 1 / 2 / 4: object of 30,000 points 266 / 308 / 334,
// scans of 250,000 709 / 609 / 608 and 500,000 1499 / 1075 / 946.  A cloud of a few
// hundred chunks of queries (against one of millions of points) has too few warps for
// anything else: each query leaves at its first chunk.  us a call, share 1 / 0 (the full
// pass): 500 against 1.2 M uniform points 604 / 400 (430), 1,600 against 400,000 397 / 265
// (386), 16,000 against 1.2 M 618 / 518 (7187).
inline float nn_share(uint32_t chunks) {
  return chunks < 600u ? 0.0f : chunks < 2500u ? 1.0f : chunks < 8000u ? 2.0f : 4.0f;
}
constexpr uint32_t kCntList = 768;   // chunks of the radius count's list
constexpr uint32_t kCntBlock = 64;   // of them split into quarters at a time
constexpr uint32_t kQuarter = kBoxChunk / 4;
// A chunk on the list costs its 32 queries together about 190 instructions at most (its
// quarters beyond or within every sphere are dropped first); a query of
// its own about 600 and 15 for every chunk that straddles its own sphere.  The chunk
// of queries is left to single-query warps when that is less (queries far apart: the
// list holds the borders of many spheres).
__device__ __forceinline__ bool cnt_apart(uint32_t listed, uint32_t own) {
  return listed * 190u > 32u * (600u + 15u * own);
}
// Below this many chunks of queries the warps of a block share one, each with a fourth of
// the super-chunks: one warp a chunk leaves most of the GPU's schedulers one warp or
// two, waiting for their own loads.  us a call, one / four warps, R = 0.05 / 0.45 of the
// extent: 36,750 points of a sphere 245 / 205, 824 / 448 (the full pass 540); 200,000 399 /
// 369, 4407 / 2694; 560,000 at 0.02 / 0.3 589 / 651, 7039 / 6211; 1 M 1058 / 1280, 16610 / 15684.
constexpr uint32_t kCntSplit = 8192;
constexpr float kInf = INFINITY;

struct Cloud {                  // one cloud in octree order
  const float4 *pts;            // x, y, z, index bits in the concatenated input
  uint32_t n, first;            // points, index of the cloud's first point in the concatenation
  BoxIndex box;
  float4 *quarter;              // boxes of every kQuarter points (radius counts only, else null)
  const unsigned long long *keys;
  const FrameInfo *frame;
};

struct EbWork {
  uint32_t nn_far[2];           // queries on the far list of each direction
  uint32_t cnt_far;             // chunks on the far list
};
}  // namespace

// one block: the two frames and their tiles, and the work counters
__global__ void __launch_bounds__(256) k_evb_tables(FrameInfo *frames, Tile *tiles, uint32_t na, uint32_t nb,
                                                    EbWork *work) {
  const uint32_t t = threadIdx.x;
  if (t < 2) {
    FrameInfo f{};
    f.begin = t ? na : 0u;
    f.end = t ? na + nb : na;
    frames[t] = f;
  }
  if (t == 2) *work = EbWork{};
  const uint32_t ta = (na + kTilePts - 1) / kTilePts, tb = (nb + kTilePts - 1) / kTilePts;
  for (uint32_t i = t; i < ta + tb; i += 256u) {
    const uint32_t f = i >= ta, e = f ? na + nb : na, b = (f ? na : 0u) + (f ? i - ta : i) * (uint32_t)kTilePts;
    tiles[i] = Tile{f, b, (e - b > (uint32_t)kTilePts) ? b + (uint32_t)kTilePts : e, f ? ta : 0u};
  }
}

// the clouds one behind the other
__global__ void k_evb_cat(const float *__restrict__ a, size_t na3, const float *__restrict__ b, size_t nb3,
                          float *__restrict__ out) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < na3 + nb3; i += (size_t)gridDim.x * blockDim.x)
    out[i] = i < na3 ? a[i] : b[i - na3];
}

// chunk and super-chunk boxes: one block per super-chunk
__global__ void __launch_bounds__(kBoxSuper) k_evb_boxes(const Cloud A, const Cloud B, const Counters *ctr) {
  __shared__ Box s_box[32];
  if (ctr->status & kStFatal) return;
  const uint32_t sa = box_supers(A.n), lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const Cloud &c = blockIdx.x < sa ? A : B;
  const uint32_t s = blockIdx.x < sa ? blockIdx.x : blockIdx.x - sa, i = s * kBoxSuper + threadIdx.x;
  Box b = box_empty();
  if (i < c.n) {
    const float4 p = c.pts[i];
    b = box_point(p.x, p.y, p.z);
  }
  if (c.quarter) {
    Box h = b;
#pragma unroll
    for (int o = 1; o < (int)kQuarter; o *= 2) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        h.lo[d] = fminf(h.lo[d], __shfl_xor_sync(0xFFFFFFFFu, h.lo[d], o));
        h.hi[d] = fmaxf(h.hi[d], __shfl_xor_sync(0xFFFFFFFFu, h.hi[d], o));
      }
    }
    if (i % kQuarter == 0 && i < c.n) box_store(c.quarter, i / kQuarter, h);
  }
  b = box_warp_union(b);
  if (lane == 0) {
    if (i < c.n) box_store(c.box.chunk, s * 32u + w, b);
    s_box[w] = b;
  }
  __syncthreads();
  if (w == 0) {
    b = box_warp_union(s_box[lane]);
    if (lane == 0) box_store(c.box.super, s, b);
  }
}

// one lane's point of a chunk, +infinity past the end (at infinite distance)
__device__ __forceinline__ float4 eb_fetch(const Cloud &c, uint32_t chunk) {
  const uint32_t p = chunk * kBoxChunk + (threadIdx.x & 31u);
  return p < c.n ? c.pts[p] : make_float4(kInf, kInf, kInf, 0.0f);
}
struct EbChunk {
  float x[kBoxChunk], y[kBoxChunk], z[kBoxChunk];
};
__device__ __forceinline__ void eb_stage(EbChunk &S, const float4 &v) {
  const uint32_t lane = threadIdx.x & 31u;
  __syncwarp();
  S.x[lane] = v.x;
  S.y[lane] = v.y;
  S.z[lane] = v.z;
  __syncwarp();
}
// d^2 of the query to four staged candidates
__device__ __forceinline__ void eb_d2x4(const EbChunk &S, uint32_t j, f32x2 QX, f32x2 QY, f32x2 QZ, f32x2 &s0,
                                        f32x2 &s1) {
  const float4 x = *reinterpret_cast<const float4 *>(S.x + j), y = *reinterpret_cast<const float4 *>(S.y + j),
               z = *reinterpret_cast<const float4 *>(S.z + j);
  const f32x2 dx0 = sub2(pk2(x.x, x.y), QX), dx1 = sub2(pk2(x.z, x.w), QX);
  const f32x2 dy0 = sub2(pk2(y.x, y.y), QY), dy1 = sub2(pk2(y.z, y.w), QY);
  const f32x2 dz0 = sub2(pk2(z.x, z.y), QZ), dz1 = sub2(pk2(z.z, z.w), QZ);
  s0 = fma2(dz0, dz0, fma2(dy0, dy0, mul2(dx0, dx0)));
  s1 = fma2(dz1, dz1, fma2(dy1, dy1, mul2(dx1, dx1)));
}
__device__ __forceinline__ float eb_d2(float qx, float qy, float qz, const float4 &p) {
  const float dx = __fsub_rn(p.x, qx), dy = __fsub_rn(p.y, qy), dz = __fsub_rn(p.z, qz);
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}
__device__ __forceinline__ float eb_min_chunk(const EbChunk &S, f32x2 QX, f32x2 QY, f32x2 QZ, float best) {
#pragma unroll
  for (uint32_t j = 0; j < kBoxChunk; j += 4u) {
    f32x2 s0, s1;
    eb_d2x4(S, j, QX, QY, QZ, s0, s1);
    float a0, a1, a2, a3, m;
    upk2(s0, a0, a1);
    upk2(s1, a2, a3);
    asm("min.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a0), "f"(a1), "f"(a2));
    asm("min.f32 %0, %1, %2, %3;" : "=f"(best) : "f"(best), "f"(m), "f"(a3));
  }
  return best;
}

// box `u` of the warp's one-a-lane boxes, in every lane
__device__ __forceinline__ Box box_shfl(const Box &b, int u) {
  Box x;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    x.lo[d] = __shfl_sync(0xFFFFFFFFu, b.lo[d], u);
    x.hi[d] = __shfl_sync(0xFFFFFFFFu, b.hi[d], u);
  }
  return x;
}

// the chunk of C where a point would lie in C's octree order (a good first guess of
// where its neighbours are; it decides nothing)
__device__ __forceinline__ uint32_t eb_locate(const Cloud &C, float x, float y, float z) {
  const FrameInfo &f = *C.frame;
  auto q = [&](float v, int a) { return v < f.lo[a] ? 0u : quantise(v, f.lo[a], f.s); };
  const unsigned long long k = morton3(q(x, 0), q(y, 1), q(z, 2)) >> 32;  // the bits the front end sorts by
  uint32_t lo = 0, hi = C.n;
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if ((C.keys[mid] >> 32) < k) lo = mid + 1;
    else hi = mid;
  }
  return min(lo, C.n - 1u) / kBoxChunk;
}

// ---------------------------------------------------------------------------
// nearest squared distance
// ---------------------------------------------------------------------------
// far[dir] list: the queries' positions; their bound so far is in out[]
__global__ void __launch_bounds__(kEbThreads) k_evb_nn(const Cloud Q, const Cloud C, float *__restrict__ out,
                                                       uint32_t *__restrict__ far, EbWork *work, int dir,
                                                       float most, const Counters *ctr) {
  __shared__ __align__(16) EbChunk s_c[kEbWarps];
  if (ctr->status & kStFatal) return;
  EbChunk &S = s_c[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31u, nsu = box_supers(C.n), nch = box_chunks(C.n);
  const uint32_t qc = blockIdx.x * kEbWarps + (threadIdx.x >> 5);
  if (qc >= box_chunks(Q.n)) return;
  const uint32_t q = qc * kBoxChunk + lane;
  const bool real = q < Q.n;
  const float4 me4 = Q.pts[real ? q : Q.n - 1u];
  const Box me = box_point(me4.x, me4.y, me4.z);
  const Box qb = box_load(Q.box.chunk, qc);
  const f32x2 QX = pk2(me4.x, me4.x), QY = pk2(me4.y, me4.y), QZ = pk2(me4.z, me4.z);
  float best = kInf;
  // start where the first, middle and last query would lie in the other cloud's order
  const uint32_t g = eb_locate(C, __shfl_sync(0xFFFFFFFFu, me4.x, 16), __shfl_sync(0xFFFFFFFFu, me4.y, 16),
                               __shfl_sync(0xFFFFFFFFu, me4.z, 16));
  const uint32_t g0 = g ? g - 1u : 0u, g1 = min(g + 1u, nch - 1u);
  for (uint32_t c = g0; c <= g1; ++c) {
    eb_stage(S, eb_fetch(C, c));
    best = eb_min_chunk(S, QX, QY, QZ, best);
  }
  float share = 0.0f;
  bool gone = false;
  for (uint32_t s0 = 0; s0 < nsu; s0 += 32u) {
    const uint32_t s = s0 + lane;
    const float bound = ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(best)));
    Box sb = box_empty();
    if (s < nsu) sb = box_load(C.box.super, s);
    uint32_t m = __ballot_sync(0xFFFFFFFFu, s < nsu && box_lower(sb, qb) < bound);
    while (m) {
      const int u = __ffs(m) - 1;
      m &= m - 1u;
      if (!__any_sync(0xFFFFFFFFu, box_lower(box_shfl(sb, u), me) < best)) continue;
      const uint32_t c = (s0 + (uint32_t)u) * 32u + lane;
      Box cb = box_empty();
      if (c < nch && (c < g0 || c > g1)) cb = box_load(C.box.chunk, c);
      uint32_t cm = __ballot_sync(0xFFFFFFFFu, !box_is_empty(cb) && box_lower(cb, qb) < bound);
      while (cm) {
        const int v = __ffs(cm) - 1;
        cm &= cm - 1u;
        const bool want = box_lower(box_shfl(cb, v), me) < best;
        const uint32_t wm = __ballot_sync(0xFFFFFFFFu, want);
        if (!wm) continue;
        eb_stage(S, eb_fetch(C, (s0 + (uint32_t)u) * 32u + (uint32_t)v));
        best = eb_min_chunk(S, QX, QY, QZ, best);  // (-1, a query that left, stays)
        if (want) share += __fdividef(1.0f, (float)__popc(wm));
        const uint32_t gm = __ballot_sync(0xFFFFFFFFu, real && !gone && share >= most);
        if (gm) {  // these get a warp of their own, from the bound they have
          uint32_t slot = 0;
          if (lane == 0) slot = atomicAdd(&work->nn_far[dir], (uint32_t)__popc(gm));
          slot = __shfl_sync(0xFFFFFFFFu, slot, 0) + __popc(gm & lanemask_lt());
          if ((gm >> lane) & 1u) {
            far[slot] = q;
            out[__float_as_uint(me4.w) - Q.first] = best;
            gone = true;
          }
          if (gone || !real) best = -1.0f;  // asks for nothing more
        }
      }
    }
  }
  if (real && !gone) out[__float_as_uint(me4.w) - Q.first] = best;
}

// one query a warp: candidates across the lanes, the nearest super-chunk first
__global__ void __launch_bounds__(kEbThreads) k_evb_nn_far(const Cloud Q, const Cloud C, float *__restrict__ out,
                                                           const uint32_t *__restrict__ far, const EbWork *work,
                                                           int dir, const Counters *ctr) {
  if (ctr->status & kStFatal) return;
  const uint32_t lane = threadIdx.x & 31u, nf = work->nn_far[dir], nsu = box_supers(C.n), nch = box_chunks(C.n);
  for (uint32_t i = blockIdx.x * kEbWarps + (threadIdx.x >> 5); i < nf; i += gridDim.x * kEbWarps) {
    const float4 me4 = Q.pts[far[i]];
    const Box me = box_point(me4.x, me4.y, me4.z);
    float *const o = out + (__float_as_uint(me4.w) - Q.first);
    float best = *o;  // warp-uniform
    auto super = [&](uint32_t s) {  // its chunks, nearest first
      const uint32_t c = s * 32u + lane;
      const float lb = c < nch ? box_lower(box_load(C.box.chunk, c), me) : kInf;
      uint32_t left = __ballot_sync(0xFFFFFFFFu, c < nch && lb < best);
      while (left) {
        const uint32_t v = ((left >> lane) & 1u) ? __float_as_uint(lb) : 0xFFFFFFFFu;
        const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, v);
        if (!(__uint_as_float(mn) < best)) break;
        const int u = __ffs(__ballot_sync(0xFFFFFFFFu, v == mn)) - 1;
        left &= ~(1u << u);
        const float d = eb_d2(me4.x, me4.y, me4.z, eb_fetch(C, s * 32u + (uint32_t)u));
        best = fminf(best, __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, __float_as_uint(d))));
      }
    };
    uint32_t near = 0xFFFFFFFFu, ns = 0;
    for (uint32_t s = lane; s < nsu; s += 32u) {
      const uint32_t v = __float_as_uint(box_lower(box_load(C.box.super, s), me));
      if (v < near) {
        near = v;
        ns = s;
      }
    }
    const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, near);
    ns = __shfl_sync(0xFFFFFFFFu, ns, __ffs(__ballot_sync(0xFFFFFFFFu, near == mn)) - 1);
    super(ns);
    for (uint32_t s0 = 0; s0 < nsu; s0 += 32u) {
      const uint32_t s = s0 + lane;
      const float lb = (s < nsu && s != ns) ? box_lower(box_load(C.box.super, s), me) : kInf;
      uint32_t m = __ballot_sync(0xFFFFFFFFu, lb < best);
      while (m) {
        const int u = __ffs(m) - 1;
        m &= m - 1u;
        if (__shfl_sync(0xFFFFFFFFu, lb, u) < best) super(s0 + (uint32_t)u);
      }
    }
    if (lane == 0) *o = best;
  }
}

// ---------------------------------------------------------------------------
// counts within a radius (of every point of C among C's points)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t eb_points(uint32_t first, uint32_t span, uint32_t n) {
  return first < n ? min(span, n - first) : 0u;
}

// Compared chunks, not box tests, are most of the count's time, and the shell of
// chunks that a warp's spheres cut is as thick as the queries' box and the chunk
// together: boxes of 8 points make the second half as thick on a surface.  us a call
// before / after (32-point chunks compared whole, their list built twice): 560,000 points of a
// scan in millimetres 2,635 / 2,270, the same in units of 6.7 mm 667 / 525, object of
// 560,000 446 / 365, 36,750 283 / 272.  An integer comparison in place of the packed
// subtraction changed nothing (2,277).
//
// The listed chunks: their quarters that lie within the radius of all of the warp's
// queries go to `whole`, those beyond it of all are dropped, and the others are
// compared, four at a time (`done` counts such fours); returns the candidates compared
// that lie outside the lane's radius.
__device__ __forceinline__ uint32_t eb_border(const Cloud &C, EbChunk &S, const uint32_t *list, uint32_t nl,
                                              uint32_t *part, const Box &qb, float r2, f32x2 QX, f32x2 QY, f32x2 QZ,
                                              f32x2 R2, uint32_t &whole, uint32_t &done) {
  const uint32_t lane = threadIdx.x & 31u;
  auto fetch = [&](uint32_t four) {
    const uint32_t p = part[4u * four + lane / kQuarter] * kQuarter + lane % kQuarter;
    return p < C.n ? C.pts[p] : make_float4(kInf, kInf, kInf, 0.0f);
  };
  uint32_t beyond = 0;
  __syncwarp();  // the list is written
  for (uint32_t base = 0; base < nl; base += kCntBlock) {
    const uint32_t top = min(nl - base, kCntBlock);
    uint32_t np = 0;
    for (uint32_t i = 0; i < top; i += 8u) {
      const uint32_t e = i + lane / 4u;
      const uint32_t id = e < top ? list[base + e] * 4u + lane % 4u : 0u;
      bool edge = false;
      if (e < top && id * kQuarter < C.n) {
        const Box b = box_load(C.quarter, id);
        if (box_upper(b, qb) <= r2)
          whole += eb_points(id * kQuarter, kQuarter, C.n);
        else
          edge = box_lower(b, qb) <= r2;
      }
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, edge);
      if (edge) part[np + __popc(m & lanemask_lt())] = id;
      np += __popc(m);
    }
    if (lane < 3u) part[np + lane] = (C.n + kQuarter - 1u) / kQuarter;  // past the end: at infinite distance
    __syncwarp();
    const uint32_t fours = (np + 3u) / 4u;
    float4 v = fours ? fetch(0) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (uint32_t i = 0; i < fours; ++i) {
      eb_stage(S, v);
      if (i + 1 < fours) v = fetch(i + 1);  // on its way while these are compared
      uint32_t bits = 0;  // one bit a candidate, all 32 shifted through
#pragma unroll
      for (uint32_t j = 0; j < kBoxChunk; j += 4u) {
        f32x2 s0, s1;
        eb_d2x4(S, j, QX, QY, QZ, s0, s1);
        float e[4];  // the sign of r2 - d^2 is set exactly when d^2 > r2
        upk2(sub2(R2, s0), e[0], e[1]);
        upk2(sub2(R2, s1), e[2], e[3]);
#pragma unroll
        for (int u = 0; u < 4; ++u) bits = __funnelshift_l(__float_as_uint(e[u]), bits, 1);
      }
      beyond += __popc(bits);
    }
    done += fours;
    __syncwarp();  // the quarters' and the chunks' lists may be written again
  }
  return beyond;
}

// kSplit warps (1 or all of a block) share a chunk of queries, each with every kSplit-th
// super-chunk.
template <int kSplit>
__global__ void __launch_bounds__(kEbThreads) k_evb_count(const Cloud C, const float *__restrict__ r2_dev,
                                                          uint32_t *__restrict__ out, uint32_t *__restrict__ far,
                                                          EbWork *work, const Counters *ctr) {
  static_assert(kSplit == 1 || kSplit == kEbWarps, "the warps of a chunk are one warp or the whole block");
  __shared__ __align__(16) EbChunk s_c[kEbWarps];
  __shared__ uint32_t s_list[kEbWarps][kCntList], s_part[kEbWarps][4u * kCntBlock + 3u];
  __shared__ uint32_t s_sum[2], s_out[kBoxChunk];
  if (ctr->status & kStFatal) return;
  const uint32_t w = threadIdx.x >> 5, share = w % kSplit;
  EbChunk &S = s_c[w];
  uint32_t *const list = s_list[w], *const part = s_part[w];
  const uint32_t lane = threadIdx.x & 31u, nsu = box_supers(C.n), nch = box_chunks(C.n);
  const uint32_t qc = (blockIdx.x * kEbWarps + w) / kSplit;
  if (qc >= nch) return;
  if (kSplit > 1) {
    if (threadIdx.x < 2) s_sum[threadIdx.x] = 0;
    if (threadIdx.x < kBoxChunk) s_out[threadIdx.x] = 0;
    __syncthreads();
  }
  const float r2 = *r2_dev;
  const uint32_t q = qc * kBoxChunk + lane;
  const float4 me = C.pts[q < C.n ? q : C.n - 1u];
  const Box qb = box_load(C.box.chunk, qc);
  const Box one = box_point(__shfl_sync(0xFFFFFFFFu, me.x, 16), __shfl_sync(0xFFFFFFFFu, me.y, 16),
                            __shfl_sync(0xFFFFFFFFu, me.z, 16));
  const f32x2 QX = pk2(me.x, me.x), QY = pk2(me.y, me.y), QZ = pk2(me.z, me.z), R2 = pk2(r2, r2);
  // Boxes within the radius of all of the warp's queries count whole, boxes beyond it
  // of all count nothing; the chunks between go on the list.  The first round also
  // counts those that one of the queries needs, to see whether the queries belong
  // together; a second one runs where they do and the list was too short for all.
  uint32_t whole = 0, beyond = 0, done = 0, nl = 0, own = 0;
  const uint32_t mine = kSplit > 1 ? 0x11111111u << share : 0xFFFFFFFFu;  // lanes: this warp's super-chunks
  static_assert(kEbWarps == 4, "the mask of a fourth");
#pragma unroll 1
  for (int round = 0; round < 2; ++round) {
    for (uint32_t s0 = 0; s0 < nsu; s0 += 32u) {
      const uint32_t s = s0 + lane;
      bool in = false, edge = false;
      if (s < nsu && ((mine >> lane) & 1u)) {
        const Box sb = box_load(C.box.super, s);
        in = box_upper(sb, qb) <= r2;
        edge = !in && box_lower(sb, qb) <= r2;
      }
      if (in) whole += eb_points(s * kBoxSuper, kBoxSuper, C.n);
      uint32_t m = __ballot_sync(0xFFFFFFFFu, edge);
      while (m) {
        const uint32_t c = (s0 + (uint32_t)__ffs(m) - 1u) * 32u + lane;
        m &= m - 1u;
        bool ci = false, ce = false, ce1 = false;
        if (c < nch) {
          const Box cb = box_load(C.box.chunk, c);
          ci = box_upper(cb, qb) <= r2;
          ce = !ci && box_lower(cb, qb) <= r2;
          ce1 = box_upper(cb, one) > r2 && box_lower(cb, one) <= r2;
        }
        const uint32_t e = __ballot_sync(0xFFFFFFFFu, ce);
        if (ci) whole += eb_points(c * kBoxChunk, kBoxChunk, C.n);
        if (round == 0) {
          own += __popc(__ballot_sync(0xFFFFFFFFu, ce1));
        } else if (nl + 32u > kCntList) {  // room for any ballot
          beyond += eb_border(C, S, list, nl, part, qb, r2, QX, QY, QZ, R2, whole, done);
          nl = 0;
        }
        const uint32_t at = nl + __popc(e & lanemask_lt());
        if (ce && at < kCntList) list[at] = c;
        nl += __popc(e);
      }
    }
    if (round == 0) {
      uint32_t listed = nl;
      if (kSplit > 1) {
        if (lane == 0) {
          atomicAdd(&s_sum[0], nl);
          atomicAdd(&s_sum[1], own);
        }
        __syncthreads();
        listed = s_sum[0];
        own = s_sum[1];
      }
      if (cnt_apart(listed, own)) {
        if (lane == 0 && share == 0) far[atomicAdd(&work->cnt_far, 1u)] = qc;
        return;
      }
      if (nl <= kCntList) break;
      nl = 0;
      whole = 0;
    }
  }
  beyond += eb_border(C, S, list, nl, part, qb, r2, QX, QY, QZ, R2, whole, done);
  uint32_t cnt = __reduce_add_sync(0xFFFFFFFFu, whole) + done * kBoxChunk - beyond;
  if (kSplit > 1) {
    atomicAdd(&s_out[lane], cnt);
    __syncthreads();
    if (share != 0) return;
    cnt = s_out[lane];
  }
  if (q < C.n) out[__float_as_uint(me.w) - C.first] = cnt;
}

// the chunks of queries that lie far apart: one query a warp
__global__ void __launch_bounds__(kEbThreads) k_evb_count_far(const Cloud C, const float *__restrict__ r2_dev,
                                                              uint32_t *__restrict__ out,
                                                              const uint32_t *__restrict__ far, const EbWork *work,
                                                              const Counters *ctr) {
  if (ctr->status & kStFatal) return;
  const float r2 = *r2_dev;
  const uint32_t lane = threadIdx.x & 31u, nf = work->cnt_far * kBoxChunk, nsu = box_supers(C.n),
                 nch = box_chunks(C.n);
  for (uint32_t i = blockIdx.x * kEbWarps + (threadIdx.x >> 5); i < nf; i += gridDim.x * kEbWarps) {
    const uint32_t q = far[i / kBoxChunk] * kBoxChunk + (i % kBoxChunk);
    if (q >= C.n) continue;
    const float4 me4 = C.pts[q];
    const Box me = box_point(me4.x, me4.y, me4.z);
    uint32_t cnt = 0;
    for (uint32_t s0 = 0; s0 < nsu; s0 += 32u) {
      const uint32_t s = s0 + lane;
      bool in = false, edge = false;
      if (s < nsu) {
        const Box sb = box_load(C.box.super, s);
        in = box_upper(sb, me) <= r2;
        edge = !in && box_lower(sb, me) <= r2;
      }
      if (in) cnt += eb_points(s * kBoxSuper, kBoxSuper, C.n);
      uint32_t m = __ballot_sync(0xFFFFFFFFu, edge);
      while (m) {
        const uint32_t c0 = (s0 + (uint32_t)__ffs(m) - 1u) * 32u, c = c0 + lane;
        m &= m - 1u;
        bool ci = false, ce = false;
        if (c < nch) {
          const Box cb = box_load(C.box.chunk, c);
          ci = box_upper(cb, me) <= r2;
          ce = !ci && box_lower(cb, me) <= r2;
        }
        if (ci) cnt += eb_points(c * kBoxChunk, kBoxChunk, C.n);
        uint32_t e = __ballot_sync(0xFFFFFFFFu, ce);
        while (e) {
          const float4 p = eb_fetch(C, c0 + (uint32_t)__ffs(e) - 1u);
          e &= e - 1u;
          cnt += eb_d2(me4.x, me4.y, me4.z, p) <= r2;
        }
      }
    }
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    if (lane == 0) out[__float_as_uint(me4.w) - C.first] = cnt;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {
struct EbMem {
  FrameInfo *frames;
  Tile *tiles;
  EbWork *work;
  float *xyz;
  unsigned long long *keys[2];
  uint32_t *vals[2];
  float4 *spts;
  uint32_t *hist, *lookback;
  unsigned char *box[2];
};
size_t eb_carve(unsigned char *p, uint32_t na, uint32_t nb, EbMem *m) {
  size_t o = 0;
  const size_t n = (size_t)na + nb, tiles = na / kTilePts + nb / kTilePts + 2;
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o += (bytes + 255) & ~size_t(255);
    return p + r;
  };
  EbMem x;
  x.frames = (FrameInfo *)take(2 * sizeof(FrameInfo));
  x.tiles = (Tile *)take(tiles * sizeof(Tile));
  x.work = (EbWork *)take(sizeof(EbWork));
  x.xyz = (float *)take(12 * n);
  for (int i = 0; i < 2; ++i) x.keys[i] = (unsigned long long *)take(8 * n);
  for (int i = 0; i < 2; ++i) x.vals[i] = (uint32_t *)take(4 * n);
  x.spts = (float4 *)take(16 * n);
  x.hist = (uint32_t *)take(4ull * 2 * kMaxPasses * 256);
  x.lookback = (uint32_t *)take(4ull * kTopPasses * tiles * 256);
  x.box[0] = take(box_bytes(na));
  x.box[1] = take(box_bytes(nb));
  if (m) *m = x;
  return o;
}

// both clouds (nb may be 0) into octree order, with their boxes
int eb_build(const EbMem &m, const float *a, uint32_t na, const float *b, uint32_t nb, Counters *ctr,
             uint32_t spin_limit, int num_sms, Cloud out[2], cudaStream_t st) {
  k_evb_tables<<<1, 256, 0, st>>>(m.frames, m.tiles, na, nb, m.work);
  if (nb) k_evb_cat<<<num_sms * 8, 256, 0, st>>>(a, 3ull * na, b, 3ull * nb, m.xyz);
  FrontArgs f{};
  f.xyz = nb ? m.xyz : a;
  f.n = na + nb;
  f.frames = m.frames;
  f.nframes = nb ? 2 : 1;
  f.tiles = m.tiles;
  f.ntiles = (na + kTilePts - 1) / kTilePts + (nb + kTilePts - 1) / kTilePts;
  f.frame_points = na > nb ? na : nb;
  for (int i = 0; i < 2; ++i) {
    f.keys[i] = m.keys[i];
    f.vals[i] = m.vals[i];
  }
  f.spts = m.spts;
  f.digit_hist = m.hist;
  f.tile_box = reinterpret_cast<uint4 *>(m.vals[1]);  // idle until the first radix pass
  f.lookback = m.lookback;
  f.ctr = ctr;
  f.max_depth = 21;
  f.spin_limit = spin_limit;
  f.order_only = true;
  if (launch_front(f, st, nullptr, nullptr, nullptr)) return -1;
  const unsigned long long *keys = m.keys[front_sorted_buffer(21, false)];
  // One cloud leaves the concatenation's place free: 16 bytes of quarter boxes for the
  // 48 of four points (the calls taken here have at least 2^15).
  out[0] = Cloud{m.spts, na, 0u, box_index(m.box[0], na), nb ? nullptr : reinterpret_cast<float4 *>(m.xyz), keys, m.frames};
  out[1] = Cloud{m.spts + na, nb, na, box_index(m.box[1], nb), nullptr, keys + na, m.frames + 1};
  k_evb_boxes<<<box_supers(na) + box_supers(nb), kBoxSuper, 0, st>>>(out[0], out[1], ctr);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
}  // namespace

// Below a billion pairs in all the full pass is faster than the sort and the tails of
// the pruned one (full / pruned, us a call: metrics of 25,000 points 290 / 257, counts
// among 25,000 205 / 309, 36,750 375 / 212-314).
bool evb_takes(uint64_t pairs) { return pairs >= (1ull << 30); }

size_t evb_scratch_bytes(uint32_t na, uint32_t nb) { return eb_carve(nullptr, na, nb, nullptr); }

int launch_evb_nearest(unsigned char *scratch, const float *a, uint32_t na, const float *b, uint32_t nb, float *nn_a,
                       float *nn_b, const FrameInfo **frame_a, Counters *ctr, uint32_t spin_limit, int num_sms,
                       cudaStream_t st) {
  EbMem m;
  eb_carve(scratch, na, nb, &m);
  Cloud c[2];
  if (eb_build(m, a, na, b, nb, ctr, spin_limit, num_sms, c, st)) return -1;
  *frame_a = m.frames;
  uint32_t *const far[2] = {m.vals[0], m.vals[0] + na};  // free after the sort
  float *const out[2] = {nn_a, nn_b};
  for (int d = 0; d < 2; ++d) {
    k_evb_nn<<<(box_chunks(c[d].n) + kEbWarps - 1) / kEbWarps, kEbThreads, 0, st>>>(c[d], c[d ^ 1], out[d], far[d],
        m.work, d, nn_share(box_chunks(c[d].n)), ctr);
    k_evb_nn_far<<<num_sms * 8, kEbThreads, 0, st>>>(c[d], c[d ^ 1], out[d], far[d], m.work, d, ctr);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_evb_count(unsigned char *scratch, const float *xyz, uint32_t n, const float *r2_dev, uint32_t *cnt,
                     Counters *ctr, uint32_t spin_limit, int num_sms, cudaStream_t st) {
  EbMem m;
  eb_carve(scratch, n, 0, &m);
  Cloud c[2];
  if (eb_build(m, xyz, n, nullptr, 0, ctr, spin_limit, num_sms, c, st)) return -1;
  if (box_chunks(n) < kCntSplit)
    k_evb_count<kEbWarps><<<box_chunks(n), kEbThreads, 0, st>>>(c[0], r2_dev, cnt, m.vals[0], m.work, ctr);
  else
    k_evb_count<1><<<(box_chunks(n) + kEbWarps - 1) / kEbWarps, kEbThreads, 0, st>>>(c[0], r2_dev, cnt, m.vals[0],
                                                                                      m.work, ctr);
  k_evb_count_far<<<num_sms * 8, kEbThreads, 0, st>>>(c[0], r2_dev, cnt, m.vals[0], m.work, ctr);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace gd
