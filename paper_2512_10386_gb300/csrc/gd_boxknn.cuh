// gd_boxknn.cuh -- the exact k nearest of 32 queries by one warp (one query a
// lane), over candidates in 32-point chunks that are skipped by their boxes
// (gd_boxes.cuh).  The selection is the counting selection of the fused leaf
// kernel (gd_knn_select.cuh); only the chunks that can hold a neighbour of one of
// the warp's queries are read.
//
//   theta_0  the largest d^2 to the k valid points around the query in octree order
//   near     the bucket counts over the chunks around the queries' own one: the top
//            of the boundary bucket bounds the k-th distance closely
//   count    the same counts over every chunk whose box is within that bound
//            (refined where the boundary bucket is too full, as in the leaf kernel)
//   emit     the neighbours below the boundary bucket, in position order, and the
//            bucket's members parked; these are sorted and the missing ones taken
//
// A chunk is needed if its box is within the largest bound of the warp from the
// box of the warp's queries, and within the own bound of at least one of them.
// A query that alone asks for many chunks (an outlier: its bound reaches far) would
// have the whole warp read them; it is put on a list instead, and a warp of its own
// finds its neighbours with the chunk's points across the lanes (bk_knn_far).
#pragma once

#include "gd_boxes.cuh"
#include "gd_leaf_kernel.cuh"

namespace gd {

constexpr int kBkWarps = 4;          // warps per CTA, each on its own
constexpr int kBkPlanes = 21;        // counts < 2^21 candidates
constexpr int kBkLowPlanes = 11;     // rippled always; the carry above them is rare
// A chunk costs the warp about 700 instructions (count and emit), a query with a
// warp of its own about 2,000: a query is left to its own once its share of the
// chunks it wants (each split evenly over the queries that want it) is this many.
// With few points the last warp's time counts, and queries leave earlier.  Measured,
// cross-leaf calls in us at shares 2 / 4 / 8 / never: 30k points 532 / 661 / 976 / 1015,
// 100k 839 / 1050 / 1389 / 2674, 300k 1877 / 1895 / 2271 / 4893, 560k 3683 / 3009 / 3251 / 8951.
__device__ __forceinline__ float bk_share(uint32_t n) { return n < 150000u ? 2.0f : 4.0f; }
constexpr uint32_t kBkFarK = 32;     // its list has one entry per lane

// One warp's shared memory.
template <int KROW>
struct BkShared {
  float x[kBoxChunk], y[kBoxChunk], z[kBoxChunk];  // the chunk being compared
  uint32_t pend_key[kSelBuf][32];                  // parked: (d^2 offset << 4) | slot
  uint32_t pend_pos[kSelBuf][32];
  uint32_t row[32][KROW + 1];                      // neighbours (positions), ascending; odd stride
};

// What the warp's queries need of the candidate set.  Src:
//   uint32_t entries()                                super-chunk entries
//   void entry(e, &super, &a, &b)                     entry e covers the positions [a, b) of super-chunk `super`
//   float4 load(p)                                    point p (x, y, z, input index bits), NaN if it is no candidate
//   BoxIndex box                                      boxes over the positions
// The queries (lanes) to leave to a warp of their own.
template <typename Src>
__device__ __forceinline__ uint32_t bk_costly(const Src &src, const Box &qb, float qx, float qy, float qz, bool act,
                                              float mine, float most) {
  const uint32_t lane = threadIdx.x & 31u;
  const Box me = box_point(qx, qy, qz);
  float share = 0.0f;
  float want = act ? mine : -1.0f;  // no chunk is within a bound of -1
  float bound = ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(want)));
  const uint32_t ne = src.entries();
  for (uint32_t e0 = 0; e0 < ne; e0 += 32u) {
    const uint32_t e = e0 + lane;
    uint32_t s = 0, a = 0, b = 0;
    Box sb = box_empty();
    if (e < ne) {
      src.entry(e, s, a, b);
      sb = box_load(src.box.super, s);
    }
    uint32_t em = __ballot_sync(0xFFFFFFFFu, !box_is_empty(sb) && box_lower(sb, qb) <= bound);
    while (em) {
      const int o = __ffs(em) - 1;
      em &= em - 1u;
      const uint32_t es = __shfl_sync(0xFFFFFFFFu, s, o), ea = __shfl_sync(0xFFFFFFFFu, a, o),
                     eb = __shfl_sync(0xFFFFFFFFu, b, o);
      const uint32_t c = es * 32u + lane;
      Box cb = box_empty();
      if (c * kBoxChunk < eb && (c + 1u) * kBoxChunk > ea) cb = box_load(src.box.chunk, c);
      uint32_t cand = __ballot_sync(0xFFFFFFFFu, !box_is_empty(cb) && box_lower(cb, qb) <= bound);
      while (cand) {
        const int u = __ffs(cand) - 1;
        cand &= cand - 1u;
        Box x;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          x.lo[d] = __shfl_sync(0xFFFFFFFFu, cb.lo[d], u);
          x.hi[d] = __shfl_sync(0xFFFFFFFFu, cb.hi[d], u);
        }
        const bool w = box_lower(x, me) <= want;
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, w);
        if (w) share += rcp_hw((float)__popc(m));
        if (__any_sync(0xFFFFFFFFu, share >= most && want >= 0.0f)) {
          if (share >= most) want = -1.0f;
          bound = ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(want)));
          if (bound < 0.0f) return __ballot_sync(0xFFFFFFFFu, act);
        }
      }
    }
  }
  return __ballot_sync(0xFFFFFFFFu, act && want < 0.0f);
}

template <typename Src, typename F>
__device__ __forceinline__ void bk_traverse(const Src &src, const Box &qb, float qx, float qy, float qz, float mine,
                                            float (&sx)[kBoxChunk], float (&sy)[kBoxChunk], float (&sz)[kBoxChunk],
                                            F body) {
  const uint32_t lane = threadIdx.x & 31u;
  const float bound = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mine)));
  const Box me = box_point(qx, qy, qz);
  const uint32_t ne = src.entries();
  for (uint32_t e0 = 0; e0 < ne; e0 += 32u) {
    const uint32_t e = e0 + lane;
    uint32_t s = 0, a = 0, b = 0;
    bool need = false;
    if (e < ne) {
      src.entry(e, s, a, b);
      const Box sb = box_load(src.box.super, s);
      need = !box_is_empty(sb) && box_lower(sb, qb) <= bound;
    }
    uint32_t em = __ballot_sync(0xFFFFFFFFu, need);
    while (em) {
      const int o = __ffs(em) - 1;
      em &= em - 1u;
      const uint32_t es = __shfl_sync(0xFFFFFFFFu, s, o), ea = __shfl_sync(0xFFFFFFFFu, a, o),
                     eb = __shfl_sync(0xFFFFFFFFu, b, o);
      const uint32_t c = es * 32u + lane;
      Box cb = box_empty();
      if (c * kBoxChunk < eb && (c + 1u) * kBoxChunk > ea) cb = box_load(src.box.chunk, c);
      uint32_t cand = __ballot_sync(0xFFFFFFFFu, !box_is_empty(cb) && box_lower(cb, qb) <= bound);
      uint32_t cm = 0;
      while (cand) {  // within the bound of one of the queries
        const int u = __ffs(cand) - 1;
        cand &= cand - 1u;
        Box x;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          x.lo[d] = __shfl_sync(0xFFFFFFFFu, cb.lo[d], u);
          x.hi[d] = __shfl_sync(0xFFFFFFFFu, cb.hi[d], u);
        }
        if (__any_sync(0xFFFFFFFFu, box_lower(x, me) <= mine)) cm |= 1u << u;
      }
      if (!cm) continue;
      auto fetch = [&](uint32_t cc) {
        const uint32_t p = cc * kBoxChunk + lane;
        return (p >= ea && p < eb) ? src.load(p) : make_float4(__int_as_float(0x7FFFFFFF), 0.f, 0.f, 0.f);
      };
      uint32_t cc = es * 32u + (uint32_t)__ffs(cm) - 1u;
      float4 v = fetch(cc);
      while (cm) {
        cm &= cm - 1u;
        __syncwarp();
        sx[lane] = v.x;
        sy[lane] = v.y;
        sz[lane] = v.z;
        __syncwarp();
        const uint32_t cur = cc;
        if (cm) {  // the next chunk is on its way while this one is compared
          cc = es * 32u + (uint32_t)__ffs(cm) - 1u;
          v = fetch(cc);
        }
        body(cur);
      }
    }
  }
}

// Bucket counts of the staged chunk into the bit-sliced counters.
__device__ __forceinline__ void bk_count(const float *sx, const float *sy, const float *sz, f32x2 QX, f32x2 QY,
                                         f32x2 QZ, const SelLevel &L, uint32_t (&c)[kBkPlanes]) {
  uint32_t(&low)[kBkLowPlanes] = reinterpret_cast<uint32_t(&)[kBkLowPlanes]>(c);
#pragma unroll 1
  for (uint32_t s = 0; s < kBoxChunk; s += 16u) {
    uint32_t m[16];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float d[4];
      sqdist4(sx, sy, sz, s + 4u * u, QX, QY, QZ, d);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int32_t db = __float_as_int(d[v]);
        m[4 * u + v] = db > L.lo ? sel_bucket_bit(L.tb, db, L.S) : 0u;
      }
    }
    uint32_t carry = sel_add16<kBkLowPlanes>(low, m);
    if (__any_sync(0xFFFFFFFFu, carry)) {
#pragma unroll
      for (int p = kBkLowPlanes; p < kBkPlanes; ++p) {
        const uint32_t t = c[p] & carry;
        c[p] ^= carry;
        carry = t;
      }
    }
  }
}

// One query by one warp: the chunk's points across the lanes, the sorted list of
// the k nearest (d^2, input index) too (lane t: rank t).
struct BkList {
  unsigned long long key;  // (d^2 bits << 32) | input index, ~0 = none
  uint32_t pos;
  unsigned long long thr;  // what a candidate has to beat (warp-uniform)
};

__device__ __forceinline__ void bk_cmpx(unsigned long long &k, uint32_t &p, int j, bool keep_min) {
  const unsigned long long ok = __shfl_xor_sync(0xFFFFFFFFu, k, j);
  const uint32_t op = __shfl_xor_sync(0xFFFFFFFFu, p, j);
  const bool take = keep_min ? (ok < k) : (k < ok);
  if (take) {
    k = ok;
    p = op;
  }
}

// ascending sort of one (key, position) a lane
__device__ __forceinline__ void bk_sort(unsigned long long &k, uint32_t &p, uint32_t lane) {
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1) bk_cmpx(k, p, j, ((lane & j) == 0) == ((lane & size) == 0));
  }
}

// The candidates of the lanes in `mask` into the list: a few one by one (a shuffle
// step each), many sorted across the lanes and merged.
__device__ __forceinline__ void bk_add(BkList &L, uint32_t mask, uint32_t dbits, uint32_t idx, uint32_t pos,
                                       uint32_t lane, uint32_t k) {
  const unsigned long long open = L.thr;
  if (__popc(mask) <= 10) {
    while (mask) {
      const int b = __ffs(mask) - 1;
      mask &= mask - 1u;
      const unsigned long long K = ((unsigned long long)__shfl_sync(0xFFFFFFFFu, dbits, b) << 32) |
                                   __shfl_sync(0xFFFFFFFFu, idx, b);
      if (K >= L.thr) continue;
      const uint32_t P = __shfl_sync(0xFFFFFFFFu, pos, b);
      const unsigned long long prev = __shfl_up_sync(0xFFFFFFFFu, L.key, 1);
      const uint32_t pprev = __shfl_up_sync(0xFFFFFFFFu, L.pos, 1);
      if (lane < k) {
        if (lane > 0 && prev > K) {
          L.key = prev;
          L.pos = pprev;
        } else if (L.key > K) {
          L.key = K;
          L.pos = P;
        }
      }
      const unsigned long long kth = __shfl_sync(0xFFFFFFFFu, L.key, k - 1);
      L.thr = kth < open ? kth : open;
    }
    return;
  }
  unsigned long long c = ((mask >> lane) & 1u) ? (((unsigned long long)dbits << 32) | idx) : ~0ull;
  uint32_t p = pos;
  bk_sort(c, p, lane);
  // the 32 smallest of two sorted lists: elementwise minimum with one reversed, then a bitonic merge
  const unsigned long long rc = __shfl_sync(0xFFFFFFFFu, c, 31 - lane);
  const uint32_t rp = __shfl_sync(0xFFFFFFFFu, p, 31 - lane);
  if (rc < L.key) {
    L.key = rc;
    L.pos = rp;
  }
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) bk_cmpx(L.key, L.pos, j, (lane & j) == 0);
  if (lane >= k) L.key = ~0ull;
  const unsigned long long kth = __shfl_sync(0xFFFFFFFFu, L.key, k - 1);
  L.thr = kth < open ? kth : open;
}

// `bound`: an upper bound of the k-th smallest d^2.  Nearest chunks of the nearest
// super-chunk first (their points bring the threshold down), then whatever is left
// within it.
template <typename Src>
__device__ __forceinline__ void bk_knn_far(const Src &src, uint32_t q, float qx, float qy, float qz, uint32_t k,
                                           float bound, BkList &L) {
  const uint32_t lane = threadIdx.x & 31u;
  const Box me = box_point(qx, qy, qz);
  L.key = ~0ull;
  L.pos = 0;
  L.thr = ((unsigned long long)__float_as_uint(bound) << 32) | 0xFFFFFFFFull;  // every index passes at the bound
  auto thr_f = [&]() { return __uint_as_float((uint32_t)(L.thr >> 32)); };
  auto entry = [&](uint32_t es, uint32_t ea, uint32_t eb, bool nearest) {
    const uint32_t c = es * 32u + lane;
    Box cb = box_empty();
    if (c * kBoxChunk < eb && (c + 1u) * kBoxChunk > ea) cb = box_load(src.box.chunk, c);
    const float lb = box_lower(cb, me);
    uint32_t cm = __ballot_sync(0xFFFFFFFFu, !box_is_empty(cb) && lb <= thr_f());
    while (cm) {
      int o = __ffs(cm) - 1;
      if (nearest) {
        const uint32_t v = ((cm >> lane) & 1u) ? __float_as_uint(lb) : 0xFFFFFFFFu;
        o = __ffs(__ballot_sync(0xFFFFFFFFu, v == __reduce_min_sync(0xFFFFFFFFu, v))) - 1;
      }
      cm &= ~(1u << o);
      if (__shfl_sync(0xFFFFFFFFu, lb, o) > thr_f()) {
        if (nearest) break;
        continue;
      }
      const uint32_t p = (es * 32u + (uint32_t)o) * kBoxChunk + lane;
      float4 v = make_float4(__int_as_float(0x7FFFFFFF), 0.f, 0.f, 0.f);
      if (p >= ea && p < eb) v = src.load(p);
      const uint32_t db = __float_as_uint(sqdist(qx, qy, qz, v.x, v.y, v.z)) & 0x7FFFFFFFu;  // NaN stays above
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, db <= (uint32_t)(L.thr >> 32) && p != q);
      if (m) bk_add(L, m, db, __float_as_uint(v.w), p, lane, k);
    }
  };
  const uint32_t ne = src.entries();
  // the nearest entry
  uint32_t best = 0xFFFFFFFFu, be = 0;
  for (uint32_t e = lane; e < ne; e += 32u) {
    uint32_t s, a, b;
    src.entry(e, s, a, b);
    const Box sb = box_load(src.box.super, s);
    const uint32_t v = __float_as_uint(box_lower(sb, me));
    if (!box_is_empty(sb) && v < best) {
      best = v;
      be = e;
    }
  }
  const uint32_t bm = __reduce_min_sync(0xFFFFFFFFu, best);
  be = __shfl_sync(0xFFFFFFFFu, be, __ffs(__ballot_sync(0xFFFFFFFFu, best == bm)) - 1);
  if (bm != 0xFFFFFFFFu) {
    uint32_t s, a, b;
    src.entry(be, s, a, b);
    entry(s, a, b, true);
  }
  for (uint32_t e0 = 0; e0 < ne; e0 += 32u) {
    const uint32_t e = e0 + lane;
    uint32_t s = 0, a = 0, b = 0;
    float lb = INFINITY;
    bool need = false;
    if (e < ne && e != be) {
      src.entry(e, s, a, b);
      const Box sb = box_load(src.box.super, s);
      lb = box_lower(sb, me);
      need = !box_is_empty(sb) && lb <= thr_f();
    }
    uint32_t em = __ballot_sync(0xFFFFFFFFu, need);
    while (em) {
      const int o = __ffs(em) - 1;
      em &= em - 1u;
      if (__shfl_sync(0xFFFFFFFFu, lb, o) > thr_f()) continue;
      entry(__shfl_sync(0xFFFFFFFFu, s, o), __shfl_sync(0xFFFFFFFFu, a, o), __shfl_sync(0xFFFFFFFFu, b, o), false);
    }
  }
}

// The k nearest of the lane's query (qx, qy, qz) at position q (a lane without a
// query shadows another lane's, act = false) into S.row[lane][0..k), ascending
// positions.  [w0, w1) is the range of positions around q to take theta_0 from
// (all of them candidates or NaN), `share` what makes a query costly.
// theta receives the k-th squared distance; `far` the lanes whose queries are left
// to a warp of their own (none where k > kBkFarK), theta then a bound of it.
// Returns false if the passes disagree (cannot happen).
template <typename Src, int KROW>
__device__ __forceinline__ bool bk_knn(const Src &src, BkShared<KROW> &S, bool act, uint32_t q, float qx, float qy,
                                       float qz, uint32_t k, uint32_t w0, uint32_t w1, float share,
                                       float &theta, uint32_t &far) {
  const uint32_t lane = threadIdx.x & 31u;
  f32x2 QX = pk2(qx, qx), QY = pk2(qy, qy), QZ = pk2(qz, qz);
  Box qb = box_warp_union(box_point(qx, qy, qz));
  far = 0;
  // theta_0: outward from q until k valid others are seen, but no further than where a
  // candidate in sixteen positions would have done: each step waits for its loads, and
  // where the voxel gate left few points of a large leaf the walk would cross it (one leaf
  // of 1 M points, 200 of them candidates, K = 32: 46.9 -> 1.5 ms)
  float t0 = 0.0f;
  {
    uint32_t found = 0;
    const uint32_t steps = 8u * k + 32u;
    for (uint32_t d = 1; d <= steps && __any_sync(0xFFFFFFFFu, found < k && (q >= w0 + d || q + d < w1)); ++d) {
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const bool in = found < k && (side ? q + d < w1 : q >= w0 + d);
        if (in) {
          const float4 p = src.load(side ? q + d : q - d);
          const float v = sqdist(qx, qy, qz, p.x, p.y, p.z);
          if (v == v) {
            t0 = fmaxf(t0, v);
            ++found;
          }
        }
      }
    }
    if (__any_sync(0xFFFFFFFFu, found < k)) {
      // too few points around the query: no candidate lies beyond the far corners of
      // the super-chunks' boxes
      const Box me = box_point(qx, qy, qz);
      float far = 0.0f;
      for (uint32_t e = 0; e < src.entries(); ++e) {
        uint32_t s, a, b;
        src.entry(e, s, a, b);
        const Box sb = box_load(src.box.super, s);
        if (!box_is_empty(sb)) far = fmaxf(far, box_upper(sb, me));
      }
      if (found < k) t0 = far;
    }
  }
  SelLevel L{__float_as_int(t0), -1, kSelS0, 0u, 0};
  uint32_t c[kBkPlanes];
  // near: the chunks around q's own one, inside [w0, w1)
  {
#pragma unroll
    for (int p = 0; p < kBkPlanes; ++p) c[p] = 0u;
    const uint32_t own = __reduce_min_sync(0xFFFFFFFFu, q) / kBoxChunk;
    const uint32_t n0 = max(own > 2u ? own - 2u : 0u, w0 / kBoxChunk), n1 = min(own + 2u, (w1 - 1u) / kBoxChunk);
    for (uint32_t cc = n0; cc <= n1; ++cc) {
      const uint32_t p = cc * kBoxChunk + lane;
      const float4 v = (p >= w0 && p < w1) ? src.load(p) : make_float4(__int_as_float(0x7FFFFFFF), 0.f, 0.f, 0.f);
      __syncwarp();
      S.x[lane] = v.x;
      S.y[lane] = v.y;
      S.z[lane] = v.z;
      __syncwarp();
      bk_count(S.x, S.y, S.z, QX, QY, QZ, L, c);
    }
    L.tb = sel_walk<kBkPlanes>(c, L, k).hi;  // (all counts below k: the top itself)
  }
  float far_bound = 0.0f;
  if (KROW <= (int)kBkFarK) {
    far = bk_costly(src, qb, qx, qy, qz, act, __int_as_float(L.tb), share);
    if (far) {  // they shadow one of the queries that stay
      const uint32_t stay = __ballot_sync(0xFFFFFFFFu, act) & ~far;
      const bool gone = (far >> lane) & 1u;
      far_bound = __int_as_float(L.tb);
      theta = far_bound;
      if (!stay) return true;
      act = act && !gone;
      const int f = __ffs(stay) - 1;
      const float x = __shfl_sync(0xFFFFFFFFu, qx, f), y = __shfl_sync(0xFFFFFFFFu, qy, f),
                  z = __shfl_sync(0xFFFFFFFFu, qz, f);
      const uint32_t nq = __shfl_sync(0xFFFFFFFFu, q, f);
      const int32_t ntb = __shfl_sync(0xFFFFFFFFu, L.tb, f);
      if (!act) {
        qx = x;
        qy = y;
        qz = z;
        q = nq;
        L.tb = ntb;
      }
      QX = pk2(qx, qx);
      QY = pk2(qy, qy);
      QZ = pk2(qz, qz);
      qb = box_warp_union(box_point(qx, qy, qz));
    }
  }
  SelCut cut;
  bool ok = true;
#pragma unroll 1
  for (int level = 0;; ++level) {
#pragma unroll
    for (int p = 0; p < kBkPlanes; ++p) c[p] = 0u;
    bk_traverse(src, qb, qx, qy, qz, __int_as_float(L.tb), S.x, S.y, S.z,
                [&](uint32_t) { bk_count(S.x, S.y, S.z, QX, QY, QZ, L, c); });
    cut = sel_walk<kBkPlanes>(c, L, k);
    const bool single = cut.hi == cut.lo + 1;
    const bool again = act && !single && (cut.c_at > kSelBuf || !sel_fits(cut, 4u));
    if (!__any_sync(0xFFFFFFFFu, again)) break;
    if (level > kSelMaxLevels) {
      ok = false;
      break;
    }
    if (again) L = sel_refine(L, cut);
  }
  const uint32_t need = k - cut.c_below;
  const bool ties_only = cut.c_at > kSelBuf;
  const int32_t kbase = cut.lo + 1;
  const float lo_f = cut.lo >= 0 ? __int_as_float(cut.lo) : -1.0f, hi_f = __int_as_float(cut.hi);
  uint32_t a = 0, np = 0;
  bk_traverse(src, qb, qx, qy, qz, hi_f, S.x, S.y, S.z, [&](uint32_t cur) {
    uint32_t gtlo = 0, gthi = 0;
#pragma unroll 2
    for (uint32_t st = 0; st < 8; ++st) {
      float d[4];
      sqdist4(S.x, S.y, S.z, 4u * st, QX, QY, QZ, d);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        // the sign of v - d^2 is set exactly when d^2 > v (a NaN, no candidate, is canonical:
        // its sign is clear, so it is dropped by the test below)
        gtlo = __funnelshift_l(__float_as_uint(__fsub_rn(lo_f, d[u])), gtlo, 1);
        gthi = __funnelshift_l(__float_as_uint(__fsub_rn(hi_f, d[u])), gthi, 1);
      }
    }
    uint32_t le_lo = ~__brev(gtlo), le_hi = ~__brev(gthi);
    const uint32_t valid = __ballot_sync(0xFFFFFFFFu, S.x[lane] == S.x[lane]);
    uint32_t keep = (q - cur * kBoxChunk < kBoxChunk) ? valid & ~(1u << (q & 31u)) : valid;
    if (!act) keep = 0;
    uint32_t em = le_lo & keep, pm = le_hi & ~le_lo & keep;
    uint32_t t = a;
    a += __popc(em);
    if (a > k) em = 0;  // counts disagree: reported below
    while (em) {
      const uint32_t b = (uint32_t)__ffs(em) - 1u;
      em &= em - 1u;
      S.row[lane][t++] = cur * kBoxChunk + b;
    }
    uint32_t slot = np;
    np += __popc(pm);
    if (ties_only || np > kSelBuf) pm = 0;
    while (pm) {
      const uint32_t b = (uint32_t)__ffs(pm) - 1u;
      pm &= pm - 1u;
      const int32_t db = __float_as_int(sqdist(qx, qy, qz, S.x[b], S.y[b], S.z[b]));
      S.pend_key[slot][lane] = ((uint32_t)(db - kbase) << 4) | slot;
      S.pend_pos[slot][lane] = cur * kBoxChunk + b;
      ++slot;
    }
  });
  if (act && (a != cut.c_below || np != cut.c_at)) ok = false;
  // the `need` smallest of the boundary bucket
  theta = hi_f;
  const bool parked = act && !ties_only && ok;
  uint32_t take = 0;
  {
    uint32_t K[kSelBuf];
#pragma unroll
    for (int i = 0; i < (int)kSelBuf; ++i) K[i] = (parked && (uint32_t)i < np) ? S.pend_key[i][lane] : 0xFFFFFFFFu;
    if (__reduce_max_sync(0xFFFFFFFFu, parked ? np : 0u) <= kSelBuf / 2) regsort_head<kSelBuf / 2>(K);
    else regsort_u<kSelBuf>(K);
    uint32_t th_off = 0;
#pragma unroll
    for (int i = 0; i < (int)kSelBuf; ++i) {
      th_off = ((uint32_t)i + 1u == need) ? (K[i] >> 4) : th_off;
      if (parked) S.pend_key[i][lane] = K[i];
    }
    uint32_t n_lt = 0, n_eq = 0;
#pragma unroll
    for (int i = 0; i < (int)kSelBuf; ++i) {
      n_lt += (K[i] >> 4) < th_off;
      n_eq += (K[i] >> 4) == th_off;
    }
    if (parked) {
      theta = __int_as_float(kbase + (int32_t)th_off);
      take = (1u << need) - 1u;  // need <= kSelBuf
      const uint32_t need_eq = need - n_lt;
      if (n_eq > need_eq) {  // ties straddle the cut: by input index
        take = (1u << n_lt) - 1u;
#pragma unroll 1
        for (uint32_t i = n_lt; i < n_lt + n_eq; ++i) {
          const uint32_t gi = __float_as_uint(src.load(S.pend_pos[S.pend_key[i][lane] & 15u][lane]).w);
          uint32_t before = 0;
#pragma unroll 1
          for (uint32_t j = n_lt; j < n_lt + n_eq; ++j)
            before += __float_as_uint(src.load(S.pend_pos[S.pend_key[j][lane] & 15u][lane]).w) < gi;
          if (before < need_eq) take |= 1u << i;
        }
      }
    }
  }
  // into the row at its place (positions ascending)
  auto insert = [&](uint32_t v) {
    uint32_t u = a++;
    while (u > 0 && S.row[lane][u - 1] > v) {
      S.row[lane][u] = S.row[lane][u - 1];
      --u;
    }
    S.row[lane][u] = v;
  };
  while (take) {
    const uint32_t i = (uint32_t)__ffs(take) - 1u;
    take &= take - 1u;
    insert(S.pend_pos[S.pend_key[i][lane] & 15u][lane]);
  }
  // more members at one d^2 than the buffer holds: one scan per missing neighbour
  // takes the smallest input index above the last one taken
  const uint32_t rounds = (act && ties_only && ok) ? need : 0u;
  const uint32_t max_rounds = __reduce_max_sync(0xFFFFFFFFu, rounds);
  uint32_t last = 0;
#pragma unroll 1
  for (uint32_t r = 0; r < max_rounds; ++r) {
    uint32_t bg = 0xFFFFFFFFu, bp = 0xFFFFFFFFu;
    bk_traverse(src, qb, qx, qy, qz, hi_f, S.x, S.y, S.z, [&](uint32_t cur) {
#pragma unroll 1
      for (uint32_t j = 0; j < kBoxChunk; ++j) {
        const float d2 = sqdist(qx, qy, qz, S.x[j], S.y[j], S.z[j]);
        const uint32_t p = cur * kBoxChunk + j;
        if (r < rounds && p != q && d2 == hi_f) {
          const uint32_t g = __float_as_uint(src.load(p).w);
          if ((r == 0 || g > last) && (g < bg || bp == 0xFFFFFFFFu)) {
            bg = g;
            bp = p;
          }
        }
      }
    });
    if (r < rounds) {
      if (bp == 0xFFFFFFFFu) ok = false;
      else insert(bp);
      last = bg;
    }
  }
  if (act && a != k) ok = false;
  if ((far >> lane) & 1u) theta = far_bound;
  __syncwarp();
  return ok;
}

}  // namespace gd
