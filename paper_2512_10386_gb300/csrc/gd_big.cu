// gd_big.cu -- leaves that one CTA should not process alone: the per-leaf steps of
// Sec. 3 (voxel gate, kNN, density gate, score, selection) spread over the whole
// GPU, one kernel a step (big_leaf_above says which: large leaf capacities, with
// "without octree" as their extreme, and depth limits that leave many points to a
// cell).
//
// The fused kernel makes a leaf one CTA's work and compares every pair of its
// points: 36,750 points in one leaf (K = 16) took 1.17 s on one SM, here 0.45 ms,
// 0.19 ms of it the kNN (its last warps: the chunks with many outliers; issue in 39 % of
// the cycles, 12 % of the warp slots occupied).  A leaf is
// cut into units of 1,024 points (gate, score) and 32 queries (kNN), and the kNN
// skips the 32-point chunks of the octree order whose bounding box lies farther than
// a bound of the query's k-th distance (gd_boxes.cuh; exact, so the neighbour sets
// are those of the full comparison).  The order statistics are radix selects over the
// leaf instead of sorts.  Every value that decides something, and the order in
// which a score sums its terms (neighbour positions ascending, even and odd ranks
// apart), is the fused kernel's, so results are identical bit for bit.
#include "gd_boxknn.cuh"

namespace gd {

constexpr int kBigUnit = (int)kBoxSuper;  // points per unit of the gate and the score: one super-chunk, one per thread
constexpr uint32_t kBigChunks = kBigUnit / kBoxChunk;  // kNN units (one chunk of queries, one warp) per unit
constexpr int kSelectThreads = 1024;
// values of one leaf that the selects keep in shared memory (larger leaves re-read L2)
constexpr uint32_t kSelectCap = 40960;

// What a big leaf's steps share; at the start of the leaf's slice of the spill area.
struct BigHead {
  uint32_t lo_ord[3], hi_ord[3];  // box of the leaf's points (ordered integers)
  uint32_t units_done;            // units whose box has been merged (the last one computes h)
  uint32_t n1;                    // |P_1|
  uint32_t Rb;                    // Eq. 14: bits of the largest r_K^2 that stays
  uint32_t m;                     // |P_2|
  float r2ref, Lref;              // the score's per-leaf constants (Eq. 16-17)
  uint32_t cut, needed, at;       // selection: key of the cut, points needed at it, points at it
  uint32_t pad;
};

// The leaf's arrays inside its slice, all by the point's offset in the leaf.
struct BigMem {
  BigHead *head;
  float4 *pts;       // P_1 points (x, y, z, input index bits); the others have NaN coordinates
  float *r2;         // r_K^2 (0xFFFFFFFF bits outside P_1)
  float *wa;         // voxel hash slots, then the score weight (alpha/2) ell
  float *F;          // score
  uint8_t *flag;     // 0 outside P_2, 1 scored
  uint32_t *nbr;     // [count][k] neighbours (leaf offsets), ascending
  BoxIndex box;
  unsigned long long *hkey;
  uint32_t *hcnt, hcap;
};

__host__ __device__ __forceinline__ size_t big_carve(unsigned char *base, uint32_t n, uint32_t k, BigMem *m) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o = al16(o + bytes);
    return r;
  };
  const size_t head = take(sizeof(BigHead)), pts = take(16ull * n), r2 = take(4ull * n), wa = take(4ull * n),
               f = take(4ull * n), fl = take(n), bx = take(box_bytes(n));
  // the hash table of the voxel gate, later (lifetimes disjoint) the neighbours
  const uint32_t hcap = pow2ceil(2 * n);
  const size_t hk = o, hc = hk + al16(8ull * hcap), nb = o;
  const size_t hash = al16(8ull * hcap) + al16(4ull * hcap), nbr = al16(4ull * n * k);
  o += hash > nbr ? hash : nbr;
  if (m) {
    m->head = (BigHead *)(base + head);
    m->pts = (float4 *)(base + pts);
    m->r2 = (float *)(base + r2);
    m->wa = (float *)(base + wa);
    m->F = (float *)(base + f);
    m->flag = (uint8_t *)(base + fl);
    m->nbr = (uint32_t *)(base + nb);
    m->box = box_index(base + bx, n);
    m->hkey = (unsigned long long *)(base + hk);
    m->hcnt = (uint32_t *)(base + hc);
    m->hcap = hcap;
  }
  return o;
}

__device__ __forceinline__ BigMem big_mem(const LeafArgs &A, const Leaf &lf) {
  BigMem m;
  big_carve(A.big_scratch + (size_t)lf.start * A.big_bpp, lf.count, A.p.k, &m);
  return m;
}

// the big leaf whose units hold unit u (unit_start ascending), and u's index in it
__device__ __forceinline__ uint32_t big_find(const uint32_t *__restrict__ unit_start, uint32_t nbig, uint32_t u) {
  uint32_t lo = 0, hi = nbig - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (unit_start[mid] <= u) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// one block: the leaves' first units (prefix over the class-0 leaves of the order), and their heads reset
__global__ void __launch_bounds__(1024) k_big_setup(const LeafArgs A) {
  __shared__ uint32_t s_w[32], s_run;
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t nbig = A.ctr->cls_count[0], tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  if (tid == 0) s_run = 0;
  __syncthreads();
  for (uint32_t base = 0; base < nbig; base += 1024u) {
    const uint32_t i = base + tid;
    uint32_t c = 0;
    if (i < nbig) {
      const Leaf lf = A.leaves[A.order[i]];
      c = (lf.count + kBigUnit - 1u) / kBigUnit;
      BigHead *h = big_mem(A, lf).head;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        h->lo_ord[a] = 0xFFFFFFFFu;
        h->hi_ord[a] = 0u;
      }
      h->units_done = 0;
      h->n1 = 0;
    }
    uint32_t inc = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= (uint32_t)o) inc += y;
    }
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    if (w == 0) {
      const uint32_t v = s_w[lane];
      uint32_t x = v;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      s_w[lane] = x - v;
    }
    __syncthreads();
    const uint32_t run = s_run;
    if (i < nbig) A.unit_start[i] = run + s_w[w] + inc - c;
    __syncthreads();
    if (tid == 1023) s_run = run + s_w[w] + inc;
    __syncthreads();
  }
  if (tid == 0) {
    A.ctr->big_units = s_run;
    A.ctr->big_work = 0;
    A.ctr->far_count = 0;
  }
}

// Eq. 10-11: the leaf's box (exact FP32 min / max); the unit that finishes a leaf
// computes h as the prep kernel does.  The unit also clears its share of the hash.
__global__ void __launch_bounds__(kBigUnit) k_big_box(const LeafArgs A) {
  __shared__ uint32_t s_mn[3], s_mx[3];
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t nu = A.ctr->big_units, nbig = A.ctr->cls_count[0], tid = threadIdx.x;
  for (uint32_t u = blockIdx.x; u < nu; u += gridDim.x) {
    const uint32_t b = big_find(A.unit_start, nbig, u), li = A.order[b], part = u - A.unit_start[b];
    const Leaf lf = A.leaves[li];
    const BigMem M = big_mem(A, lf);
    const uint32_t nun = (lf.count + kBigUnit - 1u) / kBigUnit, i = part * kBigUnit + tid;
    if (tid < 3) {
      s_mn[tid] = 0xFFFFFFFFu;
      s_mx[tid] = 0u;
    }
    for (uint32_t s = part * kBigUnit + tid; s < M.hcap; s += nun * kBigUnit) {
      M.hkey[s] = kEmpty;
      M.hcnt[s] = 0;
    }
    __syncthreads();
    uint32_t mn[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu}, mx[3] = {0u, 0u, 0u};
    if (i < lf.count) {
      const float4 p = A.spts[lf.start + i];
      mn[0] = mx[0] = f2ord(p.x);
      mn[1] = mx[1] = f2ord(p.y);
      mn[2] = mx[2] = f2ord(p.z);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const uint32_t l = __reduce_min_sync(0xFFFFFFFFu, mn[a]), h = __reduce_max_sync(0xFFFFFFFFu, mx[a]);
      if ((tid & 31u) == 0) {
        atomicMin(&s_mn[a], l);
        atomicMax(&s_mx[a], h);
      }
    }
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        atomicMin(&M.head->lo_ord[a], s_mn[a]);
        atomicMax(&M.head->hi_ord[a], s_mx[a]);
      }
      __threadfence();
      if (atomicAdd(&M.head->units_done, 1u) == nun - 1u) {
        __threadfence();
        const float delta = A.frames[lf.frame].delta;
        float lo[3], e[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          // read past the cache: other units' atomics wrote them
          lo[a] = ord2f(ld_volatile(&M.head->lo_ord[a]));
          e[a] = __fsub_rn(ord2f(ld_volatile(&M.head->hi_ord[a])), lo[a]);
        }
        Leaf *out = const_cast<Leaf *>(A.leaves) + li;
        out->h = leaf_voxel_size(e, delta, lf.count, A.p.beta);
#pragma unroll
        for (int a = 0; a < 3; ++a) out->lo[a] = lo[a];
      }
    }
    __syncthreads();
  }
}

// Eq. 12: voxel occupancy in the leaf's hash table (global memory, warp-aggregated)
__global__ void __launch_bounds__(kBigUnit) k_big_voxels(const LeafArgs A) {
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t nu = A.ctr->big_units, nbig = A.ctr->cls_count[0], tid = threadIdx.x;
  const uint32_t lt = lanemask_lt();
  for (uint32_t u = blockIdx.x; u < nu; u += gridDim.x) {
    const uint32_t b = big_find(A.unit_start, nbig, u);
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t i = (u - A.unit_start[b]) * kBigUnit + tid;
    unsigned long long key = kInvalid;
    if (i < lf.count) {
      const float4 p = A.spts[lf.start + i];
      key = voxel_key(p, lf.lo, lf.h);
    }
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, key);
    uint32_t sl = 0;
    if (i < lf.count && (peers & lt) == 0) {
      sl = hash_insert(M.hkey, M.hcap, key, A.ctr);
      atomicAdd(M.hcnt + sl, (uint32_t)__popc(peers));
    }
    sl = __shfl_sync(0xFFFFFFFFu, sl, __ffs(peers) - 1);
    if (i < lf.count) reinterpret_cast<uint32_t *>(M.wa)[i] = sl;
  }
}

// the voxel gate; P_1 points packed for the kNN, their chunk and super-chunk boxes
__global__ void __launch_bounds__(kBigUnit) k_big_p1(const LeafArgs A) {
  __shared__ Box s_box[32];
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t nu = A.ctr->big_units, nbig = A.ctr->cls_count[0], tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  for (uint32_t u = blockIdx.x; u < nu; u += gridDim.x) {
    const uint32_t b = big_find(A.unit_start, nbig, u), part = u - A.unit_start[b];
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t i = part * kBigUnit + tid;
    Box bx = box_empty();
    bool in1 = false;
    if (i < lf.count) {
      float4 p = A.spts[lf.start + i];
      in1 = M.hcnt[reinterpret_cast<const uint32_t *>(M.wa)[i]] >= A.p.min_vox_count;
      if (in1) {
        bx = box_point(p.x, p.y, p.z);
      } else {
        write_point<false>(A, __float_as_uint(p.w), 0, 0.0f, 1);
        p.x = p.y = p.z = __int_as_float(0x7FFFFFFF);
        M.r2[i] = __uint_as_float(0xFFFFFFFFu);
      }
      M.pts[i] = p;
      M.flag[i] = 0;
    }
    const uint32_t cnt = __popc(__ballot_sync(0xFFFFFFFFu, in1));
    bx = box_warp_union(bx);
    if (lane == 0) {
      if (part * kBigUnit + 32u * w < lf.count) box_store(M.box.chunk, part * 32u + w, bx);
      s_box[w] = bx;
      if (cnt) atomicAdd(&M.head->n1, cnt);
    }
    __syncthreads();
    if (w == 0) {
      const Box s = box_warp_union(s_box[lane]);
      if (lane == 0) box_store(M.box.super, part, s);
    }
    __syncthreads();
  }
}

// kNN of the P_1 points within the leaf: one warp per chunk of queries
struct BigSrc {
  const float4 *pts;
  uint32_t n;
  BoxIndex box;
  __device__ __forceinline__ uint32_t entries() const { return box_supers(n); }
  __device__ __forceinline__ void entry(uint32_t e, uint32_t &s, uint32_t &a, uint32_t &b) const {
    s = e;
    a = 0;
    b = n;
  }
  __device__ __forceinline__ float4 load(uint32_t p) const { return pts[p]; }
};

template <int KROW, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_big_knn(const LeafArgs A) {
  __shared__ BkShared<KROW> s_w[WARPS];
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  BkShared<KROW> &S = s_w[threadIdx.x >> 5];
  const uint32_t nbig = A.ctr->cls_count[0], lane = threadIdx.x & 31u;
  const uint32_t nunits = A.ctr->big_units * kBigChunks;
  for (;;) {
    uint32_t u = 0;
    if (lane == 0) u = atomicAdd(&A.ctr->big_work, 1u);
    u = __shfl_sync(0xFFFFFFFFu, u, 0);
    if (u >= nunits) break;
    const uint32_t b = big_find(A.unit_start, nbig, u / kBigChunks);
    const Leaf lf = A.leaves[A.order[b]];
    const uint32_t c = u - A.unit_start[b] * kBigChunks, n = lf.count;
    if (c * kBoxChunk >= n) continue;  // the last unit's tail
    const BigMem M = big_mem(A, lf);
    const uint32_t n1 = M.head->n1;
    if (n1 <= 1) continue;
    if (n1 >= (1u << kBkPlanes)) {  // beyond the counters: refuse, do not guess
      if (lane == 0) atomicOr(&A.ctr->status, kStInternal);
      return;
    }
    const uint32_t k = A.p.k < n1 - 1 ? A.p.k : n1 - 1;
    uint32_t q = c * kBoxChunk + lane;
    float4 me = make_float4(__int_as_float(0x7FFFFFFF), 0.f, 0.f, 0.f);
    if (q < n) me = M.pts[q];
    const bool act = me.x == me.x;
    const uint32_t any = __ballot_sync(0xFFFFFFFFu, act);
    if (!any) continue;
    const int first = __ffs(any) - 1;  // lanes without a P_1 point shadow its query
    const float fx = __shfl_sync(0xFFFFFFFFu, me.x, first), fy = __shfl_sync(0xFFFFFFFFu, me.y, first),
                fz = __shfl_sync(0xFFFFFFFFu, me.z, first);
    if (!act) {
      q = c * kBoxChunk + (uint32_t)first;
      me.x = fx;
      me.y = fy;
      me.z = fz;
    }
    const BigSrc src{M.pts, n, M.box};
    float theta;
    uint32_t far;
    if (!bk_knn(src, S, act, q, me.x, me.y, me.z, k, 0u, n, bk_share(n), theta, far)) atomicOr(&A.ctr->status, kStInternal);
    const float delta = A.frames[lf.frame].delta, delta2 = __fmul_rn(delta, delta);
    const bool gone = (far >> lane) & 1u;
    if (act) M.r2[q] = (theta < delta2 && !gone) ? delta2 : theta;  // (a far query's bound, for its own warp)
    if (far) {
      uint32_t slot = 0;
      if (lane == 0) slot = atomicAdd(&A.ctr->far_count, (uint32_t)__popc(far));
      slot = __shfl_sync(0xFFFFFFFFu, slot, 0) + __popc(far & lanemask_lt());
      if (gone) A.far_queue[slot] = make_uint2(b, q);
    }
    for (uint32_t m = any & ~far; m; m &= m - 1u) {
      const uint32_t l = (uint32_t)__ffs(m) - 1u;
      for (uint32_t t = lane; t < k; t += 32u) M.nbr[(size_t)(c * kBoxChunk + l) * A.p.k + t] = S.row[l][t];
    }
    __syncwarp();
  }
}

// the queries that were left to a warp of their own
__global__ void __launch_bounds__(128) k_big_knn_far(const LeafArgs A) {
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t lane = threadIdx.x & 31u, nq = A.ctr->far_count;
  for (uint32_t i = blockIdx.x * 4u + (threadIdx.x >> 5); i < nq; i += gridDim.x * 4u) {
    const uint2 e = A.far_queue[i];
    const Leaf lf = A.leaves[A.order[e.x]];
    const BigMem M = big_mem(A, lf);
    const uint32_t n1 = M.head->n1, k = A.p.k < n1 - 1 ? A.p.k : n1 - 1, q = e.y;
    const float4 me = M.pts[q];
    const BigSrc src{M.pts, lf.count, M.box};
    BkList L;
    bk_knn_far(src, q, me.x, me.y, me.z, k, M.r2[q], L);
    // the neighbours in position order: the order in which the score sums them
    uint32_t v = lane < k ? L.pos : 0xFFFFFFFFu;
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
      for (int o = size >> 1; o > 0; o >>= 1) {
        const uint32_t x = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        v = (((lane & o) == 0) == ((lane & size) == 0)) ? min(v, x) : max(v, x);
      }
    }
    if (lane < k) M.nbr[(size_t)q * A.p.k + lane] = v;
    const uint32_t kth = (uint32_t)(__shfl_sync(0xFFFFFFFFu, L.key, k - 1) >> 32);
    if (lane == 0) {
      if (kth > 0x7F800000u) atomicOr(&A.ctr->status, kStInternal);  // the list did not fill: cannot happen
      const float delta = A.frames[lf.frame].delta, delta2 = __fmul_rn(delta, delta), rk = __uint_as_float(kth);
      M.r2[q] = rk < delta2 ? delta2 : rk;
    }
  }
}

// ---------------------------------------------------------------------------
// order statistics of one leaf by one CTA
// ---------------------------------------------------------------------------
struct SelectShared {
  uint32_t hist[2048];
  uint32_t wsum[32];
  uint32_t bin, below, mn, mx, cnt;
};

// The value of rank `rank` (0-based, ascending) among val(i), i < n, where val is
// at most `top` (values above it do not count), and how many lie below it and at it.
// Histograms of 11 bits of (value - smallest value), from the highest bit of the
// range down: three passes at most, and bins that spread over the range.
template <typename F>
__device__ uint32_t block_select(SelectShared &S, F val, uint32_t n, uint32_t top, uint32_t rank, uint32_t *below,
                                 uint32_t *at) {
  const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  if (tid == 0) {
    S.mn = 0xFFFFFFFFu;
    S.mx = 0;
  }
  __syncthreads();
  uint32_t mn = 0xFFFFFFFFu, mx = 0;
  for (uint32_t i = tid; i < n; i += kSelectThreads) {
    const uint32_t v = val(i);
    if (v <= top) {
      mn = min(mn, v);
      mx = max(mx, v);
    }
  }
  mn = __reduce_min_sync(0xFFFFFFFFu, mn);
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  if (lane == 0) {
    atomicMin(&S.mn, mn);
    atomicMax(&S.mx, mx);
  }
  __syncthreads();
  uint32_t base = S.mn, range = S.mx - base;  // candidates: base <= v <= base + range
  uint32_t nb = 0;
  for (;;) {
    const int bits = 32 - __clz(range);
    const int sh = bits > 11 ? bits - 11 : 0;
    for (uint32_t i = tid; i < 2048u; i += kSelectThreads) S.hist[i] = 0;
    __syncthreads();
    for (uint32_t i = tid; i < n; i += kSelectThreads) {
      const uint32_t v = val(i);
      const bool in = v <= top && v >= base && v - base <= range;
      if (in) atomicAdd(&S.hist[(v - base) >> sh], 1u);
    }
    __syncthreads();
    // the bin that holds the rank: scan of 2 bins a thread
    const uint32_t h0 = S.hist[2 * tid], h1 = S.hist[2 * tid + 1];
    uint32_t inc = h0 + h1;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= (uint32_t)o) inc += y;
    }
    if (lane == 31) S.wsum[w] = inc;
    __syncthreads();
    uint32_t pre = inc - h0 - h1;
    for (uint32_t i = 0; i < w; ++i) pre += S.wsum[i];
    const uint32_t r = rank - nb;
    if (pre <= r && r < pre + h0) {
      S.bin = 2 * tid;
      S.below = pre;
      S.cnt = h0;
    } else if (pre + h0 <= r && r < pre + h0 + h1) {
      S.bin = 2 * tid + 1;
      S.below = pre + h0;
      S.cnt = h1;
    }
    __syncthreads();
    nb += S.below;
    const uint32_t cnt = S.cnt;
    base += S.bin << sh;
    if (sh == 0) {
      if (below) *below = nb;
      if (at) *at = cnt;
      return base;
    }
    range = (1u << sh) - 1u;
    __syncthreads();
  }
}

// a leaf's values in shared memory, eight loads in flight a thread; false: too many
template <typename F>
__device__ __forceinline__ bool stage_values(uint32_t *sv, F val, uint32_t n) {
  if (n > kSelectCap) return false;
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 8u * kSelectThreads) {
    uint32_t v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t i = i0 + u * kSelectThreads;
      if (i < n) v[u] = val(i);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t i = i0 + u * kSelectThreads;
      if (i < n) sv[i] = v[u];
    }
  }
  __syncthreads();
  return true;
}

// Eq. 14 cut and Eq. 16 median of one leaf per CTA
__global__ void __launch_bounds__(kSelectThreads) k_big_gate(const LeafArgs A) {
  extern __shared__ uint32_t s_val[];
  __shared__ SelectShared S;
  __shared__ uint32_t s_next;
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t nbig = A.ctr->cls_count[0], tid = threadIdx.x;
  const denoise_params &P = A.p;
  for (uint32_t b = blockIdx.x; b < nbig; b += gridDim.x) {
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t n = lf.count, n1 = M.head->n1;
    if (n1 <= 1) continue;
    const uint32_t keff = P.k < n1 - 1 ? P.k : n1 - 1;
    auto global = [&](uint32_t i) { return __float_as_uint(M.r2[i]); };
    auto run = [&](auto r2bits) {
      const double pos = __dadd_rn(__ddiv_rn(__dmul_rn((double)n1, (double)P.rho_percentile), 100.0), 0.5);
      const double cc = ceil(pos);
      const uint32_t crank = (cc < 1.0) ? 1u : (cc > (double)n1) ? n1 : (uint32_t)cc;
      uint32_t below, at;
      const uint32_t Rb = block_select(S, r2bits, n, 0x7F800000u, n1 - crank, &below, &at);
      const uint32_t m = below + at;  // |P_2|: every r_K^2 up to the cut
      __syncthreads();
      const uint32_t rab = block_select(S, r2bits, n, Rb, (m - 1) / 2, &below, &at);
      uint32_t rbb = rab;
      if (!(m & 1u) && below + at <= m / 2) {  // the upper middle value is the next larger one
        if (tid == 0) s_next = 0xFFFFFFFFu;
        __syncthreads();
        uint32_t nx = 0xFFFFFFFFu;
        for (uint32_t i = tid; i < n; i += kSelectThreads) {
          const uint32_t v = r2bits(i);
          if (v > rab) nx = min(nx, v);
        }
        nx = __reduce_min_sync(0xFFFFFFFFu, nx);
        if ((tid & 31u) == 0) atomicMin(&s_next, nx);
        __syncthreads();
        rbb = s_next;
      }
      if (tid == 0) {
        M.head->Rb = Rb;
        M.head->m = m;
        M.head->r2ref = __uint_as_float(rab);
        M.head->Lref = leaf_lref(__uint_as_float(rab), __uint_as_float(rbb), m, keff, P.eps_rho);
        atomicAdd(&A.ctr->knn_pairs, (unsigned long long)n1 * (unsigned long long)(n1 - 1));
        atomicAdd(&A.ctr->n_p1, (unsigned long long)n1);
        atomicAdd(&A.ctr->n_p2, (unsigned long long)m);
        atomicAdd(&A.ctr->score_terms, (unsigned long long)m * keff);
      }
    };
    if (stage_values(s_val, global, n)) run([&](uint32_t i) { return s_val[i]; });
    else run(global);
    __syncthreads();
  }
}

// the density gate and the score's per-point weights
__global__ void __launch_bounds__(256) k_big_weight(const LeafArgs A) {
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  constexpr uint32_t kPart = kBigUnit / 256;
  const uint32_t nu = A.ctr->big_units * kPart, nbig = A.ctr->cls_count[0];
  const float half_alpha = __fmul_rn(0.5f, A.p.alpha);
  for (uint32_t u = blockIdx.x; u < nu; u += gridDim.x) {
    const uint32_t b = big_find(A.unit_start, nbig, u / kPart);
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t i = (u - A.unit_start[b] * kPart) * 256u + threadIdx.x;
    if (i >= lf.count || M.head->n1 <= 1) continue;
    const uint32_t v = __float_as_uint(M.r2[i]);
    if (v > 0x7F800000u) continue;  // outside P_1
    M.wa[i] = __fmul_rn(half_alpha, score_ell(__uint_as_float(v), M.head->r2ref, M.head->Lref));
    M.flag[i] = v <= M.head->Rb;
  }
}

// Eq. 15-21: the score of every P_2 point, in the fused kernel's operation order
__global__ void __launch_bounds__(256) k_big_score(const LeafArgs A) {
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  constexpr uint32_t kPart = kBigUnit / 256;
  const uint32_t nu = A.ctr->big_units * kPart, nbig = A.ctr->cls_count[0], tid = threadIdx.x;
  const denoise_params &P = A.p;
  const bool g2 = (P.gamma == 2.0f);
  const float hg = 0.5f * P.gamma, ek = P.eps_k;
  const float c2 = __fdiv_rn(1.4426950408889634f, __fmul_rn(__fmul_rn(2.0f, P.sigma), P.sigma));
  for (uint32_t u = blockIdx.x; u < nu; u += gridDim.x) {
    const uint32_t b = big_find(A.unit_start, nbig, u / kPart);
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t i = (u - A.unit_start[b] * kPart) * 256u + tid, n1 = M.head->n1;
    if (i >= lf.count || !M.flag[i]) continue;
    const uint32_t keff = P.k < n1 - 1 ? P.k : n1 - 1;
    const float4 me = M.pts[i];
    const float ai = M.wa[i], ci = __fdiv_rn(c2, M.r2[i]);
    const uint32_t *row = M.nbr + (size_t)i * P.k;
    float F[2] = {0.0f, 0.0f};
    for (uint32_t t = 0; t < keff; t += 2) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (t + h >= keff) continue;  // (the fused kernel adds +0 here)
        const uint32_t j = row[t + h];
        const float4 p = M.pts[j];
        const float d2 = sqdist(me.x, me.y, me.z, p.x, p.y, p.z);
        const float wt = ex2_hw(__fmaf_rn(d2, -ci, __fadd_rn(ai, M.wa[j])));
        const float D = g2 ? d2 : pow_half_gamma(d2, hg);
        F[h] = __fadd_rn(F[h], __fmul_rn(wt, rcp_hw(__fadd_rn(D, ek))));
      }
    }
    M.F[i] = __fadd_rn(F[0], F[1]);
  }
}

// the selection's cut of one leaf per CTA
__global__ void __launch_bounds__(kSelectThreads) k_big_select(const LeafArgs A) {
  extern __shared__ uint32_t s_val[];
  __shared__ SelectShared S;
  __shared__ uint32_t s_real;
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t nbig = A.ctr->cls_count[0], tid = threadIdx.x;
  for (uint32_t b = blockIdx.x; b < nbig; b += gridDim.x) {
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t n = lf.count;
    if (M.head->n1 <= 1) continue;
    const uint32_t m = M.head->m;
    // ~F orders like (F descending); points outside P_2 are above every select's top
    auto global = [&](uint32_t i) {
      const float F = M.F[i];
      return M.flag[i] ? 0xFFFFFFFFu - __float_as_uint(F) : 0xFFFFFFFFu;
    };
    auto run = [&](auto key) {
      uint32_t keep_n = (uint32_t)ceil((double)A.p.lambda * (double)m);
      if (keep_n > m) keep_n = m;
      // a P_2 key can be 0xFFFFFFFF too (F = +0): where the others run out, every such point is at the cut
      if (tid == 0) s_real = 0;
      __syncthreads();
      uint32_t real = 0;
      for (uint32_t i = tid; i < n; i += kSelectThreads) real += key(i) != 0xFFFFFFFFu;
      real = __reduce_add_sync(0xFFFFFFFFu, real);
      if ((tid & 31u) == 0 && real) atomicAdd(&s_real, real);
      __syncthreads();
      real = s_real;
      uint32_t cut = 0xFFFFFFFFu, below = real, at = m - real;
      if (keep_n <= real) cut = block_select(S, key, n, 0xFFFFFFFEu, keep_n - 1, &below, &at);
      if (tid == 0) {
        M.head->cut = cut;
        M.head->needed = keep_n - below;
        M.head->at = at;
      }
    };
    if (stage_values(s_val, global, n)) run([&](uint32_t i) { return s_val[i]; });
    else run(global);
    __syncthreads();
  }
}

// the results (points outside P_1 were written by the voxel gate)
__global__ void __launch_bounds__(256) k_big_out(const LeafArgs A) {
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  constexpr uint32_t kPart = kBigUnit / 256;
  const uint32_t nu = A.ctr->big_units * kPart, nbig = A.ctr->cls_count[0];
  const denoise_params &P = A.p;
  for (uint32_t u = blockIdx.x; u < nu; u += gridDim.x) {
    const uint32_t b = big_find(A.unit_start, nbig, u / kPart);
    const Leaf lf = A.leaves[A.order[b]];
    const BigMem M = big_mem(A, lf);
    const uint32_t n = lf.count, i = (u - A.unit_start[b] * kPart) * 256u + threadIdx.x;
    if (i >= n) continue;
    const float4 p = M.pts[i];
    if (!(p.x == p.x)) continue;
    const uint32_t g = __float_as_uint(p.w);
    if (M.head->n1 <= 1 || !M.flag[i]) {  // the density gate (a lone point of P_1 has no neighbour)
      write_point<false>(A, g, 0, 0.0f, 2);
      continue;
    }
    const float F = M.F[i];
    bool keep;
    if (P.select_mode == DENOISE_SELECT_TOPRATIO) {
      const uint32_t kk = 0xFFFFFFFFu - __float_as_uint(F), cut = M.head->cut;
      keep = kk < cut || (kk == cut && M.head->needed >= M.head->at);
      if (kk == cut && M.head->needed < M.head->at) {  // exact score ties at the cut: rank by input index
        uint32_t before = 0;
        for (uint32_t j = 0; j < n; ++j)
          before += M.flag[j] && 0xFFFFFFFFu - __float_as_uint(M.F[j]) == cut && __float_as_uint(M.pts[j].w) < g;
        keep = before < M.head->needed;
      }
    } else {
      keep = logf(F) >= P.tau;
    }
    write_point<false>(A, g, keep ? 1 : 0, F, keep ? 0 : 3);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// The size above which a call's leaves are taken here, 0 = never (the options below,
// or no leaf can be that large but for duplicates).  The fused kernel compares all
// pairs of a leaf, but from shared memory and without this path's launches.  Dense
// scans, us a call, fused (256 or 512 threads) / this path for leaves above 512:
// capacity 1,000, 200k points 377 / 416, 560k 589 / 751; capacity 2,048, 10k 661 / 271,
// 100k 937 / 376, 560k 1299 / 873.  Where a call is one leaf, its serial time on one
// CTA decides: from 512 points.
// `frame`: points of the largest frame, which no leaf exceeds (64 frames of 600 points at
// depth 1, judged by all their points: 11 launches for nothing, 172 us a call instead of 162).
uint32_t big_leaf_above(const denoise_params &p, uint32_t n, uint32_t frame, bool rec) {
  if (p.stage_off || p.rescore_p2 || p.cross_leaf || rec) return 0;
  const uint32_t above = p.leaf_capacity >= n ? 512u : 1024u;
  if (frame <= above) return 0;
  if (p.leaf_capacity > above) return above;
  // a depth limit that leaves more than `above` points to some cell
  return (p.max_depth < 8 && (frame >> (3 * p.max_depth)) > above) ? above : 0u;
}

int launch_big(const LeafArgs &a, int num_sms, cudaStream_t st, int *launches) {
  const dim3 per_leaf(num_sms), units(num_sms * 2), parts(num_sms * 8);
  // no leaf is larger than the call: the selects' shared memory (their limit is the
  // same for every call, as other contexts' threads launch the same kernels)
  const size_t sel = 4ull * (a.n < kSelectCap ? a.n : kSelectCap);
  constexpr int kSelLimit = 4 * (int)kSelectCap;
  if (cudaFuncSetAttribute(k_big_gate, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelLimit) != cudaSuccess ||
      cudaFuncSetAttribute(k_big_select, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelLimit) != cudaSuccess)
    return -1;
  launch_pdl(k_big_setup, 1, 1024, 0, st, a);
  launch_pdl(k_big_box, units, kBigUnit, 0, st, a);
  launch_pdl(k_big_voxels, units, kBigUnit, 0, st, a);
  launch_pdl(k_big_p1, units, kBigUnit, 0, st, a);
  if (a.p.k <= 32) launch_pdl(k_big_knn<32, 4>, num_sms * 6, 128, 0, st, a);
  else launch_pdl(k_big_knn<64, 2>, num_sms * 8, 64, 0, st, a);
  if (a.p.k <= kBkFarK) launch_pdl(k_big_knn_far, num_sms * 8, 128, 0, st, a);
  launch_pdl(k_big_gate, per_leaf, kSelectThreads, sel, st, a);
  launch_pdl(k_big_weight, parts, 256, 0, st, a);
  launch_pdl(k_big_score, parts, 256, 0, st, a);
  if (a.p.select_mode == DENOISE_SELECT_TOPRATIO) launch_pdl(k_big_select, per_leaf, kSelectThreads, sel, st, a);
  launch_pdl(k_big_out, parts, 256, 0, st, a);
  if (launches) *launches += 9 + (a.p.k <= kBkFarK) + (a.p.select_mode == DENOISE_SELECT_TOPRATIO);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace gd
