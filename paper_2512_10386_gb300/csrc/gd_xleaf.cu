// gd_xleaf.cu -- the cross-leaf kNN variant: neighbours searched over the
// octree cells adjacent to a point's leaf, not only within the leaf (the
// leaf-local search of Sec. 3 gives the points on a leaf's border an r_K
// inflated by the missing points across it).
//
// Candidates of the points of a leaf at level L: the P_1 points of the 27
// cells of level L around (and including) the leaf's cell.  A cell of level L
// is a contiguous range of the Morton-sorted points, found by binary search of
// its key prefix, so the candidate set is at most 27 ranges, shared by every
// query of the leaf.  They are streamed through shared memory in tiles; each
// thread keeps its query's k_eff smallest (d^2, input index) keys in a sorted
// list (d^2 in FP32 with the method's operation order, ties by input index:
// the exact rule).  Outputs by sorted position: the neighbours (sorted
// positions), the floored r_K^2 and k_eff.  The per-leaf gate, median, score and
// selection then run in the fused leaf kernel's cross-leaf phase.
//
// For K <= 32 the P_1 points get chunk boxes (k_xleaf_boxes), every leaf its 27 ranges
// and |C_t| once (k_xleaf_ranges), and one warp finds the neighbours of 32 queries by
// counting, reading only the chunks of the ranges that can hold one (gd_boxknn.cuh;
// k_xleaf_knn_box, k_xleaf_knn_far; small calls: k_xleaf_knn_far alone).  A 560,000-point scan, K = 32: 3.2 G pairs in the
// ranges, 8.5 ms with every candidate compared, 3.0 ms so (1.7 the box search, 0.8 the
// far queries), issue in 67 % of the cycles at 29 % of the warp slots.  Larger K keep the per-thread list (k_xleaf_knn).
#include <cuda_runtime.h>

#include "gd_boxknn.cuh"

namespace gd {

constexpr int kXThreads = 128;
constexpr int kXTile = 1024;  // candidates staged per round

__device__ __forceinline__ uint32_t compact3(unsigned long long k) {  // bits 0, 3, 6, ... -> 0, 1, 2, ...
  k &= 0x1249249249249249ull;
  k = (k | (k >> 2)) & 0x10C30C30C30C30C3ull;
  k = (k | (k >> 4)) & 0x100F00F00F00F00Full;
  k = (k | (k >> 8)) & 0x1F0000FF0000FFull;
  k = (k | (k >> 16)) & 0x1F00000000FFFFull;
  k = (k | (k >> 32)) & 0x1FFFFFull;
  return (uint32_t)k;
}

__device__ __forceinline__ float xsqdist(float xi, float yi, float zi, const float4 &b) {
  const float dx = __fsub_rn(b.x, xi), dy = __fsub_rn(b.y, yi), dz = __fsub_rn(b.z, zi);
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// first position in [lo, hi) whose key is >= key
__device__ __forceinline__ uint32_t lower_key(const unsigned long long *keys, uint32_t lo, uint32_t hi,
                                              unsigned long long key) {
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (keys[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

template <int KMAX, bool kRec>
__global__ void __launch_bounds__(kXThreads) k_xleaf_knn(const XleafArgs A) {
  __shared__ float4 s_pts[kXTile];
  __shared__ uint32_t s_pos[kXTile];
  __shared__ uint32_t s_rng[27][2];
  __shared__ uint32_t s_leaf, s_cnt, s_fill;
  const uint32_t tid = threadIdx.x;
  pdl_wait();
  const uint32_t n_leaves = A.ctr->n_leaves;
  for (;;) {
    if (tid == 0) s_leaf = (ld_volatile(&A.ctr->status) & kStFatal) ? 0xFFFFFFFFu : atomicAdd(&A.ctr->xleaf_work, 1u);
    __syncthreads();
    const uint32_t li = s_leaf;
    if (li >= n_leaves) break;
    const Leaf lf = A.leaves[li];
    const FrameInfo fr = A.frames[lf.frame];
    // the 27 cell ranges (level-0 leaf: the whole frame)
    if (tid < 27) {
      uint32_t a = 0, b = 0;
      const uint32_t L = leaf_level(lf);
      if (L == 0) {
        if (tid == 13) { a = fr.begin; b = fr.end; }
      } else {
        const unsigned long long k0 = A.keys[lf.start];
        const int sh = 3 * (21 - (int)L);
        const int64_t cx = compact3(k0 >> 2) >> (21 - L), cy = compact3(k0 >> 1) >> (21 - L),
                      cz = compact3(k0) >> (21 - L);
        const int64_t x = cx + (int64_t)(tid / 9) - 1, y = cy + (int64_t)((tid / 3) % 3) - 1,
                      z = cz + (int64_t)(tid % 3) - 1;
        const int64_t side = (int64_t)1 << L;
        if (x >= 0 && y >= 0 && z >= 0 && x < side && y < side && z < side) {
          const unsigned long long pre = morton3((uint32_t)x, (uint32_t)y, (uint32_t)z);
          a = lower_key(A.keys, fr.begin, fr.end, pre << sh);
          b = lower_key(A.keys, a, fr.end, (pre + 1ull) << sh);
        }
      }
      s_rng[tid][0] = a;
      s_rng[tid][1] = b;
    }
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    // |C_t|: the P_1 points of the block
    uint32_t cnt = 0;
    for (int r = 0; r < 27; ++r)
      for (uint32_t p = s_rng[r][0] + tid; p < s_rng[r][1]; p += kXThreads) cnt += A.xflag[p];
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    if ((tid & 31) == 0) atomicAdd(&s_cnt, cnt);
    __syncthreads();
    const uint32_t nc = s_cnt;
    const uint32_t keff = nc <= 1 ? 0u : (A.k < nc - 1 ? A.k : nc - 1);
    const float delta2 = __fmul_rn(fr.delta, fr.delta);
    uint32_t nq = 0;
    for (uint32_t qb = 0; qb < lf.count; qb += kXThreads) {
      const uint32_t qi = qb + tid;
      const bool act = qi < lf.count && A.xflag[lf.start + qi];
      const uint32_t qp = lf.start + (qi < lf.count ? qi : 0);
      const float4 me = A.spts[qp];
      unsigned long long L[KMAX];
      uint32_t Pp[KMAX];
#pragma unroll
      for (int s = 0; s < KMAX; ++s) {
        L[s] = ~0ull;
        Pp[s] = 0;
      }
      unsigned long long thr = ~0ull;  // the k_eff-th key so far
      for (int r = 0; r < 27; ++r) {
        for (uint32_t c0 = s_rng[r][0]; c0 < s_rng[r][1]; c0 += kXTile) {
          const uint32_t len = min((uint32_t)kXTile, s_rng[r][1] - c0);
          __syncthreads();
          for (uint32_t u = tid; u < len; u += kXThreads) {
            s_pts[u] = A.spts[c0 + u];
            s_pos[u] = A.xflag[c0 + u] ? c0 + u : 0xFFFFFFFFu;
          }
          __syncthreads();
          if (!act || keff == 0) continue;
          for (uint32_t u = 0; u < len; ++u) {
            const uint32_t pu = s_pos[u];
            if (pu == 0xFFFFFFFFu || pu == qp) continue;
            const float4 c = s_pts[u];
            const float d2 = xsqdist(me.x, me.y, me.z, c);
            const unsigned long long key = ((unsigned long long)__float_as_uint(d2) << 32) | __float_as_uint(c.w);
            if (key >= thr) continue;
            // insert into the sorted list of k_eff keys
            int s = (int)keff - 1;
            while (s > 0 && L[s - 1] > key) {
              L[s] = L[s - 1];
              Pp[s] = Pp[s - 1];
              --s;
            }
            L[s] = key;
            Pp[s] = pu;
            thr = L[keff - 1];
          }
        }
      }
      if (act) {
        ++nq;
        A.xkeff[qp] = keff;
        if (keff) {
          const float rk = __uint_as_float((uint32_t)(L[keff - 1] >> 32));
          A.xr2[qp] = rk < delta2 ? delta2 : rk;
        }
        for (uint32_t t = 0; t < keff; ++t) A.xnbr[(size_t)qp * A.k + t] = Pp[t];
        if (kRec && A.use_dbg) {
          const uint32_t g = __float_as_uint(me.w);
          if (g < A.n) {
            for (uint32_t t = 0; t < A.k; ++t) {
              const bool v = t < keff;
              if (A.dbg.nbr) A.dbg.nbr[(size_t)g * A.k + t] = v ? (uint32_t)L[t] : 0xFFFFFFFFu;
              if (A.dbg.nbr_d2) A.dbg.nbr_d2[(size_t)g * A.k + t] = v ? __uint_as_float((uint32_t)(L[t] >> 32)) : 0.f;
            }
            if (A.dbg.r2 && keff) A.dbg.r2[g] = A.xr2[qp];
          } else {
            atomicOr(&A.ctr->status, kStInternal);
          }
        }
      }
    }
    nq = __reduce_add_sync(0xFFFFFFFFu, nq);
    if ((tid & 31) == 0 && nq && nc > 1) atomicAdd(&A.ctr->knn_pairs, (unsigned long long)nq * (nc - 1));
    __syncthreads();
  }
}

// ---- K <= 32: work units of (leaf, 32 queries), one warp each
constexpr uint32_t kXWUnit = 32;

// unit_start[l] = first work unit of leaf l (ceil(count / kXWUnit) units per leaf),
// ctr->x_units = the total: one block scans the leaf table
__global__ void __launch_bounds__(1024) k_xleaf_units(const Leaf *__restrict__ leaves, Counters *ctr,
                                                      uint32_t *__restrict__ unit_start) {
  __shared__ uint32_t s_w[32];
  __shared__ uint32_t s_run;
  pdl_wait();
  const uint32_t nl = ctr->n_leaves, tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  if (tid == 0) s_run = 0;
  __syncthreads();
  for (uint32_t base = 0; base < nl; base += 1024u) {
    const uint32_t i = base + tid;
    const uint32_t c = i < nl ? (leaves[i].count + kXWUnit - 1u) / kXWUnit : 0u;
    uint32_t inc = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= (uint32_t)o) inc += y;
    }
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    if (w == 0) {
      uint32_t v = s_w[lane], x = v;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      s_w[lane] = x - v;  // exclusive prefix of the warps
    }
    __syncthreads();
    const uint32_t run = s_run;
    if (i < nl) unit_start[i] = run + s_w[w] + inc - c;
    __syncthreads();
    if (tid == 1023) s_run = run + s_w[w] + inc;
    __syncthreads();
  }
  if (tid == 0) ctr->x_units = s_run;
}

// A leaf's candidate ranges, at the start of its slice of the spill area (idle
// between the fused kernel's cross-leaf phases; 320 bytes a point).
struct XRanges {
  uint32_t rng[27][2];
  uint32_t nc;  // |C_t|: the P_1 points in them
};
static_assert(sizeof(XRanges) <= 256, "a one-point leaf's slice holds its ranges");
__device__ __forceinline__ XRanges *x_ranges(const XleafArgs &A, const Leaf &lf) {
  return reinterpret_cast<XRanges *>(A.slices + (size_t)lf.start * A.slice_bpp);
}

// boxes of the P_1 points by sorted position, and each chunk's P_1 members as a bit mask
__global__ void __launch_bounds__(kBoxSuper) k_xleaf_boxes(const XleafArgs A) {
  __shared__ Box s_box[32];
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const BoxIndex bx = box_index(A.boxes, A.n);
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, i = blockIdx.x * kBoxSuper + threadIdx.x;
  if (i == 0) A.ctr->far_count = 0;
  Box b = box_empty();
  const bool in = i < A.n && A.xflag[i];
  if (in) {
    const float4 p = A.spts[i];
    b = box_point(p.x, p.y, p.z);
  }
  const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
  b = box_warp_union(b);
  if (lane == 0) {
    if (i < A.n) {
      box_store(bx.chunk, blockIdx.x * 32u + w, b);
      A.masks[blockIdx.x * 32u + w] = mask;
    }
    s_box[w] = b;
  }
  __syncthreads();
  if (w == 0) {
    b = box_warp_union(s_box[lane]);
    if (lane == 0) box_store(bx.super, blockIdx.x, b);
  }
}

// Calls of at most this many points give every query a warp of its own at once: they have
// too few warps of 32 queries to fill the GPU, and each is a chain of four passes.  us a
// call, warps of 32 queries / of one (K = 12, leaves of 64; K = 32, 256): 1,500 points 265 / 158,
// 271 / 160; 6,000 327 / 212, 387 / 237; 10,000 347 / 224, 488 / 272.
constexpr uint32_t kXSmall = 16384;

// the 27 ranges of every leaf and |C_t|: one warp a leaf; with `queue` its queries too go
// on the list of those with a warp of their own
__global__ void __launch_bounds__(128) k_xleaf_ranges(const XleafArgs A, const bool queue) {
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  const uint32_t lane = threadIdx.x & 31u, nl = A.ctr->n_leaves;
  for (uint32_t li = blockIdx.x * 4u + (threadIdx.x >> 5); li < nl; li += gridDim.x * 4u) {
    const Leaf lf = A.leaves[li];
    const FrameInfo &fr = A.frames[lf.frame];
    uint32_t a = 0, b = 0;
    const uint32_t L = leaf_level(lf);
    if (L == 0) {
      if (lane == 13) {  // a level-0 leaf: the whole frame
        a = fr.begin;
        b = fr.end;
      }
    } else if (lane < 27) {
      const unsigned long long k0 = A.keys[lf.start];
      const int sh = 3 * (21 - (int)L);
      const int64_t cx = compact3(k0 >> 2) >> (21 - L), cy = compact3(k0 >> 1) >> (21 - L),
                    cz = compact3(k0) >> (21 - L);
      const int64_t x = cx + (int64_t)(lane / 9) - 1, y = cy + (int64_t)((lane / 3) % 3) - 1,
                    z = cz + (int64_t)(lane % 3) - 1;
      const int64_t side = (int64_t)1 << L;
      if (x >= 0 && y >= 0 && z >= 0 && x < side && y < side && z < side) {
        const unsigned long long pre = morton3((uint32_t)x, (uint32_t)y, (uint32_t)z);
        a = lower_key(A.keys, fr.begin, fr.end, pre << sh);
        b = lower_key(A.keys, a, fr.end, (pre + 1ull) << sh);
      }
    }
    uint32_t cnt = 0;
    for (int r = 0; r < 27; ++r) {
      const uint32_t ra = __shfl_sync(0xFFFFFFFFu, a, r), rb = __shfl_sync(0xFFFFFFFFu, b, r);
      if (ra >= rb) continue;
      for (uint32_t c = ra / kBoxChunk + lane; c * kBoxChunk < rb; c += 32u) {
        uint32_t m = A.masks[c];
        const uint32_t p = c * kBoxChunk;
        if (p < ra) m &= 0xFFFFFFFFu << (ra - p);
        if (rb - p < 32u) m &= (1u << (rb - p)) - 1u;
        cnt += __popc(m);
      }
    }
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    XRanges *const x = x_ranges(A, lf);
    if (lane < 27) {
      x->rng[lane][0] = a;
      x->rng[lane][1] = b;
    }
    if (lane == 0) x->nc = cnt;
    if (queue) {
      uint32_t nq = 0;
      for (uint32_t q0 = 0; q0 < lf.count; q0 += 32u) {
        const uint32_t q = lf.start + q0 + lane;
        const bool act = q0 + lane < lf.count && A.xflag[q];
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, act);
        if (!m) continue;
        uint32_t slot = 0;
        if (lane == 0) slot = atomicAdd(&A.ctr->far_count, (uint32_t)__popc(m));
        slot = __shfl_sync(0xFFFFFFFFu, slot, 0) + __popc(m & lanemask_lt());
        if (act) {
          A.far_queue[slot] = make_uint2(li, q);
          A.xr2[q] = INFINITY;  // no bound yet
        }
        nq += __popc(m);
      }
      if (lane == 0 && nq && cnt > 1) atomicAdd(&A.ctr->knn_pairs, (unsigned long long)nq * (cnt - 1));
    }
  }
}

// The candidates of one leaf: super-chunk entries of its 27 ranges, the leaf's own
// cell first.
struct XSrc {
  const float4 *spts;
  const uint8_t *flag;
  BoxIndex box;
  const uint32_t (*rng)[2];  // in shared memory, in entry order
  const uint32_t *off;       // [28] first entry of each range
  __device__ __forceinline__ uint32_t entries() const { return off[27]; }
  __device__ __forceinline__ void entry(uint32_t e, uint32_t &s, uint32_t &a, uint32_t &b) const {
    uint32_t lo = 0, hi = 26;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (off[mid] <= e) lo = mid;
      else hi = mid - 1;
    }
    a = rng[lo][0];
    b = rng[lo][1];
    s = a / kBoxSuper + (e - off[lo]);
  }
  __device__ __forceinline__ float4 load(uint32_t p) const {
    float4 v = spts[p];
    if (!flag[p]) v.x = __int_as_float(0x7FFFFFFF);
    return v;
  }
};

struct XWarp {
  uint32_t rng[27][2];
  uint32_t off[28];
};

// a leaf's ranges into the warp's shared memory
__device__ __forceinline__ void x_load(XWarp &X, const XRanges *x, uint32_t lane) {
  __syncwarp();
  uint32_t cnt = 0;
  if (lane < 27) {
    const uint32_t r = lane == 0 ? 13u : (lane <= 13u ? lane - 1u : lane);  // own cell first
    const uint32_t a = x->rng[r][0], b = x->rng[r][1];
    X.rng[lane][0] = a;
    X.rng[lane][1] = b;
    if (a < b) cnt = (b - 1u) / kBoxSuper - a / kBoxSuper + 1u;
  }
  uint32_t inc = cnt;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= (uint32_t)o) inc += y;
  }
  if (lane < 28) X.off[lane] = inc - cnt;
  __syncwarp();
}

// one query's result: the sorted list (lane t: rank t) and r_K^2
template <bool kRec>
__device__ __forceinline__ void x_emit(const XleafArgs &A, uint32_t qp, uint32_t keff, unsigned long long key,
                                       uint32_t pos, float r2, uint32_t lane) {
  if (lane == 0) {
    A.xkeff[qp] = keff;
    if (keff) A.xr2[qp] = r2;
    // the point with log2 of its density beside it, for the score's neighbour reads
    const float4 p = A.spts[qp];
    A.xrho[qp] = make_float4(p.x, p.y, p.z, keff ? log2_density(keff, r2) : -INFINITY);
  }
  if (lane < keff) A.xnbr[(size_t)qp * A.k + lane] = pos;
  if (kRec && A.use_dbg) {
    const uint32_t g = __float_as_uint(A.spts[qp].w);
    if (g < A.n) {
      if (lane < A.k) {
        const bool v = lane < keff;
        if (A.dbg.nbr) A.dbg.nbr[(size_t)g * A.k + lane] = v ? (uint32_t)key : 0xFFFFFFFFu;
        if (A.dbg.nbr_d2) A.dbg.nbr_d2[(size_t)g * A.k + lane] = v ? __uint_as_float((uint32_t)(key >> 32)) : 0.f;
      }
      if (lane == 0 && A.dbg.r2 && keff) A.dbg.r2[g] = r2;
    } else if (lane == 0) {
      atomicOr(&A.ctr->status, kStInternal);
    }
  }
}

template <bool kRec>
__global__ void __launch_bounds__(32 * kBkWarps) k_xleaf_knn_box(const XleafArgs A) {
  __shared__ BkShared<32> s_w[kBkWarps];
  __shared__ XWarp s_x[kBkWarps];
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  BkShared<32> &S = s_w[threadIdx.x >> 5];
  XWarp &X = s_x[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31u, n_leaves = A.ctr->n_leaves, n_units = A.ctr->x_units;
  const BoxIndex bx = box_index(A.boxes, A.n);
  for (;;) {
    uint32_t u = 0;
    if (lane == 0) u = atomicAdd(&A.ctr->xleaf_work, 1u);
    u = __shfl_sync(0xFFFFFFFFu, u, 0);
    if (u >= n_units) break;
    uint32_t lo = 0, hi = n_leaves - 1;  // the leaf whose units hold u: the last start <= u
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (A.unit_start[mid] <= u) lo = mid;
      else hi = mid - 1;
    }
    const Leaf lf = A.leaves[lo];
    const uint32_t q0 = (u - A.unit_start[lo]) * kXWUnit;
    uint32_t q = lf.start + q0 + lane;
    bool act = q0 + lane < lf.count && A.xflag[q];
    const uint32_t any = __ballot_sync(0xFFFFFFFFu, act);
    if (!any) continue;
    const XRanges *const xr = x_ranges(A, lf);
    const uint32_t nc = xr->nc, keff = nc <= 1 ? 0u : (A.k < nc - 1 ? A.k : nc - 1);
    if (lane == 0 && nc > 1)
      atomicAdd(&A.ctr->knn_pairs, (unsigned long long)__popc(any) * (nc - 1));
    if (keff == 0) {
      for (uint32_t m = any; m; m &= m - 1u)
        x_emit<kRec>(A, lf.start + q0 + (uint32_t)__ffs(m) - 1u, 0u, 0ull, 0u, 0.f, lane);
      continue;
    }
    x_load(X, xr, lane);
    if (!act) q = lf.start + q0 + (uint32_t)__ffs(any) - 1u;  // shadows a query of the warp
    const float4 me = A.spts[q];
    const XSrc src{A.spts, A.xflag, bx, X.rng, X.off};
    const float delta = A.frames[lf.frame].delta, delta2 = __fmul_rn(delta, delta);
    float theta = INFINITY;
    uint32_t far = any;  // more candidates than the counters hold: a warp for every query
    if (nc < (1u << kBkPlanes) &&
        !bk_knn(src, S, act, q, me.x, me.y, me.z, keff, lf.start, lf.start + lf.count, bk_share(A.n), theta, far))
      atomicOr(&A.ctr->status, kStInternal);
    if (far) {
      uint32_t slot = 0;
      if (lane == 0) slot = atomicAdd(&A.ctr->far_count, (uint32_t)__popc(far));
      slot = __shfl_sync(0xFFFFFFFFu, slot, 0) + __popc(far & lanemask_lt());
      if ((far >> lane) & 1u) {
        A.far_queue[slot] = make_uint2(lo, q);
        A.xr2[q] = theta;  // its bound, for its own warp
      }
    }
    // rank order (d^2, input index): the order in which the score sums them
    for (uint32_t m = any & ~far; m; m &= m - 1u) {
      const uint32_t l = (uint32_t)__ffs(m) - 1u, qp = lf.start + q0 + l;
      const float qx = __shfl_sync(0xFFFFFFFFu, me.x, l), qy = __shfl_sync(0xFFFFFFFFu, me.y, l),
                  qz = __shfl_sync(0xFFFFFFFFu, me.z, l);
      unsigned long long key = ~0ull;
      uint32_t pos = 0;
      if (lane < keff) {
        pos = S.row[l][lane];
        const float4 p = A.spts[pos];
        key = ((unsigned long long)__float_as_uint(sqdist(qx, qy, qz, p.x, p.y, p.z)) << 32) | __float_as_uint(p.w);
      }
      bk_sort(key, pos, lane);
      const float th = __shfl_sync(0xFFFFFFFFu, theta, l);
      x_emit<kRec>(A, qp, keff, key, pos, th < delta2 ? delta2 : th, lane);
    }
    __syncwarp();
  }
}

// the queries that were left to a warp of their own
template <bool kRec>
__global__ void __launch_bounds__(128) k_xleaf_knn_far(const XleafArgs A) {
  __shared__ XWarp s_x[4];
  pdl_wait();
  if (A.ctr->status & kStFatal) return;
  XWarp &X = s_x[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31u, nf = A.ctr->far_count;
  const BoxIndex bx = box_index(A.boxes, A.n);
  for (uint32_t i = blockIdx.x * 4u + (threadIdx.x >> 5); i < nf; i += gridDim.x * 4u) {
    const uint2 e = A.far_queue[i];
    const Leaf lf = A.leaves[e.x];
    const XRanges *const xr = x_ranges(A, lf);
    const uint32_t nc = xr->nc, keff = nc <= 1 ? 0u : A.k < nc - 1 ? A.k : nc - 1;
    if (keff == 0) {  // alone in its block of cells
      x_emit<kRec>(A, e.y, 0u, 0ull, 0u, 0.f, lane);
      continue;
    }
    x_load(X, xr, lane);
    const float4 me = A.spts[e.y];
    const XSrc src{A.spts, A.xflag, bx, X.rng, X.off};
    BkList L;
    bk_knn_far(src, e.y, me.x, me.y, me.z, keff, A.xr2[e.y], L);
    const uint32_t kth = (uint32_t)(__shfl_sync(0xFFFFFFFFu, L.key, keff - 1) >> 32);
    if (kth > 0x7F800000u && lane == 0) atomicOr(&A.ctr->status, kStInternal);  // the list did not fill: cannot happen
    const float delta = A.frames[lf.frame].delta, delta2 = __fmul_rn(delta, delta), rk = __uint_as_float(kth);
    x_emit<kRec>(A, e.y, keff, L.key, L.pos, rk < delta2 ? delta2 : rk, lane);
  }
}

template <bool kRec>
int launch_x(const XleafArgs &a, int num_sms, cudaStream_t st, int *launches) {
  auto go = [&](auto kern) { return launch_pdl(kern, num_sms * 4, kXThreads, 0, st, a); };
  cudaError_t e;
  if (a.k <= 32) {
    e = launch_pdl(k_xleaf_boxes, box_supers(a.n), kBoxSuper, 0, st, a);
    const bool small = a.n <= kXSmall;
    if (e == cudaSuccess && !small) e = launch_pdl(k_xleaf_units, 1, 1024, 0, st, a.leaves, a.ctr, a.unit_start);
    if (e == cudaSuccess) e = launch_pdl(k_xleaf_ranges, num_sms * 8, 128, 0, st, a, small);
    if (e == cudaSuccess && !small) e = launch_pdl(k_xleaf_knn_box<kRec>, num_sms * 6, 32 * kBkWarps, 0, st, a);
    if (e == cudaSuccess) e = launch_pdl(k_xleaf_knn_far<kRec>, num_sms * 8, 128, 0, st, a);
    if (launches) *launches += small ? 3 : 5;
  } else {
    e = go(k_xleaf_knn<64, kRec>);
    if (launches) *launches += 1;
  }
  return e == cudaSuccess ? 0 : -1;
}

int launch_xleaf_knn(const XleafArgs &a, int num_sms, cudaStream_t st, int *launches) {
  return a.use_dbg ? launch_x<true>(a, num_sms, st, launches) : launch_x<false>(a, num_sms, st, launches);
}

}  // namespace gd
