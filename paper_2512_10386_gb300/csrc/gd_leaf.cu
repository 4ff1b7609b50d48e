// gd_leaf.cu -- the per-leaf part of the method, fused into one persistent kernel
// (device code in gd_leaf_kernel.cuh), its prep kernels and host launchers.
//
// Each CTA pulls octree leaves from a device work counter and runs, for one
// leaf at a time, every per-leaf step of Sec. 3 in shared memory:
//   (extents and adaptive voxel size h, Eq. 10-11, come from the prep kernel) ->
//   voxel occupancy in counters addressed by the grid cell, or a hash table where
//   the grid is large, with warp-aggregated atomics; voxel gate (Eq. 12) and
//   compaction of P_1 -> kNN of every P_1 point against the leaf's P_1 (counting
//   selection, gd_knn_select.cuh; candidates broadcast from shared memory, ties
//   broken by input index), r_K (Eq. 13) -> exact percentile gate
//   (Eq. 14) as a rank cut on r_K^2 -> median density (Eq. 16) -> dual-weight
//   gravitational score (Eq. 15-21) -> Top-lambda or log-threshold selection,
//   scattered to input order (Eq. 22).
// The leaf's points arrive in shared memory by one TMA bulk copy
// (cp.async.bulk + mbarrier).  Leaves larger than the shared-memory layout (leaf
// capacities above 2,048 points, nodes at the maximum depth) run the same code
// on a per-point spill area in global memory, or, where the call allows it, in
// kernels over the whole GPU (gd_big.cu).
//
// FP32 steps that decide integers (voxel indices, neighbour order, the density
// rank cut) use explicitly rounded intrinsics so no FMA contraction can change
// them; FP64 per-leaf scalars (V_t, h, rho_med) use explicitly rounded FP64.
#include "gd_leaf_kernel.cuh"

namespace gd {

// ---------------------------------------------------------------------------
// leaf prep: Eq. 10-11 for every leaf (all leaves in parallel)
// ---------------------------------------------------------------------------
// A warp takes 8 leaves at a time: the FP32 bounding boxes (exact min/max) one after
// the other, their descriptors and first points loaded ahead, then lane l evaluates
// leaf l's voxel size and scatters the leaf's index into the largest-first order: the
// leaf finder has counted the size classes and left each leaf its place in its class.
// With few leaves a warp takes one.  (32 leaves a block, the FP64 cube root's ten
// steps and a kernel of its own for the order took 15.4 + 3.0 us for 8 leaves and 18.2
// + 3.8 us for 5,700; this one 5.2 and 12.1 us,
// and for 93,566 leaves 74.1 + 7.9 -> 47.9 us.)
constexpr int kPrepThreads = 128;
constexpr uint32_t kPrepLeaves = 8;  // per warp

__global__ void __launch_bounds__(kPrepThreads) k_leaf_prep(const float4 *__restrict__ spts, Leaf *leaves,
                                                            const FrameInfo *__restrict__ frames, Counters *ctr,
                                                            uint32_t *__restrict__ order, float beta, uint32_t lmax,
                                                            bool skip_big) {
  pdl_wait();
  if (ctr->status & kStFatal) return;
  const uint32_t nl = ctr->n_leaves;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // first place of each size class (lane c: class c)
  const uint32_t cc = lane < kLeafClasses ? ctr->cls_count[lane] : 0u;
  uint32_t first = cc;
  for (int o = 1; o < 16; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, first, o);
    if (lane >= (uint32_t)o) first += y;
  }
  first -= cc;
  // the smallest classes (64 points each, up to kSmallLeaf points) come last
  if (blockIdx.x == 0 && threadIdx.x == kLeafClasses - kSmallLeaf / 64) ctr->split_leaf = first;
  if (blockIdx.x == 0 && threadIdx.x == 0 && skip_big) ctr->leaf_work = cc;  // the fused kernel starts behind class 0
  const uint32_t warps = gridDim.x * (kPrepThreads / 32), wi = blockIdx.x * (kPrepThreads / 32) + w;
  uint32_t per = (nl + warps - 1) / warps;
  per = per < kPrepLeaves ? per : kPrepLeaves;
  if (per == 0) return;
  for (uint32_t g = wi * per; g < nl; g += warps * per) {
    const uint32_t lj = g + lane;
    const bool on = lane < per && lj < nl;
    Leaf lf{};
    if (on) lf = leaves[lj];
    const bool box = on && !(skip_big && lf.count > lmax);  // (a big leaf's own kernels take its box, gd_big.cu)
    float lo[3] = {0.0f, 0.0f, 0.0f}, ext[3] = {0.0f, 0.0f, 0.0f};
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, box); todo; todo &= todo - 1u) {
      const int t = __ffs(todo) - 1;
      const uint32_t start = __shfl_sync(0xFFFFFFFFu, lf.start, t), cnt = __shfl_sync(0xFFFFFFFFu, lf.count, t);
      float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
      for (uint32_t i0 = lane; i0 < cnt; i0 += 256) {  // eight loads in flight per lane
        float4 p[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t i = i0 + 32u * u;
          if (i < cnt) p[u] = spts[start + i];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (i0 + 32u * u < cnt) {
            mn[0] = fminf(mn[0], p[u].x); mn[1] = fminf(mn[1], p[u].y); mn[2] = fminf(mn[2], p[u].z);
            mx[0] = fmaxf(mx[0], p[u].x); mx[1] = fmaxf(mx[1], p[u].y); mx[2] = fmaxf(mx[2], p[u].z);
          }
        }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float l = ord2f(__reduce_min_sync(0xFFFFFFFFu, f2ord(mn[a])));
        const float h = ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(mx[a])));
        if (lane == (uint32_t)t) {
          lo[a] = l;
          ext[a] = __fsub_rn(h, l);
        }
      }
    }
    const uint32_t cls = on ? leaf_class(lf.count, lmax) : 0u;
    const uint32_t base = __shfl_sync(0xFFFFFFFFu, first, cls);
    if (on) {
      const uint32_t slot = base + __float_as_uint(lf.h);  // its place in its class, from the leaf finder
      if (slot < nl) order[slot] = lj;
      else atomicOr(&ctr->status, kStInternal);
    }
    if (box) {
#pragma unroll
      for (int a = 0; a < 3; ++a) leaves[lj].lo[a] = lo[a];
      const float h = leaf_voxel_size(ext, frames[lf.frame].delta, lf.count, beta);
      leaves[lj].h = h;
      // cells a side: the index of the farthest point (vox_index is monotonic), plus one
      uint32_t g[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) g[a] = vox_index(ext[a], 0.0f, h) + 1u;
      if (g[0] < 1024u && g[1] < 1024u && g[2] < 1024u && g[0] * g[1] * g[2] <= 2u * lf.count)
        leaves[lj].level = (lf.level & 31u) | (g[1] << 5) | (g[2] << 15) | kLeafGrid;
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int leaf_kmax(uint32_t k) { return k <= 8 ? 8 : k <= 16 ? 16 : k <= 32 ? 32 : 64; }

size_t leaf_smem_bytes(uint32_t lmax, int kmax, int threads) {
  return carve<uint16_t>(nullptr, lmax, kmax, threads, nullptr);
}

namespace {
// max over spill-path leaf sizes (cap > 64) of carve<uint32_t>(cap)/cap, rounded
// up to a multiple of 16 so that every leaf's area starts 16-byte aligned.  The
// ratio is largest for small caps (fixed-size parts); beyond 2^16 points it only
// falls, so scanning 65..65536 bounds every size.
uint32_t big_bpp_scan(int kmax) {
  size_t worst = 4u * ((kLeafSmemMax + 31u) / 32u);
  for (uint32_t cap = 65; cap <= 65536; ++cap) {
    const size_t b = carve<uint32_t>(nullptr, cap, kmax, 128, nullptr);
    const size_t per = (b + cap - 1) / cap;
    if (per > worst) worst = per;
  }
  return (uint32_t)((worst + 15) & ~size_t(15));
}
}  // namespace

uint32_t leaf_big_bpp(int kmax) {
  // computed once, on first use, for the four list sizes (thread-safe static init);
  // at least the neighbour bitmap of a shared-memory leaf (one word a point per
  // 32 points of the leaf), which may be kept in the spill area
  static const uint32_t table[4] = {big_bpp_scan(8), big_bpp_scan(16), big_bpp_scan(32), big_bpp_scan(64)};
  return table[kmax <= 8 ? 0 : kmax <= 16 ? 1 : kmax <= 32 ? 2 : 3];
}

uint32_t leaf_pick_lmax(uint32_t leaf_capacity, int kmax, size_t smem_limit) {
  const uint32_t cap = leaf_capacity < 64 ? 64 : (leaf_capacity > kLeafSmemMax ? kLeafSmemMax : leaf_capacity);
  uint32_t l = pow2ceil(cap);
  while (l > 64 && leaf_smem_bytes(l, kmax, 512) > smem_limit) l >>= 1;
  return l;
}

int launch_leaf_prep(const LeafArgs &a, int num_sms, cudaStream_t st, int *launches) {
  launch_pdl(k_leaf_prep, num_sms * 8, kPrepThreads, 0, st, a.spts, const_cast<Leaf *>(a.leaves), a.frames, a.ctr, a.order,
             a.p.beta, a.lmax, a.skip_big != 0);
  if (launches) *launches += 1;
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Threads of a leaf CTA where the caller leaves the choice open.  A leaf is one
// CTA's work, so a call takes at least the time of its largest leaf; a wider CTA
// shortens that (32 queries a warp) but waits longer at the leaf's barriers and
// leaves fewer CTAs per SM to fill the waits.  Wide CTAs therefore pay while the
// points are too few to keep every SM busy, or where one leaf's shared memory
// leaves room for one to three CTAs per SM anyway.  Measured, us a call (K = 24,
// dense scans unless noted; leaf CTAs of 128 / 256 / 512 threads):
//   up to 64-point leaves: 64 threads, 300k points 376 -> 289
//   256-point leaves:  40k 148 / 136 / 165, 70k (LiDAR) 159 / 155 / 223, 100k 158 / 177 / 289
//   512-point leaves:  40k 229 / 185 / 162, 100k 270 / 232 / 228, 130k (LiDAR) 299 / 242 / 272,
//                      200k 291 / 231 / 368, 300k 294 / 292 / 463, 560k 402 / 484 / 886
//   1,024-point leaves: 200k 672 / 527 / 377, 300k 671 / 508 / 457, 560k 753 / 589 / 747
//   2,048-point leaves: 10k 1184 / 838 / 661, 560k 2362 / 1612 / 1299
// A batch of many frames a little above the capacity has leaves of an eighth of a frame
// (one octree level): where they are two or more an SM, the width is chosen for a sixth
// of the largest frame.  us a call, by the capacity's size / so (capacity 512, 64 frames):
// 600 points 175 / 128, 800 186 / 148, 1,300 207 / 168; 200 frames of 600 216 / 191.
static uint32_t leaf_auto_threads(const LeafArgs &a, int num_sms) {
  const uint32_t n = a.n;
  uint32_t lmax = a.lmax;
  if (lmax <= 512 && a.frame > a.p.leaf_capacity && 8ull * n >= 2ull * (uint32_t)num_sms * a.frame) {
    const uint32_t size = pow2ceil(a.frame / 6u);
    if (size < lmax) lmax = size;
  }
  if (lmax <= 64) return 64;
  if (lmax <= 128) return 128;
  if (lmax <= 256) return n <= (64u << 10) ? 256 : 128;
  if (lmax <= 512) return n <= (96u << 10) ? 512 : n <= (280u << 10) ? 256 : 128;
  if (lmax <= 1024) return n <= (384u << 10) ? 512 : 256;
  return 512;
}

// Whether leaves of at most kSmallLeaf points get a warp each (gd_leaf_tiny.cu).  That
// kernel needs a fifth of the instructions of the fused one for such a leaf, but its
// long straight code makes the first leaf of a warp slow (50 us: instruction
// fetches), and its warps take registers from the CTAs of the larger leaves: it pays
// where small leaves are many.  us a call, fused / tiny: leaf capacity 64, 40k points 113
// / 128, 100k 162 / 140, 560k 555 / 322; capacity 128, 100k 134 / 151, 200k 191 / 189, 560k
// 371 / 345; capacity 256, 300k 226 / 230, 560k 347 / 346, 720k (8 LiDAR frames) 463 / 453,
// 6.1M (64 frames) 3445 / 3221; capacity 512, 560k 400 / 403, 1.1M 837 / 841.
static bool leaf_tiny_pays(uint32_t n, uint32_t lmax) {
  return lmax <= 64 ? n >= 80000u : lmax <= 128 ? n >= 250000u : lmax <= 256 && n >= 600000u;
}

int launch_leaf(const LeafArgs &args, int num_sms, cudaStream_t st, int *launches, cudaStream_t side, cudaEvent_t fork,
                cudaEvent_t join) {
  LeafArgs a = args;
  if (a.skip_big) {
    // the big leaves' kernels on `st`; the other leaves, which need nothing of
    // theirs, beside them on the side stream where there is one
    const bool beside = side && fork && join;
    if (a.threads == 0 && a.ctas_per_sm == 0) a.threads = leaf_auto_threads(a, num_sms);
    if (launches) ++*launches;
    if (beside && (cudaEventRecord(fork, st) != cudaSuccess || cudaStreamWaitEvent(side, fork, 0) != cudaSuccess))
      return -1;
    if (launch_big(a, num_sms, st, launches) || launch_threads<false, false>(a, num_sms, beside ? side : st)) return -1;
    if (beside && (cudaEventRecord(join, side) != cudaSuccess || cudaStreamWaitEvent(st, join, 0) != cudaSuccess))
      return -1;
    return 0;
  }
  const bool chosen = a.threads == 0 && a.ctas_per_sm == 0;  // the caller leaves the choice open
  if (chosen) a.threads = leaf_auto_threads(a, num_sms);
  if (a.xphase != 0) {  // the cross-leaf phases: their own instantiation
    if (launches) ++*launches;
    return launch_leaf_xl(a, num_sms, st);
  }
  auto go = [&](const LeafArgs &x, cudaStream_t s) {
    return (x.use_dbg || x.use_train) ? launch_leaf_rec(x, num_sms, s) : launch_threads<false, false>(x, num_sms, s);
  };
  // Leaves of at most kSmallLeaf points beside the others, one warp each
  // (gd_leaf_tiny.cu), or, where the recording or a structural variant needs the fused
  // kernel, on 64-thread CTAs of a 64-point shared-memory layout; the others keep their
  // CTAs, and the order of the leaves and every result are the same as with one launch.
  const bool tiny = chosen && leaf_tiny_pays(a.n, a.lmax) && !a.use_dbg && !a.use_train && !a.p.stage_off && !a.p.rescore_p2;
  const bool split = side && fork && join && a.ctas_per_sm == 0 &&
                     (a.lmax > kSmallLeaf ? a.threads == 0 || a.threads == 128 : tiny);
  if (!split) {
    if (launches) ++*launches;
    return go(a, st);
  }
  LeafArgs big = a, small = a;
  big.part = 1;
  small.part = 2;
  small.threads = 64;
  small.lmax = kSmallLeaf;
  if (launches) *launches += 2;
  if (cudaEventRecord(fork, st) != cudaSuccess || cudaStreamWaitEvent(side, fork, 0) != cudaSuccess) return -1;
  if (go(big, st) || (tiny ? launch_leaf_tiny(small, num_sms, side) : go(small, side))) return -1;
  if (cudaEventRecord(join, side) != cudaSuccess || cudaStreamWaitEvent(st, join, 0) != cudaSuccess) return -1;
  return 0;
}

}  // namespace gd
