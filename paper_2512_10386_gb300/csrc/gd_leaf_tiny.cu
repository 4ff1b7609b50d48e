// gd_leaf_tiny.cu -- the per-leaf steps of Sec. 3 for leaves of at most kSmallLeaf (64)
// points, one warp a leaf and without a block barrier: a lane owns the points at
// positions lane and 32 + lane, order statistics are warp sorts, counts are ballots.
//
// The fused kernel (gd_leaf_kernel.cuh) spends a small leaf on per-leaf fixed costs:
// some twenty barriers, a bulk copy, a hash table and sorts that keep few lanes busy,
// 7,700 warp instructions a leaf.  Here the neighbours are found by a register sort of
// the leaf's squared distances (none where k_eff takes every other point), and a leaf
// takes 2,000 to 4,000 instructions.  Every value that decides something and the order
// in which a score sums its terms are the fused kernel's: results are identical bit
// for bit.  64 LiDAR frames (K = 24): 597 -> 370 us for these leaves in the launch
// list (capacity 256); bound by instruction fetch (64 frames at capacity 128: the top stall, 7.0
// warps an issued instruction, issue in 31 % of the cycles).
#include "gd_leaf_kernel.cuh"

namespace gd {

namespace {
constexpr int kTinyThreads = 128;
constexpr int kTinyWarps = kTinyThreads / 32;
constexpr uint32_t kFull = 0xFFFFFFFFu;

struct TinyShared {
  float x[64], y[64], z[64];  // P_1, then NaN
  float4 p[64];               // P_1 (x, y, z, score weight)
  uint32_t w[64];             // input index
  uint32_t key[64];           // selection keys (ties only)
};

// ascending sort of 64 keys, element e at slot e / 32 of lane e % 32
__device__ __forceinline__ void warp_sort64(uint32_t (&v)[2], uint32_t lane) {
#pragma unroll 1
  for (uint32_t size = 2; size <= 64; size <<= 1) {
#pragma unroll 1
    for (uint32_t j = size >> 1; j > 0; j >>= 1) {
      if (j == 32) {  // partners in the lane (size 64: ascending)
        const uint32_t a = min(v[0], v[1]), b = max(v[0], v[1]);
        v[0] = a;
        v[1] = b;
      } else {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const uint32_t e = 32u * s + lane, o = __shfl_xor_sync(kFull, v[s], j);
          v[s] = (((e & j) == 0) == ((e & size) == 0)) ? min(v[s], o) : max(v[s], o);
        }
      }
    }
  }
}
__device__ __forceinline__ void warp_sort32(uint32_t &v, uint32_t lane) {
#pragma unroll 1
  for (uint32_t size = 2; size <= 32; size <<= 1) {
#pragma unroll 1
    for (uint32_t j = size >> 1; j > 0; j >>= 1) {
      const uint32_t o = __shfl_xor_sync(kFull, v, j);
      v = (((lane & j) == 0) == ((lane & size) == 0)) ? min(v, o) : max(v, o);
    }
  }
}
__device__ __forceinline__ uint32_t pick(const uint32_t (&v)[2], uint32_t e) {  // element e of a sorted pair of slots
  const uint32_t a = __shfl_sync(kFull, v[0], e & 31u), b = __shfl_sync(kFull, v[1], e & 31u);
  return e < 32u ? a : b;
}

// Neighbour mask of the query at position q (coordinates x, y, z) among the n1 points,
// and its k_eff-th squared distance.  N = 32 or 64 candidates (NaN past n1).
// Out of line, one copy for both of a lane's queries: the kernel runs straight
// through its code once a leaf, so its size is instruction fetches.
template <int N>
__device__ __noinline__ unsigned long long tiny_knn(const TinyShared &S, uint32_t q, float x, float y, float z,
                                                       uint32_t n1, uint32_t keff, float &theta) {
  const f32x2 QX = pk2(x, x), QY = pk2(y, y), QZ = pk2(z, z);
  const unsigned long long all = n1 >= 64u ? ~0ull : (1ull << n1) - 1ull, self = 1ull << (q & 63u);
  if (keff + 1u == n1) {  // every other point
    float t = 0.0f;
#pragma unroll
    for (int j = 0; j < N; j += 4) {
      float d[4];
      sqdist4(S.x, S.y, S.z, j, QX, QY, QZ, d);
      t = fmaxf(fmaxf(t, d[0]), fmaxf(fmaxf(d[1], d[2]), d[3]));
    }
    theta = t;
    return all & ~self;
  }
  {
    // the query's own d^2 = 0 is the smallest (or ties with it): its k_eff-th neighbour
    // is at rank k_eff; NaN bits sort behind every number's
    uint32_t L[N];
#pragma unroll
    for (int j = 0; j < N; j += 4) {
      float d[4];
      sqdist4(S.x, S.y, S.z, j, QX, QY, QZ, d);
#pragma unroll
      for (int u = 0; u < 4; ++u) L[j + u] = __float_as_uint(d[u]) & 0x7FFFFFFFu;
    }
    regsort_u<N>(L);
    uint32_t th = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) th = (uint32_t)j == keff ? L[j] : th;
    theta = __uint_as_float(th);
  }
  const f32x2 T2 = pk2(theta, theta);
  uint32_t gt[2] = {0u, 0u};
#pragma unroll
  for (int j = 0; j < N; j += 4) {
    float d[4], e[4];
    sqdist4(S.x, S.y, S.z, j, QX, QY, QZ, d);
    // the sign of theta - d^2 is set exactly when d^2 > theta
    upk2(sub2(T2, pk2(d[0], d[1])), e[0], e[1]);
    upk2(sub2(T2, pk2(d[2], d[3])), e[2], e[3]);
#pragma unroll
    for (int u = 0; u < 4; ++u) gt[j / 32] = __funnelshift_l(__float_as_uint(e[u]), gt[j / 32], 1);
  }
  unsigned long long le = ~(unsigned long long)__brev(gt[0]);
  if (N == 64) le = (le & 0xFFFFFFFFull) | ((unsigned long long)~__brev(gt[1]) << 32);
  le &= all & ~self;
  if ((uint32_t)__popcll(le) > keff) {  // ties at the k_eff-th distance: by input index
    unsigned long long eq = 0;
    for (uint32_t j = 0; j < n1; ++j)
      if (((le >> j) & 1ull) && sqdist(x, y, z, S.x[j], S.y[j], S.z[j]) == theta) eq |= 1ull << j;
    le &= ~eq;
    const uint32_t need = keff - (uint32_t)__popcll(le);
    for (unsigned long long a = eq; a; a &= a - 1ull) {
      const uint32_t i = (uint32_t)__ffsll((long long)a) - 1u;
      uint32_t before = 0;
      for (unsigned long long b = eq; b; b &= b - 1ull) before += S.w[__ffsll((long long)b) - 1] < S.w[i];
      if (before < need) le |= 1ull << i;
    }
  }
  return le;
}

}  // namespace

__global__ void __launch_bounds__(kTinyThreads, 4) k_leaf_tiny(const LeafArgs A) {
  __shared__ TinyShared s_w[kTinyWarps];
  pdl_wait();
  if (ld_volatile(&A.ctr->status) & kStFatal) return;
  TinyShared &S = s_w[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31u, lt = lanemask_lt();
  const denoise_params &P = A.p;
  const uint32_t n_all = A.ctr->n_leaves, split = A.ctr->split_leaf;
  const bool g2 = (P.gamma == 2.0f);
  const float hg = 0.5f * P.gamma, ek = P.eps_k, half_alpha = __fmul_rn(0.5f, P.alpha);
  const float c2 = __fdiv_rn(1.4426950408889634f, __fmul_rn(__fmul_rn(2.0f, P.sigma), P.sigma));
  unsigned long long st_pairs = 0, st_n1 = 0, st_n2 = 0, st_terms = 0;  // lane 0's
  uint32_t next = 0;
  if (lane == 0) next = atomicAdd(&A.ctr->leaf_work3, 1u);
  for (;;) {
    const uint32_t wi = split + __shfl_sync(kFull, next, 0);
    if (wi >= n_all) break;
    if (lane == 0) next = atomicAdd(&A.ctr->leaf_work3, 1u);  // the next leaf's number is on its way
    const Leaf lf = A.leaves[A.order[wi]];
    const uint32_t nt = lf.count;
    if (nt > kSmallLeaf) {  // cannot happen: the class holds at most kSmallLeaf points
      if (lane == 0) atomicOr(&A.ctr->status, kStInternal);
      break;
    }
    const float delta = A.frames[lf.frame].delta;
    // ---- Eq. 12: voxel occupancy, one round per occupied voxel
    float4 p[2];
    unsigned long long vk[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint32_t i = 32u * s + lane;
      p[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      vk[s] = kInvalid;
      if (i < nt) {
        p[s] = A.spts[lf.start + i];
        vk[s] = voxel_key(p[s], lf.lo, lf.h);
      }
    }
    bool in1[2] = {false, false};
    uint32_t left0 = __ballot_sync(kFull, lane < nt), left1 = __ballot_sync(kFull, 32u + lane < nt);
    while (left0 | left1) {
      const bool first = left0 != 0;
      const unsigned long long k = __shfl_sync(kFull, first ? vk[0] : vk[1], __ffs(first ? left0 : left1) - 1);
      const uint32_t b0 = __ballot_sync(kFull, vk[0] == k), b1 = __ballot_sync(kFull, vk[1] == k);
      const bool keep = (uint32_t)(__popc(b0) + __popc(b1)) >= P.min_vox_count;
      if (vk[0] == k) in1[0] = keep;
      if (vk[1] == k) in1[1] = keep;
      left0 &= ~b0;
      left1 &= ~b1;
    }
    // ---- P_1, order kept
    const uint32_t m0 = __ballot_sync(kFull, in1[0]), m1 = __ballot_sync(kFull, in1[1]);
    const uint32_t n1 = __popc(m0) + __popc(m1);
    __syncwarp();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (32u * s + lane < nt && !in1[s]) write_point<false>(A, __float_as_uint(p[s].w), 0, 0.0f, 1);
      if (in1[s]) {
        const uint32_t pos = s ? __popc(m0) + __popc(m1 & lt) : __popc(m0 & lt);
        S.x[pos] = p[s].x;
        S.y[pos] = p[s].y;
        S.z[pos] = p[s].z;
        S.w[pos] = __float_as_uint(p[s].w);
      }
      const uint32_t i = 32u * s + lane;
      if (i >= n1) {
        S.x[i] = S.y[i] = S.z[i] = __int_as_float(0x7FFFFFFF);
        S.w[i] = 0u;
      }
    }
    __syncwarp();
    if (n1 <= 1) {  // no neighbour exists: the density gate cannot keep it
      if (lane < n1) write_point<false>(A, S.w[lane], 0, 0.0f, 2);
      continue;
    }
    const uint32_t keff = P.k < n1 - 1 ? P.k : n1 - 1;
    const bool wide = n1 > 32u;  // warp-uniform
    // ---- kNN
    bool act[2];
    float qx[2], qy[2], qz[2], r2[2];
    unsigned long long nb[2] = {0, 0};
    const float delta2 = __fmul_rn(delta, delta);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint32_t q = 32u * s + lane;
      act[s] = q < n1;
      const uint32_t qq = act[s] ? q : n1 - 1;
      qx[s] = S.x[qq];
      qy[s] = S.y[qq];
      qz[s] = S.z[qq];
      r2[s] = __uint_as_float(0xFFFFFFFFu);
    }
#pragma unroll 1
    for (uint32_t s = 0; s < (wide ? 2u : 1u); ++s) {
      const uint32_t q = 32u * s + lane, qq = q < n1 ? q : n1 - 1;
      const float x = s ? qx[1] : qx[0], y = s ? qy[1] : qy[0], z = s ? qz[1] : qz[0];
      float th;
      const unsigned long long b = wide ? tiny_knn<64>(S, qq, x, y, z, n1, keff, th)
                                        : tiny_knn<32>(S, qq, x, y, z, n1, keff, th);
      const float r = th < delta2 ? delta2 : th;
      if (s) {
        nb[1] = b;
        if (act[1]) r2[1] = r;
      } else {
        nb[0] = b;
        if (act[0]) r2[0] = r;
      }
    }
    // ---- Eq. 14 cut and Eq. 16 median, from the sorted r_K^2 (lanes without a point sort last)
    uint32_t v[2] = {__float_as_uint(r2[0]), __float_as_uint(r2[1])};
    if (wide) warp_sort64(v, lane);
    else warp_sort32(v[0], lane);
    const double pos = __dadd_rn(__ddiv_rn(__dmul_rn((double)n1, (double)P.rho_percentile), 100.0), 0.5);
    const double cc = ceil(pos);
    const uint32_t crank = (cc < 1.0) ? 1u : (cc > (double)n1) ? n1 : (uint32_t)cc;
    const uint32_t Rb = pick(v, n1 - crank);
    bool in2[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) in2[s] = act[s] && __float_as_uint(r2[s]) <= Rb;
    const uint32_t m = __popc(__ballot_sync(kFull, in2[0])) + __popc(__ballot_sync(kFull, in2[1]));
    const float ra = __uint_as_float(pick(v, (m - 1) / 2)), rb = (m & 1u) ? ra : __uint_as_float(pick(v, m / 2));
    const float Lref = leaf_lref(ra, rb, m, keff, P.eps_rho);
    float wa[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      wa[s] = 0.0f;
      if (act[s]) {
        wa[s] = __fmul_rn(half_alpha, score_ell(r2[s], ra, Lref));
        S.p[32 * s + lane] = make_float4(qx[s], qy[s], qz[s], wa[s]);
      }
    }
    __syncwarp();
    // ---- Eq. 15-21: the score (even and odd ranks in the lanes of packed FP32, positions ascending)
    float F[2] = {0.0f, 0.0f};
#pragma unroll 1
    for (uint32_t s = 0; s < (wide ? 2u : 1u); ++s) {
      if (!(s ? in2[1] : in2[0])) continue;
      const float ci = __fdiv_rn(c2, s ? r2[1] : r2[0]);
      const float4 me = S.p[32u * s + lane];
      const f32x2 XI = pk2(me.x, me.x), YI = pk2(me.y, me.y), ZI = pk2(me.z, me.z), AI = pk2(me.w, me.w);
      const f32x2 NCI = pk2(-ci, -ci), EK = pk2(ek, ek);
      f32x2 FF = pk2(0.0f, 0.0f);
      unsigned long long b = s ? nb[1] : nb[0];
#pragma unroll 1
      for (uint32_t t = 0; t < keff; t += 2) {
        const bool two = t + 1 < keff;
        const uint32_t ja = b ? (uint32_t)__ffsll((long long)b) - 1u : 0u;
        b &= b - 1ull;
        uint32_t jb = ja;
        if (two) {
          jb = b ? (uint32_t)__ffsll((long long)b) - 1u : 0u;
          b &= b - 1ull;
        }
        const float4 pa = S.p[ja], pb = S.p[jb];
        const f32x2 DX = sub2(pk2(pa.x, pb.x), XI), DY = sub2(pk2(pa.y, pb.y), YI), DZ = sub2(pk2(pa.z, pb.z), ZI);
        const f32x2 D2 = fma2(DZ, DZ, fma2(DY, DY, mul2(DX, DX)));
        float ea, eb, da, db;
        upk2(fma2(D2, NCI, add2(AI, pk2(pa.w, pb.w))), ea, eb);
        upk2(D2, da, db);
        const f32x2 DG = g2 ? D2 : pk2(pow_half_gamma(da, hg), pow_half_gamma(db, hg));
        float qa, qb;
        upk2(add2(DG, EK), qa, qb);
        float ta, tb;
        upk2(mul2(pk2(ex2_hw(ea), ex2_hw(eb)), pk2(rcp_hw(qa), rcp_hw(qb))), ta, tb);
        FF = add2(FF, pk2(ta, two ? tb : 0.0f));
      }
      float f0, f1;
      upk2(FF, f0, f1);
      if (s) F[1] = __fadd_rn(f0, f1);
      else F[0] = __fadd_rn(f0, f1);
    }
    // ---- selection
    bool keep[2] = {false, false};
    if (P.select_mode == DENOISE_SELECT_TOPRATIO) {
      uint32_t keep_n = (uint32_t)ceil((double)P.lambda * (double)m);
      if (keep_n > m) keep_n = m;
      uint32_t key[2], kv[2];
#pragma unroll
      for (int s = 0; s < 2; ++s) kv[s] = key[s] = in2[s] ? 0xFFFFFFFFu - __float_as_uint(F[s]) : 0xFFFFFFFFu;
      if (wide) warp_sort64(kv, lane);
      else warp_sort32(kv[0], lane);
      const uint32_t cut = pick(kv, keep_n - 1);
      uint32_t less = 0, tied = 0;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        less += __popc(__ballot_sync(kFull, in2[s] && key[s] < cut));
        tied += __popc(__ballot_sync(kFull, in2[s] && key[s] == cut));
      }
      const uint32_t needed = keep_n - less;  // 1 <= needed <= tied
      const bool rank = needed < tied;        // exact score ties at the cut: by input index
      if (rank) {
#pragma unroll
        for (int s = 0; s < 2; ++s)
          if (32u * s + lane < 64u) S.key[32 * s + lane] = (in2[s] && key[s] == cut) ? 1u : 0u;
        __syncwarp();
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        keep[s] = in2[s] && key[s] <= cut;
        if (rank && in2[s] && key[s] == cut) {
          const uint32_t g = S.w[32 * s + lane];
          uint32_t before = 0;
          for (uint32_t j = 0; j < n1; ++j) before += S.key[j] && S.w[j] < g;
          keep[s] = before < needed;
        }
      }
    } else {
#pragma unroll
      for (int s = 0; s < 2; ++s) keep[s] = in2[s] && logf(F[s]) >= P.tau;
    }
    // ---- Eq. 22: results in input order
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!act[s]) continue;
      const uint32_t g = S.w[32 * s + lane];
      if (!in2[s]) write_point<false>(A, g, 0, 0.0f, 2);
      else write_point<false>(A, g, keep[s] ? 1 : 0, F[s], keep[s] ? 0 : 3);
    }
    st_pairs += (unsigned long long)n1 * (n1 - 1u);
    st_n1 += n1;
    st_n2 += m;
    st_terms += (unsigned long long)m * keff;
  }
  if (lane == 0 && st_n1) {
    atomicAdd(&A.ctr->knn_pairs, st_pairs);
    atomicAdd(&A.ctr->n_p1, st_n1);
    atomicAdd(&A.ctr->n_p2, st_n2);
    atomicAdd(&A.ctr->score_terms, st_terms);
  }
}

int launch_leaf_tiny(const LeafArgs &a, int num_sms, cudaStream_t st) {
  return launch_pdl(k_leaf_tiny, num_sms * 4, kTinyThreads, 0, st, a) == cudaSuccess ? 0 : -1;
}

}  // namespace gd
