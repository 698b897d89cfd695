// GPU index build: Insert (Algorithm 3) and JointRobustPrune (Algorithm 4)
// over a deterministic batch schedule.
//
// Schedule (the paper inserts points one at a time; batch insertion with a
// frozen graph per batch is how parallel builders run Insert):
//   entry vertex s = the point nearest (fp64) to the fp64 centroid, lowest id
//   on a tie; insertion order s, then the other points by increasing id;
//   after s, each batch takes the next min(#inserted, max(1, n/50)) points.
//   Within a batch: (1) every point p runs GreedySearch with D_A(t) for each
//   of its thresholds t on the graph as it stood when the batch began and
//   keeps the expanded set V_t; (2) p's out-list = JointRobustPrune over the
//   union of its V_t; (3) back-edges v -> p are grouped by target v: v's list
//   gets the new sources in increasing id order, and a list that would
//   exceed R is pruned once over the old list plus the new sources.
// Thresholds: per point p, S = min(sample, n-1) points drawn uniformly (with
// replacement) from the others by SplitMix64 on counter (p << 20) | i; the
// threshold for percentile q is the sorted sample's element floor(q(S-1)/100)
// of dist_A(a_p, .) (implementation-details appendix).
// Pruning: for each threshold t in order, candidates ranked by
// (capped dist_A, distance, id); v joins the bucket if it was chosen for an
// earlier threshold, else if alpha^2 d(u,v) > d(p,v) (fp32 product) for every
// member u so far; a bucket stops at 0.9 R / |T| members; the out-list is the
// union of the buckets in the order first chosen.
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <vector>

#include "launch.h"
#include "launch_util.cuh"
#include "search_core.cuh"

namespace jag {

constexpr int kPruneWarps = 2;

__device__ __forceinline__ uint64_t sm64(uint64_t seed, uint64_t ctr) {
  uint64_t z = seed + (ctr + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ int64_t order_id(int64_t k, int64_t entry) {
  if (k == 0) return entry;
  const int64_t j = k - 1;
  return j < entry ? j : j + 1;
}

// Warp bitonic sort of M (power of two) (key, id) pairs in shared memory.
__device__ void warp_sort_smem(uint64_t *key, uint32_t *id, int M) {
  const int lane = threadIdx.x & 31;
  for (int k = 2; k <= M; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = lane; i < M; i += 32) {
        const int l = i ^ j;
        if (l > i) {
          const bool up = (i & k) == 0;
          const uint64_t a = key[i], b = key[l];
          const uint32_t ai = id[i], bi = id[l];
          const bool gt = key_less(b, bi, a, ai);
          if (gt == up) { key[i] = b; key[l] = a; id[i] = bi; id[l] = ai; }
        }
      }
      __syncwarp();
    }
  }
}

__device__ void warp_sort_u32(uint32_t *v, int M) {
  const int lane = threadIdx.x & 31;
  for (int k = 2; k <= M; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = lane; i < M; i += 32) {
        const int l = i ^ j;
        if (l > i) {
          const bool up = (i & k) == 0;
          const uint32_t a = v[i], b = v[l];
          if ((a > b) == up) { v[i] = b; v[l] = a; }
        }
      }
      __syncwarp();
    }
  }
}

__host__ __device__ inline int next_pow2(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

// ---------------------------------------------------------------------------
// thresholds and entry vertex
// ---------------------------------------------------------------------------

constexpr int kThrWarps = 8;
constexpr int kMaxSample = 1024;

struct Pct { int32_t v[4]; };

__global__ void __launch_bounds__(kThrWarps * 32)
thresholds_kernel(DevIndex ix, int S, uint64_t seed, int nT, Pct pct, uint32_t *thr) {
  __shared__ uint32_t buf[kThrWarps][kMaxSample];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t *b = buf[warp];
  const int64_t Ss = ix.n - 1 < S ? ix.n - 1 : S;
  const int M = next_pow2((int)(Ss > 0 ? Ss : 1));
  for (int64_t p = (int64_t)blockIdx.x * kThrWarps + warp; p < ix.n; p += (int64_t)gridDim.x * kThrWarps) {
    for (int i = lane; i < M; i += 32) {
      uint32_t v = 0xFFFFFFFFu;
      if (i < Ss) {
        const uint64_t r = sm64(seed, ((uint64_t)p << 20) | (uint64_t)i) % (uint64_t)(ix.n - 1);
        const int64_t o = (int64_t)r < p ? (int64_t)r : (int64_t)r + 1;
        v = attribute_distance(ix, p, o);
      }
      b[i] = v;
    }
    __syncwarp();
    warp_sort_u32(b, M);
    if (lane < nT) thr[p * nT + lane] = Ss > 0 ? b[(int64_t)pct.v[lane] * (Ss - 1) / 100] : 0u;
    __syncwarp();
  }
}

// Weight-JAG weights (implementation-details appendix): over the threshold
// sample of S points v, h = sigma / sigma_A with sigma the population standard
// deviation of dist(x_p, x_v) (canonical fp32 distances) and sigma_A that of
// dist_A(a_p, a_v) as a real number; sums in fp64, in sample order (the order
// fixes the rounding); h = 0 if sigma_A = 0.  The weights of p are
// w_i = fp32(c_i h).
//
// In two kernels over chunks of points: one warp per point writes the sample's
// distances, sample by sample across the points; then one thread per point
// runs its chains of additions.  (An fp64 instruction holds its pipe for 64
// cycles whether one lane or 32 take part: with the chains on one lane of each
// point's warp, 30,011 points x 500 samples took 11.1 ms.)
struct Mult { double v[8]; };
constexpr int kWgtWarps = 4;

template <int P, int CPL>
__global__ void __launch_bounds__(kWgtWarps * 32)
weights_sample_kernel(DevIndex ix, int64_t p0, int64_t np, int64_t stride, int64_t Ss, uint64_t seed, float *sa,
                      float *sd) {
  __shared__ uint32_t sid[kWgtWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t i = (int64_t)blockIdx.x * kWgtWarps + warp; i < np; i += (int64_t)gridDim.x * kWgtWarps) {
    const int64_t p = p0 + i;
    QChunks<CPL, JAG_VEC_F32> q;
    load_row<P, CPL>(ix, p, q);
    for (int64_t i0 = 0; i0 < Ss; i0 += 32) {
      const int nc = (int)min64(32, Ss - i0);
      if (lane < nc) {
        const uint64_t r = sm64(seed, ((uint64_t)p << 20) | (uint64_t)(i0 + lane)) % (uint64_t)(ix.n - 1);
        const int64_t o = (int64_t)r < p ? (int64_t)r : (int64_t)r + 1;
        sid[warp][lane] = (uint32_t)o;
        const uint32_t da = attribute_distance(ix, p, o);
        sa[(i0 + lane) * stride + i] = ix.dist_a == JAG_F_RANGE_F32 ? u2f(da) : __uint2float_rn(da);
      }
      __syncwarp();
      const float dist = candidate_distances<P, CPL, CPL == 1 ? 8 : 4, JAG_VEC_F32, true>(ix, q, sid[warp], nc);
      if (lane < nc) sd[(i0 + lane) * stride + i] = dist;
      __syncwarp();
    }
  }
}

__global__ void __launch_bounds__(64)
weights_kernel(int64_t p0, int64_t np, int64_t stride, int64_t Ss, int nW, Mult mult, const float *sa, const float *sd,
               uint32_t *wout) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  double ma = 0.0, md = 0.0, va = 0.0, vd = 0.0;
#pragma unroll 4
  for (int64_t i = 0; i < Ss; ++i) {
    ma = __dadd_rn(ma, (double)sa[i * stride + p]);
    md = __dadd_rn(md, (double)sd[i * stride + p]);
  }
  if (Ss > 0) { ma = __ddiv_rn(ma, (double)Ss); md = __ddiv_rn(md, (double)Ss); }
#pragma unroll 4
  for (int64_t i = 0; i < Ss; ++i) {
    const double ta = __dsub_rn((double)sa[i * stride + p], ma), td = __dsub_rn((double)sd[i * stride + p], md);
    va = __dadd_rn(va, __dmul_rn(ta, ta));
    vd = __dadd_rn(vd, __dmul_rn(td, td));
  }
  if (Ss > 0) { va = __ddiv_rn(va, (double)Ss); vd = __ddiv_rn(vd, (double)Ss); }
  const double s_a = __dsqrt_rn(va), s_d = __dsqrt_rn(vd);
  const double h = s_a > 0.0 ? __ddiv_rn(s_d, s_a) : 0.0;
  for (int j = 0; j < nW; ++j) wout[(p0 + p) * nW + j] = f2u(__double2float_rn(__dmul_rn(mult.v[j], h)));
}

// Column sums in index order (fp64): one lane per coordinate, one CTA per 32
// coordinates.  The sum is a chain of n dependent additions (the order fixes
// the rounding), 64 cycles each on this part, and a conversion from fp32 takes
// the same pipe for as long; so warp 0 does nothing but the additions, while
// the other three warps, on the SM's other partitions, copy the rows through
// a ring of asynchronous copies and widen them one tile ahead.  (200K x 128:
// 23.5 ms with a thread per coordinate and plain loads, 14.1 ms with the
// conversion in the adding warp, 8.0 ms so.)
constexpr int kCenRows = 32, kCenStages = 8, kCenThreads = 128;
constexpr size_t kCenSmem = sizeof(float) * kCenStages * kCenRows * 32 + sizeof(double) * 2 * kCenRows * 32;

__global__ void __launch_bounds__(kCenThreads) centroid_kernel(DevIndex ix, double *c) {
  extern __shared__ __align__(16) uint8_t csm[];
  double *wide = reinterpret_cast<double *>(csm);                          // [2][kCenRows][32]
  float *tile = reinterpret_cast<float *>(wide + 2 * kCenRows * 32);       // [kCenStages][kCenRows][32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = threadIdx.x - 32;
  const int col0 = blockIdx.x * 32;
  const int64_t nt = (ix.n + kCenRows - 1) / kCenRows;
  auto request = [&](int64_t t) {   // warps 1..3: the 16-byte chunks of tile t
    if (t < nt) {
      float *dst = tile + (size_t)(t % kCenStages) * kCenRows * 32;
      for (int i = w; i < kCenRows * 8; i += kCenThreads - 32) {
        const int r = i >> 3, col = 4 * (i & 7);
        const int64_t row = t * kCenRows + r;
        if (row < ix.n && col0 + col < ix.xs) cp_async<16>(dst + r * 32 + col, ix.x + row * ix.xs + col0 + col);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto widen = [&](int64_t t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kCenStages - 2) : "memory");
    asm volatile("bar.sync 1, 96;" ::: "memory");   // the copies of all three warps
    if (t < nt) {
      const float *src = tile + (size_t)(t % kCenStages) * kCenRows * 32;
      double *dst = wide + (size_t)(t & 1) * kCenRows * 32;
      for (int i = w; i < kCenRows * 32; i += kCenThreads - 32) dst[i] = (double)src[i];
    }
  };
  if (warp > 0) {
    for (int t = 0; t < kCenStages - 1; ++t) request(t);
    widen(0);
  }
  __syncthreads();
  double s = 0.0;
  for (int64_t t = 0; t < nt; ++t) {
    if (warp > 0) {
      request(t + kCenStages - 1);   // into the tile widened before the last barrier
      widen(t + 1);
    } else {
      const double *src = wide + (size_t)(t & 1) * kCenRows * 32 + lane;
      const int rows = (int)min64(kCenRows, ix.n - t * kCenRows);
      if (rows == kCenRows) {
#pragma unroll
        for (int r = 0; r < kCenRows; ++r) s = __dadd_rn(s, src[r * 32]);
      } else {
        for (int r = 0; r < rows; ++r) s = __dadd_rn(s, src[r * 32]);
      }
    }
    __syncthreads();
  }
  if (warp == 0 && col0 + lane < ix.d) c[col0 + lane] = __ddiv_rn(s, (double)ix.n);
}

// fp64 squared distances from the centroid and their minimum; then the lowest
// id that has it.
__global__ void medoid_kernel(DevIndex ix, const double *c, unsigned long long *best, unsigned long long *dist) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ix.n) return;
  double s = 0.0;
  for (int j = 0; j < ix.d; ++j) {
    const double t = __dsub_rn((double)ix.x[i * ix.xs + j], c[j]);
    s = __dadd_rn(s, __dmul_rn(t, t));
  }
  const unsigned long long bits = (unsigned long long)__double_as_longlong(s);
  dist[i] = bits;
  atomicMin(&best[0], bits);
}

__global__ void medoid_id_kernel(int64_t n, unsigned long long *best, const unsigned long long *dist) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && dist[i] == best[0]) atomicMin(&best[1], (unsigned long long)i);
}

// ---------------------------------------------------------------------------
// batch searches with D_A(t)
// ---------------------------------------------------------------------------

template <int CAP, int P, int CPL>
__global__ void __launch_bounds__(kSearchWarps * 32)
build_search_kernel(DevIndex ix, int64_t pos0, int64_t nb, int nT, const uint32_t *thr, int weighted, int lb,
                    int hbits, uint32_t *vis_ids, float *vis_d, int32_t *vis_n, int vcap, unsigned long long *work,
                    uint32_t *status) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WarpSmem S = carve_warp_smem(smem + warp * warp_smem_bytes(CAP, hbits), CAP, hbits);
  const unsigned long long total = (unsigned long long)nb * nT;
  for (;;) {
    unsigned long long it = 0;
    if (lane == 0) it = atomicAdd(work, 1ull);
    it = __shfl_sync(kFull, it, 0);
    if (it >= total) return;
    const int64_t bi = (int64_t)(it / nT);
    const int ti = (int)(it % nT);
    const int64_t p = order_id(pos0 + bi, ix.entry);
    QChunks<CPL, JAG_VEC_F32> q;
    load_row<P, CPL>(ix, p, q);
    VisitSink sink{vis_ids + it * vcap, vis_d + it * vcap, vcap, 0};
    SearchStats st;
    if (weighted) {
      const WeightKey key{p, u2f(thr[p * nT + ti])};
      greedy_search<CAP, P, CPL, JAG_VEC_F32>(ix, key, q, lb, hbits, S, sink, st);
    } else {
      const BuildKey key{p, thr[p * nT + ti]};
      greedy_search<CAP, P, CPL, JAG_VEC_F32>(ix, key, q, lb, hbits, S, sink, st);
    }
    if (lane == 0) {
      vis_n[it] = sink.n;
      if (sink.n > vcap) atomicOr(status, kErrVisitedOverflow);
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// JointRobustPrune
// ---------------------------------------------------------------------------

// Candidate arrays of one prune: a slice of shared memory, or a per-warp
// region of global scratch when the candidate set is larger than the slice.
struct PruneSmem {
  uint32_t *cid;     // [cmax] candidate ids
  float *cdist;      // [cmax] d(p, candidate)
  uint64_t *skey;    // [cmax] sort keys
  uint32_t *sid;     // [cmax]
  uint32_t *bucket;  // [64] (always shared)
  uint32_t *chosen;  // [64]
  uint32_t *tmp;     // [64]
  float4 *rows;      // [bucket_members][nchunks] rows of the bucket's members (first launch only)
};

__host__ __device__ inline size_t cand_bytes(int cmax) { return (size_t)cmax * (4 + 4 + 8 + 4); }

__host__ __device__ inline size_t prune_smem_bytes(int cmax) { return cand_bytes(cmax) + 64 * 4 * 3; }

__device__ inline void carve_cands(uint8_t *base, int cmax, PruneSmem &s) {
  s.skey = reinterpret_cast<uint64_t *>(base);
  s.cid = reinterpret_cast<uint32_t *>(base + (size_t)cmax * 8);
  s.cdist = reinterpret_cast<float *>(s.cid + cmax);
  s.sid = reinterpret_cast<uint32_t *>(s.cdist + cmax);
}

__device__ inline PruneSmem carve_prune(uint8_t *base, int cmax) {
  PruneSmem s;
  carve_cands(base, cmax, s);
  s.bucket = s.sid + cmax;
  s.chosen = s.bucket + 64;
  s.tmp = s.chosen + 64;
  s.rows = reinterpret_cast<float4 *>(s.tmp + 64);   // 16-byte aligned: cmax is a power of two >= 4
  return s;
}

// The same small arrays, candidate arrays moved to global scratch.
__device__ inline PruneSmem spill_prune(const PruneSmem &sm, uint8_t *gbase, int cmax_g) {
  PruneSmem s = sm;
  carve_cands(gbase, cmax_g, s);
  return s;
}

__device__ __forceinline__ bool in_list(const uint32_t *list, int n, uint32_t v) {
  const int lane = threadIdx.x & 31;
  bool hit = false;
  for (int i = lane; i < n; i += 32) hit |= (list[i] == v);
  return __any_sync(kFull, hit);
}

// Members of a bucket at most: it stops at 0.9 R / nT.
__host__ __device__ inline int bucket_members(int R, int nT) { return (9 * R + 10 * nT - 1) / (10 * nT); }

// The alpha test of one candidate (row chunks xv, distance dpv from p) against
// the nb members of the bucket: true if some member u has
// alpha^2 d(u, v) <= d(p, v).
template <int P, int CPL, bool STAGE>
__device__ __forceinline__ bool pruned_by(const DevIndex &ix, const QChunks<CPL, JAG_VEC_F32> &xv, float dpv,
                                          float alpha2, const PruneSmem &S, int nb) {
  constexpr int VPW = 32 / P;
  constexpr int U = VPW >= 4 ? 1 : 4 / VPW;   // rows per lane and round
  constexpr int F = 32 / P;
  constexpr int NA = CPL < F ? CPL : F;
  const int lane = threadIdx.x & 31, grp = lane / P, lig = lane % P;
  for (int b = 0; b < nb; b += VPW * U) {
    float acc[U];
#pragma unroll
    for (int s = 0; s < U; ++s) {
      const int r = b + s * VPW + grp;
      const bool ok = r < nb;
      float a[NA];
#pragma unroll
      for (int i = 0; i < NA; ++i) a[i] = 0.f;
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        const int ch = lig + j * P;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok && ch < ix.nchunks)
          x = STAGE ? S.rows[(size_t)r * ix.nchunks + ch] : ld_chunk(ix.x + (int64_t)S.bucket[r] * ix.xs + ch * 4);
        a[j % F] = chunk_accumulate(a[j % F], xv.v[j][0], x);
      }
#pragma unroll
      for (int h = F / 2; h >= 1; h >>= 1) {
#pragma unroll
        for (int i = 0; i < h; ++i)
          if (i + h < NA) a[i] = __fadd_rn(a[i], a[i + h]);
      }
      acc[s] = a[0];
    }
    const float duv = group_reduce_spread<P, U>(acc);
    const int r = b + (lig / (P / U)) * VPW + grp;   // the row whose sum this lane holds
    if (__any_sync(kFull, r < nb && !(__fmul_rn(alpha2, duv) > dpv))) return true;
  }
  return false;
}

// JointRobustPrune for base point p over candidates S.cid/S.cdist[0..nc).
// Writes the new out-list (-1 padded) to row.
//
// Weight-JAG (weighted != 0): T holds fp32 weights w and the ranking is by
// D_A^w(p, v) = fma(w, dist_A, dist(p, v)), then id.  The candidates are first
// put in id order, so that a candidate's index breaks ties like its id, and
// the ranking sorts indices; dist(p, v) for the alpha test comes from cdist.
template <int P, int CPL, bool STAGE>
__device__ __forceinline__ void joint_prune(const DevIndex &ix, int64_t p, const PruneSmem &S, int nc,
                            const uint32_t *T, int nT, float alpha2, int weighted, int32_t *row) {
  const int lane = threadIdx.x & 31;
  const int R = ix.R;
  const int M = next_pow2(nc > 0 ? nc : 1);
  int nchosen = 0;
  if (weighted) {
    for (int i = lane; i < M; i += 32) {
      S.skey[i] = i < nc ? (uint64_t)S.cid[i] : kNoKey;
      S.sid[i] = i < nc ? f2u(S.cdist[i]) : kEmptySlot;
    }
    __syncwarp();
    warp_sort_smem(S.skey, S.sid, M);
    for (int i = lane; i < nc; i += 32) { S.cid[i] = (uint32_t)S.skey[i]; S.cdist[i] = u2f(S.sid[i]); }
    __syncwarp();
  }
  for (int ti = 0; ti < nT; ++ti) {
    const uint32_t t = T[ti];
    for (int i = lane; i < M; i += 32) {
      if (i < nc) {
        const uint32_t c = S.cid[i];
        if (weighted) {
          const uint32_t da = attribute_distance(ix, p, c);
          const float a = ix.dist_a == JAG_F_RANGE_F32 ? u2f(da) : __uint2float_rn(da);
          S.skey[i] = make_key(0u, __fmaf_rn(u2f(t), a, S.cdist[i]));
          S.sid[i] = (uint32_t)i;
        } else {
          S.skey[i] = make_key(capped_distance(ix.dist_a, attribute_distance(ix, p, c), t), S.cdist[i]);
          S.sid[i] = c;
        }
      } else {
        S.skey[i] = kNoKey;
        S.sid[i] = kEmptySlot;
      }
    }
    __syncwarp();
    warp_sort_smem(S.skey, S.sid, M);
    // The candidates in order; the row of the next one is on its way while one
    // is tested.  The members' rows are kept in shared memory (STAGE) and
    // tested a few at a time, the nearest first, up to the first that prunes
    // the candidate.  (Read from L2 for every candidate, all members at once,
    // the insert prunes of a 200K x 128 label build took 34 ms, now 23; testing
    // a new member against 32 candidates at once instead: back-edge prunes
    // 25 -> 37 ms.)
    int nb = 0;
    QChunks<CPL, JAG_VEC_F32> xn;
    if (nc > 0) load_row<P, CPL>(ix, weighted ? S.cid[S.sid[0]] : S.sid[0], xn);
    for (int i = 0; i < nc; ++i) {
      const uint32_t v = weighted ? S.cid[S.sid[i]] : S.sid[i];
      const float dpv = weighted ? S.cdist[S.sid[i]] : u2f((uint32_t)S.skey[i]);
      const QChunks<CPL, JAG_VEC_F32> xv = xn;
      if (i + 1 < nc) load_row<P, CPL>(ix, weighted ? S.cid[S.sid[i + 1]] : S.sid[i + 1], xn);
      bool keep = true;
      if (nb > 0 && !(nchosen > 0 && in_list(S.chosen, nchosen, v)))
        keep = !pruned_by<P, CPL, STAGE>(ix, xv, dpv, alpha2, S, nb);
      if (keep) {
        if (lane == 0) S.bucket[nb] = v;
        if (STAGE && lane < P) {
#pragma unroll
          for (int j = 0; j < CPL; ++j) {
            const int ch = lane + j * P;
            if (ch < ix.nchunks) S.rows[(size_t)nb * ix.nchunks + ch] = xv.v[j][0];
          }
        }
        ++nb;
        __syncwarp();
      }
      if ((int64_t)nb * nT * 10 >= (int64_t)9 * R) break;
    }
    for (int j = 0; j < nb; ++j) {
      const uint32_t v = S.bucket[j];
      if (!in_list(S.chosen, nchosen, v)) {
        if (lane == 0) S.chosen[nchosen] = v;
        ++nchosen;
        __syncwarp();
      }
    }
  }
  const int m = nchosen < R ? nchosen : R;
  for (int r = lane; r < R; r += 32) row[r] = r < m ? (int32_t)S.chosen[r] : -1;
  __syncwarp();
}

// The prunes of a batch run in two launches.  They are bound by the latency of
// each warp's chain of row loads, so what counts is warps in flight: with
// 1,024-candidate slices (20 KB) ten fit an SM.  The first launch gives a warp
// a slice of shared memory that holds the usual candidate set and lists the
// larger ones; the second, with few warps of large slices and a global spill,
// takes the list (usually empty: its warps read the count and leave).
// Measured on a 200K x 128 label build: back-edge prunes 57 -> 25 ms.
struct PruneList {
  int32_t *items;              // oversized items of the first launch
  unsigned long long *count;
};

// Union of batch point bi's visited sets (`total` entries, repeats among them)
// and its new out-list; false if the union has more than cmax vertices.
template <int P, int CPL, bool STAGE>
__device__ __forceinline__ bool insert_point(const DevIndex &ix, int64_t bi, int64_t p, int nT, const uint32_t *thr,
                                             int weighted, float alpha2, const uint32_t *vis_ids, const float *vis_d,
                                             const int32_t *vis_n, int vcap, int total, const PruneSmem &S, int cmax,
                                             int32_t *row) {
  const int lane = threadIdx.x & 31;
  // the union of the visited sets: a hash table in the sort keys' place
  // (joint_prune sorts by key and id, so the order here is free; the sets of
  // a point's thresholds share most of their vertices)
  uint32_t *tab = reinterpret_cast<uint32_t *>(S.skey);
  const int H = min(2 * cmax, next_pow2(2 * max(total, 32)));
  const int shift = 33 - __ffs(H);   // 32 - log2 H
  for (int i = lane; i < H; i += 32) tab[i] = kEmptySlot;
  __syncwarp();
  int w = 0;
  for (int ti = 0; ti < nT && w <= cmax; ++ti) {
    const int64_t it = bi * nT + ti;
    const int m = min(vis_n[it], vcap);
    for (int i0 = 0; i0 < m && w <= cmax; i0 += 32) {
      const bool in = i0 + lane < m;
      const uint32_t id = in ? vis_ids[it * vcap + i0 + lane] : kEmptySlot;
      const float dv = in ? vis_d[it * vcap + i0 + lane] : 0.f;
      bool fresh = false;
      if (in) {
        uint32_t h = (id * 0x9E3779B1u) >> shift;
        for (;;) {   // at most cmax + 32 of the 2 cmax slots are taken
          const uint32_t old = atomicCAS(&tab[h], kEmptySlot, id);
          fresh = old == kEmptySlot;
          if (fresh | (old == id)) break;
          h = (h + 1) & (H - 1);
        }
      }
      const uint32_t fm = __ballot_sync(kFull, fresh);
      const int pos = w + __popc(fm & lanemask_lt());
      if (fresh && pos < cmax) {
        S.cid[pos] = id;
        S.cdist[pos] = dv;   // Weight-JAG lists hold D_A^w, not dist: recomputed below
      }
      w += __popc(fm);
    }
  }
  __syncwarp();
  if (w > cmax) return false;
  if (weighted) {
    QChunks<CPL, JAG_VEC_F32> xp;
    load_row<P, CPL>(ix, p, xp);
    for (int b = 0; b < w; b += 32) {
      const int m = min(32, w - b);
      const float dv = candidate_distances<P, CPL, 4, JAG_VEC_F32, true>(ix, xp, S.cid + b, m);
      if (lane < m) S.cdist[b + lane] = dv;
    }
    __syncwarp();
  }
  joint_prune<P, CPL, STAGE>(ix, p, S, w, thr + p * nT, nT, alpha2, weighted, row);
  return true;
}

// The same with the candidate arrays in global scratch (a copy of its own, so
// that the usual one addresses shared memory).
template <int P, int CPL, bool STAGE>
__device__ __noinline__ bool insert_point_spilled(const DevIndex &ix, int64_t bi, int64_t p, int nT,
                                                  const uint32_t *thr, int weighted, float alpha2,
                                                  const uint32_t *vis_ids, const float *vis_d, const int32_t *vis_n,
                                                  int vcap, int total, const PruneSmem &S, int cmax, int32_t *row) {
  return insert_point<P, CPL, STAGE>(ix, bi, p, nT, thr, weighted, alpha2, vis_ids, vis_d, vis_n, vcap, total, S, cmax,
                                     row);
}

// Union of a batch point's visited sets (deduplicated), then its new
// out-list; emits its back-edges.
// LARGE: the second launch, over the listed points.
// STAGE: the members' rows go to shared memory.
template <int P, int CPL, bool LARGE, bool STAGE>
__global__ void __launch_bounds__(kPruneWarps * 32)
prune_insert_kernel(DevIndex ix, int32_t *graph, int64_t pos0, int64_t nb, int nT, const uint32_t *thr,
                    int weighted, float alpha2, const uint32_t *vis_ids, const float *vis_d, const int32_t *vis_n,
                    int vcap, PruneList big,
                    int cmax_s, int cmax_g, size_t warp_bytes, uint8_t *gscratch, int32_t *etgt, int32_t *esrc) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PruneSmem Ss = carve_prune(smem + warp * warp_bytes, cmax_s);
  const int64_t gw = (int64_t)blockIdx.x * kPruneWarps + warp;
  const PruneSmem Sg = spill_prune(Ss, gscratch + gw * cand_bytes(cmax_g), cmax_g);
  const int64_t ni = LARGE ? (int64_t)*big.count : nb;
  for (int64_t ii = gw; ii < ni; ii += (int64_t)gridDim.x * kPruneWarps) {
    const int64_t bi = LARGE ? big.items[ii] : ii;
    const int64_t p = order_id(pos0 + bi, ix.entry);
    int total = 0;
    for (int ti = 0; ti < nT; ++ti) total += min(vis_n[bi * nT + ti], vcap);
    int32_t *row = graph + p * ix.R;
    bool done = insert_point<P, CPL, STAGE>(ix, bi, p, nT, thr, weighted, alpha2, vis_ids, vis_d, vis_n, vcap, total, Ss,
                                            cmax_s, row);
    if (!done)
      done = insert_point_spilled<P, CPL, STAGE>(ix, bi, p, nT, thr, weighted, alpha2, vis_ids, vis_d, vis_n, vcap,
                                                 total, Sg, cmax_g, row);
    if (!done) {   // (not in the second launch: its spill holds every visited set)
      if (lane == 0 && !LARGE) big.items[atomicAdd(big.count, 1ull)] = (int32_t)bi;
      continue;
    }
    for (int r = lane; r < ix.R; r += 32) {
      const int32_t v = row[r];
      etgt[bi * ix.R + r] = v;
      esrc[bi * ix.R + r] = v >= 0 ? (int32_t)p : -1;
    }
    __syncwarp();
  }
}

// Back-edges: count per target, reserve, scatter, apply.
struct EdgeState {
  int32_t *tcount, *tfill;   // [n], zero between batches
  int64_t *toff;             // [n]
  int32_t *tlist;            // [nb*R]
  int32_t *srcbuf;           // [nb*R]
  unsigned long long *ctr;   // [0] targets, [1] cursor, [3] most sources of a target, [4], [5] listed items
};

__global__ void edge_count_kernel(const int32_t *etgt, int64_t ne, EdgeState E) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const int32_t v = etgt[e];
  if (v < 0) return;
  if (atomicAdd(&E.tcount[v], 1) == 0) {
    const unsigned long long i = atomicAdd(&E.ctr[0], 1ull);
    E.tlist[i] = v;
  }
}

// Largest number of new back-edges of one target in the batch (ctr[3]).
__global__ void edge_max_kernel(int64_t cap, EdgeState E) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool ok = i < cap && (unsigned long long)i < E.ctr[0];
  const unsigned most = __reduce_max_sync(kFull, ok ? (unsigned)E.tcount[E.tlist[i]] : 0u);
  if ((threadIdx.x & 31) == 0 && most > 0) atomicMax(&E.ctr[3], (unsigned long long)most);
}

__global__ void edge_offset_kernel(int64_t cap, EdgeState E) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool ok = i < cap && (unsigned long long)i < E.ctr[0];
  const int32_t v = ok ? E.tlist[i] : 0;
  const int own = ok ? E.tcount[v] : 0;
  int sum = own;   // inclusive sum over the warp: one reservation per warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, sum, o);
    if (lane >= o) sum += t;
  }
  unsigned long long base = 0;
  if (lane == 31 && sum > 0) base = atomicAdd(&E.ctr[1], (unsigned long long)sum);
  base = __shfl_sync(kFull, base, 31);
  if (ok) E.toff[v] = (int64_t)base + sum - own;
}

__global__ void edge_scatter_kernel(const int32_t *etgt, const int32_t *esrc, int64_t ne, EdgeState E) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const int32_t v = etgt[e];
  if (v < 0) return;
  const int32_t slot = atomicAdd(&E.tfill[v], 1);
  E.srcbuf[E.toff[v] + slot] = esrc[e];
}

// LARGE: the second launch, over the listed targets.
template <int P, int CPL, bool LARGE, bool STAGE>
__global__ void __launch_bounds__(kPruneWarps * 32)
edge_apply_kernel(DevIndex ix, int32_t *graph, int nT, const uint32_t *thr, int weighted, float alpha2, PruneList big,
                  int cmax_s, int cmax_g, size_t warp_bytes, uint8_t *gscratch, EdgeState E, uint32_t *status) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PruneSmem Ss = carve_prune(smem + warp * warp_bytes, cmax_s);
  const int64_t gw = (int64_t)blockIdx.x * kPruneWarps + warp;
  const PruneSmem Sg = LARGE ? spill_prune(Ss, gscratch + gw * cand_bytes(cmax_g), cmax_g) : Ss;
  const int64_t ni = (int64_t)(LARGE ? *big.count : E.ctr[0]);
  for (int64_t i = gw; i < ni; i += (int64_t)gridDim.x * kPruneWarps) {
    const int32_t v = LARGE ? big.items[i] : E.tlist[i];
    const int ns = E.tcount[v];
    const int32_t *src = E.srcbuf + E.toff[v];
    int32_t *row = graph + (int64_t)v * ix.R;
    int deg = 0;
    for (int r = lane; r < ix.R; r += 32) deg += row[r] >= 0 ? 1 : 0;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) deg += __shfl_xor_sync(kFull, deg, o);
    if (!LARGE && deg + ns > cmax_s) {
      if (lane == 0) big.items[atomicAdd(big.count, 1ull)] = v;
      continue;   // its counts are cleared by the second launch
    }
    // (of the first launch neither test can fail here, but without them its copy
    // takes 64 registers, not 56, and a build 1.5 % longer)
    const PruneSmem &S = deg + ns <= cmax_s ? Ss : Sg;
    if (deg + ns > cmax_g) {
      if (lane == 0) atomicOr(status, kErrCandOverflow);
    } else if (deg + ns <= ix.R) {
      // append the new sources in increasing id order
      const int M = next_pow2(ns);
      for (int j = lane; j < M; j += 32) S.tmp[j] = j < ns ? (uint32_t)src[j] : 0xFFFFFFFFu;
      __syncwarp();
      warp_sort_u32(S.tmp, M);
      for (int j = lane; j < ns; j += 32) row[deg + j] = (int32_t)S.tmp[j];
    } else {
      const int nc = deg + ns;
      for (int j = lane; j < nc; j += 32) S.cid[j] = j < deg ? (uint32_t)row[j] : (uint32_t)src[j - deg];
      __syncwarp();
      QChunks<CPL, JAG_VEC_F32> xv;
      load_row<P, CPL>(ix, v, xv);
      for (int b = 0; b < nc; b += 32) {
        const int m = min(32, nc - b);
        const float dv = candidate_distances<P, CPL, 4, JAG_VEC_F32, true>(ix, xv, S.cid + b, m);
        if (lane < m) S.cdist[b + lane] = dv;
      }
      __syncwarp();
      joint_prune<P, CPL, STAGE>(ix, v, S, nc, thr + (int64_t)v * nT, nT, alpha2, weighted, row);
    }
    __syncwarp();
    if (lane == 0) { E.tcount[v] = 0; E.tfill[v] = 0; }
  }
}

// ---------------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------------

struct BuildScratch {
  uint32_t *vis_ids = nullptr;
  float *vis_d = nullptr;
  int32_t *vis_n = nullptr;
  int32_t *etgt = nullptr, *esrc = nullptr;
  EdgeState E{};
  unsigned long long *work = nullptr;
  uint32_t *status = nullptr;
  double *centroid = nullptr;
  unsigned long long *best = nullptr;
  uint8_t *gscratch = nullptr;   // per-warp candidate arrays of large prunes (before the first: the weights' samples)
  size_t gbytes = 0;
  int64_t prune_blocks = 0;      // CTAs of the second (large) prune launches
  int32_t *biglist = nullptr;    // oversized items listed by the first ones
  uint8_t *big = nullptr;        // per-warp arrays for a batch whose hub targets need more
  size_t big_bytes = 0;
  void *blocks[24] = {};
  int nblocks = 0;
};

static cudaError_t balloc(BuildScratch &s, void **p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes < 256 ? 256 : bytes);
  if (e == cudaSuccess) s.blocks[s.nblocks++] = *p;
  return e;
}

static void bfree(BuildScratch &s) {
  for (int i = 0; i < s.nblocks; ++i) cudaFree(s.blocks[i]);
  s.nblocks = 0;
  if (s.big) cudaFree(s.big);
  s.big = nullptr;
  s.big_bytes = 0;
}

// Budget of the per-warp candidate arrays of oversized back-edge prunes.
constexpr size_t kBigScratchBytes = size_t(1) << 30;

template <int CAP, int P, int CPL>
static cudaError_t launch_build_search(const BuildLaunch &B, int64_t pos0, int64_t nb, int hbits, BuildScratch &s,
                                       int vcap) {
  const size_t smem = (size_t)kSearchWarps * warp_smem_bytes(CAP, hbits);
  auto kern = build_search_kernel<CAP, P, CPL>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int bps = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kSearchWarps * 32, smem);
  if (bps <= 0) return cudaErrorInvalidConfiguration;
  const int64_t items = nb * B.nT;
  const int64_t grid = std::min<int64_t>((int64_t)bps * num_sms(), (items + kSearchWarps - 1) / kSearchWarps);
  kern<<<(unsigned)grid, kSearchWarps * 32, smem, B.stream>>>(B.ix, pos0, nb, B.nT, B.thr, B.weighted, B.lb, hbits,
                                                             s.vis_ids, s.vis_d, s.vis_n, vcap, s.work, s.status);
  return cudaGetLastError();
}

// Shared-memory slice of the first prune launches, in candidates: room for
// the union of the visited sets of the usual searches (l_b hops and a few more
// per threshold, most of them shared), and for a back-edge target's list and
// sources.
static int insert_slice(int nT, int lb) { return std::max(256, std::min(1024, next_pow2(nT * (lb + lb / 4)))); }
constexpr int kEdgeSlice = 128;
constexpr int kMidCands = 1024;

// A prune kernel's grid: the CTAs that fit the SMs with `smem` bytes each.  (The
// sizes differ between builds; blocks_per_sm raises the kernel's limit, which
// the whole process shares, to the most there is, so that a launch of another
// build, from another thread, stays valid.)
template <class Kern>
static cudaError_t prune_grid(Kern kern, size_t smem, int64_t items, unsigned *grid) {
  const int bps = blocks_per_sm(kern, smem, kPruneWarps);
  if (bps <= 0) return cudaErrorInvalidConfiguration;
  *grid = (unsigned)std::max<int64_t>(
      1, std::min<int64_t>((items + kPruneWarps - 1) / kPruneWarps, (int64_t)bps * num_sms()));
  return cudaSuccess;
}

template <int P, int CPL>
static cudaError_t launch_prunes(const BuildLaunch &B, int64_t pos0, int64_t nb, BuildScratch &s, int vcap,
                                 int cmax_s, int cmax_g) {
  cudaError_t e;
  const size_t wbytes = prune_smem_bytes(cmax_s), smem = kPruneWarps * wbytes;
  const int64_t ne = nb * B.ix.R;
  // bytes of a warp's shared memory with the bucket rows behind a slice, 0
  // where fewer than eight warps would fit an SM (the rows are then read from
  // memory)
  auto staged = [&](int slice) {
    const size_t v = prune_smem_bytes(slice) + (size_t)bucket_members(B.ix.R, B.nT) * (size_t)B.ix.nchunks * 16;
    return v * 8 <= 220 * 1024 ? v : 0;
  };
  unsigned grid = 0;
  {
    const int slice = insert_slice(B.nT, B.lb);
    const PruneList big{s.biglist, s.E.ctr + 4};
    const size_t st = staged(slice), wb = st ? st : prune_smem_bytes(slice);
    auto pk = st ? prune_insert_kernel<P, CPL, false, true> : prune_insert_kernel<P, CPL, false, false>;
    if ((e = prune_grid(pk, kPruneWarps * wb, nb, &grid)) != cudaSuccess) return e;
    // candidate sets past the slice spill to kMidCands per warp, in the area
    // that the second launch uses after this one
    grid = std::min(grid, (unsigned)std::max<size_t>(1, s.gbytes / (cand_bytes(kMidCands) * kPruneWarps)));
    pk<<<grid, kPruneWarps * 32, kPruneWarps * wb, B.stream>>>(
        B.ix, B.graph, pos0, nb, B.nT, B.thr, B.weighted, B.alpha2, s.vis_ids, s.vis_d, s.vis_n, vcap, big, slice,
        kMidCands, wb, s.gscratch, s.etgt, s.esrc);
    auto lk = prune_insert_kernel<P, CPL, true, false>;
    if (blocks_per_sm(lk, smem, kPruneWarps) <= 0) return cudaErrorInvalidConfiguration;
    const int64_t lgrid = std::max<int64_t>(1, std::min<int64_t>((nb + kPruneWarps - 1) / kPruneWarps, s.prune_blocks));
    lk<<<(unsigned)lgrid, kPruneWarps * 32, smem, B.stream>>>(
        B.ix, B.graph, pos0, nb, B.nT, B.thr, B.weighted, B.alpha2, s.vis_ids, s.vis_d, s.vis_n, vcap, big, cmax_s,
        cmax_g, wbytes, s.gscratch, s.etgt, s.esrc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const unsigned eb = (unsigned)((ne + 255) / 256);
  edge_count_kernel<<<eb, 256, 0, B.stream>>>(s.etgt, ne, s.E);
  // A hub can receive more back-edges in one batch than the fixed per-warp
  // arrays hold.  Size this batch's arrays from its largest target: fewer
  // warps, each with room for a whole candidate set.
  edge_max_kernel<<<eb, 256, 0, B.stream>>>(ne, s.E);
  unsigned long long most = 0;
  if ((e = cudaMemcpyAsync(&most, s.E.ctr + 3, sizeof(most), cudaMemcpyDeviceToHost, B.stream)) != cudaSuccess)
    return e;
  edge_offset_kernel<<<eb, 256, 0, B.stream>>>(ne, s.E);
  edge_scatter_kernel<<<eb, 256, 0, B.stream>>>(s.etgt, s.esrc, ne, s.E);
  const PruneList big{s.biglist, s.E.ctr + 5};
  const size_t est = staged(kEdgeSlice), ewb = est ? est : prune_smem_bytes(kEdgeSlice);
  auto ak = est ? edge_apply_kernel<P, CPL, false, true> : edge_apply_kernel<P, CPL, false, false>;
  if ((e = prune_grid(ak, kPruneWarps * ewb, ne, &grid)) != cudaSuccess) return e;
  ak<<<grid, kPruneWarps * 32, kPruneWarps * ewb, B.stream>>>(B.ix, B.graph, B.nT, B.thr, B.weighted, B.alpha2, big,
                                                             kEdgeSlice, kEdgeSlice, ewb, nullptr, s.E, s.status);
  if ((e = cudaStreamSynchronize(B.stream)) != cudaSuccess) return e;
  if ((int64_t)most + B.ix.R > kEdgeSlice) {
    uint8_t *scratch = s.gscratch;
    int cmax = cmax_g;
    int64_t agrid = std::min<int64_t>((ne + kPruneWarps - 1) / kPruneWarps, s.prune_blocks);
    if ((int64_t)most + B.ix.R > cmax_g) {
      cmax = next_pow2((int)most + B.ix.R);
      const size_t per = cand_bytes(cmax);
      const int64_t warps = std::max<int64_t>(
          kPruneWarps, std::min<int64_t>(s.prune_blocks * kPruneWarps, (int64_t)(kBigScratchBytes / per)));
      agrid = std::max<int64_t>(1, std::min<int64_t>(agrid, warps / kPruneWarps));
      const size_t need = per * (size_t)agrid * kPruneWarps;
      if (s.big_bytes < need) {
        if (s.big) cudaFree(s.big);
        s.big = nullptr;
        s.big_bytes = 0;
        if ((e = cudaMalloc((void **)&s.big, need)) != cudaSuccess) return e;
        s.big_bytes = need;
      }
      scratch = s.big;
    }
    auto lk = edge_apply_kernel<P, CPL, true, false>;
    if (blocks_per_sm(lk, smem, kPruneWarps) <= 0) return cudaErrorInvalidConfiguration;
    lk<<<(unsigned)std::max<int64_t>(agrid, 1), kPruneWarps * 32, smem, B.stream>>>(
        B.ix, B.graph, B.nT, B.thr, B.weighted, B.alpha2, big, cmax_s, cmax, wbytes, scratch, s.E, s.status);
  }
  return cudaGetLastError();
}

static cudaError_t launch_weights(const BuildLaunch &B, const Mult &mult, float *scratch, int64_t chunk) {
  int P, CPL;
  if (!row_mapping(B.ix.nchunks, &P, &CPL)) return cudaErrorInvalidValue;
  const int64_t n = B.ix.n, Ss = std::min<int64_t>(n - 1, B.sample);
  float *sa = scratch, *sd = scratch + chunk * std::max<int64_t>(Ss, 1);
  for (int64_t p0 = 0; p0 < n; p0 += chunk) {
    const int64_t np = std::min<int64_t>(chunk, n - p0);
    const unsigned blocks =
        (unsigned)std::min<int64_t>((np + kWgtWarps - 1) / kWgtWarps, (int64_t)num_sms() * 16);
    bool done = false;
#define JAG_WCASE(PP, CC)                                                                                          \
  if (P == PP && CPL == CC) {                                                                                      \
    weights_sample_kernel<PP, CC><<<blocks, kWgtWarps * 32, 0, B.stream>>>(B.ix, p0, np, chunk, Ss, B.seed, sa, sd); \
    done = true;                                                                                                   \
  }
    JAG_WCASE(8, 1)
    JAG_WCASE(16, 1)
    JAG_WCASE(32, 1)
    JAG_WCASE(32, 2)
    JAG_WCASE(32, 4)
    JAG_WCASE(32, 8)
#undef JAG_WCASE
    if (!done) return cudaErrorInvalidValue;
    weights_kernel<<<(unsigned)((np + 63) / 64), 64, 0, B.stream>>>(p0, np, chunk, Ss, B.nT, mult, sa, sd, B.thr);
  }
  return cudaGetLastError();
}

template <int CAP>
static cudaError_t dispatch_build(const BuildLaunch &B, int P, int CPL, int64_t pos0, int64_t nb, int hbits,
                                  BuildScratch &s, int vcap, int cmax_s, int cmax_g) {
  cudaError_t e = cudaErrorInvalidValue;
#define JAG_BCASE(PP, CC)                                                   \
  if (P == PP && CPL == CC) {                                               \
    e = launch_build_search<CAP, PP, CC>(B, pos0, nb, hbits, s, vcap);      \
    if (e == cudaSuccess) e = launch_prunes<PP, CC>(B, pos0, nb, s, vcap, cmax_s, cmax_g); \
    return e;                                                               \
  }
  JAG_BCASE(8, 1)
  JAG_BCASE(16, 1)
  JAG_BCASE(32, 1)
  JAG_BCASE(32, 2)
  JAG_BCASE(32, 4)
  JAG_BCASE(32, 8)
#undef JAG_BCASE
  return e;
}

int run_build(BuildLaunch &B, int32_t *entry_out, char *msg, size_t msg_len) {
  const int64_t n = B.ix.n;
  const int R = B.ix.R;
  int P, CPL;
  if (!row_mapping(B.ix.nchunks, &P, &CPL)) { snprintf(msg, msg_len, "dimension too large"); return JAG_EINVAL; }
  const int cap_list = list_capacity(B.lb);
  if (!cap_list) { snprintf(msg, msg_len, "l_b must be <= 256"); return JAG_EINVAL; }
  BuildScratch s;
  cudaError_t e = cudaSuccess;
  const int64_t bcap = std::max<int64_t>(1, n / 50);
  // visited lists: hop counts are ~l_b plus a few, but a search may expand
  // more; 16 l_b leaves a wide margin and an overflow is reported, not cut
  const int vcap = std::max(1024, 16 * B.lb);
  const int cmax_s = 1024;                                   // shared-memory slice
  const int cmax_g = std::max(8192, next_pow2(B.nT * vcap)); // global spill
  const int bps = (int)std::max<size_t>(1, (227 * 1024) / (kPruneWarps * prune_smem_bytes(cmax_s)));
  s.prune_blocks = (int64_t)bps * num_sms();
  // visited-set slots: about twice the distances of a search of l_b hops; the
  // set may forget, and a smaller one leaves room for more warps (2^11 -> 2^10
  // at l_b = 64: 24 -> 36 warps per SM)
  const int hbits = B.lb <= 64 ? 10 : (B.lb <= 128 ? 11 : 12);
#define JAG_TRY(x) do { e = (x); if (e != cudaSuccess) goto fail; } while (0)
  JAG_TRY(balloc(s, (void **)&s.vis_ids, sizeof(uint32_t) * (size_t)bcap * B.nT * vcap));
  JAG_TRY(balloc(s, (void **)&s.vis_d, sizeof(float) * (size_t)bcap * B.nT * vcap));
  JAG_TRY(balloc(s, (void **)&s.vis_n, sizeof(int32_t) * (size_t)bcap * B.nT));
  JAG_TRY(balloc(s, (void **)&s.etgt, sizeof(int32_t) * (size_t)bcap * R));
  JAG_TRY(balloc(s, (void **)&s.esrc, sizeof(int32_t) * (size_t)bcap * R));
  JAG_TRY(balloc(s, (void **)&s.E.tcount, sizeof(int32_t) * (size_t)n));
  JAG_TRY(balloc(s, (void **)&s.E.tfill, sizeof(int32_t) * (size_t)n));
  JAG_TRY(balloc(s, (void **)&s.E.toff, sizeof(int64_t) * (size_t)n));
  JAG_TRY(balloc(s, (void **)&s.E.tlist, sizeof(int32_t) * (size_t)bcap * R));
  JAG_TRY(balloc(s, (void **)&s.E.srcbuf, sizeof(int32_t) * (size_t)bcap * R));
  JAG_TRY(balloc(s, (void **)&s.E.ctr, 256));
  JAG_TRY(balloc(s, (void **)&s.work, 256));
  JAG_TRY(balloc(s, (void **)&s.status, 256));
  JAG_TRY(balloc(s, (void **)&s.centroid, sizeof(double) * (size_t)B.ix.d));
  JAG_TRY(balloc(s, (void **)&s.best, 256));
  JAG_TRY(balloc(s, (void **)&s.biglist, sizeof(int32_t) * (size_t)bcap * R));
  s.gbytes = cand_bytes(cmax_g) * (size_t)s.prune_blocks * kPruneWarps;   // 160 KB a warp at least
  JAG_TRY(balloc(s, (void **)&s.gscratch, s.gbytes));
  JAG_TRY(cudaMemsetAsync(s.E.tcount, 0, sizeof(int32_t) * (size_t)n, B.stream));
  JAG_TRY(cudaMemsetAsync(s.E.tfill, 0, sizeof(int32_t) * (size_t)n, B.stream));
  JAG_TRY(cudaMemsetAsync(s.status, 0, 256, B.stream));
  JAG_TRY(cudaMemsetAsync(B.graph, 0xFF, sizeof(int32_t) * (size_t)n * R, B.stream));
  {
    Pct pct;
    for (int i = 0; i < 4; ++i) pct.v[i] = B.pct[i];
    const int64_t blocks = std::min<int64_t>((n + kThrWarps - 1) / kThrWarps, (int64_t)num_sms() * 8);
    if (B.weighted) {
      Mult mult;
      for (int i = 0; i < 8; ++i) mult.v[i] = B.mult[i];
      const int64_t Ss = std::max<int64_t>(1, std::min<int64_t>(n - 1, B.sample));
      const int64_t chunk = std::min<int64_t>(n, (int64_t)(s.gbytes / (size_t)(8 * Ss)));
      JAG_TRY(launch_weights(B, mult, reinterpret_cast<float *>(s.gscratch), chunk));
    } else {
      thresholds_kernel<<<(unsigned)blocks, kThrWarps * 32, 0, B.stream>>>(B.ix, B.sample, B.seed, B.nT, pct, B.thr);
    }
    JAG_TRY(cudaGetLastError());
    JAG_TRY(cudaFuncSetAttribute(centroid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCenSmem));
    centroid_kernel<<<(B.ix.d + 31) / 32, kCenThreads, kCenSmem, B.stream>>>(B.ix, s.centroid);
    JAG_TRY(cudaMemsetAsync(s.best, 0xFF, 16, B.stream));
    auto *dist = reinterpret_cast<unsigned long long *>(s.E.toff);   // free until the first batch
    medoid_kernel<<<(unsigned)((n + 255) / 256), 256, 0, B.stream>>>(B.ix, s.centroid, s.best, dist);
    medoid_id_kernel<<<(unsigned)((n + 255) / 256), 256, 0, B.stream>>>(n, s.best, dist);
    JAG_TRY(cudaGetLastError());
    unsigned long long best[2];
    JAG_TRY(cudaMemcpyAsync(best, s.best, 16, cudaMemcpyDeviceToHost, B.stream));
    JAG_TRY(cudaStreamSynchronize(B.stream));
    B.ix.entry = (int32_t)best[1];
    *entry_out = B.ix.entry;
  }
  {
    int64_t pos = 1, inserted = 1;
    while (pos < n) {
      int64_t nb = std::min<int64_t>(inserted, bcap);
      nb = std::min<int64_t>(nb, n - pos);
      JAG_TRY(cudaMemsetAsync(s.work, 0, 256, B.stream));
      JAG_TRY(cudaMemsetAsync(s.E.ctr, 0, 256, B.stream));
      switch (cap_list) {
        case 64: e = dispatch_build<64>(B, P, CPL, pos, nb, hbits, s, vcap, cmax_s, cmax_g); break;
        case 128: e = dispatch_build<128>(B, P, CPL, pos, nb, hbits, s, vcap, cmax_s, cmax_g); break;
        default: e = dispatch_build<256>(B, P, CPL, pos, nb, hbits, s, vcap, cmax_s, cmax_g); break;
      }
      if (e != cudaSuccess) goto fail;
      pos += nb;
      inserted += nb;
    }
    uint32_t status = 0;
    JAG_TRY(cudaMemcpyAsync(&status, s.status, 4, cudaMemcpyDeviceToHost, B.stream));
    JAG_TRY(cudaStreamSynchronize(B.stream));
    bfree(s);
    if (status & kErrVisitedOverflow) {
      snprintf(msg, msg_len, "build search visited more than %d vertices", vcap);
      return JAG_EUNSUPPORTED;
    }
    if (status & kErrCandOverflow) {
      snprintf(msg, msg_len, "back-edge candidates exceeded %d", cmax_g);
      return JAG_EUNSUPPORTED;
    }
    return JAG_OK;
  }
fail:
  cudaStreamSynchronize(B.stream);
  bfree(s);
  snprintf(msg, msg_len, "CUDA error in build: %s", cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? JAG_ENOMEM : JAG_ECUDA;
#undef JAG_TRY
}

}  // namespace jag
