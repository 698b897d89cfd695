// Training of the beam / stop network of the learned search policy: forward
// pass, back-propagation and Adam, all on the GPU.
//
// Network: 12 features -> 64 ReLU -> 64 ReLU -> nl + 1 outputs (nl logits
// over the beam ladder, one stop-hop output).  Loss of a batch of B rows:
// mean cross-entropy of the logits against the beam class plus lam * mean
// squared error of the stop output against its target.
//
// K_mlp1 (mlp_grad_kernel): one cluster of 8 CTAs per 64-row slice of the
//   batch.  A CTA runs 8 of the rows, one warp each, forward and backward with
//   the weights in its shared memory; then the cluster trades activations
//   through distributed shared memory and every CTA sums an eighth of the
//   parameters over the slice's 64 rows, in row order.  The chains of 64
//   dependent additions, not the arithmetic, set the time of a slice, so it is
//   spread over as many threads as it has chains.  With few slices the last
//   CTA to finish an eighth sums its partials over the slices, in order, and
//   applies Adam: one launch per mini-batch (a 512-row step: 82 us as one CTA
//   per slice and a second launch, 22 us so).
// K_mlp2 (mlp_reduce_kernel): the same sums over many slices, one thread per
//   parameter.  Either way the result does not depend on scheduling.
//
// The network is a few thousand parameters and trains offline; every sum keeps
// a fixed order.
#include <cooperative_groups.h>

#include <cmath>
#include <vector>

#include "launch.h"

namespace jag {

constexpr int kMlpRows = 64;       // rows per slice
constexpr int kMlpCtas = 8;        // CTAs per slice (a cluster)
constexpr int kMlpThreads = 256;
constexpr int kMlpOwn = kMlpRows / kMlpCtas;   // rows per CTA, one per warp
constexpr int kMlpFused = 64;      // slices up to which the last CTAs reduce
constexpr int kMaxLadder = 16;
constexpr int kF = JAG_MLP_FEATURES, kH = JAG_MLP_HIDDEN;
constexpr int kCols = kH / kMlpCtas;           // hidden units per CTA in the parameter sums
static_assert(kMlpOwn * 32 == kMlpThreads && kH == 64, "a warp per row, two hidden units per lane");

__host__ __device__ inline int64_t mlp_params(int nl) {
  return (int64_t)kH * kF + kH + kH * kH + kH + (int64_t)(nl + 1) * kH + (nl + 1);
}

// Shared memory of K_mlp1 (floats).  Weight rows are padded by one float, so
// that the lanes of a warp, one row each, read different banks.
struct MlpSmem {
  float *w1, *w2, *w3;                  // [64][kF + 1], [64][65], [no][65]
  float *b1, *b2, *b3;
  float *x, *a1, *a2, *d1, *d2, *z;     // the CTA's own rows: [8][kF], [8][64] x 4, [8][no]
  float *rl;                            // [8] row losses
  float *ga1, *gx, *gz;                 // the slice's rows: [64][64], [64][kF], [64][no]
  float *gd1, *gd2, *ga2;               // [64][kCols]: the CTA's hidden units
  __host__ __device__ static size_t carve(MlpSmem *s, float *p, int no) {
    float *const p0 = p;
    auto take = [&](size_t n) { float *r = p; p += n; return r; };
    s->w1 = take(kH * (kF + 1)); s->w2 = take(kH * (kH + 1)); s->w3 = take(no * (kH + 1));
    s->b1 = take(kH); s->b2 = take(kH); s->b3 = take(no);
    s->x = take(kMlpOwn * kF);
    s->a1 = take(kMlpOwn * kH); s->a2 = take(kMlpOwn * kH); s->d1 = take(kMlpOwn * kH); s->d2 = take(kMlpOwn * kH);
    s->z = take(kMlpOwn * no); s->rl = take(kMlpOwn);
    s->ga1 = take(kMlpRows * kH); s->gx = take(kMlpRows * kF); s->gz = take(kMlpRows * no);
    s->gd1 = take(kMlpRows * kCols); s->gd2 = take(kMlpRows * kCols); s->ga2 = take(kMlpRows * kCols);
    return (size_t)(p - p0);
  }
};

inline size_t mlp_smem_bytes(int nl) {
  MlpSmem s;
  return MlpSmem::carve(&s, nullptr, nl + 1) * sizeof(float);
}

// What a mini-batch's sums end in.
struct MlpUpdate {
  float *grad, *loss, *loss_acc;   // each may be NULL
  int adam;
  float *params, *am, *av;
  float lr, c1, c2;
};

// Parameter p from the slices' partials in slice order; with u.adam the Adam
// step theta -= lr * (m c1) / (sqrt(v c2) + eps) follows (c1, c2: the bias
// corrections 1 / (1 - beta^t)).
__device__ __forceinline__ void mlp_reduce_one(int64_t p, int64_t P, int nslices, const float *part,
                                               const MlpUpdate &u) {
  float g = 0.f;
#pragma unroll 8
  for (int b = 0; b < nslices; ++b) g += __ldcg(part + (int64_t)b * P + p);
  if (u.grad) u.grad[p] = g;
  if (u.adam) {
    const float m = 0.9f * u.am[p] + 0.1f * g;
    const float v = 0.999f * u.av[p] + 0.001f * g * g;
    u.am[p] = m;
    u.av[p] = v;
    u.params[p] -= u.lr * (m * u.c1) / (sqrtf(v * u.c2) + 1e-8f);
  }
}

__device__ __forceinline__ void mlp_reduce_loss(int nslices, const float *lpart, int64_t B, const MlpUpdate &u) {
  float l = 0.f;
  for (int b = 0; b < nslices; ++b) l += __ldcg(lpart + b);
  l /= (float)B;
  if (u.loss) *u.loss = l;
  if (u.loss_acc) *u.loss_acc += l;
}

// The parameters CTA `rank` of a cluster sums, e-th of mlp_share(no, rank):
// rows [8 rank, 8 rank + 8) of W2 and W1 with their biases, the same columns
// of W3, and b3 for rank 0.
__device__ __forceinline__ int mlp_share(int no, int rank) {
  return kCols * kH + kCols * kF + no * kCols + 2 * kCols + (rank == 0 ? no : 0);
}

__global__ void __cluster_dims__(kMlpCtas, 1, 1) __launch_bounds__(kMlpThreads)
mlp_grad_kernel(int nl, const float *params, const float *__restrict__ X, const int32_t *__restrict__ Y,
                const float *__restrict__ T, int64_t row0, int64_t B, float lam, int nslices, int fused, float *part,
                float *lpart, unsigned int *done, const MlpUpdate upd) {
  extern __shared__ __align__(16) float sm[];
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int no = nl + 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster.block_rank();
  const int64_t slice = blockIdx.x / kMlpCtas;
  const int64_t P = mlp_params(nl);
  const int64_t oW2 = (int64_t)kH * kF + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH, oB3 = oW3 + (int64_t)no * kH;
  MlpSmem s;
  MlpSmem::carve(&s, sm, no);
  const int64_t r0 = slice * kMlpRows;
  const int rows = (int)min64(kMlpRows, B - r0);
  const float inv_b = 1.f / (float)B;
  const int row = rank * kMlpOwn + warp;   // of the slice
  const bool live = row < rows;
  const int64_t g = row0 + r0 + row;
  {
    // every load leaves before the first value is stored
    constexpr int N1 = kH * kF / kMlpThreads, N2 = kH * kH / kMlpThreads, N3 = (kMaxLadder + 1) * kH / kMlpThreads + 1;
    float v1[N1], v2[N2], v3[N3];
    const float xv = live && lane < kF ? X[g * kF + lane] : 0.f;
    const float bv = tid < kH ? params[kH * kF + tid] : tid < 2 * kH ? params[oB2 + tid - kH]
                     : tid < 2 * kH + no ? params[oB3 + tid - 2 * kH] : 0.f;
#pragma unroll
    for (int i = 0; i < N2; ++i) v2[i] = params[oW2 + tid + i * kMlpThreads];
#pragma unroll
    for (int i = 0; i < N1; ++i) v1[i] = params[tid + i * kMlpThreads];
#pragma unroll
    for (int i = 0; i < N3; ++i) {
      const int e = tid + i * kMlpThreads;
      v3[i] = e < no * kH ? params[oW3 + e] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < N2; ++i) {
      const int e = tid + i * kMlpThreads;
      s.w2[(e / kH) * (kH + 1) + e % kH] = v2[i];
    }
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const int e = tid + i * kMlpThreads;
      s.w1[(e / kF) * (kF + 1) + e % kF] = v1[i];
    }
#pragma unroll
    for (int i = 0; i < N3; ++i) {
      const int e = tid + i * kMlpThreads;
      if (e < no * kH) s.w3[(e / kH) * (kH + 1) + e % kH] = v3[i];
    }
    if (tid < 2 * kH + no) (tid < kH ? s.b1[tid] : tid < 2 * kH ? s.b2[tid - kH] : s.b3[tid - 2 * kH]) = bv;
    if (live && lane < kF) s.x[warp * kF + lane] = xv;
  }
  __syncthreads();
  if (live) {
    // forward: lane j and j + 32 of each hidden layer
    const float *x = s.x + warp * kF;
    float *a1 = s.a1 + warp * kH, *a2 = s.a2 + warp * kH, *d1 = s.d1 + warp * kH, *d2 = s.d2 + warp * kH;
    float *z = s.z + warp * no;
    float p0 = s.b1[lane], p1 = s.b1[lane + 32];
#pragma unroll
    for (int i = 0; i < kF; ++i) {
      p0 = fmaf(s.w1[lane * (kF + 1) + i], x[i], p0);
      p1 = fmaf(s.w1[(lane + 32) * (kF + 1) + i], x[i], p1);
    }
    a1[lane] = p0;
    a1[lane + 32] = p1;
    __syncwarp();
    float q0 = s.b2[lane], q1 = s.b2[lane + 32];
#pragma unroll 16
    for (int i = 0; i < kH; ++i) {
      const float h = fmaxf(a1[i], 0.f);
      q0 = fmaf(s.w2[lane * (kH + 1) + i], h, q0);
      q1 = fmaf(s.w2[(lane + 32) * (kH + 1) + i], h, q1);
    }
    a2[lane] = q0;
    a2[lane + 32] = q1;
    __syncwarp();
    float o = -INFINITY;
    if (lane < no) {
      o = s.b3[lane];
#pragma unroll 16
      for (int i = 0; i < kH; ++i) o = fmaf(s.w3[lane * (kH + 1) + i], fmaxf(a2[i], 0.f), o);
    }
    // loss of the row and d loss / d z; the exponentials are summed in class order
    float mx = lane < nl ? o : -INFINITY;
#pragma unroll
    for (int k = 16; k >= 1; k >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, k));
    const float ex = lane < nl ? expf(o - mx) : 0.f;
    float se = 0.f;
    for (int c = 0; c < nl; ++c) se += __shfl_sync(kFull, ex, c);
    const float lse = mx + logf(se);
    const int y = Y[g];
    const bool yok = y >= 0 && y < nl;
    const float zy = __shfl_sync(kFull, o, yok ? y : 0), dz = __shfl_sync(kFull, o, nl) - T[g];
    if (lane == 0) s.rl[warp] = (yok ? lse - zy : NAN) + lam * dz * dz;
    if (lane < nl) z[lane] = (ex / se - (lane == y ? 1.f : 0.f)) * inv_b;
    if (lane == nl) z[lane] = 2.f * lam * dz * inv_b;
    __syncwarp();
    // d loss / d a2 and d loss / d a1
    float e0 = 0.f, e1 = 0.f;
    for (int c = 0; c < no; ++c) {
      e0 = fmaf(z[c], s.w3[c * (kH + 1) + lane], e0);
      e1 = fmaf(z[c], s.w3[c * (kH + 1) + lane + 32], e1);
    }
    d2[lane] = q0 > 0.f ? e0 : 0.f;
    d2[lane + 32] = q1 > 0.f ? e1 : 0.f;
    __syncwarp();
    float f0 = 0.f, f1 = 0.f;
#pragma unroll 16
    for (int j = 0; j < kH; ++j) {
      f0 = fmaf(d2[j], s.w2[j * (kH + 1) + lane], f0);
      f1 = fmaf(d2[j], s.w2[j * (kH + 1) + lane + 32], f1);
    }
    d1[lane] = p0 > 0.f ? f0 : 0.f;
    d1[lane + 32] = p1 > 0.f ? f1 : 0.f;
  }
  cluster.sync();   // every row of the slice is done, and every CTA of the cluster has read the weights
  // the slice's activations that this CTA's parameters need
  // (row 8 k + warp is row `warp` of CTA k; four rows' loads in flight at once)
#pragma unroll
  for (int k0 = 0; k0 < kMlpCtas; k0 += 4) {
    float va[4], vb[4], vx[4], vz[4], v1[4], v2[4], v3[4];
    const int at = warp * kH + rank * kCols + (lane & (kCols - 1));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float *a1 = cluster.map_shared_rank(s.a1, k0 + k) + warp * kH;
      va[k] = a1[lane];
      vb[k] = a1[lane + 32];
      vx[k] = cluster.map_shared_rank(s.x, k0 + k)[warp * kF + (lane < kF ? lane : 0)];
      vz[k] = cluster.map_shared_rank(s.z, k0 + k)[warp * no + (lane < no ? lane : 0)];
      v1[k] = cluster.map_shared_rank(s.d1, k0 + k)[at];
      v2[k] = cluster.map_shared_rank(s.d2, k0 + k)[at];
      v3[k] = cluster.map_shared_rank(s.a2, k0 + k)[at];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = (k0 + k) * kMlpOwn + warp;   // rows past the batch are copied too and never read
      s.ga1[r * kH + lane] = fmaxf(va[k], 0.f);
      s.ga1[r * kH + lane + 32] = fmaxf(vb[k], 0.f);
      if (lane < kF) s.gx[r * kF + lane] = vx[k];
      if (lane < no) s.gz[r * no + lane] = vz[k];
      if (lane < kCols) {
        s.gd1[r * kCols + lane] = v1[k];
        s.gd2[r * kCols + lane] = v2[k];
        s.ga2[r * kCols + lane] = fmaxf(v3[k], 0.f);
      }
    }
  }
  if (rank == 0 && tid == 0) {
    float l = 0.f;
    for (int r = 0; r < rows; ++r) l += cluster.map_shared_rank(s.rl, r / kMlpOwn)[r % kMlpOwn];
    lpart[slice] = l;
  }
  cluster.sync();   // no CTA leaves (or reuses its rows) while another reads them
  // partial gradient of the CTA's parameters over the slice's rows, in order
  const int share = mlp_share(no, rank);
  auto param = [&](int e, int *i, int *k) -> int64_t {   // e-th parameter; the indices of its two factors
    if (e < kCols * kH) { *i = e / kH; *k = e % kH; return oW2 + (int64_t)(rank * kCols + *i) * kH + *k; }
    e -= kCols * kH;
    if (e < kCols * kF) { *i = e / kF; *k = e % kF; return (int64_t)(rank * kCols + *i) * kF + *k; }
    e -= kCols * kF;
    if (e < no * kCols) { *i = e / kCols; *k = e % kCols; return oW3 + (int64_t)*i * kH + rank * kCols + *k; }
    e -= no * kCols;
    if (e < kCols) { *i = e; *k = -1; return (int64_t)kH * kF + rank * kCols + e; }
    e -= kCols;
    if (e < kCols) { *i = e; *k = -2; return oB2 + rank * kCols + e; }
    *i = e - kCols; *k = -3;
    return oB3 + *i;
  };
  float *out = part + slice * P;
  for (int e = tid; e < share; e += kMlpThreads) {
    int i, k;
    const int64_t p = param(e, &i, &k);
    const float *u, *v = nullptr;
    int su, sv = 0;
    if (e < kCols * kH) { u = s.gd2 + i; su = kCols; v = s.ga1 + k; sv = kH; }
    else if (e < kCols * (kH + kF)) { u = s.gd1 + i; su = kCols; v = s.gx + k; sv = kF; }
    else if (e < kCols * (kH + kF + no)) { u = s.gz + i; su = no; v = s.ga2 + k; sv = kCols; }
    else { u = k == -1 ? s.gd1 + i : k == -2 ? s.gd2 + i : s.gz + i; su = k == -3 ? no : kCols; }
    float acc = 0.f;
    if (v) {
#pragma unroll 8
      for (int r = 0; r < rows; ++r) acc = fmaf(u[r * su], v[r * sv], acc);
    } else {
      for (int r = 0; r < rows; ++r) acc += u[r * su];
    }
    out[p] = acc;
  }
  if (!fused) return;
  // the last slice to finish this eighth reduces it (the parameters may change
  // now: a CTA counts itself only after its whole cluster has read them)
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    last = atomicAdd(done + rank, 1u) == (unsigned)nslices - 1u;
    if (last) done[rank] = 0u;   // for the next mini-batch
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  for (int e = tid; e < share; e += kMlpThreads) {
    int i, k;
    mlp_reduce_one(param(e, &i, &k), P, nslices, part, upd);
  }
  if (rank == 0 && tid == 0) mlp_reduce_loss(nslices, lpart, B, upd);
}

__global__ void __launch_bounds__(256)
mlp_reduce_kernel(int64_t P, int nslices, const float *part, const float *lpart, int64_t B, const MlpUpdate upd) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p == 0) mlp_reduce_loss(nslices, lpart, B, upd);
  if (p < P) mlp_reduce_one(p, P, nslices, part, upd);
}

__global__ void mlp_export_kernel(int64_t nw, int nl, const float *params, uint16_t *w, float *b) {
  const int no = nl + 1;
  const int64_t n1 = (int64_t)kH * kF, n2 = (int64_t)kH * kH;
  const int64_t nb = 2 * kH + no;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nw + nb; i += (int64_t)gridDim.x * blockDim.x) {
    if (i < nw) {
      // weight i of W1 | W2 | W3 -> its place in the flat parameter vector
      const int64_t src = i < n1 ? i : i < n1 + n2 ? i + kH : i + 2 * kH;
      w[i] = __bfloat16_as_ushort(__float2bfloat16_rn(params[src]));
    } else {
      const int64_t j = i - nw;
      const int64_t src = j < kH ? n1 + j : j < 2 * kH ? n1 + kH + n2 + (j - kH) : n1 + 2 * kH + n2 + no * kH + (j - 2 * kH);
      b[j] = params[src];
    }
  }
}

// Device scratch of a call: partial gradients and losses of ns slices, the
// cluster counters (zero before the first batch), and `extra` floats.
struct MlpScratch {
  float *part, *lpart, *extra;
  unsigned int *done;
  static size_t bytes(int64_t ns, int64_t P, int64_t extra) {
    return (size_t)(ns * P + ns + kMlpCtas + extra) * sizeof(float);
  }
  MlpScratch(void *buf, int64_t ns, int64_t P) {
    part = (float *)buf;
    lpart = part + ns * P;
    done = (unsigned int *)(lpart + ns);
    extra = lpart + ns + kMlpCtas;
  }
};

// One batch (rows [row0, row0 + B)).
static cudaError_t mlp_batch(int nl, const float *params, const float *X, const int32_t *y, const float *t,
                             int64_t row0, int64_t B, float lam, const MlpScratch &w, const MlpUpdate &upd,
                             cudaStream_t st) {
  const int64_t P = mlp_params(nl);
  const int ns = (int)((B + kMlpRows - 1) / kMlpRows);
  const int fused = ns <= kMlpFused;
  mlp_grad_kernel<<<(unsigned)ns * kMlpCtas, kMlpThreads, mlp_smem_bytes(nl), st>>>(
      nl, params, X, y, t, row0, B, lam, ns, fused, w.part, w.lpart, w.done, upd);
  if (!fused)
    mlp_reduce_kernel<<<(unsigned)((P + 255) / 256), 256, 0, st>>>(P, ns, w.part, w.lpart, B, upd);
  return cudaGetLastError();
}

// The kernel's shared-memory limit, which the whole process shares, is set to
// what the longest ladder takes: a call with another ladder, from another
// thread, must not lower it before this one's launches.
static jag_status mlp_setup() {
  const size_t smem = mlp_smem_bytes(kMaxLadder);
  if (cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return set_error(JAG_ECUDA, "cannot reserve shared memory for the network kernels");
  return JAG_OK;
}

}  // namespace jag

using namespace jag;

extern "C" JAG_API jag_status jag_mlp_loss_grad(int32_t n_ladder, const float *params, const float *X,
                                                const int32_t *y, const float *t, int64_t m, float lam,
                                                float *grad, float *loss, void *stream) {
  if (n_ladder < 1 || n_ladder > kMaxLadder) return set_error(JAG_EINVAL, "n_ladder must be in [1, 16]");
  if (!params || !X || !y || !t || !grad || !loss) return set_error(JAG_EINVAL, "NULL argument");
  if (m < 1) return set_error(JAG_EINVAL, "m must be >= 1");
  if (!(lam >= 0.f) || !std::isfinite(lam)) return set_error(JAG_EINVAL, "lam must be finite and >= 0");
  if (jag_status s = mlp_setup()) return s;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t P = mlp_params(n_ladder);
  const int64_t ns = (m + kMlpRows - 1) / kMlpRows;
  void *buf = nullptr;
  if (cudaMallocAsync(&buf, MlpScratch::bytes(ns, P, 0), st) != cudaSuccess)
    return set_error(JAG_ENOMEM, "cannot allocate the gradient partials");
  const MlpScratch w(buf, ns, P);
  MlpUpdate upd{};
  upd.grad = grad;
  upd.loss = loss;
  cudaError_t e = cudaMemsetAsync(w.done, 0, kMlpCtas * sizeof(unsigned int), st);
  if (e == cudaSuccess) e = mlp_batch(n_ladder, params, X, y, t, 0, m, lam, w, upd, st);
  cudaFreeAsync(buf, st);
  if (e != cudaSuccess) return set_error(JAG_ECUDA, cudaGetErrorString(e));
  return JAG_OK;
}

extern "C" JAG_API jag_status jag_mlp_train(int32_t n_ladder, float *params, float *adam_m, float *adam_v,
                                            int64_t *adam_step, const float *X, const int32_t *y, const float *t,
                                            int64_t m, int32_t epochs, int32_t batch, float lr, float lam,
                                            float *loss_trace, void *stream) {
  if (n_ladder < 1 || n_ladder > kMaxLadder) return set_error(JAG_EINVAL, "n_ladder must be in [1, 16]");
  if (!params || !adam_m || !adam_v || !adam_step || !X || !y || !t) return set_error(JAG_EINVAL, "NULL argument");
  if (m < 1 || epochs < 0 || batch < 1) return set_error(JAG_EINVAL, "m, batch must be >= 1 and epochs >= 0");
  if (!(lam >= 0.f) || !std::isfinite(lam) || !(lr > 0.f) || !std::isfinite(lr))
    return set_error(JAG_EINVAL, "lr must be > 0 and lam >= 0, both finite");
  if (*adam_step < 0) return set_error(JAG_EINVAL, "adam_step must be >= 0");
  if (jag_status s = mlp_setup()) return s;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t P = mlp_params(n_ladder);
  const int64_t B = batch < m ? batch : m;
  const int64_t ns = (B + kMlpRows - 1) / kMlpRows;
  const int64_t nb = (m + B - 1) / B;
  void *buf = nullptr;
  const int64_t nacc = epochs > 0 ? epochs : 1;
  if (cudaMallocAsync(&buf, MlpScratch::bytes(ns, P, nacc), st) != cudaSuccess)
    return set_error(JAG_ENOMEM, "cannot allocate the training scratch");
  const MlpScratch w(buf, ns, P);
  float *acc = w.extra;
  MlpUpdate upd{};
  upd.adam = 1;
  upd.params = params;
  upd.am = adam_m;
  upd.av = adam_v;
  upd.lr = lr;
  cudaError_t e = cudaMemsetAsync(w.done, 0, sizeof(float) * (size_t)(kMlpCtas + nacc), st);   // counters and acc
  int64_t step = *adam_step;
  for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
    for (int64_t b = 0; b < nb && e == cudaSuccess; ++b) {
      const int64_t row0 = b * B, rows = row0 + B <= m ? B : m - row0;
      ++step;
      upd.c1 = (float)(1.0 / (1.0 - std::pow(0.9, (double)step)));
      upd.c2 = (float)(1.0 / (1.0 - std::pow(0.999, (double)step)));
      upd.loss_acc = acc + ep;
      e = mlp_batch(n_ladder, params, X, y, t, row0, rows, lam, w, upd, st);
    }
  }
  std::vector<float> tr((size_t)(epochs > 0 ? epochs : 1));
  if (e == cudaSuccess && loss_trace && epochs > 0)
    e = cudaMemcpyAsync(tr.data(), acc, sizeof(float) * (size_t)epochs, cudaMemcpyDeviceToHost, st);
  cudaFreeAsync(buf, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return set_error(JAG_ECUDA, cudaGetErrorString(e));
  if (loss_trace)
    for (int ep = 0; ep < epochs; ++ep) loss_trace[ep] = tr[(size_t)ep] / (float)nb;
  *adam_step = step;
  return JAG_OK;
}

extern "C" JAG_API jag_status jag_mlp_export(int32_t n_ladder, const float *params, uint16_t *w_bf16, float *b_f32,
                                             void *stream) {
  if (n_ladder < 1 || n_ladder > kMaxLadder) return set_error(JAG_EINVAL, "n_ladder must be in [1, 16]");
  if (!params || !w_bf16 || !b_f32) return set_error(JAG_EINVAL, "NULL argument");
  const int64_t nw = (int64_t)kH * kF + (int64_t)kH * kH + (int64_t)(n_ladder + 1) * kH;
  mlp_export_kernel<<<32, 256, 0, (cudaStream_t)stream>>>(nw, n_ladder, params, w_bf16, b_f32);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return set_error(JAG_ECUDA, cudaGetErrorString(e));
  return JAG_OK;
}
