// K1t: GreedySearch (Algorithm 1) with several warps per query.
//
// One CTA owns one search; L, the visited set and a hop's candidates are in
// its shared memory.  A hop is a chain of dependent steps (out-list, visited
// test, rows, distances, merge) that one warp runs in about 860 instructions
// and two memory latencies.  Here TM warps share the steps of a hop:
//   A  warp 0 (and 1 when R > 32): the out-list of the expanded vertex, first
//      keys, early rejection, visited test, compaction; meanwhile every
//      thread reads the EPT entries of L that it owns;
//   B  the candidates' distances, split over the warps; each candidate's rank
//      in L by two ballots (the last key of 32 equal parts of L, then 32
//      consecutive entries), which also finds a repeat;
//   C  merge: an entry moves by the number of candidates whose rank is at or
//      before it, straight to its new position (every read of L happened
//      before the barrier that ended B).  The next vertex to expand is the
//      lower of the smallest rank and the next unexpanded entry.
// TS more warps work one hop ahead: they take the next unexpanded entry of L,
// the next vertex in about 85 % of hops, and compute the distances of its
// neighbours that are not yet visited (its out-list they loaded a hop
// earlier, when it was the entry after the next); so on a hit step A finds
// the candidates' keys in shared memory and step B reads no rows.  A
// neighbour they reject (visited, or a first key past L's last) would be
// rejected later too: visited ids are in L or left it for good, and L's last
// key only decreases.  So the hops, the list and the answers are those of
// greedy_search.
#pragma once

#include <algorithm>

#include "launch.h"
#include "launch_util.cuh"
#include "search_core.cuh"

namespace jag {

// Shared memory of one team search.  The keys and ranks of a hop's
// candidates are padded with kNoKey / kNoRank to a multiple of four.
constexpr int kNoRank = 0x7FFFFFFF;
struct TeamSmem {
  uint64_t *bkey;    // [cap] keys of L
  uint64_t *ckey;    // [64] keys of the candidates (kNoKey: dropped)
  uint32_t *bid;     // [cap] ids of L, bit 31 = expanded
  uint32_t *cid;     // [64] candidate ids of the hop
  uint32_t *ck1;     // [64] their first keys
  int32_t *crk;      // [64] their ranks in L
  int32_t *sp_u;     // [2][64] out-list of the predicted vertex (-1: none or rejected)
  uint32_t *sp_k1;   // [2][64] first keys
  float *sp_d;       // [2][64] distances
  uint64_t *nx_w;    // [2][64] attribute words and
  int32_t *nx_u;     // [2][64] out-list of the vertex after the predicted one
  uint32_t *scid;    // [4][32] rows of a look-ahead warp
  uint32_t *ctl;     // [kTcWords] control words, see below
  uint32_t *hash;    // [1 << hbits] visited set
};

enum TeamCtl { kTcCount = 0, kTcNext = 1, kTcSel = 2, kTcCnt = 3, kTcQuery = 6 /* and 7 */, kTcLs = 8,
               kTcLim = 9, kTcWords = 16 };

__host__ __device__ inline size_t team_smem_bytes(int cap, int hbits) {
  return (size_t)cap * 12 + 64 * 8 + 64 * 2 * 8 + (64 * 3 + 128 * 4 + 4 * 32 + kTcWords) * 4 + ((size_t)4 << hbits);
}

__device__ inline TeamSmem carve_team_smem(uint8_t *base, int cap) {
  TeamSmem s;
  s.bkey = reinterpret_cast<uint64_t *>(base);
  s.ckey = s.bkey + cap;
  s.nx_w = s.ckey + 64;
  s.bid = reinterpret_cast<uint32_t *>(s.nx_w + 128);
  s.cid = s.bid + cap;
  s.ck1 = s.cid + 64;
  s.crk = reinterpret_cast<int32_t *>(s.ck1 + 64);
  s.sp_u = s.crk + 64;
  s.sp_k1 = reinterpret_cast<uint32_t *>(s.sp_u + 128);
  s.sp_d = reinterpret_cast<float *>(s.sp_k1 + 128);
  s.nx_u = reinterpret_cast<int32_t *>(s.sp_d + 128);
  s.scid = reinterpret_cast<uint32_t *>(s.nx_u + 128);
  s.ctl = s.scid + 4 * 32;
  s.hash = s.ctl + kTcWords;
  return s;
}

template <int N>
__device__ __forceinline__ void bar_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
}
template <int N>
__device__ __forceinline__ void bar_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(N) : "memory");
}

// Visited-set probe with one atomic: both slots are read first, then the id
// goes to the first empty one, or replaces the first slot's id.  An id that
// another lane's exchange overwrites is forgotten, which only costs a
// recomputed distance; the same id from another lane of this warp is caught,
// since both choose the same slot.
__device__ __forceinline__ bool team_visit(uint32_t *tab, int hbits, uint32_t id, bool cand) {
  const uint32_t mask = (1u << hbits) - 1;
  const uint32_t h = (id * 0x9E3779B1u) >> (32 - hbits), h2 = (h + 1) & mask;
  const uint32_t a = *(volatile uint32_t *)&tab[h], b = *(volatile uint32_t *)&tab[h2];
  bool fresh = cand & (a != id) & (b != id);
  if (fresh) fresh = atomicExch(&tab[(a != kEmptySlot) & (b == kEmptySlot) ? h2 : h], id) != id;
  return fresh;
}

__device__ __forceinline__ bool team_visited(const uint32_t *tab, int hbits, uint32_t id) {
  const uint32_t mask = (1u << hbits) - 1;
  const uint32_t h = (id * 0x9E3779B1u) >> (32 - hbits);
  return (*(const volatile uint32_t *)&tab[h] == id) | (*(const volatile uint32_t *)&tab[(h + 1) & mask] == id);
}

// One batch of candidate_distances in two halves: the chunks of the rows of
// candidates c0 + s * stride + grp (s < U, below c1), and their sums: lane
// s * VPW + g returns the distance of candidate c0 + s * stride + g.
template <int P, int CPL, int U, int FMT>
struct RowBatch {
  uint4 xv[U][CPL];
  float sc[U];
  __device__ __forceinline__ void load(const DevIndex &ix, const uint32_t *cid, int c0, int stride, int c1) {
    const int lane = threadIdx.x & 31, grp = lane / P, lig = lane % P;
    const int nch = FMT == JAG_VEC_F32 ? ix.nchunks : ix.qchunks;
#pragma unroll
    for (int s = 0; s < U; ++s) {
      const int c = c0 + s * stride + grp;
      const bool ok = c < c1;
      const uint32_t id = ok ? cid[c] : 0u;
      const uint8_t *row = static_cast<const uint8_t *>(row_address<FMT>(ix, id));
      sc[s] = 1.f;
      if (FMT == JAG_VEC_FP8) sc[s] = ok ? __ldg(ix.qscale + id) : 1.f;
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        const int ch = lig + j * P;
        xv[s][j] = (ok && ch < nch) ? ld_chunk_u4(row + ch * 16) : make_uint4(0, 0, 0, 0);
      }
    }
  }
  __device__ __forceinline__ float reduce(const QChunks<CPL, FMT> &q) {
    constexpr int VPW = 32 / P;
    constexpr int F = 32 / P;
    constexpr int NA = CPL < F ? CPL : F;
    const int lane = threadIdx.x & 31;
    float acc[U];
#pragma unroll
    for (int s = 0; s < U; ++s) {
      float a[NA];
#pragma unroll
      for (int i = 0; i < NA; ++i) a[i] = 0.f;
#pragma unroll
      for (int j = 0; j < CPL; ++j) a[j % F] = chunk_acc<FMT>(a[j % F], q.v[j], xv[s][j], sc[s]);
#pragma unroll
      for (int h = F / 2; h >= 1; h >>= 1) {
#pragma unroll
        for (int i = 0; i < h; ++i)
          if (i + h < NA) a[i] = __fadd_rn(a[i], a[i + h]);
      }
      acc[s] = a[0];
    }
    const float tot = group_reduce_spread<P, U>(acc);
    const bool mine = lane < VPW * U;
    return __shfl_sync(kFull, tot, mine ? spread_source<P, U>(lane / VPW, lane % VPW) : 0);
  }
};

// Where a team search stands between two calls.
struct TeamCursor {
  int cnt, sel;
};

// Algorithm 1 for one search by the calling CTA of TM + TS warps (every
// thread calls it; the count of L is returned to all).  Stops before a hop
// once st.hops >= max_hops; cur->cnt > 0 on entry resumes such a search with
// L as it stands (the caller may have shortened it).  Only st.hops is counted.
template <int EPT, int TM, int TS, int P, int CPL, int FMT>
__device__ __forceinline__ int team_search(const DevIndex &ix, const QueryKey &key1, const QChunks<CPL, FMT> &q, int ls,
                                           int hbits, const TeamSmem &S, SearchStats &st, int max_hops,
                                           TeamCursor *cur) {
  static_assert(TM >= 2 && TS * 16 == 64, "R <= 64 edges: 32 per warp in step A, 16 per look-ahead warp");
  constexpr int VPW = 32 / P;
  constexpr int NT = 32 * (TM + TS);
  // rows in flight per lane when one per lane does not cover the candidates
  constexpr int UB = CPL <= 2 ? 2 : 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int cnt = 1, sel = 0;
  if (cur->cnt > 0) {
    cnt = cur->cnt;
    sel = cur->sel;
  } else {
    const uint32_t hsize = 1u << hbits;
    for (uint32_t i = tid; i < hsize; i += NT) S.hash[i] = kEmptySlot;
    const uint32_t s = (uint32_t)ix.entry;
    if (tid == 0) {
      S.cid[0] = s;
      S.ctl[kTcCount] = 0u;
    }
    __syncthreads();
    if (warp == 0) {
      RowBatch<P, CPL, 1, FMT> rb;
      rb.load(ix, S.cid, 0, 0, 1);
      const uint32_t k0 = key1(ix, s);
      const float d0 = rb.reduce(q);
      if (lane == 0) {
        S.hash[(s * 0x9E3779B1u) >> (32 - hbits)] = s;
        S.bkey[0] = key1.key(k0, d0);
        S.bid[0] = s;
      }
    }
    __syncthreads();
    st.hops = 0;
  }
  int par = 0;
  if (warp >= TM) {
    // ---- one hop ahead ----
    const int sw = warp - TM, r = lane * TS + sw;   // neighbours spread over the warps: survivors cluster
    uint32_t nv = kEmptySlot;   // the vertex whose edges are in nx_u, nx_w (of the current parity)
    while (sel < cnt && st.hops < max_hops) {
      st.hops += 1;
      const bool full = cnt == ls;
      const uint32_t tail1 = full ? (uint32_t)(S.bkey[ls - 1] >> 32) : 0xFFFFFFFFu;
      // the first two unexpanded entries after sel: the predicted vertex v
      // and the one after it
      int nx = kNoRank;
      uint32_t v = kEmptySlot, v2 = kEmptySlot;
      for (int b = sel + 1; b < cnt; b += 32) {
        const uint32_t un = __ballot_sync(kFull, b + lane < cnt && !(S.bid[b + lane] & kExpanded));
        if (un) {
          const uint32_t un2 = un & (un - 1);
          nx = b + __ffs(un) - 1;
          v = S.bid[nx];
          if (un2) v2 = S.bid[b + __ffs(un2) - 1];
          break;
        }
      }
      if (sw == 0 && lane == 0) S.ctl[kTcNext] = (uint32_t)nx;
      bar_arrive<NT>(1);
      par ^= 1;
      const bool slot = lane < 16 && r < ix.R;
      if (v == kEmptySlot) {
        nv = kEmptySlot;
      } else {
        int u = -1;
        uint64_t aw = 0;
        asm volatile("cp.async.wait_all;" ::: "memory");   // each lane reads what it copied itself
        if (slot) {
          if (v == nv) {
            u = S.nx_u[(par ^ 1) * 64 + r];
            aw = S.nx_w[(par ^ 1) * 64 + r];
          } else {
            const int64_t e = (int64_t)v * ix.R + r;
            u = __ldg(ix.graph + e);
            aw = key1.edge_word(ix, e);
          }
        }
        // v2's edges for the next hop, straight to shared memory
        nv = v2;
        if (slot && v2 != kEmptySlot) {
          const int64_t e = (int64_t)v2 * ix.R + r;
          cp_async<4>(S.nx_u + par * 64 + r, ix.graph + e);
          key1.copy_edge_word(ix, e, S.nx_w + par * 64 + r);
        }
        bool cand = u >= 0;
        const uint32_t k1 = key1.from_word(aw);
        cand = cand & !(full & (k1 > tail1));
        if (cand) cand = !team_visited(S.hash, hbits, (uint32_t)u);
        const uint32_t km = __ballot_sync(kFull, cand);
        const int nc = __popc(km);
        uint32_t *cid = S.scid + sw * 32;
        const int pos = __popc(km & lanemask_lt());
        if (cand) cid[pos] = (uint32_t)u;
        __syncwarp();
        float dist = 0.f;
        if (nc <= VPW) {
          if (nc > 0) {
            RowBatch<P, CPL, 1, FMT> rb;
            rb.load(ix, cid, 0, VPW, nc);
            dist = __shfl_sync(kFull, rb.reduce(q), pos & 31);
          }
        } else {
          for (int b = 0; b < nc; b += VPW * UB) {
            RowBatch<P, CPL, UB, FMT> rb;
            rb.load(ix, cid, b, VPW, nc);
            const float mine = __shfl_sync(kFull, rb.reduce(q), (pos - b) & 31);
            if (pos >= b && pos < b + VPW * UB) dist = mine;
          }
        }
        if (slot) {
          S.sp_u[par * 64 + r] = cand ? u : -1;
          S.sp_k1[par * 64 + r] = k1;
          S.sp_d[par * 64 + r] = dist;
        }
      }
      __syncthreads();
      sel = (int)S.ctl[kTcSel];
      cnt = (int)S.ctl[kTcCnt];
    }
  } else {
    const int G = list_slots(ls) >> 5;   // entries per part of L in the rank search
    bool hit = false;                    // the look-ahead warps have the vertex at sel
    while (sel < cnt && st.hops < max_hops) {
      st.hops += 1;
      // ---- A ----
      if (32 * warp < ix.R) {
        const bool full = cnt == ls;
        const uint64_t tkey = full ? S.bkey[ls - 1] : kNoKey;
        const int r = 32 * warp + lane;
        const bool slot = r < ix.R;
        int u = -1;
        uint32_t k1 = 0;
        float d = 0.f;
        if (hit) {
          if (slot) {
            u = S.sp_u[par * 64 + r];
            k1 = S.sp_k1[par * 64 + r];
            d = S.sp_d[par * 64 + r];
          }
        } else {
          const int64_t e = (int64_t)(S.bid[sel] & ~kExpanded) * ix.R + r;
          uint64_t aw = 0;
          if (slot) {
            u = __ldg(ix.graph + e);
            aw = key1.edge_word(ix, e);
          }
          k1 = key1.from_word(aw);
        }
        const bool cand = (u >= 0) & !(full & (k1 > (uint32_t)(tkey >> 32)));
        bool keep = team_visit(S.hash, hbits, (uint32_t)u, cand);
        uint64_t key = kNoKey;
        if (hit) {   // its key is known: drop it here if it follows L's last entry
          key = key1.key(k1, d);
          keep = keep & (key <= tkey);
        }
        const uint32_t km = __ballot_sync(kFull, keep);
        uint32_t base = 0;
        if (ix.R > 32) {   // two parts share the list of candidates
          if (lane == 0) base = atomicAdd(&S.ctl[kTcCount], (uint32_t)__popc(km));
          base = __shfl_sync(kFull, base, 0);
        } else if (lane == 0) {
          S.ctl[kTcCount] = (uint32_t)__popc(km);
        }
        if (keep) {
          const int pos = base + __popc(km & lanemask_lt());
          S.cid[pos] = (uint32_t)u;
          S.ck1[pos] = k1;
          S.ckey[pos] = key;
        }
      }
      uint64_t ek[EPT];
      uint32_t ef[EPT];
#pragma unroll
      for (int e = 0; e < EPT; ++e) {
        const int j = (e * TM + warp) * 32 + lane;
        ek[e] = 0;
        ef[e] = 0;
        if (j < cnt) {
          ek[e] = S.bkey[j];
          ef[e] = S.bid[j];
        }
        if (j == sel) ef[e] |= kExpanded;
      }
      bar_sync<NT>(1);
      const bool ahead = hit;   // this hop's keys are known
      const int nc = (int)S.ctl[kTcCount], nx = (int)S.ctl[kTcNext];
      int uns = nx;   // first unexpanded position of L
      hit = nx != kNoRank;
      int c0 = 0;
      do {
        // ---- B ----
        const int c1 = min(nc, c0 + 32), m = c1 - c0;
        if (c0 > 0) {   // a second round of the same hop: L has changed
#pragma unroll
          for (int e = 0; e < EPT; ++e) {
            const int j = (e * TM + warp) * 32 + lane;
            if (j < cnt) {
              ek[e] = S.bkey[j];
              ef[e] = S.bid[j];
            }
          }
        }
        // rank of candidate c = (kc, ic) in L; kNoRank if L holds it already
        // (the visited set had forgotten it) or an earlier candidate of the
        // round is the same vertex (an uploaded out-list may repeat one)
        auto rank_of = [&](int c, uint64_t kc, uint32_t ic) -> int {
          const bool twin = c0 + lane < c && S.cid[c0 + lane] == ic;
          const int j1 = lane * G + G - 1;
          const bool l1 = j1 < cnt && S.bkey[j1] < kc;
          int base = __popc(__ballot_sync(kFull, l1)) * G;
          for (;;) {
            const int j2 = base + lane;
            const uint64_t k2 = j2 < cnt ? S.bkey[j2] : kNoKey;
            const uint32_t i2 = j2 < cnt ? (S.bid[j2] & ~kExpanded) : kEmptySlot;
            const uint32_t lm = __ballot_sync(kFull, key_less(k2, i2, kc, ic));
            if (__any_sync(kFull, twin | ((k2 == kc) & (i2 == ic)))) return kNoRank;
            if (lm != kFull) return base + __popc(lm);
            base += 32;
          }
        };
        if (ahead) {
          for (int c = c0 + warp; c < c1; c += TM) {
            const int rank = rank_of(c, S.ckey[c], S.cid[c]);
            if (lane == 0) {
              S.crk[c] = rank;
              if (rank == kNoRank) S.ckey[c] = kNoKey;
            }
          }
        } else {
          const bool full = cnt == ls;
          const uint64_t tkey = full ? S.bkey[ls - 1] : kNoKey;
          // key and rank of candidate c (lanes with `mine`), whose distance the lane holds
          auto place = [&](int c, bool mine, float dist) {
            uint64_t ck = kNoKey;
            uint32_t cv = 0;
            int rank = kNoRank;
            if (mine) {
              cv = S.cid[c];
              ck = key1.key(S.ck1[c], dist);
              if (ck > tkey) ck = kNoKey;
            }
            for (uint32_t w = __ballot_sync(kFull, ck != kNoKey); w; w &= w - 1) {
              const int src = __ffs(w) - 1;
              const int rk = rank_of(__shfl_sync(kFull, c, src), __shfl_sync(kFull, ck, src), __shfl_sync(kFull, cv, src));
              if (lane == src) rank = rk;
            }
            if (mine) {
              S.ckey[c] = rank == kNoRank ? kNoKey : ck;
              S.crk[c] = rank;
            }
          };
          if (m <= TM * VPW) {
            if (warp * VPW < m) {
              RowBatch<P, CPL, 1, FMT> rb;
              rb.load(ix, S.cid, c0 + warp * VPW, 0, c1);
              const int c = c0 + warp * VPW + lane;
              place(c, lane < VPW && c < c1, rb.reduce(q));
            }
          } else {
            for (int b = c0 + warp * VPW; b < c1; b += TM * VPW * UB) {
              RowBatch<P, CPL, UB, FMT> rb;
              rb.load(ix, S.cid, b, TM * VPW, c1);
              const int c = b + (lane / VPW) * (TM * VPW) + lane % VPW;
              place(c, lane < VPW * UB && c < c1, rb.reduce(q));
            }
          }
        }
        if (warp == TM - 1 && (m & 3) && lane >= (m & 3) && lane < 4) {   // pad to whole groups of four
          S.ckey[c0 + (m & ~3) + lane] = kNoKey;
          S.crk[c0 + (m & ~3) + lane] = kNoRank;
        }
        bar_sync<32 * TM>(2);
        // ---- C ----
        if (tid == 0) S.ctl[kTcCount] = 0u;
        const int rk = lane < m ? S.crk[c0 + lane] : kNoRank;
        const uint32_t vm = __ballot_sync(kFull, rk != kNoRank);
        int sh[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) sh[e] = 0;
        for (int c = c0; c < c1; c += 4) {
          const int4 r = *reinterpret_cast<const int4 *>(S.crk + c);
#pragma unroll
          for (int e = 0; e < EPT; ++e) {
            const int j = (e * TM + warp) * 32 + lane;
            sh[e] += (r.x <= j) + (r.y <= j) + (r.z <= j) + (r.w <= j);
          }
        }
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          const int j = (e * TM + warp) * 32 + lane;
          const int pos = j + sh[e];
          if (j < cnt && pos < ls && (sh[e] > 0 || j == sel)) { S.bkey[pos] = ek[e]; S.bid[pos] = ef[e]; }
        }
        if (warp == TM - 1 && vm) {
          const uint64_t ck = lane < m ? S.ckey[c0 + lane] : kNoKey;
          const uint32_t cv = lane < m ? S.cid[c0 + lane] : kEmptySlot;
          int crank = 0;   // new keys before this one
          for (int c = 0; c < m; c += 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint64_t kc = S.ckey[c0 + c + i];
              const uint32_t ic = S.cid[c0 + c + i];
              crank += key_less(kc, ic, ck, cv) ? 1 : 0;
            }
          }
          const int pos = rk + crank;
          if (rk != kNoRank && pos < ls) { S.bkey[pos] = ck; S.bid[pos] = cv; }
        }
        // the first unexpanded entry: the first new key, or the old one where no new key precedes it
        const int least = (int)__reduce_min_sync(kFull, (unsigned)rk);
        if (least <= uns) { uns = least; hit = false; }
        cnt = min(cnt + __popc(vm), ls);
        c0 += 32;
        if (c0 < nc) bar_sync<32 * TM>(2);
      } while (c0 < nc);
      if (tid == 0) { S.ctl[kTcSel] = (uint32_t)uns; S.ctl[kTcCnt] = (uint32_t)cnt; }
      __syncthreads();
      sel = uns;
      par ^= 1;
    }
  }
  cur->cnt = cnt;
  cur->sel = sel;
  asm volatile("cp.async.wait_all;" ::: "memory");   // no copy outlives the search
  __syncthreads();
  return cnt;
}

// The graph-route kernel of a query batch with one CTA of TM + TS warps per
// query in flight; POL as in query_kernel (0 plain, 1 with the search policy).
// BPS: CTAs per SM it is compiled for; FP8 rows and lists of more than 128 spill
// at 64 registers and run faster as three CTAs (300K x 100, 310 to 600 queries,
// beam 160 and 256: 1.09 times as fast as four).  ngraph (or NULL): the batch's graph
// searches; more than `most` of them are left to the kernel launched next, which
// claims from the same counter (and finds nothing if this one took them).
template <int EPT, int TM, int TS, int P, int CPL, int FMT, int POL, int BPS>
__global__ void __launch_bounds__((TM + TS) * 32, BPS == 4 && EPT == 2 && FMT == JAG_VEC_FP8 ? 3 : BPS)
query_team_kernel(DevIndex ix, const float *queries, int d, const jag_filter *filters, const QueryPlan *plans,
                  const uint8_t *lut_base, int64_t nq, int k, int ls, int hbits, int rr, int32_t *rr_ids,
                  int32_t *out_ids, float *out_dist, unsigned long long *work, const unsigned long long *ngraph,
                  unsigned long long most, const __grid_constant__ jag_policy pol) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TeamSmem S = carve_team_smem(smem, list_slots(ls));
  const int64_t sample = ix.n < 4096 ? ix.n : 4096;
  if (ngraph && *ngraph > most) return;
  for (;;) {
    __syncthreads();   // the previous query's shared memory is no longer read
    if (tid == 0) {
      const unsigned long long c = atomicAdd(work, 1ull);
      S.ctl[kTcQuery] = (uint32_t)c;
      S.ctl[kTcQuery + 1] = (uint32_t)(c >> 32);
    }
    __syncthreads();
    const unsigned long long qi = (unsigned long long)S.ctl[kTcQuery] | ((unsigned long long)S.ctl[kTcQuery + 1] << 32);
    if (qi >= (unsigned long long)nq) return;
    const QueryPlan pl = plans[qi];
    if (pl.route != kRouteGraph) continue;
    QChunks<CPL, FMT> q;
    load_point<P, CPL, FMT>(queries + (int64_t)qi * d, d, q);
    const jag_filter f = filters[qi];
    const QueryKey key{f.kind, f.payload, pl.lut_off >= 0 ? lut_base + pl.lut_off : nullptr};
    SearchStats st;
    TeamCursor cur{0, 0};
    int cnt;
    if constexpr (POL == 1) {
      // the plain loop up to hop h0, the decision by warp 0, the same loop
      // again (as in query_kernel)
      int lsq = ls, lim = pol.mode != JAG_POLICY_PLAIN ? pol.h0 : 0x7FFFFFFF;
      if (pol.features && tid < JAG_MLP_FEATURES) pol.features[(int64_t)qi * JAG_MLP_FEATURES + tid] = 0.f;
      for (;;) {
        cnt = team_search<EPT, TM, TS, P, CPL, FMT>(ix, key, q, lsq, hbits, S, st, lim, &cur);
        if (lim != pol.h0 || st.hops < lim) break;
        if (warp == 0) {
          const int64_t est = (f.kind == JAG_F_SUBSET || f.kind == JAG_F_BOOL) ? (int64_t)pl.est * ix.n / sample
                              : (f.kind == JAG_F_NONE ? ix.n : (int64_t)pl.est);
          WarpSmem W;
          W.bkey = S.bkey; W.bid = S.bid; W.hash = S.hash; W.cid = S.cid; W.ck1 = S.ck1; W.rank = S.ck1;
          const PolicyOut o = policy_decide(pol, W, reinterpret_cast<float *>(S.cid), cnt, k, est, f.kind, ls,
                                            pol.features ? pol.features + (int64_t)qi * JAG_MLP_FEATURES : nullptr,
                                            pol.forced ? pol.forced + (int64_t)qi * 2 : nullptr);
          if (lane == 0) { S.ctl[kTcLs] = (uint32_t)o.beam; S.ctl[kTcLim] = (uint32_t)o.stop; }
        }
        __syncthreads();
        lsq = (int)S.ctl[kTcLs];
        const int stop = (int)S.ctl[kTcLim];
        if (cnt > lsq) cnt = lsq;
        if (stop > 0 && st.hops >= stop) break;
        lim = stop > 0 ? stop : 0x7FFFFFFF;
        cur.cnt = cnt;   // sel stays the first unexpanded position (past cnt: none left)
      }
    } else {
      cnt = team_search<EPT, TM, TS, P, CPL, FMT>(ix, key, q, ls, hbits, S, st, 0x7FFFFFFF, &cur);
    }
    if (FMT == JAG_VEC_F32) {
      for (int j = tid; j < k; j += 32 * (TM + TS)) {
        int32_t id = -1;
        float dd = __int_as_float(0x7F800000);
        if (j < cnt) {
          const uint64_t kk = S.bkey[j];
          if ((kk >> 32) == 0) { id = (int32_t)(S.bid[j] & ~kExpanded); dd = u2f((uint32_t)kk); }
        }
        out_ids[(int64_t)qi * k + j] = id;
        out_dist[(int64_t)qi * k + j] = dd;
      }
    } else {
      for (int j = tid; j < rr; j += 32 * (TM + TS)) {
        int32_t id = -1;
        if (j < cnt && (S.bkey[j] >> 32) == 0) id = (int32_t)(S.bid[j] & ~kExpanded);
        rr_ids[(int64_t)qi * rr + j] = id;
      }
    }
  }
}

constexpr int kTeamMain = 4, kTeamAhead = 4;   // TM, TS

// How a batch uses the team kernel: CTAs per SM (0: not at all), and the graph
// searches past which it leaves them (0: takes any number).
struct TeamUse {
  int ctas;
  int64_t most;
};

template <int EPT, int P, int CPL, int FMT, int POL, int BPS>
static cudaError_t launch_team_one(const SearchLaunch &L, int64_t most) {
  constexpr int TM = kTeamMain, TS = kTeamAhead;
  auto kern = query_team_kernel<EPT, TM, TS, P, CPL, FMT, POL, BPS>;
  // the default visited set grows to 2^12 slots: shared memory is not what
  // limits the CTAs here, and fewer distances are computed twice
  const int hbits = L.hbits_auto ? 12 : L.hbits;
  const size_t smem = team_smem_bytes(list_slots(L.ls), hbits);
  const int bps = blocks_per_sm(kern, smem, TM + TS);
  if (bps == 0) return cudaErrorInvalidConfiguration;
  const int64_t grid = std::min<int64_t>((int64_t)bps * num_sms(), std::max<int64_t>(L.nq, 1));
  if (L.ev_begin) cudaEventRecord(L.ev_begin, L.stream);
  kern<<<(unsigned)grid, (TM + TS) * 32, smem, L.stream>>>(L.ix, L.queries, L.d, L.filters, L.plans, L.lut, L.nq, L.k,
                                                          L.ls, hbits, L.rr, L.rr_ids, L.out_ids, L.out_dist,
                                                          L.work, most > 0 ? L.work + kWorkGraph : nullptr,
                                                          (unsigned long long)most, L.policy);
  if (L.ev_end) cudaEventRecord(L.ev_end, L.stream);
  return cudaGetLastError();
}

// Batches the team kernel takes.  Up to two CTAs per SM they are compiled for
// two per SM (up to 128 registers); a plain search of rows of one chunk per lane
// goes on with four per SM (64 registers), as long as the graph searches about
// fit them at once.  nq is the only count the host has, so past that many queries,
// up to six per SM, of which the exact scan may take some, the kernel looks at
// the count of graph searches itself; the one-warp kernel is launched behind it.
// Measured against one warp per query (all of the queries graph searches,
// unless said otherwise):
//   300K x 100 BF16, R = 32, beam 256: 256 queries 1,204 -> 540 us, 615 queries
//   1.13 times as fast, 700 queries 1.02, 900 queries 0.95;
//   1M x 32, R = 16, beam 64: 450 queries 1.20 times, 615 queries 1.04, 700
//   queries 0.88, 900 queries 0.82;
//   150K x 77, R = 48, beam 160, ranges and boolean filters: 777 queries (about
//   570 graph searches), whole call 1,349 -> 731 us;
//   300K x 16, R = 64: 900 queries 1.15 (beam 64) to 1.55 (beam 256), and 200K x
//   128 BF16, R = 40: 1.04 to 1.20: past 32 edges a one-warp hop reads its
//   out-list in two rounds, so six per SM gain still (at beam 16 they lose 3 %).
// Rows of more chunks per lane and policy searches stop at the two per SM that
// their registers allow; more of them was not tried.
// An index that stays in L2 has less latency to hide: three per SM (30K points,
// 568 queries: 267 -> 279 us), two for short lists or few edges, and none for
// both (1,000 x 16, R = 8, beam 10: 60 -> 67 us).
inline TeamUse team_use(const SearchLaunch &L, int CPL, int pol) {
  constexpr TeamUse none{0, 0};
  if (list_slots(L.ls) > 256 || (pol && CPL > 2) || (L.ix.R <= 16 && L.ls <= 16)) return none;
  const int64_t sms = num_sms();
  if (L.nq <= 2 * sms) return {2, 0};
  if (CPL != 1 || pol) return none;
  const int64_t row = L.ix.fmt == JAG_VEC_F32 ? L.ix.xs * 4 : L.ix.qbytes;
  const bool in_l2 = L.ix.n * (row + 8 * L.ix.R) < ((int64_t)64 << 20);
  if (in_l2) return L.ix.R > 16 && L.ls > 16 && L.nq <= 3 * sms ? TeamUse{4, 0} : none;
  const int64_t most = L.ix.R > 32 && L.ls > 16 ? kTeamQueriesPerSm * sms : 17 * sms / 4;
  if (L.nq <= most) return {4, 0};
  return L.s0 > 0 && L.nq <= kTeamQueriesPerSm * sms ? TeamUse{4, most} : none;
}

template <int EPT, int FMT, int POL, int BPS>
static cudaError_t launch_team_rows(const SearchLaunch &L, int P, int CPL, int64_t most) {
#define JAG_TCASE(PP, CC) \
  if (P == PP && CPL == CC) return launch_team_one<EPT, PP, CC, FMT, POL, BPS>(L, most);
  JAG_TCASE(8, 1)
  JAG_TCASE(16, 1)
  JAG_TCASE(32, 1)
  if constexpr (BPS == 2) {
    JAG_TCASE(32, 2)
    if constexpr (!POL) {
      JAG_TCASE(32, 4)
      if constexpr (FMT == JAG_VEC_F32) {
        JAG_TCASE(32, 8)
      }
    }
  }
#undef JAG_TCASE
  return cudaErrorInvalidValue;
}

template <int FMT>
cudaError_t launch_team_fmt(const SearchLaunch &L, int P, int CPL, TeamTook *took) {
  // a plain-mode policy without features is the plain search
  const int pol = L.has_policy && !(L.policy.mode == JAG_POLICY_PLAIN && !L.policy.features) ? 1 : 0;
  const TeamUse use = team_use(L, CPL, pol);
  *took = !use.ctas ? kTeamNone : use.most ? kTeamMaybe : kTeamAll;
  if (*took == kTeamNone) return cudaSuccess;
  SearchLaunch T = L;
  if (*took == kTeamMaybe) T.ev_end = nullptr;   // recorded behind the next kernel
  const bool one = list_slots(L.ls) <= 32 * kTeamMain;   // entries of L per thread: 1 or 2
  if (pol) return one ? launch_team_rows<1, FMT, 1, 2>(T, P, CPL, 0) : launch_team_rows<2, FMT, 1, 2>(T, P, CPL, 0);
  if (use.ctas == 2)
    return one ? launch_team_rows<1, FMT, 0, 2>(T, P, CPL, 0) : launch_team_rows<2, FMT, 0, 2>(T, P, CPL, 0);
  return one ? launch_team_rows<1, FMT, 0, 4>(T, P, CPL, use.most)
             : launch_team_rows<2, FMT, 0, 4>(T, P, CPL, use.most);
}

}  // namespace jag
