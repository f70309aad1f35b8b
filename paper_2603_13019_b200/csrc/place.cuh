// Placement of what a pool's selection granted, one warp per (scenario, pool).
//   GPU pools (Section 5.3): chunks are aligned power-of-two intervals inside a node; requests
//     are served by size descending, then queue position; each takes the smallest sufficient
//     maximal free block, lowest (node, start) first, and the low end of a split block.
//   CPU pools (Section 5.2): cores are exclusive; an action's cores come from one NUMA domain
//     when one fits (fewest free cores that still fit, lowest index), lowest core ids first;
//     otherwise domains are filled in ascending order.
//   API pools (Section 5.1): the grant is accounted against the quota / concurrency limit.
#pragma once
#include "common.cuh"

// lowest start of a maximal free aligned block of size 2^bl in a node mask, or -1
__device__ __forceinline__ int find_block(u32 busy, int bl, int group) {
  const int bs = 1 << bl;
  const u32 ones = (1u << bs) - 1u;
#pragma unroll 1
  for (int st = 0; st < group; st += bs) {
    if (busy & (ones << st)) continue;
    if (bs < 8) {                                       // maximal: the enclosing block is not free
      int ps = st & ~(2 * bs - 1);
      u32 pones = ((1u << (2 * bs)) - 1u) << ps;
      if (!(busy & pones)) continue;
    }
    return st;
  }
  return -1;
}

// nm: node busy masks of the pool (updated).  keep candidates, multiplicities r[].
__device__ void place_gpu(const PoolDev& pd, u8* nm, int keep, const u8* cg, const u8* r, int* pnode, int* poff, int lane) {
  const int top = ilog2(pd.group);
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
#pragma unroll 1
  for (int lz = top; lz >= 0; --lz) {
    const int z = 1 << lz;
#pragma unroll 1
    for (int i = 0; i < keep; ++i) {
      const int g = cg[i] & 0x7f, gang = cg[i] >> 7, ri = r[i];
      const int nreq = gang ? (g * ri == z ? 1 : 0) : (g == z ? ri : 0);
#pragma unroll 1
      for (int rep = 0; rep < nreq; ++rep) {
        int node = -1, start = -1;
#pragma unroll 1
        for (int bl = lz; bl <= top && node < 0; ++bl) {
#pragma unroll 1
          for (int v0 = 0; v0 < pd.n_nodes; v0 += 32) {
            int v = v0 + lane;
            bool has = v < pd.n_nodes && ((node_levels(nm[v] | pad) >> bl) & 1u) != 0;
            u32 b = __ballot_sync(TG_FULL, has);
            if (b) { node = v0 + __ffs(b) - 1; start = find_block(nm[node] | pad, bl, pd.group); break; }
          }
        }
        if (node < 0 || start < 0) continue;            // cannot happen: the selection fits
        __syncwarp();
        if (lane == 0) {
          nm[node] |= (u8)(((1u << z) - 1u) << start);
          if (rep == 0) { pnode[i] = node; poff[i] = start; }
        }
        __syncwarp();
      }
    }
  }
}

// CPU placement on a pool nobody occupies yet (a single round).  Cores are only ever taken
// lowest id first, so the used cores of a domain are always a prefix of it: the free count per
// domain is the whole state and a grant's first core follows from it.  The rule: the domain with the fewest free
// cores that still fit, lowest index among equals; else ascending domains.
__device__ void place_cpu_fresh(const PoolDev& pd, int* dfree, int keep, const u8* cg, const u8* r,
                                int* pnode, int* poff, int lane) {
  const int D = pd.capacity / pd.group;
#pragma unroll 1
  for (int d = lane; d < D; d += 32) dfree[d] = pd.group;
  __syncwarp();
#pragma unroll 1
  for (int i0 = 0; i0 < keep; i0 += 32) {
    // this lane's candidate of the block of 32; its units are broadcast when its turn comes
    const int mine = i0 + lane < keep ? (cg[i0 + lane] & 0x7f) * r[i0 + lane] : 0;
    const int nb = min(32, keep - i0);
#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
      const int k = __shfl_sync(TG_FULL, mine, b);
      i64 key = TG_INF;
#pragma unroll 1
      for (int d = lane; d < D; d += 32) {
        int f = dfree[d];
        if (f >= k) key = min(key, ((i64)f << 32) | d);
      }
      key = warp_min64(key);
      if (lane == 0) {
        int first = -1;
        if (key != TG_INF) {
          int d = (int)(key & 0xffffffff);
          first = d * pd.group + (pd.group - dfree[d]);
          dfree[d] -= k;
        } else {
          int need = k;
#pragma unroll 1
          for (int d = 0; d < D && need > 0; ++d) {
            int f = dfree[d];
            if (f == 0) continue;
            if (first < 0) first = d * pd.group + (pd.group - f);
            int take = min(f, need);
            dfree[d] = f - take; need -= take;
          }
        }
        pnode[i0 + b] = first >= 0 ? first / pd.group : -1; poff[i0 + b] = first;
      }
      __syncwarp();
    }
  }
}

// GPU placement with a service cache (Section 5.3, evict on execution).  The rule of place_gpu, and among
// the free blocks of the level it picks, one whose granted chunk (the block's low end) caches the
// request's instance goes first, then the lowest (node, start).  An instance is (service, chunk size);
// a chunk caches it iff every GPU of the chunk remembers its tag.  ctag / cuse: the pool's entries,
// [node][8][K] (tag 0 = empty, time of last use).  A grant makes the instance the most recently used
// one on every GPU of the chunk; on a miss a GPU overwrites an empty entry (lowest index), else its
// least recently used one (lowest index among equals), and miss[i] is set: candidate i then runs its
// restoration time longer.  svc: the scenario's service column (may be null), ids: action indices.
__device__ void place_gpu_cache(const PoolDev& pd, u8* nm, int keep, const u8* cg, const u8* r, const int* ids,
                                int* pnode, int* poff, u8* miss, const unsigned short* svc, u32* ctag, i64* cuse,
                                int K, i64 now, int lane, int* owner = nullptr) {
  const int top = ilog2(pd.group);
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
#pragma unroll 1
  for (int i = lane; i < keep; i += 32) miss[i] = 0;
  __syncwarp();
#pragma unroll 1
  for (int lz = top; lz >= 0; --lz) {
    const int z = 1 << lz;
#pragma unroll 1
    for (int i = 0; i < keep; ++i) {
      const int g = cg[i] & 0x7f, gang = cg[i] >> 7, ri = r[i];
      const int nreq = gang ? (g * ri == z ? 1 : 0) : (g == z ? ri : 0);
      if (nreq == 0) continue;
      const u32 sv = svc ? svc[ids[i]] : 0xffffu;
      const u32 tag = sv == 0xffffu ? 0u : ((sv << 3) | (u32)lz) + 1u;
#pragma unroll 1
      for (int rep = 0; rep < nreq; ++rep) {
        u32 kmin = 0xffffffffu;
#pragma unroll 1
        for (int bl = lz; bl <= top && kmin == 0xffffffffu; ++bl) {
          u32 key = 0xffffffffu;
#pragma unroll 1
          for (int v = lane; v < pd.n_nodes; v += 32) {
            const NodeBlocks nb = node_blocks(nm[v] | pad);
            u32 starts = bl == 0 ? nb.s1 : (bl == 1 ? nb.s2 : (bl == 2 ? nb.s4 : nb.s8));
#pragma unroll 1
            while (starts) {
              const int st = __ffs(starts) - 1; starts &= starts - 1;
              bool hit = tag != 0;
#pragma unroll 1
              for (int b = st; b < st + z && hit; ++b) {
                bool has = false;
#pragma unroll 1
                for (int k = 0; k < K; ++k) has |= ctag[(size_t)(v * 8 + b) * K + k] == tag;
                hit = has;
              }
              key = min(key, (hit ? 0u : 1u << 30) | ((u32)v << 4) | (u32)st);
            }
          }
          kmin = __reduce_min_sync(TG_FULL, key);
        }
        if (kmin == 0xffffffffu) continue;              // cannot happen: the selection fits
        const int node = (int)((kmin >> 4) & 0x3ffffffu), start = (int)(kmin & 15u);
        const bool hit = (kmin >> 30) == 0;
        __syncwarp();
        if (lane == 0) {
          nm[node] |= (u8)(((1u << z) - 1u) << start);
          if (rep == 0) { pnode[i] = node; poff[i] = start; }
          if (owner) for (int b = 0; b < z; ++b) owner[node * pd.group + start + b] = ids[i];
          if (tag) {
            if (!hit) miss[i] = 1;
#pragma unroll 1
            for (int b = start; b < start + z; ++b) {
              u32* tg = ctag + (size_t)(node * 8 + b) * K;
              i64* us = cuse + (size_t)(node * 8 + b) * K;
              int at = -1;
#pragma unroll 1
              for (int k = 0; k < K && at < 0; ++k) if (tg[k] == tag) at = k;
#pragma unroll 1
              for (int k = 0; k < K && at < 0; ++k) if (tg[k] == 0) at = k;
              if (at < 0) { at = 0; for (int k = 1; k < K; ++k) if (us[k] < us[at]) at = k; }
              tg[at] = tag; us[at] = now;
            }
          }
        }
        __syncwarp();
      }
    }
  }
}

// ---- register-resident fast paths of a single round (fresh CPU pool, at most 128 domains /
// ---- GPU nodes): the state lives in lane registers, the arg-min is one redux, and every lane
// ---- keeps the result of "its" candidate of a block of 32 for a coalesced write.

// Same placement rule as place_gpu; requires pd.n_nodes <= 128.  busy_row: the pool's node masks before the round
// (may be null).  Lane k and register s hold node 32 s + k; lv[l][s] has bit k set where that node has a maximal
// free block of 2^l GPUs, the same in every lane, so that the lowest node of a level is one bit scan.
template <int NS>
__device__ __forceinline__ void place_gpu_masks(const PoolDev& pd, const u8* busy_row, int keep, const u8* cg, const u8* r,
                                                int* pnode, int* poff, int lane) {
  const int top = ilog2(pd.group), n_nodes = pd.n_nodes;
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
  u32 nm[NS], lv[4][NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int v = lane + 32 * s;
    nm[s] = v < n_nodes ? ((busy_row ? busy_row[v] : 0u) | pad) : 0xffu;
    const u32 lev = node_levels(nm[s]);
#pragma unroll
    for (int l = 0; l < 4; ++l) lv[l][s] = __ballot_sync(TG_FULL, (lev >> l) & 1u);
  }
#pragma unroll 1
  for (int lz = top; lz >= 0; --lz) {
    const int z = 1 << lz;
#pragma unroll 1
    for (int i0 = 0; i0 < keep; i0 += 32) {
      const int i = i0 + lane;
      int nreq = 0;
      if (i < keep) {
        const int g = cg[i] & 0x7f, gang = cg[i] >> 7, ri = r[i];
        nreq = gang ? (g * ri == z ? 1 : 0) : (g == z ? ri : 0);
      }
      int myn = -1, myo = -1;
      u32 bm = __ballot_sync(TG_FULL, nreq > 0);
#pragma unroll 1
      while (bm) {
        const int b = __ffs(bm) - 1; bm &= bm - 1;
        const int cnt = __shfl_sync(TG_FULL, nreq, b);
#pragma unroll 1
        for (int rep = 0; rep < cnt; ++rep) {
          // smallest sufficient block level, lowest node
          int bl = -1, s = 0; u32 m = 0;
#pragma unroll
          for (int l = 3; l >= 0; --l)
#pragma unroll
            for (int q = NS - 1; q >= 0; --q) if (l >= lz && lv[l][q]) { bl = l; s = q; m = lv[l][q]; }
          if (bl < 0) continue;                         // cannot happen: the selection fits
          const int k = __ffs(m) - 1;
          u32 busy = 0;
#pragma unroll
          for (int q = 0; q < NS; ++q) if (q == s) busy = nm[q];
          busy = __shfl_sync(TG_FULL, busy, k);
          const int start = node_block_start(busy, bl);
          busy |= ((1u << z) - 1u) << start;
          const u32 lev = node_levels(busy), bit = 1u << k;
#pragma unroll
          for (int q = 0; q < NS; ++q)
            if (q == s) {
              if (lane == k) nm[q] = busy;
#pragma unroll
              for (int l = 0; l < 4; ++l) lv[l][q] = ((lev >> l) & 1u) ? lv[l][q] | bit : lv[l][q] & ~bit;
            }
          if (rep == 0 && lane == b) { myn = 32 * s + k; myo = start; }
        }
      }
      if (i < keep && myn >= 0) { pnode[i] = myn; poff[i] = myo; }
    }
  }
}

// Same placement rule as place_cpu_fresh; requires at most 32 NS domains of fewer than 65536 cores.
// Lane k and register s hold domain 32 s + k's free cores; a candidate costs one warp minimum over the
// domains that still fit it.
template <int NS>
struct CpuFresh {
  u32 df[NS];
  __device__ __forceinline__ CpuFresh(const PoolDev& pd, int lane) {
    const int D = pd.capacity / pd.group;
#pragma unroll
    for (int s = 0; s < NS; ++s) df[s] = lane + 32 * s < D ? (u32)pd.group : 0u;
  }
  // places the next nb <= 32 candidates, lane b's asking for `mine` cores; node / off are the lane's results
  __device__ __forceinline__ void place(const PoolDev& pd, int mine, int nb, int lane, int& node, int& off) {
    const int G = pd.group, D = pd.capacity / G;
#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
      const u32 k = (u32)__shfl_sync(TG_FULL, mine, b);
      u32 key = 0xffffffffu;
#pragma unroll
      for (int s = 0; s < NS; ++s) if (df[s] >= k) key = min(key, (df[s] << 16) | (u32)(lane + 32 * s));
      const u32 best = __reduce_min_sync(TG_FULL, key);
      int first = -1, dom = -1;
      if (best != 0xffffffffu) {                       // best fit: fewest free cores that still fit
        const int d = (int)(best & 0xffffu), f = (int)(best >> 16);
        first = d * G + (G - f); dom = d;
#pragma unroll
        for (int s = 0; s < NS; ++s) if (d == lane + 32 * s) df[s] -= k;
      } else {                                         // no domain fits: fill domains in ascending order
        u32 need = k;
#pragma unroll 1
        for (int d = 0; d < D && need > 0; ++d) {
          u32 f = 0;
#pragma unroll
          for (int s = 0; s < NS; ++s) if (s == (d >> 5)) f = df[s];
          f = __shfl_sync(TG_FULL, f, d & 31);
          if (f == 0) continue;
          if (first < 0) { first = d * G + (G - (int)f); dom = d; }
          const u32 take = min(f, need);
          if (lane == (d & 31)) {
#pragma unroll
            for (int s = 0; s < NS; ++s) if (s == (d >> 5)) df[s] -= take;
          }
          need -= take;
        }
      }
      if (lane == b) { node = dom; off = first; }
    }
  }
};
