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

// One request after the other: where the list of place_gpu_lists finds no room.
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

// The nodes of a pool as a round keeps them (a byte of busy GPUs each), and as a replay does (a word of free ones).
struct BusyNodes {
  u8* m;
  __device__ __forceinline__ u32 busy(int v) const { return m[v]; }
  __device__ __forceinline__ void take(int v, u32 gpus) const { m[v] |= (u8)gpus; }
};
struct FreeNodes {
  u32* w;
  __device__ __forceinline__ u32 busy(int v) const { return ~w[v] & 0xffu; }
  __device__ __forceinline__ void take(int v, u32 gpus) const { w[v] &= ~gpus; }
};

// GPU placement with a service cache (Section 5.3, evict on execution).  The rule of place_gpu, and among
// the free blocks of the level it picks, one whose granted chunk (the block's low end) caches the
// request's instance goes first, then the lowest (node, start).  An instance is (service, chunk size);
// a chunk caches it iff every GPU of the chunk remembers its tag.  ctag / cuse: the pool's entries,
// [node][8][K] (tag 0 = empty, time of last use).  A grant makes the instance the most recently used
// one on every GPU of the chunk; on a miss a GPU overwrites an empty entry (lowest index), else its
// least recently used one (lowest index among equals), and miss[i] is set: candidate i then runs its
// restoration time longer.  svc: the scenario's service column (may be null), ids: action indices, scratch: keep ints.
// Per request, a lane looks at one GPU's entries and votes, four nodes a vote, then a lane per node finds the node's best block
// by bit operations on free and holding GPUs, one warp minimum picks among them, and the chunk's GPUs update their
// entries a lane each.  Bound by that chain; the entries work in shared memory (mem) where they fit, 38 nodes of two per
// GPU in the selection's work area.  A lane that walked a node's chunks entry by entry in global memory took 3600 cycles a
// request: 4096 x 1024 with two entries per GPU 400 us a call against 357.
template <class Nodes>
__device__ __forceinline__ void place_gpu_cache(const PoolDev& pd, const Nodes nodes, int keep, const u8* cg, const u8* r, const int* ids,
                                                int* pnode, int* poff, u8* miss, int* scratch, const unsigned short* svc, u32* tag_row, i64* use_row,
                                                int K, i64 now, int lane, char* mem, int mem_bytes, int* owner = nullptr) {
  const int entries = pd.n_nodes * 8 * K;
  u32* ctag = tag_row; i64* cuse = use_row;
  const bool near = entries * 12 <= mem_bytes;
  if (near) {
    cuse = (i64*)mem; ctag = (u32*)(cuse + entries);
#pragma unroll 2
    for (int e = lane; e < entries; e += 32) { cuse[e] = use_row[e]; ctag[e] = tag_row[e]; }
  }
  const int top = ilog2(pd.group), n_nodes = pd.n_nodes;
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
#pragma unroll 1
  for (int i = lane; i < keep; i += 32) { miss[i] = 0; scratch[i] = svc ? (int)svc[ids[i]] : 0xffff; }
  __syncwarp();
#pragma unroll 1
  for (int lz = top; lz >= 0; --lz) {
    const int z = 1 << lz;
#pragma unroll 1
    for (int i0 = 0; i0 < keep; i0 += 32) {
      int nreq = 0;
      if (i0 + lane < keep) {
        const int g = cg[i0 + lane] & 0x7f, gang = cg[i0 + lane] >> 7, ri = r[i0 + lane];
        nreq = gang ? (g * ri == z ? 1 : 0) : (g == z ? ri : 0);
      }
#pragma unroll 1
      for (u32 todo = __ballot_sync(TG_FULL, nreq > 0); todo; todo &= todo - 1u) {
        const int b = __ffs(todo) - 1, i = i0 + b, cnt = __shfl_sync(TG_FULL, nreq, b);
        const u32 sv = (u32)scratch[i], tag = sv == 0xffffu ? 0u : ((sv << 3) | (u32)lz) + 1u;
#pragma unroll 1
        for (int rep = 0; rep < cnt; ++rep) {
          u32 best = 0xffffffffu;                        // block level | does not cache it | node | first GPU
#pragma unroll 1
          for (int v0 = 0; v0 < n_nodes; v0 += 32) {
            u32 hold = 0;                                // GPUs of the lane's node that remember the tag
            if (tag)
#pragma unroll 1
              for (int q = 0; q < 8 && v0 + 4 * q < n_nodes; ++q) {
                const int at = (v0 + 4 * q) * 8 + lane;
                bool has = false;
                if (at < n_nodes * 8)
#pragma unroll 1
                  for (int k = 0; k < K; ++k) has |= ctag[(size_t)at * K + k] == tag;
                const u32 w = __ballot_sync(TG_FULL, has);
                if ((lane >> 2) == q) hold = (w >> (8 * (lane & 3))) & 0xffu;
              }
            const int v = v0 + lane;
            const NodeBlocks nb = node_blocks(v < n_nodes ? nodes.busy(v) | pad : 0xffu);
            // the node's smallest sufficient level, the blocks of that level, and the ones whose low end caches the tag
            const u32 s = lz <= 0 && nb.s1 ? nb.s1 : (lz <= 1 && nb.s2 ? nb.s2 : (lz <= 2 && nb.s4 ? nb.s4 : nb.s8));
            const u32 lev = lz <= 0 && nb.s1 ? 0u : (lz <= 1 && nb.s2 ? 1u : (lz <= 2 && nb.s4 ? 2u : 3u));
            u32 all = hold;                              // GPUs from which on z of them hold it
            if (lz >= 1) all &= all >> 1;
            if (lz >= 2) all &= all >> 2;
            if (lz >= 3) all &= all >> 4;
            const u32 hits = s & all;
            if (s) best = min(best, (lev << 30) | (hits ? 0u : 1u << 29) | ((u32)v << 4) | (u32)(__ffs(hits ? hits : s) - 1));
          }
          best = __reduce_min_sync(TG_FULL, best);
          if (best == 0xffffffffu) continue;              // cannot happen: the selection fits
          const int node = (int)((best >> 4) & 0x1ffffffu), start = (int)(best & 15u);
          const bool hit = ((best >> 29) & 1u) == 0u;
          __syncwarp();
          if (lane == 0) {
            nodes.take(node, ((1u << z) - 1u) << start);
            if (rep == 0) { pnode[i] = node; poff[i] = start; }
            if (tag && !hit) miss[i] = 1;
          }
          if (lane < z) {
            const int gpu = start + lane;
            if (owner) owner[node * pd.group + gpu] = ids[i];
            if (tag) {
              u32* tg = ctag + (size_t)(node * 8 + gpu) * K;
              i64* us = cuse + (size_t)(node * 8 + gpu) * K;
              int at = -1;
#pragma unroll 1
              for (int k = 0; k < K && at < 0; ++k) if (tg[k] == tag) at = k;
#pragma unroll 1
              for (int k = 0; k < K && at < 0; ++k) if (tg[k] == 0) at = k;
              if (at < 0) { at = 0; for (int k = 1; k < K; ++k) if (us[k] < us[at]) at = k; }
              tg[at] = tag; us[at] = now;
            }
          }
          __syncwarp();
        }
      }
    }
  }
  if (near)
#pragma unroll 2
    for (int e = lane; e < entries; e += 32) { use_row[e] = cuse[e]; tag_row[e] = ctag[e]; }
}

// ---- fast paths of a single round: GPU requests size by size, core pools of at most 128 domains with their
// ---- state in lane registers (the arg-min is one redux, every lane keeps the result of "its" candidate of a block of 32).

// Same placement rule as place_gpu, all requests of one size at once.  While requests of size z are served, a block of
// level L is only touched once every smaller sufficient block is used up, and then from its low end on; so the places that
// are taken, in the order in which they are taken, are the free z-aligned places by (level of their block, node, start),
// and the k-th request gets the k-th of them.  First every candidate gets the rank of its first request among those of its
// size (pnode / poff hold size and rank meanwhile), then, size by size from the largest down, every node finds the ranks of
// its places by a scan over the nodes and lists the ones that are taken, then the candidates look theirs up.
// ONE: at most 32 nodes, their masks stay in registers; else in nm.  list: room for all requests (see gpu_requests).
// One request after the other, with the nodes' levels as bit masks in registers, took about 80 instructions each, 18 % of the
// selection kernel's cycles at 16384 x 4096: 1780 us a call against 1692, 4096 x 1024 279 against 252.
template <bool ONE>
__device__ __forceinline__ void place_gpu_lists(const PoolDev& pd, const u8* busy_row, u8* nm, u32* list, const int R[4], int keep, int* pnode, int* poff,
                                                int lane) {
  const int n_nodes = pd.n_nodes;
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
  u32 reg = 0xffu;
  if (ONE) { if (lane < n_nodes) reg = (busy_row ? busy_row[lane] : 0u) | pad; }
  else
#pragma unroll 1
    for (int v = lane; v < n_nodes; v += 32) nm[v] = (u8)((busy_row ? busy_row[v] : 0u) | pad);
  const int at[4] = {R[3] + R[2] + R[1], R[3] + R[2], R[3], 0};          // where a size's part of the list begins
#pragma unroll 1
  for (int lz = 3; lz >= 0; --lz) {
    const int want = pick4(R, lz);
    u32* const mine = list + pick4(at, lz);
    const u32 zm = (1u << (1 << lz)) - 1u;
    int done = 0;                                        // places listed so far
#pragma unroll 1
    for (int L = lz; L < 4 && done < want; ++L)
#pragma unroll 1
      for (int v0 = 0; v0 < n_nodes && done < want; v0 += 32) {
        const int v = v0 + lane;
        u32 busy = ONE ? reg : (v < n_nodes ? nm[v] : 0xffu);
        const NodeBlocks nb = node_blocks(busy);
        u32 s = L == 0 ? nb.s1 : (L == 1 ? nb.s2 : (L == 2 ? nb.s4 : nb.s8));
        if (!__any_sync(TG_FULL, s != 0u)) continue;
        const int cnt = __popc(s) << (L - lz);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(TG_FULL, incl, o); if (lane >= o) incl += y; }
        int k = done + incl - cnt;                       // rank of the node's first place
        done += __shfl_sync(TG_FULL, incl, 31);
        const int per = 1 << (L - lz);
#pragma unroll 1
        for (; s && k < want; s &= s - 1u) {
          const int st = __ffs(s) - 1;
#pragma unroll 1
          for (int x = 0; x < per && k < want; ++x, ++k) {
            const int p = st + (x << lz);
            mine[k] = ((u32)v << 3) | (u32)p;
            busy |= zm << p;
          }
        }
        if (ONE) reg = busy; else if (v < n_nodes) nm[v] = (u8)busy;
      }
  }
  __syncwarp();
#pragma unroll 1
  for (int i = lane; i < keep; i += 32) {
    const u32 e = list[pick4(at, pnode[i]) + poff[i]];
    pnode[i] = (int)(e >> 3); poff[i] = (int)(e & 7u);
  }
}
// Requests per size -> R; every candidate's size and the rank of its first request among those of that size -> pnode, poff.
__device__ __forceinline__ void gpu_requests(int keep, const u8* cg, const u8* r, int* pnode, int* poff, int R[4], int lane) {
  R[0] = R[1] = R[2] = R[3] = 0;
  const u32 below = (1u << lane) - 1u;
#pragma unroll 1
  for (int i0 = 0; i0 < keep; i0 += 32) {
    const int i = i0 + lane;
    int n = 0, c = -1;
    if (i < keep) {
      const int g = cg[i] & 0x7f, gang = cg[i] >> 7, ri = r[i];
      n = gang ? 1 : ri; c = ilog2(gang ? g * ri : g);
    }
    const bool several = __any_sync(TG_FULL, n > 1);
    int rank = 0;
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const u32 b = __ballot_sync(TG_FULL, c == z);
      int before = __popc(b & below), all = __popc(b);
      if (several && b) {
        const int x = c == z ? n : 0;
        int incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(TG_FULL, incl, o); if (lane >= o) incl += y; }
        before = incl - x; all = __shfl_sync(TG_FULL, incl, 31);
      }
      if (c == z) rank = R[z] + before;
      R[z] += all;
    }
    if (i < keep) { pnode[i] = c; poff[i] = rank; }
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
