// Device-resident trace replay (workflow of Section 3: submit, queue, schedule, execute,
// return), one warp per scenario, no host round trips.  Every round at now = r * round_us
//   1. refills quota pools whose window changed (Section 5.1),
//   2. releases what has finished (cores, chunks, concurrency slots),
//   3. admits the actions that have arrived to the waiting queue,
//   4. runs the scheduler of Algorithm 1 on the queue with the running actions of a pool in
//      its completion heap (Algorithm 2), using the same per-pool routines as a single round,
//   5. starts what was selected and records the occupancy.
// Rounds in which nothing can start are jumped over: with an empty queue up to the next arrival (what ends
// meanwhile is released then), behind a head of the queue that does not fit up to the next event on its pool.
//
// A scenario is one long chain of dependent rounds, each of which handles one or two actions, so what
// counts is the latency of a round, which is the number of dependent instructions in it:
//   * the records of the waiting actions (decoded once, on arrival) and the running actions sit in the warp's shared
//     memory in 16-byte pieces; arrivals are read 32 at a time, one batch ahead;
//   * times are compared as round numbers (32 bits, one warp minimum), worked out when an action starts;
//   * free cores are bit masks, a grant is a mask of one word wherever it can be, so everything that ends in a round
//     is released at once, a lane each, by shared-memory atomics; only grants over several words or chunks are found
//     again by their owner entries, one after the other;
//   * the queue is a ring, so what starts leaves it by moving its head;
//   * occupancy is recorded as differences (two atomics per action that nobody waits for), k_occupancy adds them up;
//   * pools without a choice to make (one candidate, or none elastic) never build the arrays of the selection.
#pragma once
#include "common.cuh"
#include "arrange.cuh"
#include "evict.cuh"
#include "place.cuh"
#include "order_pin.cuh"

struct ReplayWs {
  int* wait;        // [S][N] waiting actions behind the first wcap, by queue position
  u64* wkey;        // [S][N] their sort keys (policy 1 / 2 only)
  u32* words;       // [S][W] free cores of every domain word (two of them each), free GPUs of every node
  int* dfree;       // [S][Dtot + 1] free cores per NUMA domain; the last one belongs to nobody
  int* owner;       // [S][U]  action holding each core / GPU of a grant over several words or chunks
  // running actions where they do not fit shared memory (ReplayRun)
  uint4* run_at; i64* run_fin; int* run_end; u32* run_pu; int* run_idx;
  // per pool: first unit / domain / word of a scenario's row, domains, words per domain (core pools)
  int unit0[TG_MAX_POOLS], dom0[TG_MAX_POOLS], word0[TG_MAX_POOLS], n_dom[TG_MAX_POOLS], wpd[TG_MAX_POOLS];
  int U, Dtot, W;
  i64 round_us; u64 round_recip;      // round_recip: ceil(2^64 / round_us), 0 where round_at has to divide
  int max_rounds;
  int* occupancy; int* rounds_used;   // rounds_used: never null in the kernels
  int policy;       // 0: first come first served; 1 / 2: the queue is kept in shortest / longest least-level duration order
  // trajectories pinned to CPU nodes as their actions arrive (Section 5.2); trajectory == nullptr: none of it
  const int* trajectory; const u32* traj_mem; const u8* traj_last; int max_traj;
  int* traj_node; i64* mem_free; u8* pool_rw;   // pool_rw: the pool column the kernel reads (P.a_pool) and rewrites
  int state_bytes;  // > 0: a scenario's live state (words .. owner) takes that many bytes of the warp's shared memory
  int wcap, rcap;   // waiting records / running actions in shared memory (rcap 0: running actions in global memory)
};

__host__ __device__ __forceinline__ size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }
// bytes of the live state: masks, free counts, owners (a release may touch the word behind the last one)
__host__ __device__ __forceinline__ size_t replay_state_bytes(const ReplayWs& R) {
  return align16((size_t)(R.W + 2) * 4) + align16((size_t)(R.Dtot + 1) * 4) + align16((size_t)R.U * 4);
}

#define KR_THREADS 32
#define KR_FAST_BYTES 8192        // shared-memory window of the selection's arrays
#define KR_WAIT_BYTES 60          // per waiting record: three 16-byte pieces, key, queue, free list
#define KR_RUN_BYTES 36
#define KR_STATE_MAX 16384
#define KR_MIN_WAIT 64
#define KR_PER_SM 8               // blocks of 32 threads of 255 registers that an SM holds
#define KR_SLOT_BYTES 128         // free capacity of the 32 demand slots at most
// shared memory of a block (one warp) without the parts sized by the round
#define KR_TABLE_BYTES 2048       // per free mask of a node: its free blocks by size, and where a chunk of every size goes
#define KR_BASE_BYTES (WARP_SMEM_BYTES + KR_FAST_BYTES + KR_SLOT_BYTES + KR_TABLE_BYTES + 64)
#define KR_NEVER 0x7fffffff

// Waiting records, and the queue: a ring of records, or (LIST: a queue that is kept in another order) a ring of the
// numbers of records that do not move.  sp: s, p; ta: least duration, arrival; c: action, meta, mask, unit byte
// (bit 8: the last action of its trajectory).
// meta: chunk class of the least level (2 bits) and pool (3), by which a demand slot's lane knows what it is charged; nobody
// (1), elastic (1), started in this round (1), units of the least level (24).
template <bool LIST>
struct ReplayQueue {
  uint4* sp; uint4* ta; uint4* c; u64* key; unsigned short* q; unsigned short* free;
  int cap, head;
  __device__ __forceinline__ int at(int i) const { const int k = head + i; return k >= cap ? k - cap : k; }   // ring place of position i < cap
  __device__ __forceinline__ int slot(int i) const { return LIST ? (int)q[at(i)] : at(i); }
};
#define RQ_CLASS(m) ((int)((m) & 3u))
#define RQ_POOL(m) ((int)(((m) >> 2) & 15u))        // 8 and above: nobody
#define RQ_ELASTIC 64u
#define RQ_STARTED 128u
#define RQ_UNITS(m) ((int)((m) >> 8))
#define RQ_NOBODY 32u

// Running actions.  end: the round that releases it; pu: the units it gives back (21 bits; none of a quota window's), first demand
// slot (5), pool (3), wide (1), GPU (1), a trajectory's last (1); at: what it holds - masks of two words, the first one's number, domain.  A wide grant's
// units are the ones whose owner it is, from at.x on.
struct ReplayRun { uint4* at; i64* fin; int* end; u32* pu; int* idx; };
#define RR_UNITS(v) ((int)((v) & 0x1fffffu))
#define RR_SLOT(v) ((int)(((v) >> 21) & 31u))
#define RR_POOL(v) ((int)(((v) >> 26) & 7u))
#define RR_WIDE 0x20000000u
#define RR_GPU 0x40000000u
#define RR_LAST 0x80000000u
__device__ __forceinline__ u32 rr_pack(const PoolDev& pd, int j, int units, bool wide) {
  const int back = pd.window_us > 0 ? 0 : units;          // used quota is not given back
  return (u32)back | ((u32)pd.slot0 << 21) | ((u32)j << 26) | (pd.type == TG_POOL_GPU ? RR_GPU : 0u) | (wide ? RR_WIDE : 0u);
}

__device__ __forceinline__ i64 i64_of(u32 lo, u32 hi) { return (i64)(((u64)hi << 32) | lo); }

// the first round at or after time t
__device__ __forceinline__ int round_at(const ReplayWs& R, i64 t) {
  if (t <= 0) return 0;
  const u64 d = (u64)t - 1u;
  // d * recip / 2^64 exceeds d / round_us by less than d * round_us / (round_us * 2^64) < 1 / round_us for d below 2^42 and
  // round_us below 2^22 (where recip is set), so the floor is exact
  const u64 q = R.round_recip && d < (1ull << 42) ? __umul64hi(d, R.round_recip) : d / (u64)R.round_us;
  return q >= (u64)KR_NEVER - 1u ? KR_NEVER : (int)q + 1;
}

// A decoded record
struct ReplayRec { i64 s, p, tl, arr; u32 meta, mask; u8 cg; };
__device__ __forceinline__ ReplayRec replay_decode(const Params& P, int j, u32 unit, u32 mk, i64 s, i64 p) {
  ReplayRec r;
  const PoolDev& pd = P.pool[j];
  int g, gang; u32 eff;
  decode_levels(pd, (u8)unit, mk, g, gang, eff);
  const int rmin = __ffs(eff), c = pd.type == TG_POOL_GPU ? level_of(g, gang, rmin) : 0;
  r.s = clamp_param(s); r.p = clamp_param(p); r.tl = duration(r.s, r.p, rmin);
  r.mask = eff; r.cg = (u8)(g | (gang << 7));
  r.meta = (u32)c | ((u32)j << 2) | (eff & (eff - 1) ? RQ_ELASTIC : 0u) | ((u32)(g * rmin) << 8);
  return r;
}
__device__ __forceinline__ ReplayRec replay_load(const Params& P, size_t row, int a) {
  ReplayRec r = replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], P.a_s[row + a], P.a_p[row + a]);
  r.arr = P.a_arrival ? P.a_arrival[row + a] : 0;
  return r;
}
template <bool LIST>
__device__ __forceinline__ void replay_store(const ReplayQueue<LIST>& Q, int x, const ReplayRec& r, int a, u32 last) {
  Q.sp[x] = make_uint4((u32)r.s, (u32)((u64)r.s >> 32), (u32)r.p, (u32)((u64)r.p >> 32));
  Q.ta[x] = make_uint4((u32)r.tl, (u32)((u64)r.tl >> 32), (u32)r.arr, (u32)((u64)r.arr >> 32));
  Q.c[x] = make_uint4((u32)a, r.meta, r.mask, (u32)r.cg | last);
}
// a record's bit 8: the action is marked as the last one of its trajectory (traces with trajectories, and so LIST, only)
template <bool LIST>
__device__ __forceinline__ u32 replay_last(const ReplayWs& R, size_t row, int a) {
  return LIST && R.traj_last && R.traj_last[row + a] ? 256u : 0u;
}
// action, meta, mask, unit byte and bit 8 at a queue position (any lane's own); x: its slot where it is in shared memory
template <bool LIST>
__device__ __forceinline__ uint4 replay_facts(const Params& P, const ReplayWs& R, const ReplayQueue<LIST>& Q, const int* wait, size_t row, int i, int& x) {
  if (i < Q.cap) { x = Q.slot(i); return Q.c[x]; }
  const int a = wait[i];
  const ReplayRec r = replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], 0, 0);
  x = -1;
  return make_uint4((u32)a, r.meta, r.mask, (u32)r.cg | replay_last<LIST>(R, row, a));
}
// ... and the rest of a record whose facts are known
template <bool LIST>
__device__ __forceinline__ ReplayRec replay_rec(const Params& P, const ReplayQueue<LIST>& Q, size_t row, const uint4& c, int x) {
  if (x < 0) return replay_load(P, row, (int)c.x);
  const uint4 u = Q.sp[x], v = Q.ta[x];
  ReplayRec r;
  r.s = i64_of(u.x, u.y); r.p = i64_of(u.z, u.w); r.tl = i64_of(v.x, v.y); r.arr = i64_of(v.z, v.w);
  r.meta = c.y; r.mask = c.z; r.cg = (u8)c.w;
  return r;
}

// Live state of the scenario at hand: in the warp's shared memory, or in the arrays of ReplayWs where it is large.
// slot: free capacity per demand slot; node_of: by a node's free GPUs, x: its free blocks of 1, 2, 4 and 8 GPUs (9, 8, 7
// and 6 bits, so that 32 nodes add up), y: a byte per chunk size, block level << 4 | first GPU of the smallest sufficient
// block, 0xff where there is none.
struct ReplayState { u32* words; int* dfree; int* owner; int* slot; uint2* node_of; };

__device__ __forceinline__ uint2 replay_node_entry(u32 free_mask) {
  const u32 busy = ~free_mask & 0xffu;
  const NodeBlocks b = node_blocks(busy);
  const u32 lev = node_levels(busy);
  u32 y = 0;
  for (int lz = 3; lz >= 0; --lz) {
    const u32 ok = lev & (~0u << lz);
    const int l = __ffs(ok) - 1;
    y = (y << 8) | (ok ? ((u32)l << 4) | (u32)node_block_start(busy, l) : 0xffu);
  }
  return make_uint2((u32)__popc(b.s1) | ((u32)__popc(b.s2) << 9) | ((u32)__popc(b.s4) << 17) | ((u32)__popc(b.s8) << 24), y);
}

// What a grant holds: masks of two words of the state (a core domain's, or a node's one), or owner entries (wide).
// node / off: NUMA domain or GPU node, and the first core or GPU.
struct ReplayGrant { int node, off; uint4 at; bool wide; };

// the lowest k of the 64 bits hi:lo (at least k are set); every lane looks at two of them
__device__ __forceinline__ void lowest_bits(u32 lo, u32 hi, int k, int lane, u32& tlo, u32& thi) {
  if (k == 1) { tlo = lo & (0u - lo); thi = lo ? 0u : hi & (0u - hi); return; }
  const u32 below = (1u << lane) - 1u;
  const int nlo = __popc(lo);
  tlo = __ballot_sync(TG_FULL, ((lo >> lane) & 1u) && __popc(lo & below) < k);
  thi = __ballot_sync(TG_FULL, ((hi >> lane) & 1u) && nlo + __popc(hi & below) < k);
}

// One grant of k cores on a pool with cores in use: fewest free cores that still fit, lowest domain, lowest cores first;
// else ascending domains.  For pools of many or large domains, and for grants that no domain holds; words / dfree /
// owner: the pool's own rows, which begin at word w0 and domain d0 of the scenario's.
__device__ __noinline__ ReplayGrant replay_take_cores(int group, int n_dom, int wpd, u32* words, int* dfree, int* owner, int w0, int d0,
                                                      int k, int id, int lane) {
  ReplayGrant G;
  G.node = G.off = -1; G.at = make_uint4(0u, 0u, 0u, 0u); G.wide = false;
  u32 best = 0xffffffffu; int at = -1, dom = -1;
#pragma unroll 1
  for (int d = lane; d < n_dom; d += 32) { const int f = dfree[d]; if (f >= k && (u32)f < best) { best = (u32)f; at = d; } }
  const u32 mn = __reduce_min_sync(TG_FULL, best);
  if (mn != 0xffffffffu) dom = (int)__reduce_min_sync(TG_FULL, best == mn ? (u32)at : 0xffffffffu);
  int need = k;
  const int end = dom >= 0 ? (dom + 1) * wpd : n_dom * wpd;
#pragma unroll 1
  for (int w = dom >= 0 ? dom * wpd : 0; w < end && need > 0; ++w) {
    const u32 mlo = words[2 * w], mhi = words[2 * w + 1];
    if ((mlo | mhi) == 0u) continue;
    u32 lo, hi;
    const int got = min(need, __popc(mlo) + __popc(mhi));
    lowest_bits(mlo, mhi, got, lane, lo, hi);
    const int d = w / wpd, c0 = d * group + (w - d * wpd) * 64;        // the word's first core
    if (G.off < 0) {
      G.off = c0 + (lo ? __ffs(lo) - 1 : 31 + __ffs(hi)); G.node = d;
      G.wide = got < need;
      G.at = G.wide ? make_uint4((u32)G.off, 0u, 0u, 0u) : make_uint4(lo, hi, (u32)(w0 + 2 * w), (u32)(d0 + d));
    }
    if (G.wide) {
      if ((lo >> lane) & 1u) owner[c0 + lane] = id;
      if ((hi >> lane) & 1u) owner[c0 + 32 + lane] = id;
    }
    __syncwarp();
    if (lane == 0) { words[2 * w] = mlo & ~lo; words[2 * w + 1] = mhi & ~hi; dfree[d] -= got; }
    need -= got;
    __syncwarp();
  }
  return G;
}

// nreq chunks of 2^lz GPUs for one action (Section 5.3: smallest sufficient maximal free block, lowest node, lowest start);
// node / off: the first chunk.  words / owner: the pool's own rows, which begin at word w0.
__device__ __forceinline__ ReplayGrant replay_take_gpus(int group, int n_nodes, u32* words, const uint2* node_of, int* owner, int w0, int dummy,
                                                        int lz, int nreq, int id, int lane) {
  ReplayGrant G;
  G.node = G.off = -1; G.at = make_uint4(0u, 0u, (u32)w0, (u32)dummy); G.wide = nreq > 1;
#pragma unroll 1
  for (int rep = 0; rep < nreq; ++rep) {
    u32 best = 0xffffffffu;                                // level | node | first GPU
    if (n_nodes == 1) {
      const u32 y = (node_of[words[0]].y >> (8 * lz)) & 0xffu;
      if (y != 0xffu) best = y & 15u;
    } else {
#pragma unroll 1
      for (int v = lane; v < n_nodes; v += 32) {
        const u32 y = (node_of[words[v]].y >> (8 * lz)) & 0xffu;
        if (y != 0xffu) best = min(best, ((y & 0xf0u) << 20) | ((u32)v << 4) | (y & 15u));
      }
      best = __reduce_min_sync(TG_FULL, best);
    }
    if (best == 0xffffffffu) continue;                     // cannot happen: the selection fits
    const int at = (int)((best >> 4) & 0xfffffu), start = (int)(best & 15u);
    const u32 bits = ((1u << (1 << lz)) - 1u) << start;
    __syncwarp();
    if (lane == 0) words[at] &= ~bits;
    if (G.wide && lane < (1 << lz)) owner[at * group + start + lane] = id;
    if (rep == 0) { G.node = at; G.off = start; if (!G.wide) { G.at.x = bits; G.at.z = (u32)(w0 + at); } }
    __syncwarp();
  }
  return G;
}

// free capacity of a GPU pool's four demand slots
__device__ __forceinline__ void replay_gpu_slots(const PoolDev& pd, const u32* words, const uint2* node_of, int* slot, int lane) {
  int f0 = 0, f1 = 0, f2 = 0, f3 = 0;
#pragma unroll 1
  for (int v0 = 0; v0 < pd.n_nodes; v0 += 32) {
    u32 x;
    if (pd.n_nodes == 1) x = node_of[words[0]].x;
    else x = __reduce_add_sync(TG_FULL, v0 + lane < pd.n_nodes ? node_of[words[v0 + lane]].x : 0u);
    f0 += (int)(x & 511u); f1 += (int)((x >> 9) & 255u); f2 += (int)((x >> 17) & 127u); f3 += (int)(x >> 24);
  }
  // GPUs in blocks of at least 2^lane
  const int c = f3 * 8 + (lane <= 2 ? f2 * 4 : 0) + (lane <= 1 ? f1 * 2 : 0) + (lane == 0 ? f0 : 0);
  if (lane < 4) slot[pd.slot0 + lane] = c;
  __syncwarp();
}

// The selection of a pool with a choice to make: its candidates (among the first n positions) and, where an eviction
// step can look at them, the waiting actions behind and the running ones are gathered into arrays.
template <bool LIST>
__device__ __forceinline__ bool replay_select(const Params& P, const ReplayWs& R, const ReplayQueue<LIST>& Q, const ReplayRun run, const int* wait, size_t row, int j,
                                           int n, int nw, int nr, int m, i64 now, int cap0, int cap1, int cap2, int cap3, Slab& slab,
                                           CandArrays& C, int& keep, int lane) {
  const PoolDev& pd = P.pool[j];
  C.cg = (u8*)slab.take_fast(m); C.rsel = (u8*)slab.take_fast(m); C.rkeep = (u8*)slab.take_fast(m);
  C.cmask = (u32*)slab.take_fast((u64)m * 4); C.rowcand = (int*)slab.take_fast((u64)m * 4);
  C.cs = (i64*)slab.take_fast((u64)m * 8); C.cp = (i64*)slab.take_fast((u64)m * 8);
  C.cidx = (int*)slab.take_fast((u64)m * 4); C.pnode = (int*)slab.take_fast((u64)m * 4); C.poff = (int*)slab.take_fast((u64)m * 4);
  if (!C.cg || !C.rsel || !C.rkeep || !C.cmask || !C.rowcand || !C.cs || !C.cp || !C.cidx || !C.pnode || !C.poff) return false;
  int cm = 0;
  bool elastic = false;
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    int x = -1; uint4 c = make_uint4(0u, RQ_NOBODY, 1u, 1u);
    if (i < n) c = replay_facts(P, R, Q, wait, row, i, x);
    const bool mine = RQ_POOL(c.y) == j;
    const u32 b = __ballot_sync(TG_FULL, mine);
    if (mine) {
      const ReplayRec r = replay_rec(P, Q, row, c, x);
      const int k = cm + __popc(b & ((1u << lane) - 1u));
      C.cidx[k] = (int)c.x; C.cmask[k] = r.mask; C.cg[k] = r.cg; C.cs[k] = r.s; C.cp[k] = r.p;
      C.rkeep[k] = (u8)__ffs(r.mask); C.pnode[k] = -1; C.poff[k] = -1;
      elastic |= (r.mask & (r.mask - 1)) != 0;
    }
    cm += __popc(b);
  }
  elastic = __any_sync(TG_FULL, elastic);
  __syncwarp();
  keep = m;
  if (!elastic) return true;
  PoolTask& T = warp_task();
  i64* ac = nullptr; i64* seeds = nullptr;
  int n_ac = 0, ns = 0, first = -1;
  if (m >= 2) {                                           // (a single candidate is never evicted)
    ac = (i64*)slab.take_fast((u64)(nw - n + 1) * 8);
    seeds = (i64*)slab.take_fast((u64)(nr + 1) * 8);
    if (!ac || !seeds) return false;
#pragma unroll 1
    for (int i0 = n; i0 < nw; i0 += 32) {
      const int i = i0 + lane;
      int x = -1; uint4 c = make_uint4(0u, RQ_NOBODY, 1u, 1u);
      if (i < nw) c = replay_facts(P, R, Q, wait, row, i, x);
      const u32 b = __ballot_sync(TG_FULL, RQ_POOL(c.y) == j);
      if ((b >> lane) & 1u) ac[n_ac + __popc(b & ((1u << lane) - 1u))] = replay_rec(P, Q, row, c, x).tl;
      if (first < 0 && b) first = i0 + __ffs(b) - 1;
      n_ac += __popc(b);
    }
    // completion times (relative to now) of what runs on this pool seed the heap
#pragma unroll 1
    for (int i0 = 0; i0 < nr; i0 += 32) {
      const int i = i0 + lane;
      const u32 b = __ballot_sync(TG_FULL, i < nr && RR_POOL(run.pu[i]) == j);
      if ((b >> lane) & 1u) { const i64 f = run.fin[i]; seeds[ns + __popc(b & ((1u << lane) - 1u))] = f > now ? f - now : 0; }
      ns += __popc(b);
    }
  }
  __syncwarp();
  if (lane == 0) {
    T.type = pd.type; T.group = pd.group;
    T.cap[0] = cap0; T.cap[1] = cap1; T.cap[2] = cap2; T.cap[3] = cap3;
    T.m = m; T.cs = C.cs; T.cp = C.cp; T.cmask = C.cmask; T.cg = C.cg;
    T.n_ac = n_ac; T.ac_tmin = ac;
    T.ac_first.s = T.ac_first.p = 0; T.ac_first.mask = 1; T.ac_first.g = 1; T.ac_first.gang = 0;
    if (first >= 0) {
      int x;
      const uint4 c = replay_facts(P, R, Q, wait, row, first, x);
      const ReplayRec r = replay_rec(P, Q, row, c, x);
      T.ac_first.s = r.s; T.ac_first.p = r.p; T.ac_first.mask = r.mask; T.ac_first.g = r.cg & 0x7f; T.ac_first.gang = r.cg >> 7;
    }
    T.seeds = seeds; T.n_seeds = ns;
    T.depth = P.depth;
    T.rsel = C.rsel; T.rkeep = C.rkeep; T.rowcand = C.rowcand;
    T.wk = warp_smem(); T.wk_bytes = WARP_WORK_BYTES;
  }
  __syncwarp();
  keep = evict_loop<4>(P, T, slab, lane);
  return keep >= 0;
}

// the waiting records of a block, from `at` in its shared memory on
template <bool LIST>
__device__ __forceinline__ ReplayQueue<LIST> replay_queue(const ReplayWs& R, char* at) {
  ReplayQueue<LIST> Q;
  Q.cap = R.wcap; Q.head = 0;
  Q.sp = (uint4*)at; Q.ta = Q.sp + Q.cap; Q.c = Q.ta + Q.cap; Q.key = (u64*)(Q.c + Q.cap);
  Q.q = (unsigned short*)(Q.key + Q.cap); Q.free = Q.q + Q.cap;
  return Q;
}
// `started` of the first n actions leave a queue that goes on in global memory (n <= Q.cap < nw): the ones of the prefix that
// stay move up behind the others, and records from global memory take the places that the head then leaves behind.  Only
// those are read; moving every record and every number behind them took 15000 to 260000 cycles a round, a quarter to 38 % of
// a replay whose queue stays long (3000 actions on domains of 256 cores 32.7 -> 22.9 ms, 20000 on 256 cores 943 -> 553).
// Out of line, and with few arguments, since the common path (the whole queue in shared memory) is slower with this text in
// it: 256 x 20000 40.1 ms without, 40.3 out of line, 41.4 in line.
template <bool LIST>
__device__ __noinline__ void replay_leave(const Params& P, const ReplayWs& R, int head, int off, int sc, int n, int nw, int started, int free_slots) {
  extern __shared__ __align__(16) unsigned char k2_smem[];
  const int lane = threadIdx.x;
  const u32 below = (1u << lane) - 1u;
  const size_t row = (size_t)sc * P.N;
  const int* wait = R.wait + row + off; const u64* wkey = R.wkey + row + off;
  ReplayQueue<LIST> Q = replay_queue<LIST>(R, (char*)k2_smem + WARP_SMEM_BYTES + KR_FAST_BYTES + KR_SLOT_BYTES + KR_TABLE_BYTES);
  Q.head = head;
  int to_end = n;
#pragma unroll 1
  for (int i0 = (n - 1) & ~31; i0 >= 0; i0 -= 32) {
    const int i = i0 + lane, x = i < n ? Q.slot(i) : 0;
    const bool gone = i < n && (Q.c[x].y & RQ_STARTED), stay = i < n && !gone;
    const u32 gb = __ballot_sync(TG_FULL, gone), sb = __ballot_sync(TG_FULL, stay);
    const int to = Q.at(stay ? to_end - __popc(sb >> lane) : 0);
    uint4 sp, ta, c;
    if (!LIST && stay) { sp = Q.sp[x]; ta = Q.ta[x]; c = Q.c[x]; }
    if (LIST && gone) Q.free[free_slots + __popc(gb & below)] = (unsigned short)x;
    free_slots += __popc(gb); to_end -= __popc(sb);
    __syncwarp();
    if (stay) { if (LIST) Q.q[to] = (unsigned short)x; else { Q.sp[to] = sp; Q.ta[to] = ta; Q.c[to] = c; } }
    __syncwarp();
  }
  Q.head = Q.at(started < Q.cap ? started : 0);
  const int first = Q.cap - started, end = min(Q.cap, nw - started);
#pragma unroll 1
  for (int p = first + lane; p < end; p += 32) {
    const int a = wait[p + started];
    int y = Q.at(p);
    if (LIST) {
      const int z = Q.free[free_slots - 1 - (p - first)];
      Q.q[y] = (unsigned short)z; y = z;
      if (R.policy) Q.key[y] = wkey[p + started];
    }
    replay_store(Q, y, replay_load(P, row, a), a, replay_last<LIST>(R, row, a));
  }
  __syncwarp();
}

// Two candidates (queue positions ba < bb < 32, in shared memory) on a pool with at most KR_PAIR_RUN actions running in all and
// at most KR_PAIR_WAIT waiting behind the prefix: DPArrange's answer for both (lanes try b's levels, one after
// the other a's), a's alone, and the eviction step between them, without any of the selection's arrays.  Returns how many
// are kept, their levels in ra and rb, or 0: the general path decides (a time beyond 32 bits).  Most selections of a trace
// are of two candidates: with the arrays 11400 cycles each on the `trace` cluster, and 3700 for placing them.
#define KR_PAIR_RUN 30
#define KR_PAIR_WAIT 1024
template <bool LIST>
__device__ __forceinline__ int replay_pair(const Params& P, const PoolDev& pd, const ReplayQueue<LIST>& Q, const ReplayRun& run, size_t row, int j, int ba,
                                           int bb, int n, int nw, int nr, i64 now, const int* slot, int aside, u32* list, int lane, int& ra, int& rb) {
  const int xa = Q.slot(ba), xb = Q.slot(bb);
  const uint4 ca = Q.c[xa], cb = Q.c[xb];
  const ReplayRec A = replay_rec(P, Q, row, ca, xa), B = replay_rec(P, Q, row, cb, xb);
  const bool gpu = pd.type == TG_POOL_GPU;
  const int ga = A.cg & 0x7f, anga = A.cg >> 7, gb = B.cg & 0x7f, angb = B.cg >> 7, r = lane + 1;
  int cap[4] = {slot[0] - aside, 0, 0, 0};
  if (gpu) { cap[1] = slot[1]; cap[2] = slot[2]; cap[3] = slot[3]; }
  const bool has_b = (B.mask >> lane) & 1u;
  const int ub = gb * r, lb = has_b && gpu ? level_of(gb, angb, r) : 0;
  const i64 tb = duration(B.s, B.p, has_b ? r : 1);
  i64 bv = TG_INF; u32 bt = 0xffffffffu;                  // duration sum; units << 12 | b's level << 6 | a's level
#pragma unroll 1
  for (u32 mk = A.mask; mk; mk &= mk - 1) {
    const int x = __ffs(mk), ua = ga * x, la = gpu ? level_of(ga, anga, x) : 0;
    const int m0 = cap[0] - ua, m1 = min(m0, cap[1] - (la >= 1 ? ua : 0)), m2 = min(m1, cap[2] - (la >= 2 ? ua : 0)),
              m3 = min(m2, cap[3] - (la >= 3 ? ua : 0));
    // (b's own class bounds it, a's the levels up to a's: a level that a charges and b does not has to hold a)
    const bool a_fits = la == 0 ? m0 >= 0 : la == 1 ? m1 >= 0 : la == 2 ? m2 >= 0 : m3 >= 0;
    const i64 v = duration(A.s, A.p, x) + tb;
    const u32 t = ((u32)(ua + ub) << 12) | ((u32)r << 6) | (u32)x;
    if (has_b && a_fits && ub <= (lb == 0 ? m0 : lb == 1 ? m1 : lb == 2 ? m2 : m3) && (v < bv || (v == bv && t < bt))) { bv = v; bt = t; }
  }
  const i64 both = warp_min64(bv);
  const u32 t = __reduce_min_sync(TG_FULL, bv == both ? bt : 0xffffffffu);
  const bool has_a = (A.mask >> lane) & 1u;
  const int la = has_a && gpu ? level_of(ga, anga, r) : 0;
  const u32 fits = __ballot_sync(TG_FULL, has_a && ga * r <= pick4(cap, la));
  if (both == TG_INF || !fits) return 0;                  // (cannot happen: the prefix admitted them)
  ra = (int)(t & 63u); rb = (int)((t >> 6) & 63u);
  const int alone = best_level(A.p, fits);
  const i64 t_alone = duration(A.s, A.p, alone), t_first = duration(B.s, B.p, nth_level(B.mask, min(P.depth, __popc(B.mask)) - 1));
  if (ra == alone && duration(B.s, B.p, rb) <= t_first) return 2;      // eviction_cannot_pay
  // ---- what waits on the pool behind them
  int n_ac = 0, first = -1;
#pragma unroll 1
  for (int i0 = n; i0 < nw; i0 += 32) {
    const int i = i0 + lane, x = i < nw ? Q.slot(i) : 0;
    const bool mine = i < nw && RQ_POOL(Q.c[x].y) == j;
    const u32 m = __ballot_sync(TG_FULL, mine);
    if (mine) { const uint4 v = Q.ta[x]; list[n_ac + __popc(m & ((1u << lane) - 1u))] = ev_key(i64_of(v.x, v.y)); }
    if (first < 0 && m) first = i0 + __ffs(m) - 1;
    n_ac += __popc(m);
  }
  i64 fixed = t_alone - both + t_first, first_a = 0;
  if (n_ac > 0) {
    const int x = Q.slot(first);
    const uint4 c = Q.c[x];
    const ReplayRec F = replay_rec(P, Q, row, c, x);
    first_a = duration(F.s, F.p, nth_level(F.mask, min(P.depth, __popc(F.mask)) - 1));
    fixed += F.tl - first_a;
  }
  __syncwarp();
  // ---- the heaps: what runs on the pool, and the candidates behind it
  u32 a[1] = {EV_NONE}, b[1] = {EV_NONE};
  if (lane < nr && RR_POOL(run.pu[lane]) == j) { const i64 f = run.fin[lane]; a[0] = b[0] = ev_key(f > now ? f - now : 0); }
  if (lane == nr) { a[0] = ev_key(duration(A.s, A.p, ra)); b[0] = ev_key(t_alone); }
  if (lane == nr + 1) a[0] = ev_key(duration(B.s, B.p, rb));
  const int pays = ev_run_regs<1, 4>(a, b, nr + 2, n_ac, ev_key(t_first), ev_key(first_a), fixed, [&](int k) { return list[k]; },
                                  (u32)__cvta_generic_to_shared(warp_smem()), lane);
  if (pays < 0) return 0;
  if (pays) { ra = alone; return 1; }
  return 2;
}

// EXT: the queue may be kept sorted by R.policy's key, trajectories pinned on arrival (R.trajectory), further cost-vector
// entries (n_side) and a service cache; the plain instance carries none of their code.  SMEM: live state and running
// actions are in shared memory; the other instance asks at run time.
template <bool EXT, bool SMEM>
__global__ void __launch_bounds__(KR_THREADS, 1) k_replay(const __grid_constant__ Params P, const __grid_constant__ ReplayWs R) {
  extern __shared__ __align__(16) unsigned char k2_smem[];
  const int lane = threadIdx.x;
  const u32 below = (1u << lane) - 1u;
  char* const sm = (char*)k2_smem;                         // (WARP_SMEM_BYTES from here are what warp_smem() hands out)
  char* const fast = sm + WARP_SMEM_BYTES;
  // per-warp arrays behind the selection's work area
  ReplayState Z;
  Z.slot = (int*)(fast + KR_FAST_BYTES);
  Z.node_of = (uint2*)(fast + KR_FAST_BYTES + KR_SLOT_BYTES);
  ReplayQueue<EXT> Q = replay_queue<EXT>(R, fast + KR_FAST_BYTES + KR_SLOT_BYTES + KR_TABLE_BYTES);
  char* const run_at = fast + KR_FAST_BYTES + KR_SLOT_BYTES + KR_TABLE_BYTES + align16((size_t)Q.cap * KR_WAIT_BYTES);
  char* const state_at = run_at + align16((size_t)R.rcap * KR_RUN_BYTES);
#pragma unroll 1
  for (int x = lane; x < 256; x += 32) Z.node_of[x] = replay_node_entry((u32)x);
#pragma unroll 1
  for (int sc = blockIdx.x; sc < P.S; sc += gridDim.x) {
    const size_t row = (size_t)sc * P.N;
    const int n_act = uniform(min(max(P.n_actions[sc], 0), P.N));
    int* wait = R.wait + row; u64* wkey = EXT && R.wkey ? R.wkey + row : nullptr;
    ReplayRun run;
    if (SMEM || R.rcap > 0) {
      run.at = (uint4*)run_at; run.fin = (i64*)(run.at + R.rcap); run.end = (int*)(run.fin + R.rcap); run.pu = (u32*)(run.end + R.rcap);
      run.idx = (int*)(run.pu + R.rcap);
    } else { run.at = R.run_at + row; run.fin = R.run_fin + row; run.end = R.run_end + row; run.pu = R.run_pu + row; run.idx = R.run_idx + row; }
    if (SMEM || R.state_bytes > 0) {
      Z.words = (u32*)state_at; Z.dfree = (int*)(state_at + align16((size_t)(R.W + 2) * 4));
      Z.owner = (int*)((char*)Z.dfree + align16((size_t)(R.Dtot + 1) * 4));
    } else { Z.words = R.words + (size_t)sc * (R.W + 2); Z.dfree = R.dfree + (size_t)sc * (R.Dtot + 1); Z.owner = R.owner + (size_t)sc * R.U; }
    int* occ = R.occupancy ? R.occupancy + (size_t)sc * R.max_rounds * P.P : nullptr;
    int* const o_alloc = P.o_alloc + row; int* const o_node = P.o_node + row; int* const o_off = P.o_off + row; i64* const o_act = P.o_act + row;
    // outputs and state start empty (the occupancy rows were zeroed before)
#pragma unroll 4
    for (int i = lane; i < P.N; i += 32) { o_alloc[i] = 0; o_node[i] = -1; o_off[i] = -1; o_act[i] = -1; }
    int status = 0;
#pragma unroll 2
    for (int i = lane; i < n_act; i += 32) {
      const int j = P.a_pool[row + i];
      int g, gang; u32 eff;
      if (j >= P.P || !decode_levels(P.pool[j], P.a_unit[row + i], P.a_mask[row + i], g, gang, eff)) status |= TG_ST_BAD_ACTION;
      if (EXT)
#pragma unroll 1
        for (int e = 0; e < P.n_side; ++e) {                // further entries: a quota / concurrency pool other than j, 1 .. capacity
          const int k = P.a_side_pool[e * P.side_plane + row + i];
          if (k == 0xff) continue;
          const int c = P.a_side_units[e * P.side_plane + row + i];
          if (k >= P.P || P.pool[k < P.P ? k : 0].type != TG_POOL_API || k == j || c < 1 || c > P.pool[k < P.P ? k : 0].capacity)
            status |= TG_ST_BAD_ACTION;
        }
      if (i > 0 && P.a_arrival && P.a_arrival[row + i - 1] > P.a_arrival[row + i]) status |= TG_ST_UNSORTED;
    }
    status = __reduce_or_sync(TG_FULL, status);
    if (status & TG_ST_BAD_ACTION) status = TG_ST_BAD_ACTION;
    u32 gpu_pools = 0;
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < P.P; ++j) {
      const PoolDev& pd = P.pool[j];
      if (pd.type == TG_POOL_GPU) {
        int taken = 0;
        u32* words = Z.words + R.word0[j];
#pragma unroll 1
        for (int v = lane; v < pd.n_nodes; v += 32) {
          const u32 b = (P.gpu_busy ? P.gpu_busy[(size_t)sc * P.n_nodes_total + pd.node0 + v] : 0u) & ((1u << pd.group) - 1u);
          words[v] = ~b & ((1u << pd.group) - 1u);
          taken += __popc(b);
        }
        taken = warp_sum32(taken);
        if (occ && lane == 0 && status == 0) occ[j] = taken;   // round 0's difference
        __syncwarp();
        replay_gpu_slots(pd, words, Z.node_of, Z.slot, lane);
        gpu_pools |= 1u << j;
      } else if (lane == 0) Z.slot[pd.slot0] = pd.capacity;
      if (pd.type == TG_POOL_API) continue;
#pragma unroll 1
      for (int c = lane; c < pd.capacity; c += 32) Z.owner[R.unit0[j] + c] = -1;
      if (pd.type != TG_POOL_CPU) continue;
      const int wpd = R.wpd[j];
#pragma unroll 1
      for (int w = lane; w < R.n_dom[j] * wpd; w += 32) {
        const int left = pd.group - (w % wpd) * 64;         // cores of the domain from this word on
        const u64 m = left >= 64 ? ~0ull : (1ull << left) - 1ull;
        Z.words[R.word0[j] + 2 * w] = (u32)m; Z.words[R.word0[j] + 2 * w + 1] = (u32)(m >> 32);
      }
#pragma unroll 1
      for (int d = lane; d < R.n_dom[j]; d += 32) Z.dfree[R.dom0[j] + d] = pd.group;
    }
    if (EXT)
#pragma unroll 1
      for (int i = lane; i < Q.cap; i += 32) Q.free[i] = (unsigned short)i;
    Q.head = 0;
    __syncwarp();
    int rounds = 0;
    if (status == 0) {
      int next = 0, nw = 0, nr = 0, r = 0, free_slots = Q.cap;
      bool drained = false, gated = false;                 // gated: an arrival waits for a node (Section 5.2)
      i64 total = 0; int selected = 0;
      int min_end = KR_NEVER;                              // the first round that releases something
      // arrivals, 32 at a time: lane k holds record base + k; the next batch's columns are on their way
      int base = 0;
      int l_pool = 0; u32 l_unit = 1, l_mask = 1; i64 l_s = 0, l_p = 0, l_arr = 0;
      int l_traj = -1; u32 l_mem = 0, l_last = 0;          // (trajectories)
      auto fetch = [&](int from) {
        const int i = from + lane;
        if (i < n_act) {
          if (EXT && R.trajectory) {
            l_traj = R.trajectory[row + i]; l_mem = R.traj_mem[row + i];
            l_last = replay_last<EXT>(R, row, i);
          }
          l_pool = P.a_pool[row + i]; l_unit = P.a_unit[row + i]; l_mask = P.a_mask[row + i]; l_s = P.a_s[row + i]; l_p = P.a_p[row + i];
          l_arr = P.a_arrival ? P.a_arrival[row + i] : 0;
        }
      };
      int b_traj = -1; u32 b_mem = 0, b_last = 0;
      // lane j < P: free memory and cores of node j (-1 cores: not a CPU node)
      i64 node_mem = 0; int node_cores = -1;
      if (EXT && R.trajectory && lane < P.P) {
        node_mem = R.mem_free[(size_t)sc * P.P + lane];
        if (P.pool[lane].type == TG_POOL_CPU) node_cores = P.pool[lane].capacity;
      }
      int* const traj_node = EXT && R.trajectory ? R.traj_node + (size_t)sc * R.max_traj : nullptr;
      ReplayRec b_rec; int b_at = KR_NEVER;                // b_at: the round that admits the lane's arrival
      int next_at = KR_NEVER;
      auto refill = [&](int from) {                        // the batch that was fetched becomes the current one
        base = from;
        b_rec = replay_decode(P, l_pool, l_unit, l_mask, l_s, l_p);
        b_rec.arr = l_arr;
        if (EXT) { b_traj = l_traj; b_mem = l_mem; b_last = l_last; }
        b_at = from + lane < n_act ? round_at(R, l_arr) : KR_NEVER;
        next_at = __shfl_sync(TG_FULL, b_at, 0);
        fetch(from + 32);
      };
      fetch(0);
      refill(0);
      // lane v < 32: free capacity of demand slot v is Z.slot[v]; lane j < P: where pool j's is, and the round in which its
      // quota window turns
      const int D = P.V - P.P;
      const int my_slot = lane < P.P ? P.pool[lane].slot0 : 0;
      const i64 my_window = lane < P.P && P.pool[lane].type == TG_POOL_API ? P.pool[lane].window_us : 0;
      int my_turn = my_window > 0 ? round_at(R, my_window) : KR_NEVER;
      int next_turn = warp_min32(my_turn);
      u32 charged = 0;                                     // bit pool << 2 | class: such a request asks this lane's demand slot
#pragma unroll 1
      for (int j = 0; j < P.P; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (lane >= P.pool[j].slot0 && lane <= P.pool[j].slot0 + c && (c == 0 || P.pool[j].type == TG_POOL_GPU)) charged |= 1u << (4 * j + c);
      while (r < R.max_rounds) {
        const i64 now = (i64)r * R.round_us;
        // 1. quota refill: usage restarts with its window
        if (r >= next_turn) {
          if (r >= my_turn) {
            const int cap = P.pool[lane].capacity, used = cap - Z.slot[my_slot];
            if (occ && used) atomicSub(&occ[(size_t)my_turn * P.P + lane], used);
            Z.slot[my_slot] = cap;
            my_turn = round_at(R, (now / my_window + 1) * my_window);
          }
          next_turn = warp_min32(my_turn);
          __syncwarp();
        }
        // 2. release what has finished, a lane each; the running list is compacted in place
        while (min_end <= r) {
          // (the memory of a trajectory that ends goes back in the order of the rounds)
          const int until = EXT && R.trajectory && R.traj_last ? min_end : r;
          int kept = 0, me = KR_NEVER;
          bool gpus = false;
#pragma unroll 1
          for (int i0 = 0; i0 < nr; i0 += 32) {
            const int i = i0 + lane;
            const int end = i < nr ? run.end[i] : KR_NEVER;
            const bool done = end <= until, stay = i < nr && !done;
            const u32 bd = __ballot_sync(TG_FULL, done), bk = __ballot_sync(TG_FULL, stay);
            if (stay) me = min(me, end);
            if (bd || kept != i0) {
              uint4 at = make_uint4(0u, 0u, 0u, 0u); u32 pu = 0; int a = 0; i64 fin = 0;
              if (i < nr) { at = run.at[i]; pu = run.pu[i]; a = run.idx[i]; fin = run.fin[i]; }
              if (done) {
                // (a GPU pool's slots are worked out again below; its domain, and a quota call's, is nobody's)
                const int units = RR_UNITS(pu);
                gpus |= (pu & RR_GPU) != 0;
                atomicAdd(&Z.slot[RR_SLOT(pu)], units);
                if (!(pu & RR_WIDE)) {
                  atomicOr(Z.words + at.z, at.x);
                  if (at.y) atomicOr(Z.words + at.z + 1, at.y);
                  atomicAdd(Z.dfree + at.w, units);
                }
                if (EXT)
#pragma unroll 1
                  for (int e = 0; e < P.n_side; ++e) {     // a concurrency pool held the action's further amounts until now
                    const int k = P.a_side_pool[e * P.side_plane + row + a];
                    if (k != 0xff && P.pool[k].window_us == 0) atomicAdd(&Z.slot[P.pool[k].slot0], (int)P.a_side_units[e * P.side_plane + row + a]);
                  }
              }
#pragma unroll 1
              for (u32 wide = __ballot_sync(TG_FULL, done && (pu & RR_WIDE)); wide; wide &= wide - 1) {
                const int b = __ffs(wide) - 1, fa = __shfl_sync(TG_FULL, a, b);
                const u32 fpu = __shfl_sync(TG_FULL, pu, b);
                const int from = (int)__shfl_sync(TG_FULL, at.x, b), j = RR_POOL(fpu);
                const PoolDev& pd = P.pool[j];
                const bool cpu = pd.type == TG_POOL_CPU;
                int* ow = Z.owner + R.unit0[j];
                int left = RR_UNITS(fpu);
#pragma unroll 1
                for (int c0 = from & ~31; c0 < pd.capacity && left > 0; c0 += 32) {
                  const int c = c0 + lane;
                  const bool mine = c < pd.capacity && ow[c] == fa;
                  const u32 mb = __ballot_sync(TG_FULL, mine);
                  if (!mb) continue;
                  left -= __popc(mb);
                  if (mine) {
                    ow[c] = -1;
                    const int d = c / pd.group, x = c - d * pd.group;
                    const int w = cpu ? 2 * (d * R.wpd[j] + (x >> 6)) + ((x >> 5) & 1) : d;
                    atomicOr(Z.words + R.word0[j] + w, 1u << (x & 31));
                    if (cpu) atomicAdd(&Z.dfree[R.dom0[j] + d], 1);
                  }
                }
              }
              if (EXT)
#pragma unroll 1
                for (u32 rest = __ballot_sync(TG_FULL, done && (pu & RR_LAST)); rest; rest &= rest - 1) {
                  // the trajectory's last action has ended: its memory goes back to its node
                  const int fa = __shfl_sync(TG_FULL, a, __ffs(rest) - 1), t = R.trajectory[row + fa];
                  const u32 mem = R.traj_mem[row + fa];
                  const int node = t >= 0 && t < R.max_traj ? traj_node[t] : -1;
                  if (lane == node) node_mem += (i64)mem;
                  __syncwarp();
                  if (lane == 0 && node >= 0) traj_node[t] = -1;
                  __syncwarp();
                }
              __syncwarp();
              const int k = kept + __popc(bk & below);
              if (stay && k != i) { run.at[k] = at; run.fin[k] = fin; run.end[k] = end; run.pu[k] = pu; run.idx[k] = a; }
            }
            kept += __popc(bk);
            __syncwarp();
          }
          nr = kept;
          min_end = warp_min32(me);
          gated = false;
          if (__any_sync(TG_FULL, gpus))
#pragma unroll 1
            for (u32 g = gpu_pools; g; g &= g - 1) {
              const int j = __ffs(g) - 1;
              replay_gpu_slots(P.pool[j], Z.words + R.word0[j], Z.node_of, Z.slot, lane);
            }
        }
        // 3. admit arrivals
        bool was_gated = gated;
#pragma unroll 1
        while (next_at <= r && !was_gated) {
          int cnt = __popc(__ballot_sync(TG_FULL, base + lane >= next && b_at <= r));   // sorted: the lanes from next - base on
          const int k0 = next - base;
          if (EXT && R.trajectory) {
            // per-node CPU scheduling: an arrival joins the queue once its trajectory has a node; the first one
            // that finds none waits outside, with everything that arrived after it
            int pool_of = 0xff;
            const bool have = lane >= k0 && lane < k0 + cnt;
            const int pj = RQ_POOL(b_rec.meta);
            const bool mine = have && b_traj >= 0 && b_traj < R.max_traj && P.pool[pj].type == TG_POOL_CPU;
            const int out = pin_chunk(mine, b_traj, b_mem, RQ_UNITS(b_rec.meta), pj, have, traj_node, node_mem, node_cores, lane, pool_of);
            if (have && lane < out) {
              R.pool_rw[row + base + lane] = (u8)pool_of;
              b_rec.meta = (b_rec.meta & ~(7u << 2)) | ((u32)pool_of << 2);
            }
            __syncwarp();
            if (out < k0 + cnt) { cnt = out - k0; was_gated = true; gated = true; }   // the gate
          }
          const bool in = lane >= k0 && lane < k0 + cnt;
          const int pos = nw + lane - k0;                  // queue position of this lane's arrival
          const bool fits = in && pos < Q.cap;
          if (EXT && R.policy) {
            // Other queue orders (Section 4.2): the queue stays sorted by the policy's key, equal keys in arrival order.
            // Each arrival goes behind the last entry whose key is not larger; the tail moves up by one.
#pragma unroll 1
            for (int b = k0; b < k0 + cnt; ++b) {
              const i64 tl = __shfl_sync(TG_FULL, b_rec.tl, b);
              const u64 key = R.policy == 2 ? (u64)((1ll << 42) - tl) : (u64)tl;
              int p = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < nw; i0 += 32) {
                const int i = i0 + lane;
                const u64 ki = i >= nw ? ~0ull : (i < Q.cap ? Q.key[Q.q[Q.at(i)]] : wkey[i]);
                const u32 le = __ballot_sync(TG_FULL, i < nw && ki <= key);
                p += __popc(le);
                if (le != TG_FULL) break;                  // (sorted)
              }
              // what lies in global memory moves up first; the last record in shared memory follows it there
              if (nw >= Q.cap) {
#pragma unroll 1
                for (int hi = nw; hi > max(p, Q.cap);) {
                  const int lo = max(max(p, Q.cap), hi - 32), i = lo + lane;
                  int va = 0; u64 vk = 0;
                  if (i < hi) { va = wait[i]; vk = wkey[i]; }
                  __syncwarp();
                  if (i < hi) { wait[i + 1] = va; wkey[i + 1] = vk; }
                  __syncwarp();
                  hi = lo;
                }
                if (p < Q.cap) {
                  const int x = Q.q[Q.at(Q.cap - 1)];
                  if (lane == 0) { wait[Q.cap] = (int)Q.c[x].x; wkey[Q.cap] = Q.key[x]; Q.free[free_slots] = (unsigned short)x; }
                  ++free_slots;
                  __syncwarp();
                }
              }
              if (p < Q.cap) {
#pragma unroll 1
                for (int hi = min(nw, Q.cap - 1); hi > p;) {
                  const int lo = max(p, hi - 32), i = lo + lane;
                  unsigned short v = 0;
                  if (i < hi) v = Q.q[Q.at(i)];
                  __syncwarp();
                  if (i < hi) Q.q[Q.at(i + 1)] = v;
                  __syncwarp();
                  hi = lo;
                }
                const int x = Q.free[--free_slots];
                __syncwarp();
                if (lane == b) { Q.q[Q.at(p)] = (unsigned short)x; Q.key[x] = key; replay_store(Q, x, b_rec, base + b, EXT ? b_last : 0u); }
              } else if (lane == b) { wait[p] = base + b; wkey[p] = key; }
              __syncwarp();
              ++nw;
            }
          } else {
            if (fits) {
              int x = Q.at(pos);
              if (EXT) { const int y = Q.free[free_slots - 1 - (lane - k0)]; Q.q[x] = (unsigned short)y; x = y; }
              replay_store(Q, x, b_rec, base + lane, EXT ? b_last : 0u);
            } else if (in) wait[pos] = base + lane;
            if (EXT) free_slots -= min(cnt, max(Q.cap - nw, 0));
            nw += cnt;
          }
          next += cnt;
          __syncwarp();
          if (next == base + 32 || next == n_act) {
            next_at = KR_NEVER;
            if (next < n_act) refill(next);
          } else next_at = __shfl_sync(TG_FULL, b_at, next - base);
        }
        // 4. schedule
        int blocked_pool = -1;                             // pool of a head-of-line action that does not fit
        if (nw > 0) {
          const int capreg = lane < D ? Z.slot[lane] : 0;
          __syncwarp();                                    // (before other lanes write the slots, in this round or the next worked one)
          // Candidate prefix (Algorithm 1, line 2): lane v adds up the demand on slot v, action by action
          int n = 0, run_dem = 0, stop_pool = -1, aside = 0;
          u32 present = 0;                                 // pools with candidates; << 8: with elastic ones
          uint4 c0 = make_uint4(0u, RQ_NOBODY, 1u, 1u); int x0 = -1;   // the first 32 positions
#pragma unroll 1
          for (int i0 = 0; i0 < nw; i0 += 32) {
            uint4 c = make_uint4(0u, RQ_NOBODY, 1u, 1u); int x = -1;
            if (i0 + lane < nw) c = replay_facts(P, R, Q, wait, row, i0 + lane, x);
            if (i0 == 0) { c0 = c; x0 = x; }
            const int nb = min(32, nw - i0);
            int k0 = 0xff, u0 = 0, k1 = 0xff, u1 = 0;      // further entries of the cost vector
            if (EXT && P.n_side > 0 && lane < nb) {
              const size_t o = row + (int)c.x;
              k0 = P.a_side_pool[o]; u0 = P.a_side_units[o];
              if (P.n_side > 1) { k1 = P.a_side_pool[P.side_plane + o]; u1 = P.a_side_units[P.side_plane + o]; }
            }
            // (lanes without a record ask for nothing; four steps at a time need one vote)
            int over = 32;                                 // this slot's first action that does not fit
#pragma unroll 1
            for (int b0 = 0; b0 < nb; b0 += 4) {
#pragma unroll
              for (int z = 0; z < 4; ++z) {
                const int b = b0 + z;
                const u32 mb = __shfl_sync(TG_FULL, c.y, b);
                if ((charged >> (mb & 31u)) & 1u) run_dem += RQ_UNITS(mb);
                if (EXT && P.n_side > 0) {
                  const int a0 = __shfl_sync(TG_FULL, k0, b), d0 = __shfl_sync(TG_FULL, u0, b);
                  const int a1 = __shfl_sync(TG_FULL, k1, b), d1 = __shfl_sync(TG_FULL, u1, b);
                  if (a0 != 0xff && lane == P.pool[a0].slot0) run_dem += d0;
                  if (a1 != 0xff && lane == P.pool[a1].slot0) run_dem += d1;
                }
                if (run_dem > capreg) over = min(over, b);
              }
              if (__any_sync(TG_FULL, over < 32)) break;
            }
            over = min(warp_min32(over), nb);
            n += over;
            u32 mine = 0;
            if (lane < over) mine = (1u << RQ_POOL(c.y)) | (c.y & RQ_ELASTIC ? 256u << RQ_POOL(c.y) : 0u);
            present |= __reduce_or_sync(TG_FULL, mine);
            if (EXT && P.n_side > 0)                       // lane j: what is set aside of pool j for the others
#pragma unroll 1
              for (int j = 0; j < P.P; ++j) {
                const int a = warp_sum32(lane < over ? (k0 == j ? u0 : 0) + (k1 == j ? u1 : 0) : 0);
                if (lane == j) aside += a;
              }
            if (over < nb) { stop_pool = RQ_POOL(__shfl_sync(TG_FULL, c.y, over)); break; }
          }
          const int nr0 = nr;
          bool ok = true;
          int my_end = KR_NEVER;                           // first release among what this lane starts
          // the lane's candidate starts (Eq. 2: completion - arrival = waited so far + execution)
          auto start = [&](const PoolDev& pd, int j, int k, int a, int units, i64 fin, i64 arr, const ReplayGrant& G, bool last) {
            const i64 act = fin - arr;
            const int end = max(round_at(R, fin), r + 1);
            o_alloc[a] = units; o_node[a] = G.node; o_off[a] = G.off; o_act[a] = act;
            run.at[k] = G.at; run.pu[k] = rr_pack(pd, j, units, G.wide) | (EXT && last && pd.type == TG_POOL_CPU ? RR_LAST : 0u); run.fin[k] = fin; run.end[k] = end; run.idx[k] = a;
            if (occ) {
              atomicAdd(&occ[(size_t)r * P.P + j], units);
              if (end < R.max_rounds && pd.window_us == 0) atomicSub(&occ[(size_t)end * P.P + j], units);
            }
            total += act; my_end = min(my_end, end);
          };
          // Algorithm 1, line 3: pool by pool
#pragma unroll 1
          for (u32 pools = present & 255u; pools && ok; pools &= pools - 1) {
            const int j = __ffs(pools) - 1;
            const PoolDev& pd = P.pool[j];
            const int slot0 = pd.slot0, aside_j = EXT ? __shfl_sync(TG_FULL, aside, j) : 0;
            int* ow = Z.owner + R.unit0[j];
            int m = 0;
            if (n <= 32) m = __popc(__ballot_sync(TG_FULL, lane < n && RQ_POOL(c0.y) == j));
            else
#pragma unroll 1
              for (int i0 = 0; i0 < n; i0 += 32) {
                int x; u32 meta = RQ_NOBODY;
                if (i0 + lane < n) meta = replay_facts(P, R, Q, wait, row, i0 + lane, x).y;
                m += __popc(__ballot_sync(TG_FULL, RQ_POOL(meta) == j));
              }
            const bool el = (present >> (8 + j)) & 1u;
            const bool cached = EXT && pd.type == TG_POOL_GPU && P.cache_slots > 0;
            int units_now = 0;                             // core pools: what the candidates take
            int pair = 0, ra = 1, rb = 1;                  // of two candidates: how many are kept, their levels
            if (m == 2 && el && n <= 32 && !cached && nr <= KR_PAIR_RUN && nw <= Q.cap && nw - n <= KR_PAIR_WAIT) {
              const u32 mb = __ballot_sync(TG_FULL, lane < n && RQ_POOL(c0.y) == j);
              pair = replay_pair(P, pd, Q, run, row, j, __ffs(mb) - 1, 31 - __clz(mb), n, nw, nr, now, Z.slot + slot0, aside_j, (u32*)fast, lane, ra, rb);
            }
            if ((m == 1 || pair || (!el && (pd.type != TG_POOL_GPU || n <= 32))) && !cached) {
              // Nothing left to choose: each candidate takes its level (a lone one DPArrange's answer in closed form: the
              // feasible level of least duration, the smallest among equals) and is placed in queue order.
              int seen = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < n && seen < m; i0 += 32) {
                uint4 c = c0; int x = x0;
                if (i0 > 0) {
                  c = make_uint4(0u, RQ_NOBODY, 1u, 1u); x = -1;
                  if (i0 + lane < n) c = replay_facts(P, R, Q, wait, row, i0 + lane, x);
                }
                bool mine = i0 + lane < n && RQ_POOL(c.y) == j;
                u32 mb = __ballot_sync(TG_FULL, mine);
                if (!mb) continue;
                if (pair == 1) { mb &= 0u - mb; mine = (mb >> lane) & 1u; }
                ReplayRec rec; rec.s = rec.p = rec.arr = 0;
                if (mine) rec = replay_rec(P, Q, row, c, x);
                int rr = __ffs(c.z);
                if (pair) rr = (mb & below) ? rb : ra;
                else if (m == 1 && el) {
                  const int b = __ffs(mb) - 1;
                  const u32 mk = __shfl_sync(TG_FULL, c.z, b), cg = __shfl_sync(TG_FULL, c.w, b);
                  const int g = cg & 0x7f, gang = (cg >> 7) & 1, rl = lane + 1;
                  const bool has = (mk >> lane) & 1u;
                  const int cl = has && pd.type == TG_POOL_GPU ? level_of(g, gang, rl) : 0;
                  const int room = Z.slot[slot0 + cl] - (cl == 0 ? aside_j : 0);
                  const u32 fits = __ballot_sync(TG_FULL, has && g * rl <= room);
                  if (lane == b && fits) rr = best_level(rec.p, fits);   // (durations do not grow with the level)
                }
                const int units = mine ? (int)(c.w & 0x7f) * rr : 0;
                const i64 fin = now + duration(rec.s, rec.p, rr);
                ReplayGrant G; G.node = 0; G.off = -1; G.at = make_uint4(0u, 0u, 0u, (u32)R.Dtot); G.wide = false;
                if (pd.type == TG_POOL_API) {
                  // Section 5.1: the offset is what was in use before
                  const int incl = warp_incl_scan32(units, lane), free_now = Z.slot[slot0];
                  G.off = pd.capacity - free_now + incl - units;
                  const int all = __shfl_sync(TG_FULL, incl, 31);
                  __syncwarp();                            // every lane has read the slot (a shuffle orders no memory)
                  if (lane == 0) Z.slot[slot0] = free_now - all;
                } else if (pd.type == TG_POOL_GPU) {       // largest chunks first, then queue position
                  const int g = (int)(c.w & 0x7fu), gang = (int)(c.w >> 7) & 1, lz = ilog2(gang ? g * rr : g), nreq = gang ? 1 : rr;
#pragma unroll 1
                  for (u32 todo = mb; todo;) {
                    int b = __ffs(todo) - 1;
                    if (todo & (todo - 1)) b = 31 - (int)(__reduce_max_sync(TG_FULL, (todo >> lane) & 1u ? ((u32)lz << 5) | (u32)(31 - lane) : 0u) & 31u);
                    todo &= ~(1u << b);
                    const ReplayGrant g1 = replay_take_gpus(pd.group, pd.n_nodes, Z.words + R.word0[j], Z.node_of, ow, R.word0[j], R.Dtot,
                                                            __shfl_sync(TG_FULL, lz, b), __shfl_sync(TG_FULL, nreq, b), __shfl_sync(TG_FULL, (int)c.x, b), lane);
                    if (lane == b) G = g1;
                  }
                } else {
                  // lane d: free cores and masks of domain d
                  const int n_dom = R.n_dom[j];
                  u32* words = Z.words + R.word0[j]; int* dfree = Z.dfree + R.dom0[j];
                  const bool direct = R.wpd[j] == 1 && n_dom <= 32;
                  int f = -1; u32 lo = 0, hi = 0;
                  auto load = [&]() { if (direct && lane < n_dom) { f = dfree[lane]; lo = words[2 * lane]; hi = words[2 * lane + 1]; } };
                  auto save = [&]() { if (direct && lane < n_dom) { dfree[lane] = f; words[2 * lane] = lo; words[2 * lane + 1] = hi; } __syncwarp(); };
                  load();
#pragma unroll 1
                  for (u32 todo = mb; todo; todo &= todo - 1) {
                    const int b = __ffs(todo) - 1, k = __shfl_sync(TG_FULL, units, b);
                    const u32 mn = __reduce_min_sync(TG_FULL, f >= k ? ((u32)f << 5) | (u32)lane : 0xffffffffu);
                    units_now += k;
                    if (mn != 0xffffffffu) {               // fewest free cores that still fit, lowest domain, lowest cores
                      const int d = (int)(mn & 31u);
                      u32 tlo, thi;
                      lowest_bits(__shfl_sync(TG_FULL, lo, d), __shfl_sync(TG_FULL, hi, d), k, lane, tlo, thi);
                      if (lane == d) { f -= k; lo &= ~tlo; hi &= ~thi; }
                      if (lane == b) { G.node = d; G.at = make_uint4(tlo, thi, (u32)(R.word0[j] + 2 * d), (u32)(R.dom0[j] + d)); }
                    } else {
                      save();
                      const ReplayGrant g1 = replay_take_cores(pd.group, n_dom, R.wpd[j], words, dfree, ow, R.word0[j], R.dom0[j],
                                                               k, __shfl_sync(TG_FULL, (int)c.x, b), lane);
                      if (lane == b) G = g1;
                      load();
                    }
                  }
                  save();
                  if (G.off < 0) G.off = G.node * pd.group + (G.at.x ? __ffs(G.at.x) - 1 : 31 + __ffs(G.at.y));
                }
                if (mine) {
                  if (x >= 0) Q.c[x].y = c.y | RQ_STARTED;
                  start(pd, j, nr + __popc(mb & below), (int)c.x, units, fin, rec.arr, G, c.w & 256u);
                }
                nr += __popc(mb); seen += __popc(mb); selected += __popc(mb);
                __syncwarp();
              }
            } else {
              Slab slab;
              slab.base = P.slabs + (u64)blockIdx.x * P.slab_bytes; slab.cap = P.slab_bytes; slab.used = 0;
              slab.fbase = fast; slab.fcap = KR_FAST_BYTES; slab.fused = 0;
              CandArrays C; int keep = 0;
              ok = replay_select(P, R, Q, run, wait, row, j, n, nw, nr, m, now, Z.slot[slot0] - aside_j, Z.slot[(slot0 + 1) & 31],
                                 Z.slot[(slot0 + 2) & 31], Z.slot[(slot0 + 3) & 31], slab, C, keep, lane);
              if (!ok) break;
              const u8* missed = nullptr;                  // candidates whose chunk did not cache their service
              if (cached) {
                const size_t cbase = ((size_t)sc * P.n_nodes_total + pd.node0) * 8 * P.cache_slots;
                place_gpu_cache(pd, FreeNodes{Z.words + R.word0[j]}, keep, C.cg, C.rkeep, C.cidx, C.pnode, C.poff, C.rsel, C.rowcand,
                                P.a_service ? P.a_service + row : nullptr, P.cache_tag + cbase, P.cache_use + cbase, P.cache_slots, now, lane,
                                warp_smem(), WARP_WORK_BYTES, ow);
                missed = C.rsel;
              } else if (pd.type == TG_POOL_GPU) {
                // Section 5.3: by size, largest first, then queue position
#pragma unroll 1
                for (int lz = 3; lz >= 0; --lz)
#pragma unroll 1
                  for (int i0 = 0; i0 < keep; i0 += 32) {
                    const int i = i0 + lane;
                    int nreq = 0;
                    if (i < keep) {
                      const int g = C.cg[i] & 0x7f, ri = C.rkeep[i];
                      nreq = C.cg[i] >> 7 ? (g * ri == 1 << lz ? 1 : 0) : (g == 1 << lz ? ri : 0);
                    }
#pragma unroll 1
                    for (u32 todo = __ballot_sync(TG_FULL, nreq > 0); todo; todo &= todo - 1) {
                      const int b = __ffs(todo) - 1;
                      const ReplayGrant G = replay_take_gpus(pd.group, pd.n_nodes, Z.words + R.word0[j], Z.node_of, ow, R.word0[j], R.Dtot, lz,
                                                             __shfl_sync(TG_FULL, nreq, b), C.cidx[i0 + b], lane);
                      if (lane == b) { C.pnode[i] = G.node; C.poff[i] = G.off; }
                    }
                  }
              } else if (pd.type == TG_POOL_CPU) {
#pragma unroll 1
                for (int i = 0; i < keep; ++i) {
                  const int units = (C.cg[i] & 0x7f) * C.rkeep[i];
                  const ReplayGrant G = replay_take_cores(pd.group, R.n_dom[j], R.wpd[j], Z.words + R.word0[j], Z.dfree + R.dom0[j], ow,
                                                          R.word0[j], R.dom0[j], units, C.cidx[i], lane);
                  if (lane == 0) { C.pnode[i] = G.node; C.poff[i] = G.off; run.at[nr + i] = G.at; C.rsel[i] = G.wide ? 1 : 0; }
                  units_now += units;
                }
              } else if (lane == 0) {
                int used = pd.capacity - Z.slot[slot0];
#pragma unroll 1
                for (int i = 0; i < keep; ++i) { C.pnode[i] = 0; C.poff[i] = used; used += (C.cg[i] & 0x7f) * C.rkeep[i]; }
                Z.slot[slot0] = pd.capacity - used;
              }
              __syncwarp();
#pragma unroll 1
              for (int i = lane; i < keep; i += 32) {
                const int g = C.cg[i] & 0x7f, rr = C.rkeep[i], units = g * rr, a = C.cidx[i];
                i64 fin = now + duration(C.cs[i], C.cp[i], rr);
                if (EXT && missed && missed[i] && P.a_restore) fin += clamp_param(P.a_restore[row + a]);   // restoration precedes execution
                ReplayGrant G;
                G.node = C.pnode[i]; G.off = C.poff[i]; G.wide = false; G.at = make_uint4(0u, 0u, 0u, (u32)R.Dtot);
                if (pd.type == TG_POOL_CPU) { G.at = run.at[nr + i]; G.wide = C.rsel[i] != 0; }
                else if (pd.type == TG_POOL_GPU) {
                  G.wide = !(C.cg[i] >> 7) && rr > 1;      // chunks of replicas lie anywhere
                  G.at.x = G.wide ? 0u : ((1u << units) - 1u) << G.off; G.at.z = (u32)(R.word0[j] + G.node);
                }
                start(pd, j, nr + i, a, units, fin, P.a_arrival ? P.a_arrival[row + a] : 0, G, replay_last<EXT>(R, row, a) != 0u);
              }
              // the kept ones are the pool's first `keep` in queue order
              int seen = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < n && seen < keep; i0 += 32) {
                int x = -1; u32 meta = RQ_NOBODY;
                if (i0 + lane < n) meta = replay_facts(P, R, Q, wait, row, i0 + lane, x).y;
                const bool mine = RQ_POOL(meta) == j;
                const u32 mb = __ballot_sync(TG_FULL, mine);
                if (mine && seen + __popc(mb & below) < keep && x >= 0) Q.c[x].y = meta | RQ_STARTED;
                seen += __popc(mb);
              }
              nr += keep; selected += keep;
              __syncwarp();
            }
            if (pd.type == TG_POOL_GPU) replay_gpu_slots(pd, Z.words + R.word0[j], Z.node_of, Z.slot, lane);
            else if (pd.type == TG_POOL_CPU && lane == 0) Z.slot[slot0] -= units_now;
            __syncwarp();
          }
          if (!ok) { status = TG_ST_WORKSPACE; break; }
          const int started = nr - nr0;
          if (EXT && P.n_side > 0 && started) {             // the started actions consume their further amounts
#pragma unroll 1
            for (int i = nr0 + lane; i < nr; i += 32)
#pragma unroll 1
              for (int e = 0; e < P.n_side; ++e) {
                const size_t o = e * P.side_plane + row + run.idx[i];
                const int k = P.a_side_pool[o];
                if (k == 0xff) continue;
                const int c = (int)P.a_side_units[o];
                atomicSub(&Z.slot[P.pool[k].slot0], c);
                if (occ) {
                  atomicAdd(&occ[(size_t)r * P.P + k], c);
                  if (P.pool[k].window_us == 0 && run.end[i] < R.max_rounds) atomicSub(&occ[(size_t)run.end[i] * P.P + k], c);
                }
              }
            __syncwarp();
          }
          if (started) min_end = min(min_end, warp_min32(my_end));
          // What does not fit behind candidates that all started does not fit until something ends on its pool: they hold at
          // least what the prefix counted for them.
          if (started == n) blocked_pool = stop_pool;
          // the started actions leave the queue
          if (started && nw <= Q.cap) {
            if (EXT || started < n) {
              int to_end = n;                              // the ones that stay move up behind the others, last first
#pragma unroll 1
              for (int i0 = (n - 1) & ~31; i0 >= 0; i0 -= 32) {
                const int i = i0 + lane, x = i < n ? Q.slot(i) : 0;
                const bool gone = i < n && (started == n || (Q.c[x].y & RQ_STARTED));
                const u32 gb = __ballot_sync(TG_FULL, gone);
                if (EXT) {
                  if (gone) Q.free[free_slots + __popc(gb & below)] = (unsigned short)x;
                  free_slots += __popc(gb);
                }
                if (started < n) {
                  const bool stay = i < n && !gone;
                  const u32 sb = __ballot_sync(TG_FULL, stay);
                  const int to = Q.at(stay ? to_end - __popc(sb >> lane) : 0);
                  uint4 sp, ta, c;
                  if (!EXT && stay) { sp = Q.sp[x]; ta = Q.ta[x]; c = Q.c[x]; }
                  __syncwarp();
                  if (stay) { if (EXT) Q.q[to] = (unsigned short)x; else { Q.sp[to] = sp; Q.ta[to] = ta; Q.c[to] = c; } }
                  to_end -= __popc(sb);
                  __syncwarp();
                }
              }
            }
            Q.head = Q.at(started < Q.cap ? started : 0);
            nw -= started;
            __syncwarp();
          } else if (started && n <= Q.cap) {               // a queue that goes on in global memory
            // `wait` and `wkey` point to where queue position 0 would be, so that nothing moves there (what started since that
            // part was last empty and what waits are different actions: it never outgrows its row)
            replay_leave<EXT>(P, R, Q.head, (int)(wait - (R.wait + row)), sc, n, nw, started, free_slots);
            Q.head = Q.at(started < Q.cap ? started : 0);
            nw -= started;
            if (EXT) free_slots += Q.cap - min(Q.cap, nw);
            if (nw > Q.cap) { wait += started; if (EXT && R.policy) wkey += started; }
            else { wait = R.wait + row; if (EXT && R.policy) wkey = R.wkey + row; }
          } else if (started) {                             // ... as the prefix does: all of it moves up
            int kw = 0;
#pragma unroll 1
            for (int i0 = 0; i0 < nw; i0 += 32) {
              const int i = i0 + lane;
              bool stay = false; int x = 0, a = 0; u64 kk = 0;
              if (i < min(nw, Q.cap)) { x = Q.slot(i); stay = !(Q.c[x].y & RQ_STARTED); }
              else if (i < nw) { a = wait[i]; stay = o_act[a] < 0; if (EXT && R.policy) kk = wkey[i]; }
              const u32 b = __ballot_sync(TG_FULL, stay), gone = __ballot_sync(TG_FULL, i < min(nw, Q.cap) && !stay);
              const int to = kw + __popc(b & below);
              uint4 sp, ta, c;
              if (!EXT && stay && i < Q.cap) { sp = Q.sp[x]; ta = Q.ta[x]; c = Q.c[x]; }
              __syncwarp();
              if (stay && i < Q.cap) {
                const int y = Q.at(to);
                if (EXT) Q.q[y] = (unsigned short)x; else { Q.sp[y] = sp; Q.ta[y] = ta; Q.c[y] = c; }
              } else if (stay && to >= Q.cap) { wait[to] = a; if (EXT && R.policy) wkey[to] = kk; }
              if (EXT) {
                if ((gone >> lane) & 1u) Q.free[free_slots + __popc(gone & below)] = (unsigned short)x;
                free_slots += __popc(gone);
              }
              __syncwarp();
              const u32 mv = __ballot_sync(TG_FULL, stay && i >= Q.cap && to < Q.cap);
              if ((mv >> lane) & 1u) {                      // a record moves up into shared memory
                int y = Q.at(to);
                if (EXT) { const int z = Q.free[free_slots - 1 - __popc(mv & below)]; Q.q[y] = (unsigned short)z; y = z; Q.key[y] = kk; }
                replay_store(Q, y, replay_load(P, row, a), a, replay_last<EXT>(R, row, a));
              }
              if (EXT) free_slots -= __popc(mv);
              __syncwarp();
              kw += __popc(b);
            }
            nw = kw;
            if (nw <= Q.cap) { wait = R.wait + row; if (EXT && R.policy) wkey = R.wkey + row; }
          }
        }
        // 5. the next round in which something can start
        if (next == n_act && nw == 0 && nr == 0) { drained = true; ++r; break; }
        int r_next = r + 1;
        if (nw == 0) {
          // empty queue: the next arrival (a gated one waits for a completion), after the last one the last completion
          r_next = gated ? min_end : next_at;
          if (next == n_act) {
            int last = 0;
#pragma unroll 1
            for (int i = lane; i < nr; i += 32) last = max(last, run.end[i]);
            r_next = warp_max32(last);
          }
        } else if (blocked_pool >= 0) {
          // The action at the head of the queue does not fit, so nothing can start until an action that runs ends, a quota
          // window turns or (in a sorted queue) an arrival becomes the head.
          if (EXT && (P.n_side > 0 || R.trajectory)) {
            // (the head may wait for any pool's amounts; an arrival would be pinned against the memory free at its time)
            r_next = min(min(gated ? KR_NEVER : next_at, min_end), next_turn);
          } else {
            // ... on its pool: arrivals join behind it
            r_next = __shfl_sync(TG_FULL, my_turn, blocked_pool);
            if (EXT && R.policy) r_next = min(r_next, next_at);
            int e = KR_NEVER;
#pragma unroll 1
            for (int i = lane; i < nr; i += 32)
              if (RR_POOL(run.pu[i]) == blocked_pool) e = min(e, run.end[i]);
            r_next = min(r_next, warp_min32(e));
          }
        }
        r_next = max(r_next, r + 1);
        // (the last round still gives back what ends by then)
        if (r_next >= R.max_rounds) r_next = r < R.max_rounds - 1 ? R.max_rounds - 1 : R.max_rounds;
        r = r_next;
      }
      rounds = drained ? r : R.max_rounds;
      if (!drained && r < R.max_rounds) rounds = r;
      if (EXT && R.trajectory && lane < P.P) R.mem_free[(size_t)sc * P.P + lane] = node_mem;
      total = warp_sum64(total);
      if (lane == 0) { P.o_total[sc] = total; P.o_nsel[sc] = selected; P.o_status[sc] = status; }
    } else if (lane == 0) { P.o_total[sc] = 0; P.o_nsel[sc] = 0; P.o_status[sc] = status; }
    if (lane == 0) R.rounds_used[sc] = rounds;
    __syncwarp();
  }
}

// Occupancy: running sums of the differences that k_replay left, in place, one block per scenario; rows behind the last
// round are zero.  Every thread adds up KOCC_ROWS consecutive rounds of a pool.
#define KOCC_ROWS 8
__global__ void __launch_bounds__(256) k_occupancy(int n_pools, int max_rounds, const int* rounds_used, const int* status, int* occupancy) {
  __shared__ int part[TG_MAX_POOLS][8];
  __shared__ int carry[TG_MAX_POOLS];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int* occ = occupancy + (size_t)blockIdx.x * max_rounds * n_pools;
  const int rounds = min(rounds_used[blockIdx.x], max_rounds);
  if (t < TG_MAX_POOLS) carry[t] = 0;
  __syncthreads();
  for (int r0 = 0; r0 < rounds; r0 += 256 * KOCC_ROWS) {
    const int first = r0 + t * KOCC_ROWS;
    for (int j = 0; j < n_pools; ++j) {
      int v[KOCC_ROWS], sum = 0;
#pragma unroll
      for (int k = 0; k < KOCC_ROWS; ++k) { v[k] = first + k < rounds ? occ[(size_t)(first + k) * n_pools + j] : 0; sum += v[k]; }
      const int incl = warp_incl_scan32(sum, lane);
      if (lane == 31) part[j][warp] = incl;
      __syncthreads();
      int run = carry[j] + incl - sum, all = 0;
      for (int w = 0; w < 8; ++w) { if (w < warp) run += part[j][w]; all += part[j][w]; }
#pragma unroll
      for (int k = 0; k < KOCC_ROWS; ++k) { run += v[k]; if (first + k < rounds) occ[(size_t)(first + k) * n_pools + j] = run; }
      __syncthreads();
      if (t == 0) carry[j] += all;
      __syncthreads();
    }
  }
  if (status[blockIdx.x])                                  // (a replay that broke off leaves differences behind its last round)
    for (size_t x = (size_t)rounds * n_pools + t; x < (size_t)max_rounds * n_pools; x += 256) occ[x] = 0;
}
