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
  u32* cores;       // [S][W][2] free cores of every domain word (bit = core)
  int* dfree;       // [S][Dtot] free cores per NUMA domain
  int* owner;       // [S][U]  action holding each core / GPU of a grant over several words or chunks
  u8* nm;           // [S][nodes] GPU busy masks
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
  int state_bytes;  // > 0: a scenario's live state (cores .. nm) takes that many bytes of the warp's shared memory
  int wcap, rcap;   // waiting records / running actions in shared memory (rcap 0: running actions in global memory)
};

__host__ __device__ __forceinline__ size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }
// bytes of the live state: masks and free counts, owners, node masks
__host__ __device__ __forceinline__ size_t replay_state_bytes(const ReplayWs& R, int n_nodes) {
  return align16((size_t)R.W * 8) + align16((size_t)R.Dtot * 4) + align16((size_t)R.U * 4) + align16((size_t)n_nodes + 1);
}

#define KR_THREADS 32
#define KR_FAST_BYTES 8192        // shared-memory window of the selection's arrays
#define KR_WAIT_BYTES 60          // per waiting record: three 16-byte pieces, key, queue, free list
#define KR_RUN_BYTES 36
#define KR_STATE_MAX 16384
#define KR_SLOT_BYTES 128         // free capacity of the 32 demand slots at most
// shared memory of a block (one warp) without the parts sized by the round
#define KR_BASE_BYTES (WARP_SMEM_BYTES + KR_FAST_BYTES + KR_SLOT_BYTES + 64)
#define KR_NEVER 0x7fffffff

// Waiting records: slots that do not move, and the queue as a ring of slot numbers.  sp: s, p; ta: least duration,
// arrival; c: action, meta, mask, unit byte.  meta: pool (4 bits), first demand slot (6), chunk class of the least
// level (2), units of the least level (13), elastic (1); bit 31: started in this round.
struct ReplayQueue {
  uint4* sp; uint4* ta; uint4* c; u64* key; unsigned short* q; unsigned short* free;
  int cap, head;
  __device__ __forceinline__ int at(int i) const { const int k = head + i; return k >= cap ? k - cap : k; }   // ring place of position i < cap
};
#define RQ_POOL(m) ((int)((m) & 15u))
#define RQ_SLOT(m) ((int)(((m) >> 4) & 63u))
#define RQ_CLASS(m) ((int)(((m) >> 10) & 3u))
#define RQ_UNITS(m) ((int)(((m) >> 12) & 0x1fffu))
#define RQ_ELASTIC 0x2000000u
#define RQ_STARTED 0x80000000u
#define RQ_NOBODY 15u             // meta of a lane without a record: no pool, no demand

// Running actions.  end: the round that releases it; pu: units (21 bits), first demand slot (5), pool (3), type (2), wide
// (1); at: what it holds - mask (64 bits), word or node, domain.  A wide grant's units are the ones whose owner it is.
struct ReplayRun { uint4* at; i64* fin; int* end; u32* pu; int* idx; };
#define RR_UNITS(v) ((int)((v) & 0x1fffffu))
#define RR_SLOT(v) ((int)(((v) >> 21) & 31u))
#define RR_POOL(v) ((int)(((v) >> 26) & 7u))
#define RR_TYPE(v) ((int)(((v) >> 29) & 3u))
#define RR_WIDE 0x80000000u
__device__ __forceinline__ u32 rr_pack(const PoolDev& pd, int j, int units, bool wide) {
  return (u32)units | ((u32)pd.slot0 << 21) | ((u32)j << 26) | ((u32)pd.type << 29) | (wide ? RR_WIDE : 0u);
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
  r.meta = (u32)j | ((u32)pd.slot0 << 4) | ((u32)c << 10) | ((u32)(g * rmin) << 12) | (eff & (eff - 1) ? RQ_ELASTIC : 0u);
  return r;
}
__device__ __forceinline__ ReplayRec replay_load(const Params& P, size_t row, int a) {
  ReplayRec r = replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], P.a_s[row + a], P.a_p[row + a]);
  r.arr = P.a_arrival ? P.a_arrival[row + a] : 0;
  return r;
}
__device__ __forceinline__ void replay_store(const ReplayQueue& Q, int x, const ReplayRec& r, int a) {
  Q.sp[x] = make_uint4((u32)r.s, (u32)((u64)r.s >> 32), (u32)r.p, (u32)((u64)r.p >> 32));
  Q.ta[x] = make_uint4((u32)r.tl, (u32)((u64)r.tl >> 32), (u32)r.arr, (u32)((u64)r.arr >> 32));
  Q.c[x] = make_uint4((u32)a, r.meta, r.mask, (u32)r.cg);
}
// action, meta, mask and unit byte at a queue position (any lane's own); x: its slot where it is in shared memory
__device__ __forceinline__ uint4 replay_facts(const Params& P, const ReplayQueue& Q, const int* wait, size_t row, int i, int& x) {
  if (i < Q.cap) { x = Q.q[Q.at(i)]; return Q.c[x]; }
  const int a = wait[i];
  const ReplayRec r = replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], 0, 0);
  x = -1;
  return make_uint4((u32)a, r.meta, r.mask, (u32)r.cg);
}
// ... and the rest of a record whose facts are known
__device__ __forceinline__ ReplayRec replay_rec(const Params& P, const ReplayQueue& Q, size_t row, const uint4& c, int x) {
  if (x < 0) return replay_load(P, row, (int)c.x);
  const uint4 u = Q.sp[x], v = Q.ta[x];
  ReplayRec r;
  r.s = i64_of(u.x, u.y); r.p = i64_of(u.z, u.w); r.tl = i64_of(v.x, v.y); r.arr = i64_of(v.z, v.w);
  r.meta = c.y; r.mask = c.z; r.cg = (u8)c.w;
  return r;
}

// Live state of the scenario at hand: in the warp's shared memory, or in the arrays of ReplayWs where it is large.
// slot: free capacity per demand slot, always in shared memory.
struct ReplayState { u32* cores; int* dfree; int* owner; u8* nm; int* slot; };

// What a grant holds: a mask of one word (core pools) or node (GPU pools), or owner entries (wide).
// node / off: NUMA domain or GPU node, and the first core or GPU.
struct ReplayGrant { int node, off, word, dom; u32 lo, hi; bool wide; };

// One grant of k cores on a pool with cores in use: fewest free cores that still fit, lowest domain, lowest cores first;
// else ascending domains.  cores / dfree / owner: the pool's own rows.
__device__ __forceinline__ ReplayGrant replay_take_cores(int group, int n_dom, int wpd, u32* cores, int* dfree, int* owner,
                                                         int k, int id, int lane) {
  ReplayGrant G;
  G.node = G.off = -1; G.word = 0; G.dom = 0; G.lo = G.hi = 0; G.wide = false;
  int dom = -1;
  if (n_dom <= 32 && group < (1 << 26)) {
    const int f = lane < n_dom ? dfree[lane] : -1;
    const u32 mn = __reduce_min_sync(TG_FULL, f >= k ? ((u32)f << 5) | (u32)lane : 0xffffffffu);
    if (mn != 0xffffffffu) dom = (int)(mn & 31u);
  } else {
    u32 best = 0xffffffffu; int at = -1;
#pragma unroll 1
    for (int d = lane; d < n_dom; d += 32) { const int f = dfree[d]; if (f >= k && (u32)f < best) { best = (u32)f; at = d; } }
    const u32 mn = __reduce_min_sync(TG_FULL, best);
    if (mn != 0xffffffffu) dom = (int)__reduce_min_sync(TG_FULL, best == mn ? (u32)at : 0xffffffffu);
  }
  int need = k;
  const int end = dom >= 0 ? (dom + 1) * wpd : n_dom * wpd;
#pragma unroll 1
  for (int w = dom >= 0 ? dom * wpd : 0; w < end && need > 0; ++w) {
    const uint2 m = *(const uint2*)(cores + 2 * w);
    if ((m.x | m.y) == 0u) continue;
    // the lowest `need` free cores of the word: every lane looks at two of them
    const u32 below = (1u << lane) - 1u;
    const int nlo = __popc(m.x);
    const u32 lo = __ballot_sync(TG_FULL, ((m.x >> lane) & 1u) && __popc(m.x & below) < need);
    const u32 hi = __ballot_sync(TG_FULL, ((m.y >> lane) & 1u) && nlo + __popc(m.y & below) < need);
    const int got = __popc(lo) + __popc(hi);
    const int d = wpd == 1 ? w : w / wpd, c0 = d * group + (wpd == 1 ? 0 : (w - d * wpd) * 64);   // the word's first core
    if (G.off < 0) {
      G.off = c0 + (lo ? __ffs(lo) - 1 : 31 + __ffs(hi)); G.node = d;
      G.word = w; G.dom = d; G.lo = lo; G.hi = hi;
      G.wide = got < need;
      if (G.wide) G.dom = G.off;                           // (where the search for its cores begins)
    }
    if (G.wide) {
      if ((lo >> lane) & 1u) owner[c0 + lane] = id;
      if ((hi >> lane) & 1u) owner[c0 + 32 + lane] = id;
    }
    __syncwarp();
    if (lane == 0) { *(uint2*)(cores + 2 * w) = make_uint2(m.x & ~lo, m.y & ~hi); dfree[d] -= got; }
    need -= got;
    __syncwarp();
  }
  return G;
}

// One candidate alone on a GPU pool: nreq chunks of 2^lz GPUs (Section 5.3: smallest sufficient maximal free block,
// lowest node, lowest start); node / off: the first chunk.
__device__ __forceinline__ ReplayGrant replay_take_gpus(const PoolDev& pd, u8* nm, int* owner, int lz, int nreq, int id, int lane) {
  ReplayGrant G;
  G.node = G.off = -1; G.word = 0; G.dom = 0; G.lo = G.hi = 0; G.wide = nreq > 1;
  const int top = ilog2(pd.group), z = 1 << lz;
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
#pragma unroll 1
  for (int rep = 0; rep < nreq; ++rep) {
    u32 best = 0xffffffffu;                                // level << 24 | node
#pragma unroll 1
    for (int v = lane; v < pd.n_nodes; v += 32) {
      const u32 lev = node_levels(nm[v] | pad) & (~0u << lz);   // the smallest sufficient block of the node
      if (lev) best = min(best, ((u32)(__ffs(lev) - 1) << 24) | (u32)v);
    }
    best = __reduce_min_sync(TG_FULL, best);
    const int at = (int)(best & 0xffffffu), level = (int)(best >> 24);
    if (level > top) continue;                             // cannot happen: the selection fits
    const u32 busy = nm[at];
    const int start = node_block_start(busy | pad, level);
    const u32 bits = ((1u << z) - 1u) << start;
    __syncwarp();
    if (lane == 0) nm[at] = (u8)(busy | bits);
    if (G.wide && lane < z) owner[at * pd.group + start + lane] = id;
    if (rep == 0) { G.node = at; G.off = start; G.word = at; G.lo = bits; }
    __syncwarp();
  }
  return G;
}

// free capacity of a GPU pool's four demand slots
__device__ __forceinline__ void replay_gpu_slots(const PoolDev& pd, const u8* nm_row, int* slot, int lane) {
  int c[4];
  if (pd.n_nodes <= 32) {
    // the four counts of free blocks in one word: at most 256, 128, 64 and 32
    const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
    u32 x = 0;
    if (lane < pd.n_nodes) {
      const NodeBlocks b = node_blocks(nm_row[pd.node0 + lane] | pad);
      x = (u32)__popc(b.s1) | ((u32)__popc(b.s2) << 9) | ((u32)__popc(b.s4) << 17) | ((u32)__popc(b.s8) << 24);
    }
    x = __reduce_add_sync(TG_FULL, x);
    c[3] = (int)(x >> 24) * 8; c[2] = c[3] + (int)((x >> 17) & 127u) * 4; c[1] = c[2] + (int)((x >> 9) & 255u) * 2; c[0] = c[1] + (int)(x & 511u);
  } else gpu_caps(pd, nm_row, lane, c);
  if (lane < 4) slot[pd.slot0 + lane] = pick4(c, lane);
  __syncwarp();
}

// The selection of a pool with a choice to make: its candidates (among the first n positions) and, where an eviction
// step can look at them, the waiting actions behind and the running ones are gathered into arrays.
template <bool EXT>
__device__ __forceinline__ bool replay_select(const Params& P, const ReplayQueue Q, const ReplayRun run, const int* wait, int sc, int j,
                                           int n, int nw, int nr, int m, i64 now, int cap0, int cap1, int cap2, int cap3, Slab& slab,
                                           CandArrays& C, int& keep, int lane) {
  const size_t row = (size_t)sc * P.N;
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
    if (i < n) c = replay_facts(P, Q, wait, row, i, x);
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
      if (i < nw) c = replay_facts(P, Q, wait, row, i, x);
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
      const uint4 c = replay_facts(P, Q, wait, row, first, x);
      const ReplayRec r = replay_rec(P, Q, row, c, x);
      T.ac_first.s = r.s; T.ac_first.p = r.p; T.ac_first.mask = r.mask; T.ac_first.g = r.cg & 0x7f; T.ac_first.gang = r.cg >> 7;
    }
    T.seeds = seeds; T.n_seeds = ns;
    T.depth = P.depth;
    T.rsel = C.rsel; T.rkeep = C.rkeep; T.rowcand = C.rowcand;
    T.wk = warp_smem(); T.wk_bytes = WARP_WORK_BYTES;
  }
  __syncwarp();
  keep = evict_loop(P, T, slab, lane);
  return keep >= 0;
}

// EXT: the queue may be kept sorted by R.policy's key, trajectories pinned on arrival (R.trajectory), further cost-vector
// entries (n_side) and a service cache; the plain instance carries none of their code.
template <bool EXT>
__global__ void __launch_bounds__(KR_THREADS, 1) k_replay(const __grid_constant__ Params P, const __grid_constant__ ReplayWs R) {
  extern __shared__ __align__(16) unsigned char k2_smem[];
  const int lane = threadIdx.x;
  const u32 below = (1u << lane) - 1u;
  char* const sm = (char*)(((u64)k2_smem + 15u) & ~(u64)15);
  char* const fast = sm + WARP_SMEM_BYTES;
  // per-warp arrays behind the selection's work area
  ReplayQueue Q;
  Q.cap = R.wcap;
  {
    char* at = fast + KR_FAST_BYTES + KR_SLOT_BYTES;
    Q.sp = (uint4*)at; Q.ta = Q.sp + Q.cap; Q.c = Q.ta + Q.cap; Q.key = (u64*)(Q.c + Q.cap);
    Q.q = (unsigned short*)(Q.key + Q.cap); Q.free = Q.q + Q.cap;
  }
  char* const run_at = fast + KR_FAST_BYTES + KR_SLOT_BYTES + align16((size_t)Q.cap * KR_WAIT_BYTES);
  char* const state_at = run_at + align16((size_t)R.rcap * KR_RUN_BYTES);
#pragma unroll 1
  for (int sc = blockIdx.x; sc < P.S; sc += gridDim.x) {
    const size_t row = (size_t)sc * P.N;
    const int n_act = uniform(min(max(P.n_actions[sc], 0), P.N));
    int* wait = R.wait + row; u64* wkey = EXT && R.wkey ? R.wkey + row : nullptr;
    ReplayRun run;
    if (R.rcap > 0) {
      run.at = (uint4*)run_at; run.fin = (i64*)(run.at + R.rcap); run.end = (int*)(run.fin + R.rcap); run.pu = (u32*)(run.end + R.rcap);
      run.idx = (int*)(run.pu + R.rcap);
    } else { run.at = R.run_at + row; run.fin = R.run_fin + row; run.end = R.run_end + row; run.pu = R.run_pu + row; run.idx = R.run_idx + row; }
    ReplayState Z;
    Z.slot = (int*)(fast + KR_FAST_BYTES);
    if (R.state_bytes > 0) {
      const size_t o_df = align16((size_t)R.W * 8), o_ow = o_df + align16((size_t)R.Dtot * 4), o_nm = o_ow + align16((size_t)R.U * 4);
      Z.cores = (u32*)state_at; Z.dfree = (int*)(state_at + o_df); Z.owner = (int*)(state_at + o_ow); Z.nm = (u8*)(state_at + o_nm);
    } else {
      Z.cores = R.cores + (size_t)sc * R.W * 2; Z.dfree = R.dfree + (size_t)sc * R.Dtot; Z.owner = R.owner + (size_t)sc * R.U;
      Z.nm = R.nm + (size_t)sc * ((P.n_nodes_total + 4) & ~3);
    }
    int* occ = R.occupancy ? R.occupancy + (size_t)sc * R.max_rounds * P.P : nullptr;
    // outputs and state start empty (the occupancy rows were zeroed before)
#pragma unroll 4
    for (int i = lane; i < P.N; i += 32) { P.o_alloc[row + i] = 0; P.o_node[row + i] = -1; P.o_off[row + i] = -1; P.o_act[row + i] = -1; }
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
#pragma unroll 1
    for (int j = 0; j < P.P; ++j) {
      const PoolDev& pd = P.pool[j];
      if (pd.type == TG_POOL_GPU) {
        int taken = 0;
#pragma unroll 1
        for (int v = lane; v < pd.n_nodes; v += 32) {
          const u32 b = (P.gpu_busy ? P.gpu_busy[(size_t)sc * P.n_nodes_total + pd.node0 + v] : 0u) & ((1u << pd.group) - 1u);
          Z.nm[pd.node0 + v] = (u8)b;
          taken += __popc(b);
        }
        taken = warp_sum32(taken);
        if (occ && lane == 0 && status == 0) occ[j] = taken;   // round 0's difference
        __syncwarp();
        replay_gpu_slots(pd, Z.nm, Z.slot, lane);
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
        *(uint2*)(Z.cores + 2 * (R.word0[j] + w)) = make_uint2((u32)m, (u32)(m >> 32));
      }
#pragma unroll 1
      for (int d = lane; d < R.n_dom[j]; d += 32) Z.dfree[R.dom0[j] + d] = pd.group;
    }
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
      auto fetch = [&](int from) {
        const int i = from + lane;
        if (i < n_act) {
          l_pool = P.a_pool[row + i]; l_unit = P.a_unit[row + i]; l_mask = P.a_mask[row + i]; l_s = P.a_s[row + i]; l_p = P.a_p[row + i];
          l_arr = P.a_arrival ? P.a_arrival[row + i] : 0;
        }
      };
      ReplayRec b_rec; int b_at = KR_NEVER;                // b_at: the round that admits the lane's arrival
      int next_at = KR_NEVER;
      auto refill = [&](int from) {                        // the batch that was fetched becomes the current one
        base = from;
        b_rec = replay_decode(P, l_pool, l_unit, l_mask, l_s, l_p);
        b_rec.arr = l_arr;
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
          const int until = EXT && R.traj_last ? min_end : r;
          int kept = 0, me = KR_NEVER;
          u32 touched = 0;                                 // GPU pools
#pragma unroll 1
          for (int i0 = 0; i0 < nr; i0 += 32) {
            const int i = i0 + lane;
            const int end = i < nr ? run.end[i] : KR_NEVER;
            const bool done = i < nr && end <= until, stay = i < nr && !done;
            const u32 bd = __ballot_sync(TG_FULL, done), bk = __ballot_sync(TG_FULL, stay);
            if (stay) me = min(me, end);
            if (bd || kept != i0) {
              uint4 at = make_uint4(0u, 0u, 0u, 0u); u32 pu = 0; int a = 0; i64 fin = 0;
              if (i < nr) { at = run.at[i]; pu = run.pu[i]; a = run.idx[i]; fin = run.fin[i]; }
              if (done) {
                const int type = RR_TYPE(pu), units = RR_UNITS(pu), j = RR_POOL(pu);
                if (type == TG_POOL_GPU) {
                  touched |= 1u << j;
                  if (!(pu & RR_WIDE)) {
                    const u32 v = (u32)P.pool[j].node0 + at.z;
                    atomicAnd((u32*)Z.nm + (v >> 2), ~(at.x << (8u * (v & 3u))));
                  }
                } else if (type == TG_POOL_CPU) {
                  atomicAdd(&Z.slot[RR_SLOT(pu)], units);
                  if (!(pu & RR_WIDE)) {
                    u32* w = Z.cores + 2 * (R.word0[j] + (int)at.z);
                    if (at.x) atomicOr(w, at.x);
                    if (at.y) atomicOr(w + 1, at.y);
                    atomicAdd(&Z.dfree[R.dom0[j] + (int)at.w], units);
                  }
                } else if (P.pool[j].window_us == 0) atomicAdd(&Z.slot[RR_SLOT(pu)], units);   // (used quota is not given back)
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
                const int from = __shfl_sync(TG_FULL, (int)at.w, b), j = RR_POOL(fpu);
                const PoolDev& pd = P.pool[j];
                const bool cpu = pd.type == TG_POOL_CPU;
                int* ow = Z.owner + R.unit0[j];
                int left = RR_UNITS(fpu);
#pragma unroll 1
                for (int c0 = cpu ? from & ~31 : 0; c0 < pd.capacity && left > 0; c0 += 32) {
                  const int c = c0 + lane;
                  const bool mine = c < pd.capacity && ow[c] == fa;
                  const u32 mb = __ballot_sync(TG_FULL, mine);
                  if (!mb) continue;
                  left -= __popc(mb);
                  if (mine) {
                    ow[c] = -1;
                    const int d = c / pd.group, x = c - d * pd.group;
                    if (cpu) {
                      const int w = d * R.wpd[j] + (x >> 6);
                      atomicOr(Z.cores + 2 * (R.word0[j] + w) + ((x >> 5) & 1), 1u << (x & 31));
                      atomicAdd(&Z.dfree[R.dom0[j] + d], 1);
                    } else {
                      const u32 v = (u32)(pd.node0 + d);
                      atomicAnd((u32*)Z.nm + (v >> 2), ~(1u << (x + 8 * (int)(v & 3u))));
                    }
                  }
                }
              }
              if (EXT && R.trajectory && R.traj_last)
#pragma unroll 1
                for (u32 rest = bd; rest; rest &= rest - 1) {
                  const int b = __ffs(rest) - 1, fa = __shfl_sync(TG_FULL, a, b);
                  const u32 fpu = __shfl_sync(TG_FULL, pu, b);
                  if (lane == 0 && RR_TYPE(fpu) == TG_POOL_CPU && R.traj_last[row + fa]) {
                    // the trajectory's last action has ended: its memory goes back to its node
                    const int t = R.trajectory[row + fa];
                    if (t >= 0 && t < R.max_traj) {
                      int* tn = R.traj_node + (size_t)sc * R.max_traj;
                      if (tn[t] >= 0) { R.mem_free[(size_t)sc * P.P + tn[t]] += (i64)R.traj_mem[row + fa]; tn[t] = -1; }
                    }
                  }
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
          touched = __reduce_or_sync(TG_FULL, touched);
#pragma unroll 1
          for (; touched; touched &= touched - 1) replay_gpu_slots(P.pool[__ffs(touched) - 1], Z.nm, Z.slot, lane);
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
            __syncwarp();
            i64 mf = 0; int cores = -1;
            if (lane < P.P && P.pool[lane].type == TG_POOL_CPU) { mf = R.mem_free[(size_t)sc * P.P + lane]; cores = P.pool[lane].capacity; }
            int pool_of = 0xff;
            const bool have = lane >= k0 && lane < k0 + cnt;
            const int out = pin_chunk(P, R.pool_rw, row + base + lane, have, R.trajectory, R.traj_mem, R.max_traj,
                                      R.traj_node + (size_t)sc * R.max_traj, mf, cores, lane, pool_of);
            if (lane < P.P && cores >= 0) R.mem_free[(size_t)sc * P.P + lane] = mf;
            if (have && lane < out) {
              R.pool_rw[row + base + lane] = (u8)pool_of;
              b_rec.meta = (b_rec.meta & ~0x3ffu) | (u32)pool_of | ((u32)P.pool[pool_of].slot0 << 4);
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
                if (lane == b) { Q.q[Q.at(p)] = (unsigned short)x; Q.key[x] = key; replay_store(Q, x, b_rec, base + b); }
              } else if (lane == b) { wait[p] = base + b; wkey[p] = key; }
              __syncwarp();
              ++nw;
            }
          } else {
            if (fits) {
              const int x = Q.free[free_slots - 1 - (lane - k0)];
              Q.q[Q.at(pos)] = (unsigned short)x;
              replay_store(Q, x, b_rec, base + lane);
            } else if (in) wait[pos] = base + lane;
            free_slots -= min(cnt, max(Q.cap - nw, 0));
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
          // Candidate prefix (Algorithm 1, line 2): lane v adds up the demand on slot v, action by action
          int n = 0, run_dem = 0, stop_pool = -1, aside = 0;
          u32 present = 0;                                 // pools with candidates; << 8: with elastic ones
          uint4 c0 = make_uint4(0u, RQ_NOBODY, 1u, 1u); int x0 = -1;   // the first 32 positions
#pragma unroll 1
          for (int i0 = 0; i0 < nw; i0 += 32) {
            uint4 c = make_uint4(0u, RQ_NOBODY, 1u, 1u); int x = -1;
            if (i0 + lane < nw) c = replay_facts(P, Q, wait, row, i0 + lane, x);
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
                if ((u32)(lane - RQ_SLOT(mb)) <= (u32)RQ_CLASS(mb)) run_dem += RQ_UNITS(mb);
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
          auto start = [&](const PoolDev& pd, int j, int k, int a, int units, i64 fin, i64 arr, int node, int off) {
            const size_t o = row + a;
            const i64 act = fin - arr;
            const int end = max(round_at(R, fin), r + 1);
            P.o_alloc[o] = units; P.o_node[o] = node; P.o_off[o] = off; P.o_act[o] = act;
            run.fin[k] = fin; run.end[k] = end; run.idx[k] = a;
            if (occ) {
              atomicAdd(&occ[(size_t)r * P.P + j], units);
              if (end < R.max_rounds && (pd.type != TG_POOL_API || pd.window_us == 0)) atomicSub(&occ[(size_t)end * P.P + j], units);
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
                if (i0 + lane < n) meta = replay_facts(P, Q, wait, row, i0 + lane, x).y;
                m += __popc(__ballot_sync(TG_FULL, RQ_POOL(meta) == j));
              }
            const bool el = (present >> (8 + j)) & 1u;
            const bool cached = EXT && pd.type == TG_POOL_GPU && P.cache_slots > 0;
            int units_now = 0;                             // what this lane's candidates take
            if ((m == 1 || (!el && pd.type != TG_POOL_GPU)) && !cached) {
              // Nothing to choose between candidates: each takes its level (a lone one DPArrange's answer in closed form: the
              // feasible level of least duration, the smallest among equals) and is placed in queue order.
              int seen = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < n && seen < m; i0 += 32) {
                uint4 c = c0; int x = x0;
                if (i0 > 0) {
                  c = make_uint4(0u, RQ_NOBODY, 1u, 1u); x = -1;
                  if (i0 + lane < n) c = replay_facts(P, Q, wait, row, i0 + lane, x);
                }
                const bool mine = i0 + lane < n && RQ_POOL(c.y) == j;
                const u32 mb = __ballot_sync(TG_FULL, mine);
                if (!mb) continue;
                ReplayRec rec; rec.s = rec.p = rec.arr = 0;
                if (mine) rec = replay_rec(P, Q, row, c, x);
                int rr = __ffs(c.z);
                if (m == 1 && el) {
                  const int b = __ffs(mb) - 1;
                  const u32 mk = __shfl_sync(TG_FULL, c.z, b), cg = __shfl_sync(TG_FULL, c.w, b);
                  const int g = cg & 0x7f, gang = cg >> 7, rl = lane + 1;
                  bool fit = (mk >> lane) & 1u;
                  const int cl = fit && pd.type == TG_POOL_GPU ? level_of(g, gang, rl) : 0;
                  const int room = Z.slot[slot0 + cl] - (cl == 0 ? aside_j : 0);
                  const u32 fits = __ballot_sync(TG_FULL, fit && g * rl <= room);
                  if (lane == b && fits) rr = best_level(rec.p, fits);   // (durations do not grow with the level)
                }
                const int units = mine ? (int)(c.w & 0x7f) * rr : 0;
                const i64 fin = now + duration(rec.s, rec.p, rr);
                ReplayGrant G; G.node = 0; G.off = -1; G.word = 0; G.dom = 0; G.lo = G.hi = 0; G.wide = false;
                if (pd.type == TG_POOL_API) {
                  // Section 5.1: the offset is what was in use before
                  const int incl = warp_incl_scan32(units, lane);
                  G.off = pd.capacity - Z.slot[slot0] + incl - units;
                  const int all = __shfl_sync(TG_FULL, incl, 31);
                  if (lane == 0) Z.slot[slot0] -= all;
                } else
#pragma unroll 1
                  for (u32 todo = mb; todo; todo &= todo - 1) {
                    const int b = __ffs(todo) - 1;
                    const int k = __shfl_sync(TG_FULL, units, b), id = __shfl_sync(TG_FULL, (int)c.x, b);
                    ReplayGrant g1;
                    if (pd.type == TG_POOL_CPU)
                      g1 = replay_take_cores(pd.group, R.n_dom[j], R.wpd[j], Z.cores + 2 * R.word0[j], Z.dfree + R.dom0[j], ow, k, id, lane);
                    else {
                      const int cg = __shfl_sync(TG_FULL, (int)c.w, b), rb = __shfl_sync(TG_FULL, rr, b), g = cg & 0x7f, gang = cg >> 7;
                      g1 = replay_take_gpus(pd, Z.nm + pd.node0, ow, ilog2(gang ? g * rb : g), gang ? 1 : rb, id, lane);
                    }
                    if (lane == b) G = g1;
                  }
                if (mine) {
                  const int k = nr + __popc(mb & below);
                  run.at[k] = make_uint4(G.lo, G.hi, (u32)G.word, (u32)G.dom); run.pu[k] = rr_pack(pd, j, units, G.wide);
                  if (x >= 0) Q.c[x].y = c.y | RQ_STARTED;
                  start(pd, j, k, (int)c.x, units, fin, rec.arr, G.node, G.off);
                }
                units_now += units;
                nr += __popc(mb); seen += __popc(mb); selected += __popc(mb);
                __syncwarp();
              }
            } else {
              Slab slab;
              slab.base = P.slabs + (u64)blockIdx.x * P.slab_bytes; slab.cap = P.slab_bytes; slab.used = 0;
              slab.fbase = fast; slab.fcap = KR_FAST_BYTES; slab.fused = 0;
              CandArrays C; int keep = 0;
              ok = replay_select<EXT>(P, Q, run, wait, sc, j, n, nw, nr, m, now, Z.slot[slot0] - aside_j, Z.slot[(slot0 + 1) & 31],
                                      Z.slot[(slot0 + 2) & 31], Z.slot[(slot0 + 3) & 31], slab, C, keep, lane);
              if (!ok) break;
              const u8* missed = nullptr;                  // candidates whose chunk did not cache their service
              if (cached) {
                const size_t cbase = ((size_t)sc * P.n_nodes_total + pd.node0) * 8 * P.cache_slots;
                place_gpu_cache(pd, Z.nm + pd.node0, keep, C.cg, C.rkeep, C.cidx, C.pnode, C.poff, C.rsel,
                                P.a_service ? P.a_service + row : nullptr, P.cache_tag + cbase, P.cache_use + cbase, P.cache_slots, now, lane, ow);
                missed = C.rsel;
              } else if (pd.type == TG_POOL_GPU) {
                place_gpu(pd, Z.nm + pd.node0, keep, C.cg, C.rkeep, C.pnode, C.poff, lane, ow, C.cidx);
              } else if (pd.type == TG_POOL_CPU) {
#pragma unroll 1
                for (int i = 0; i < keep; ++i) {
                  const int units = (C.cg[i] & 0x7f) * C.rkeep[i];
                  const ReplayGrant G = replay_take_cores(pd.group, R.n_dom[j], R.wpd[j], Z.cores + 2 * R.word0[j], Z.dfree + R.dom0[j], ow,
                                                          units, C.cidx[i], lane);
                  if (lane == 0) {
                    C.pnode[i] = G.node; C.poff[i] = G.off;
                    run.at[nr + i] = make_uint4(G.lo, G.hi, (u32)G.word, (u32)G.dom); run.pu[nr + i] = rr_pack(pd, j, units, G.wide);
                  }
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
                const int g = C.cg[i] & 0x7f, gang = C.cg[i] >> 7, rr = C.rkeep[i], units = g * rr, a = C.cidx[i];
                i64 fin = now + duration(C.cs[i], C.cp[i], rr);
                if (EXT && missed && missed[i] && P.a_restore) fin += clamp_param(P.a_restore[row + a]);   // restoration precedes execution
                if (pd.type != TG_POOL_CPU) {
                  run.at[nr + i] = make_uint4(((1u << (units & 31)) - 1u) << (C.poff[i] & 31), 0u, (u32)C.pnode[i], 0u);
                  run.pu[nr + i] = rr_pack(pd, j, units, pd.type == TG_POOL_GPU && !gang && rr > 1);
                }
                start(pd, j, nr + i, a, units, fin, P.a_arrival ? P.a_arrival[row + a] : 0, C.pnode[i], C.poff[i]);
                units_now += units;
              }
              // the kept ones are the pool's first `keep` in queue order
              int seen = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < n && seen < keep; i0 += 32) {
                int x = -1; u32 meta = RQ_NOBODY;
                if (i0 + lane < n) meta = replay_facts(P, Q, wait, row, i0 + lane, x).y;
                const bool mine = RQ_POOL(meta) == j;
                const u32 mb = __ballot_sync(TG_FULL, mine);
                if (mine && seen + __popc(mb & below) < keep && x >= 0) Q.c[x].y = meta | RQ_STARTED;
                seen += __popc(mb);
              }
              nr += keep; selected += keep;
              __syncwarp();
            }
            if (pd.type == TG_POOL_GPU) replay_gpu_slots(pd, Z.nm, Z.slot, lane);
            else if (pd.type == TG_POOL_CPU) {
              const int all = warp_sum32(units_now);
              if (lane == 0) Z.slot[slot0] -= all;
            }
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
            int to_end = n;                                // the ones that stay move up behind the others, last first
#pragma unroll 1
            for (int i0 = (n - 1) & ~31; i0 >= 0; i0 -= 32) {
              const int i = i0 + lane, x = i < n ? (int)Q.q[Q.at(i)] : 0;
              const bool gone = i < n && (started == n || (Q.c[x].y & RQ_STARTED));
              const u32 gb = __ballot_sync(TG_FULL, gone);
              if (gone) Q.free[free_slots + __popc(gb & below)] = (unsigned short)x;
              free_slots += __popc(gb);
              if (started < n) {
                const u32 sb = __ballot_sync(TG_FULL, i < n && !gone);
                __syncwarp();
                if (i < n && !gone) Q.q[Q.at(to_end - __popc(sb >> lane))] = (unsigned short)x;
                to_end -= __popc(sb);
                __syncwarp();
              }
            }
            Q.head = Q.at(started < Q.cap ? started : 0);
            nw -= started;
            __syncwarp();
          } else if (started) {                             // a queue that goes on in global memory
            int kw = 0;
#pragma unroll 1
            for (int i0 = 0; i0 < nw; i0 += 32) {
              const int i = i0 + lane;
              bool stay = false; int x = 0, a = 0; u64 kk = 0;
              if (i < min(nw, Q.cap)) { x = Q.q[Q.at(i)]; stay = !(Q.c[x].y & RQ_STARTED); }
              else if (i < nw) { a = wait[i]; stay = P.o_act[row + a] < 0; if (EXT && R.policy) kk = wkey[i]; }
              const u32 b = __ballot_sync(TG_FULL, stay), gone = __ballot_sync(TG_FULL, i < min(nw, Q.cap) && !stay);
              const int to = kw + __popc(b & below);
              __syncwarp();
              if (stay && i < Q.cap) Q.q[Q.at(to)] = (unsigned short)x;
              else if (stay && to >= Q.cap) { wait[to] = a; if (EXT && R.policy) wkey[to] = kk; }
              if ((gone >> lane) & 1u) Q.free[free_slots + __popc(gone & below)] = (unsigned short)x;
              free_slots += __popc(gone);
              __syncwarp();
              const u32 mv = __ballot_sync(TG_FULL, stay && i >= Q.cap && to < Q.cap);
              if ((mv >> lane) & 1u) {                      // a record moves up into shared memory
                const int y = Q.free[free_slots - 1 - __popc(mv & below)];
                Q.q[Q.at(to)] = (unsigned short)y;
                replay_store(Q, y, replay_load(P, row, a), a);
                if (EXT) Q.key[y] = kk;
              }
              free_slots -= __popc(mv);
              __syncwarp();
              kw += __popc(b);
            }
            nw = kw;
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
